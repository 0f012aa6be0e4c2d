// Inverses of the element blocks by elimination of the species (FP32).
//
// The species of an element couple only to themselves and to the potential
// (Eq. NPDG: row k holds c_k and Phi), so a block is an arrow of n x n field
// blocks, n = (p + 1)^3: A_00, A_0k, A_k0, A_kk. With X_k = A_kk^-1 A_k0,
// Y_k = A_0k A_kk^-1 and S = A_00 - sum_k A_0k X_k its inverse is
//   (0,0): S^-1,  (k,0): -X_k S^-1,  (0,l): -S^-1 Y_l,
//   (k,l): X_k S^-1 Y_l (+ A_kk^-1 if k = l).
// Only n x n matrices are pivoted, in the registers of one to four warps, and the
// rest are products at the FP32 pipe's rate. For three fields at p = 3 that is 4.5
// instead of 7.1 million multiply-adds and 3 x 64 instead of 192 pivot steps, each
// of which cost two barriers of 512 threads: 32,768 blocks of 192 x 192 58.7 ms,
// 25 so.
//
// Pivots are searched within a field block only. A pivot below kElimPivot of the
// field block's largest entry sets *singular, and the caller inverts the whole
// blocks with full pivoting instead.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace enp {

constexpr float kElimPivot = 1e-5f;

// Gauss-Jordan inversion, in place, of the n x n matrices at blocks + e stride +
// offset + f fstride (e = blockIdx.x / nf, f = blockIdx.x % nf), leading dimension
// ld: W warps per matrix, each lane RPL whole rows in registers. Step k pivots on
// column k in the largest unused row p, without exchanging rows; the columns
// rotate by one register each step, so that the pivot column is always register
// 0 and every index is a compile-time one:
//   M_i[c-1] <- M_i[c] - (M_i[0] / v) M_p[c],  M_i[n-1] <- -M_i[0] / v  (i != p),
// row p itself only shifts, M_p[n-1] <- 1, and keeps its factor 1/v for the end.
// The pivot row passes through shared memory; with one warp there is no barrier.
template <int n, int W, int RPL>
__global__ void __launch_bounds__(32 * W)
elim_invert_kernel(float* blocks, long long stride, long long offset, long long fstride, int nf,
                   int ld, int* __restrict__ singular) {
  constexpr int NR = 32 * W * RPL;
  constexpr int LD = n % 2 ? n : n + 1;        // staging rows in different banks
  constexpr int NP4 = (n + 3) / 4 * 4;
  static_assert(NR >= n, "rows");
  __shared__ __align__(16) float prow[W > 1 ? 2 : 1][W][NP4];   // per warp: its candidate row
  __shared__ unsigned cand[W > 1 ? 2 : 1][W];
  __shared__ int piv[n], stepof[NR];
  __shared__ float wmax[W];
  extern __shared__ __align__(16) float stage[];   // [n][LD]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  float* A = blocks + (long long)(blockIdx.x / nf) * stride + offset + (blockIdx.x % nf) * fstride;
  for (int t = tid; t < n * n; t += 32 * W) {
    const int i = t / n, j = t - i * n;
    stage[i * LD + j] = A[(long long)i * ld + j];
  }
  if (W > 1) __syncthreads();
  else __syncwarp();
  float M[RPL][n];
  float amax = 0.f;
#pragma unroll
  for (int r = 0; r < RPL; ++r) {
    const int i = lane + 32 * (w + W * r);
#pragma unroll
    for (int c = 0; c < n; ++c) {
      M[r][c] = i < n ? stage[i * LD + c] : 0.f;
      amax = fmaxf(amax, fabsf(M[r][c]));
    }
  }
  amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));
  if (W > 1) {
    if (lane == 0) wmax[w] = amax;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < W; ++q) amax = fmaxf(amax, wmax[q]);
  }
  const float thr = kElimPivot * amax;
  unsigned used = 0u;
  float sc[RPL];
#pragma unroll
  for (int r = 0; r < RPL; ++r) {
    sc[r] = 1.f;
    if (lane + 32 * (w + W * r) >= n) used |= 1u << r;    // padding rows never pivot
  }
  bool bad = false;
#pragma unroll 1
  for (int k = 0; k < n; ++k) {
    const int buf = W > 1 ? k & 1 : 0;
    // this warp's largest unused row (|values| order as their bits; NaN is largest)
    unsigned key = 0u;
    int slot = 0;
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
      const unsigned b = (used >> r) & 1u ? 0u : __float_as_uint(fabsf(M[r][0]));
      if (b > key) { key = b; slot = r; }
    }
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    const unsigned who = __ballot_sync(0xffffffffu, key == top);
    const int owner = __ffs(who) - 1;
    if (lane == owner) {
      cand[buf][w] = top;
      float4* o = reinterpret_cast<float4*>(prow[buf][w]);
#pragma unroll
      for (int r = 0; r < RPL; ++r)
        if (r == slot) {
#pragma unroll
          for (int c = 0; c < NP4 / 4; ++c)
            o[c] = make_float4(M[r][4 * c], 4 * c + 1 < n ? M[r][4 * c + 1 < n ? 4 * c + 1 : 0] : 0.f,
                               4 * c + 2 < n ? M[r][4 * c + 2 < n ? 4 * c + 2 : 0] : 0.f,
                               4 * c + 3 < n ? M[r][4 * c + 3 < n ? 4 * c + 3 : 0] : 0.f);
        }
    }
    int pw = 0;
    unsigned btop = top;
    if (W > 1) {
      __syncthreads();
      btop = cand[buf][0];
#pragma unroll
      for (int q = 1; q < W; ++q) {
        const unsigned c = cand[buf][q];
        if (c > btop) { btop = c; pw = q; }         // as bits: a NaN of any warp wins
      }
    } else {
      __syncwarp();
    }
    const float best = __uint_as_float(btop);
    if (!(best > thr) || !isfinite(best)) { bad = true; break; }   // the same in every thread
    const bool mine = (W == 1 || pw == w) && lane == owner;
    const float4* pr = reinterpret_cast<const float4*>(prow[buf][pw]);
    const float4 p0 = pr[0];
    const float pinv = __frcp_rn(p0.x);
    float f[RPL];
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
      const bool own = mine && r == slot;
      f[r] = own ? 0.f : M[r][0] * pinv;
      if (own) {
        sc[r] = pinv;
        used |= 1u << r;
        const int i = lane + 32 * (w + W * r);
        piv[k] = i;
        stepof[i] = k;
      }
    }
#pragma unroll
    for (int c4 = 0; c4 < NP4 / 4; ++c4) {
      const float4 q = c4 ? pr[c4] : p0;
      const float qs[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const int c = 4 * c4 + d;
        if (c >= 1 && c < n)
#pragma unroll
          for (int r = 0; r < RPL; ++r) M[r][c - 1] = fmaf(-f[r], qs[d], M[r][c]);
      }
    }
#pragma unroll
    for (int r = 0; r < RPL; ++r) M[r][n - 1] = (mine && r == slot) ? 1.f : -f[r];
    if (W == 1) __syncwarp();      // the row is read before the next step writes it
  }
  if (bad) {
    if (tid == 0) atomicOr(singular, 1);
    return;
  }
  if (W > 1) __syncthreads();
  else __syncwarp();
  // inv[step(i)][p_c] = sc_i M_i[c]
#pragma unroll
  for (int r = 0; r < RPL; ++r) {
    const int i = lane + 32 * (w + W * r);
    if (i < n) {
      float* o = stage + stepof[i] * LD;
#pragma unroll
      for (int c = 0; c < n; ++c) o[piv[c]] = sc[r] * M[r][c];
    }
  }
  if (W > 1) __syncthreads();
  else __syncwarp();
  for (int t = tid; t < n * n; t += 32 * W) {
    const int i = t / n, j = t - i * n;
    A[(long long)i * ld + j] = stage[i * LD + j];
  }
}

// Products of n x n matrices by one thread block: TR x TC threads (row tiles
// fastest), each a TM x TM tile of C in registers, operands staged KC columns
// (rows) at a time in shared memory, A transposed.
template <int n>
struct ElimShape {
  static constexpr int TM = n <= 32 ? 4 : 8;
  static constexpr int T = (n + TM - 1) / TM;        // tiles per dimension
  static constexpr int NP = T * TM;
  static constexpr int NT = T * T;
  static constexpr int KC = 16;
  static constexpr int LD = NP + 4;
};
__device__ __forceinline__ void copy4(float* dst, const float* src, bool ok) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int size = ok ? 4 : 0;     // 0: zeros, nothing read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(size) : "memory");
}
__device__ __forceinline__ void copy16(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
// c += A B (A, B: global, leading dimension ld; written by this block before, if
// at all, so no read-only loads). As, Bs: two buffers each; the next chunk is
// copied while this one is multiplied (loads through registers left the products
// waiting on memory 80 % of the time). Barriers on both sides.
template <int n>
__device__ __forceinline__ void elim_gemm(float (&c)[ElimShape<n>::TM][ElimShape<n>::TM],
                                          const float* A, const float* B, int ld, float* As,
                                          float* Bs) {
  using S = ElimShape<n>;
  constexpr int TM = S::TM, T = S::T, NP = S::NP, NT = S::NT, KC = S::KC, LD = S::LD;
  constexpr int NCH = (n + KC - 1) / KC;
  const int tid = threadIdx.x, r0 = (tid % T) * TM, c0 = (tid / T) * TM;
  auto fetch = [&](int ch) {
    const int k0 = ch * KC;
    float *a = As + (ch & 1) * (KC * LD), *b = Bs + (ch & 1) * (KC * LD);
#pragma unroll 4
    for (int t = tid; t < NP * KC; t += NT) {
      const int i = t / KC, k = t % KC;
      const bool ok = i < n && k0 + k < n;
      copy4(a + k * LD + i, ok ? A + (long long)i * ld + k0 + k : A, ok);
    }
    if constexpr (n % KC == 0) {   // rows of 16-byte multiples: n, ld and the offsets are multiples of 4
#pragma unroll 4
      for (int t = tid; t < n / 4 * KC; t += NT) {
        const int k = t / (n / 4), j = t % (n / 4) * 4;
        copy16(b + k * LD + j, B + (long long)(k0 + k) * ld + j);
      }
    } else {
#pragma unroll 4
      for (int t = tid; t < NP * KC; t += NT) {
        const int k = t / NP, j = t % NP;
        const bool ok = j < n && k0 + k < n;
        copy4(b + k * LD + j, ok ? B + (long long)(k0 + k) * ld + j : B, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  __syncthreads();
  fetch(0);
#pragma unroll 1
  for (int ch = 0; ch < NCH; ++ch) {
    if (ch + 1 < NCH) {
      fetch(ch + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float *as = As + (ch & 1) * (KC * LD) + r0, *bs = Bs + (ch & 1) * (KC * LD) + c0;
    // four at a time: three to four products are inlined in a kernel, and whole
    // chunks of straight-line code (16 KB each) outran the instruction cache
#pragma unroll 4
    for (int k = 0; k < KC; ++k) {
      float a[TM], b[TM];
#pragma unroll
      for (int q = 0; q < TM; q += 4) {
        const float4 x = *reinterpret_cast<const float4*>(as + k * LD + q);
        const float4 y = *reinterpret_cast<const float4*>(bs + k * LD + q);
        a[q] = x.x; a[q + 1] = x.y; a[q + 2] = x.z; a[q + 3] = x.w;
        b[q] = y.x; b[q + 1] = y.y; b[q + 2] = y.z; b[q + 3] = y.w;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) c[i][j] = fmaf(a[i], b[j], c[i][j]);
    }
    __syncthreads();
  }
}
// A thread's tile of a row-major matrix (leading dimension ld) in and out; whole
// 16-byte groups where the tile rows are such (n and ld multiples of 4).
template <int n, int TM>
__device__ __forceinline__ void tile_load(float (&c)[TM][TM], const float* p, int ld, int r0, int c0) {
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    if constexpr (n % TM == 0 && n % 4 == 0) {
#pragma unroll
      for (int j = 0; j < TM; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(p + (long long)(r0 + i) * ld + c0 + j);
        c[i][j] = v.x; c[i][j + 1] = v.y; c[i][j + 2] = v.z; c[i][j + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < TM; ++j)
        c[i][j] = (r0 + i < n && c0 + j < n) ? p[(long long)(r0 + i) * ld + c0 + j] : 0.f;
    }
  }
}
template <int n, int TM>
__device__ __forceinline__ void tile_store(float* p, const float (&c)[TM][TM], int ld, int r0, int c0) {
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    if constexpr (n % TM == 0 && n % 4 == 0) {
#pragma unroll
      for (int j = 0; j < TM; j += 4)
        *reinterpret_cast<float4*>(p + (long long)(r0 + i) * ld + c0 + j) =
            make_float4(c[i][j], c[i][j + 1], c[i][j + 2], c[i][j + 3]);
    } else {
#pragma unroll
      for (int j = 0; j < TM; ++j)
        if (r0 + i < n && c0 + j < n) p[(long long)(r0 + i) * ld + c0 + j] = c[i][j];
    }
  }
}
// The tile times sign, transposed, as TS.
template <int n, int TM, class TS>
__device__ __forceinline__ void tile_emit(TS* o, float sign, const float (&c)[TM][TM], int ld, int r0,
                                          int c0) {
#pragma unroll
  for (int j = 0; j < TM; ++j) {
    TS* q = o + (long long)(c0 + j) * ld + r0;
    if constexpr (n % TM == 0 && TM == 8 && n % 8 == 0) {
      if constexpr (sizeof(TS) == 4) {
#pragma unroll
        for (int i = 0; i < TM; i += 4)
          *reinterpret_cast<float4*>(q + i) = make_float4(sign * c[i][j], sign * c[i + 1][j],
                                                          sign * c[i + 2][j], sign * c[i + 3][j]);
      } else {
        union { __nv_bfloat16 h[8]; uint4 u; } v;
#pragma unroll
        for (int i = 0; i < 8; ++i) v.h[i] = (__nv_bfloat16)(sign * c[i][j]);
        *reinterpret_cast<uint4*>(q) = v.u;
      }
    } else {
#pragma unroll
      for (int i = 0; i < TM; ++i)
        if (r0 + i < n && c0 + j < n) q[i] = (TS)(sign * c[i][j]);
    }
  }
}
template <int TM>
__device__ __forceinline__ void tile_zero(float (&c)[TM][TM]) {
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) c[i][j] = 0.f;
}

// With A_kk^-1 in place: X_k over A_k0, Y_k over A_0k, S over A_00.
template <int n, int NF>
__global__ void __launch_bounds__(ElimShape<n>::NT, 384 / ElimShape<n>::NT > 0 ? 384 / ElimShape<n>::NT : 1)
elim_schur_kernel(float* blocks) {
  using S = ElimShape<n>;
  constexpr int TM = S::TM, T = S::T, nb = NF * n;
  __shared__ __align__(16) float As[2 * S::KC * S::LD], Bs[2 * S::KC * S::LD];
  float* E = blocks + (long long)blockIdx.x * nb * nb;
  const int r0 = ((int)threadIdx.x % T) * TM, c0 = ((int)threadIdx.x / T) * TM;
  auto at = [&](int f, int g) { return E + (long long)f * n * nb + g * n; };
  float s[TM][TM], c[TM][TM];
  tile_zero(s);
#pragma unroll 1
  for (int k = 1; k < NF; ++k) {
    tile_zero(c);
    elim_gemm<n>(c, at(k, k), at(k, 0), nb, As, Bs);
    tile_store<n>(at(k, 0), c, nb, r0, c0);     // X_k
    __syncthreads();
    elim_gemm<n>(s, at(0, k), at(k, 0), nb, As, Bs);
    tile_zero(c);
    elim_gemm<n>(c, at(0, k), at(k, k), nb, As, Bs);
    tile_store<n>(at(0, k), c, nb, r0, c0);     // Y_k
  }
  tile_load<n>(c, at(0, 0), nb, r0, c0);
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) c[i][j] -= s[i][j];
  tile_store<n>(at(0, 0), c, nb, r0, c0);
}

// With S^-1 in place: the inverse, transposed, out[e][c][r] in type TS.
template <int n, int NF, class TS>
__global__ void __launch_bounds__(ElimShape<n>::NT, 512 / ElimShape<n>::NT)
elim_finish_kernel(float* blocks, TS* __restrict__ out) {
  using S = ElimShape<n>;
  constexpr int TM = S::TM, T = S::T, nb = NF * n;
  __shared__ __align__(16) float As[2 * S::KC * S::LD], Bs[2 * S::KC * S::LD];
  float* E = blocks + (long long)blockIdx.x * nb * nb;
  TS* O = out + (long long)blockIdx.x * nb * nb;
  const int r0 = ((int)threadIdx.x % T) * TM, c0 = ((int)threadIdx.x / T) * TM;
  auto at = [&](int f, int g) { return E + (long long)f * n * nb + g * n; };
  auto emit = [&](int f, int g, float sign, const float (&c)[TM][TM]) {
    tile_emit<n>(O + (long long)g * n * nb + f * n, sign, c, nb, r0, c0);
  };
  float c[TM][TM];
  tile_load<n>(c, at(0, 0), nb, r0, c0);
  emit(0, 0, 1.f, c);
#pragma unroll 1
  for (int k = 1; k < NF; ++k) {
    tile_zero(c);
    elim_gemm<n>(c, at(k, 0), at(0, 0), nb, As, Bs);
    emit(k, 0, -1.f, c);
    tile_store<n>(at(k, 0), c, nb, r0, c0);     // X_k S^-1 over X_k
    __syncthreads();
  }
#pragma unroll 1
  for (int l = 1; l < NF; ++l) {
    tile_zero(c);
    elim_gemm<n>(c, at(0, 0), at(0, l), nb, As, Bs);
    emit(0, l, -1.f, c);
#pragma unroll 1
    for (int k = 1; k < NF; ++k) {
      if (k == l) tile_load<n>(c, at(k, k), nb, r0, c0);
      else tile_zero(c);
      elim_gemm<n>(c, at(k, 0), at(0, l), nb, As, Bs);
      emit(k, l, 1.f, c);
    }
  }
}

template <int n, int W, int RPL, int NF>
static cudaError_t launch_elim_n(float* blocks, void* out, int storage, long long nblk, int* singular,
                                 cudaStream_t s) {
  using S = ElimShape<n>;
  constexpr int nb = NF * n;
  constexpr size_t stage = sizeof(float) * n * (n % 2 ? n : n + 1);
  const long long st = (long long)nb * nb, diag = (long long)n * nb + n;
  auto inv = elim_invert_kernel<n, W, RPL>;
  cudaError_t e = cudaFuncSetAttribute(inv, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stage);
  if (e != cudaSuccess) return e;
  inv<<<(unsigned)(nblk * (NF - 1)), 32 * W, stage, s>>>(blocks, st, diag, diag, NF - 1, nb, singular);
  elim_schur_kernel<n, NF><<<(unsigned)nblk, S::NT, 0, s>>>(blocks);
  inv<<<(unsigned)nblk, 32 * W, stage, s>>>(blocks, st, 0, 0, 1, nb, singular);
  if (storage == 1)
    elim_finish_kernel<n, NF, float><<<(unsigned)nblk, S::NT, 0, s>>>(blocks, (float*)out);
  else
    elim_finish_kernel<n, NF, __nv_bfloat16><<<(unsigned)nblk, S::NT, 0, s>>>(blocks, (__nv_bfloat16*)out);
  return cudaGetLastError();
}

}  // namespace enp
