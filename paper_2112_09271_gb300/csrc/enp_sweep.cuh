// The downwind block Gauss-Seidel sweep, one launch for the whole mesh.
//
// The sweep solves (D + L) z = x with D the element-diagonal blocks of J and L
// each element's coupling to its upstream neighbour along the flow axis a
// (Sec. 4: the block preconditioner of the Newton-Krylov solve, ordered along
// the advection of Eq. NPDG). L couples an element only to the one before it on
// its own line of elements along the flow, so every line is an independent
// chain: one thread block takes one line for one operating point and walks down
// it, with z of the element before in shared memory. Per element e:
//   1. the face between e and its upstream neighbour: the traces of both states
//      and of the upstream tangent z_up (e's own tangent is zero), the J v face
//      flux, and the lifting onto e's face nodes;
//   2. t = x_e minus e's side of the lifted terms;
//   3. z_e = Binv_e t, with the inverse stored transposed (BT[c][r]).
// A chain is bound by latency, so nothing on it waits on memory: the next
// element's state on the face, its x and its geometry are loaded into registers
// while this one is worked on; its inverse is started towards L2 a step ahead (where
// few lines run: the inverses of many would not fit L2) and its first columns are read
// into registers during the face stages. One launch per
// element plane took 9.5 us a plane whatever its size (192 x 48 x 16 elements,
// p = 2: 1.8 ms an application, 0.37 now; the inverses alone are 0.26 ms
// of HBM).
#pragma once
#include <cuda_bf16.h>

#include "enp_launch.cuh"
#include "enp_tile3d.cuh"

namespace enp {

// Rows of a block padded to whole warps, times COLS column pieces per row: a thread
// each (WIDE), or one after the other by the row's thread, in the same order of sums.
template <int P, int NF, bool WIDE>
struct SweepShape {
  static constexpr int N = P + 1, Q = P + 2, QP = Rows<P>::QP, FN = N * N, FQ = Q * Q;
  static constexpr int NX = N % 2 ? N : N + 1;
  static constexpr int nb = NF * N * N * N;
  static constexpr int RP = (nb + 31) / 32 * 32;
  // Pieces that let a block of few rows fill some 256 threads, and a large one the 768
  // that its registers allow. 54 rows with one, two and four, FP32 vectors: 80 lines of
  // 100 elements 151, 150 and 140 us, 640 lines 186, 192 and 420.
  static constexpr int COLS = nb <= 64 ? 1 : (nb <= 128 ? 2 : (nb <= 192 ? 4 : (nb <= 256 ? 3 : 2)));
  static constexpr int NT = WIDE ? RP * COLS : RP;
  static constexpr int CC = (nb + COLS - 1) / COLS;        // columns per piece
  // Blocks per SM the registers are sized for (0: the compiler's choice, which gives 768
  // threads 40 registers with FP64 vectors, and spills 650 bytes).
  static constexpr int MINB = WIDE ? (NT > 256 ? 1 : 0) : (RP <= 128 ? 5 : (RP <= 192 ? 4 : (RP <= 256 ? 3 : 2)));
  // Columns of the inverse held in registers (the others stream from L2).
  template <class TS> __host__ __device__ static constexpr int ahead() {
    constexpr int most = (!WIDE ? 8 : (NT > 256 ? 40 : 64)) / (sizeof(TS) == 8 ? 2 : 1);
    return CC < most ? CC : most;
  }
  static constexpr int NTR = 2 * (NF + 1) + 2 * NF;        // traces: both states, upstream tangent
  static constexpr int max2(int a, int b) { return a > b ? a : b; }
  // region A: layer data, then traces, then the first transposed contraction;
  // region B: the first contraction, the flux coefficients
  static constexpr int kA = max2(NTR * N * NX, max2(NTR * Q * QP, 2 * NF * N * QP));
  static constexpr int kB = max2(NTR * N * QP, 2 * NF * Q * QP);
  static_assert((2 + NF) * FN <= NT && FQ <= NT, "one trace item, one face point per thread");
};
template <int P, int NF, bool WIDE, class TV, class TA>
struct SweepSmem {
  using S = SweepShape<P, NF, WIDE>;
  static constexpr size_t z_off = (size_t)(S::kA + S::kB) * sizeof(TV);
  static constexpr size_t t_off = (z_off + S::nb * sizeof(TV) + 15) / 16 * 16;
  static constexpr size_t p_off = t_off + (size_t)S::RP * sizeof(TA);
  static constexpr size_t bytes = p_off + (WIDE && S::COLS > 1 ? (size_t)S::NT * sizeof(TA) : 0);
};

// TS: type of the stored inverses (FP64 accumulated in FP64, FP32 and BF16 in
// FP32). upc: the linearisation point. dir = +1: flow along +e_a, -1: along -e_a.
template <int P, int NF, bool WIDE, class TV, class TS>
__global__ void __launch_bounds__(SweepShape<P, NF, WIDE>::NT, SweepShape<P, NF, WIDE>::MINB)
sweep_line_kernel(const OpParams prm, const TS* __restrict__ binv, const TV* __restrict__ x,
                  TV* __restrict__ z, const TV* __restrict__ upc, int a, int dir,
                  int shared_blocks) {
  using TA = typename std::conditional<sizeof(TS) == 8, double, float>::type;
  using S = SweepShape<P, NF, WIDE>;
  using M = SweepSmem<P, NF, WIDE, TV, TA>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, NX = S::NX, FN = S::FN, FQ = S::FQ, NN = N * FN;
  constexpr int nb = S::nb, NT = S::NT, CC = S::CC, AH = S::template ahead<TS>();
  constexpr int NA = 2 * NF, T0 = 2 * (NF + 1);   // T0: first tangent trace
  extern __shared__ __align__(16) unsigned char sweep_raw[];
  TV* A = reinterpret_cast<TV*>(sweep_raw);
  TV* B = A + S::kA;
  TV* zs = reinterpret_cast<TV*>(sweep_raw + M::z_off);
  TA* ts = reinterpret_cast<TA*>(sweep_raw + M::t_off);
  TA* ps = reinterpret_cast<TA*>(sweep_raw + M::p_off);
  const int tid = threadIdx.x, b = blockIdx.y;
  const int b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
  const int nb0 = pick3(prm.ne, b0), nk = pick3(prm.ne, a);
  const int j0 = (int)blockIdx.x % nb0, j1 = (int)blockIdx.x / nb0;
  const int stride[3] = {1, prm.ne[0], prm.ne[0] * prm.ne[1]};
  const long long sa = pick3(stride, a);
  const long long line0 = (long long)j0 * pick3(stride, b0) + (long long)j1 * pick3(stride, b1);
  const long long EN = (long long)prm.E * NN, boff = (long long)b * prm.batch_stride;
  const TS* BT = binv + (shared_blocks ? 0 : (long long)b * prm.E) * (long long)(nb * nb);
  auto elem = [&](int step) { return line0 + (long long)(dir > 0 ? step : nk - 1 - step) * sa; };
  const int own = dir > 0 ? 1 : 0, up = 1 - own;   // sides of the face: 0 lower, 1 upper

  // this thread's piece of the block product: row r, columns [c0, c0 + cn)
  const int r = tid % S::RP, c0 = (tid / S::RP) * CC;
  const int rr = r < nb ? r : nb - 1;              // padding rows repeat the last one
  const int cn = c0 + CC <= nb ? CC : nb - c0;
  TS bv[AH];
  // chunk q of `of` of the step's inverse into registers
  auto load_inverse = [&](int step, int q, int of) {
    const TS* p = BT + elem(step) * (long long)(nb * nb) + (long long)c0 * nb + rr;
#pragma unroll
    for (int i = 0; i < AH; ++i)
      if (i >= AH * q / of && i < AH * (q + 1) / of) bv[i] = i < cn ? p[(long long)i * nb] : TS(0.f);
  };
  auto prefetch_inverse = [&](int step) {
    const char* p = reinterpret_cast<const char*>(BT + elem(step) * (long long)(nb * nb));
    for (size_t o = (size_t)tid * 128; o < (size_t)nb * nb * sizeof(TS); o += (size_t)NT * 128)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
  };
  // state on the face: thread (side, j) holds the potential's N values along the
  // normal and the species' layer values; x of the next element
  const bool state_item = tid < 2 * FN;
  const int side = tid / FN, j = tid % FN;         // also of the tangent items below
  const int jj1 = j % N, jj2 = j / N;
  const int fs = a == 0 ? 1 : (a == 1 ? N : FN);
  const int node0 = a == 0 ? N * j : (a == 1 ? jj1 + FN * jj2 : j);
  TV up0[N], us[NF - 1], xv = TV(0);
  auto load_state = [&](int step) {                // the face between step - 1 and step
    if (!state_item) return;
    const TV* p = upc + boff + elem(side == own ? step : step - 1) * NN + node0;
#pragma unroll
    for (int k = 0; k < N; ++k) up0[k] = p[k * fs];
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) us[k] = p[(k + 1) * EN + (side == 0 ? P : 0) * fs];
  };
  const int xf = tid / NN, xi = tid % NN;          // row tid < nb: field and node
  auto load_x = [&](int step) {
    if (tid < nb) xv = x[boff + xf * EN + elem(step) * NN + xi];
  };
  const int x3[3] = {xi % N, (xi / N) % N, xi / FN};
  const int xk = pick3(x3, a);

  // geometry of the next face: the elements' 2 / h, the penalty, and (threads
  // with a face point) the point's weight and velocity along the axis
  const PhysT<TV>& ph = phys<TV>(prm);
  FaceGeo<TV> G;
  G.in_plane(prm, a, j0, j1);
  const int k1 = tid % Q, k2 = (tid / Q) % Q, po = k2 * QP + k1;
  const TV wt = ctab<P, TV>(TO::W + k1) * ctab<P, TV>(TO::W + k2) * (TV(0.25f) * G.h0 * G.h1);
  const TV xb0 = G.lo0 + halfv((ctab<P, TV>(TO::X + k1) + TV(1)) * G.h0);
  const TV xb1 = G.lo1 + halfv((ctab<P, TV>(TO::X + k2) + TV(1)) * G.h1);
  TV scl = TV(0), scu = TV(0), ua = TV(0), delta = TV(0);
  auto load_geo = [&](int step) {
    const int ia = dir > 0 ? step : nk - step;
    G.along(prm, a, ia, true, true);
    scl = inv_scale<TV>(prm, a, ia - 1);
    scu = inv_scale<TV>(prm, a, ia);
  };
  auto point_geo = [&] {
    TV xp[3], uv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) xp[c] = c == a ? G.xa : (c == b0 ? xb0 : xb1);
    velocity(ph, xp, uv);
    ua = pick3(uv, a);
    const TV hh = G.h0 * G.h0 + G.h1 * G.h1;
    delta = ph.cip * TV(P * P) / halfv(sqrtv(G.hL * G.hL + hh) + sqrtv(G.hU * G.hU + hh));
  };
  // lifting coefficients of this thread's row: its node's B values in the face,
  // and its end derivative
  const int xj0 = pick3(x3, b0), xj1 = pick3(x3, b1);
  TV bt[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) bt[q] = ctab<P, TV>(TO::B + q * N + xj0);
  const TV dle = ctab<P, TV>(TO::dL + (1 - own) * N + xk);
  const bool at_face = xk == (own == 0 ? P : 0);

  TV dl[N];   // end derivatives of the side this thread takes traces of
#pragma unroll
  for (int q = 0; q < N; ++q) dl[q] = ctab<P, TV>(TO::dL + (1 - (state_item ? side : up)) * N + q);

  load_inverse(0, 0, 1);
  load_x(0);
  if (nk > 1) { load_state(1); load_geo(1); }
#pragma unroll 1
  for (int step = 0; step < nk; ++step) {
    if (WIDE && step + 1 < nk) prefetch_inverse(step + 1);
    if (step > 0) {
      // layer values and physical normal derivatives along +e_a
      if (state_item || tid < (2 + NF) * FN) {
        const int sd = state_item ? side : up;
        const TV sc = sd == 0 ? scl : scu;
        TV v[N];
        if (!state_item) {
#pragma unroll
          for (int q = 0; q < N; ++q) v[q] = zs[(side - 2) * NN + node0 + q * fs];
        } else {
#pragma unroll
          for (int q = 0; q < N; ++q) v[q] = up0[q];
        }
        Dot<TV> d(dl[0], v[0]);
#pragma unroll
        for (int q = 1; q < N; ++q) d.fma(dl[q], v[q]);
        TV* o = A + jj1 + NX * jj2;
        const int tv = state_item ? side * (NF + 1) : T0 + side - 2;
        const int td = state_item ? side * (NF + 1) + NF : T0 + NF + side - 2;
        o[tv * (N * NX)] = sd == 0 ? v[P] : v[0];
        o[td * (N * NX)] = sc * d.get();
        if (state_item) {
#pragma unroll
          for (int q = 0; q < NF - 1; ++q) o[(tv + 1 + q) * (N * NX)] = us[q];
        }
      }
      load_inverse(step, 0, 3);
      __syncthreads();
      for (int w = tid; w < S::NTR * N; w += NT)
        line<P, TO::B, false, N, Q, TV>(A + w * NX, 1, B + w * QP, 1);
      load_inverse(step, 1, 3);
      __syncthreads();
      for (int w = tid; w < S::NTR * Q; w += NT) {
        const int g = w / Q, l = w - g * Q;
        line<P, TO::B, false, N, Q, TV>(B + g * (N * QP) + l, QP, A + g * (Q * QP) + l, QP);
      }
      load_inverse(step, 2, 3);
      point_geo();
      if (step + 1 < nk) load_state(step + 1);
      __syncthreads();
      if (tid < FQ) {
        const int o = po;
        face_interior_point<P, NF, kJvp, TV>(
            ph, ua, wt, delta,
            [&](int s, int t) -> TV {
              if (t == 0) return A[s * (NF + 1) * (Q * QP) + o];
              if (t == NA) return A[(s * (NF + 1) + NF) * (Q * QP) + o];
              if (t > NF && t < NA) return A[(s * (NF + 1) + t - NF) * (Q * QP) + o];
              const TV v = A[(t <= NF ? T0 + t - 1 : T0 + NF + t - NA - 1) * (Q * QP) + o];
              return s == up ? v : TV(0);
            },
            // own side's coefficients only: values, then derivatives
            [&](int slot, TV v) {
              if (slot < NF) B[slot * (Q * QP) + o] = own == 0 ? v : -v;
              else if (slot == NF) { if (own == 0) B[slot * (Q * QP) + o] = v; }
              else if (slot == 2 * NF) { if (own == 1) B[NF * (Q * QP) + o] = v; }
              else B[slot * (Q * QP) + o] = v;
            });
      }
      __syncthreads();
      for (int w = tid; w < 2 * NF * Q; w += NT) {
        const int g = w / Q, l = w - g * Q;
        line<P, TO::B, true, Q, N, TV>(B + g * (Q * QP) + l, QP, A + g * (N * QP) + l, QP);
      }
      __syncthreads();
    }
    if (tid < nb) {
      TA t = (TA)xv;
      if (step > 0) {
        // the last contraction for this row only: its S and T at its face node
        const TV* gs = A + (xf * N + xj1) * QP;
        const TV* gt = A + ((NF + xf) * N + xj1) * QP;
        TV sv = bt[0] * gs[0], tv = bt[0] * gt[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) {
          sv = mad(bt[q], gs[q], sv);
          tv = mad(bt[q], gt[q], tv);
        }
        TA add = (TA)dle * (TA)((own == 0 ? scl : scu) * tv);
        if (at_face) add += (TA)sv;
        t -= add;
      }
      ts[tid] = t;
    }
    if (step + 1 < nk) load_geo(step + 1);
    if (step + 1 < nk) load_x(step + 1);
    __syncthreads();
    {
      // a piece's columns in four sums by turns, the pieces added in order
      const TS* p = BT + elem(step) * (long long)(nb * nb) + rr;
      auto piece = [&](int from, int n, auto first) {      // columns [from, from + n)
        constexpr int A0 = decltype(first)::value ? AH : 0;  // of them held in registers
        TA acc[4] = {TA(0), TA(0), TA(0), TA(0)};
#pragma unroll
        for (int i = 0; i < A0; ++i)
          if (i < n) acc[i & 3] += (TA)bv[i] * ts[from + i];
        if constexpr (A0 < CC) {
          const TS* pc = p + (long long)from * nb;
          constexpr int K = WIDE ? 8 : 16;      // loads in flight
          int i = A0;
          for (; i + K <= n; i += K) {
            TS v[K];
#pragma unroll
            for (int q = 0; q < K; ++q) v[q] = pc[(long long)(i + q) * nb];
#pragma unroll
            for (int q = 0; q < K; ++q) acc[q & 3] += (TA)v[q] * ts[from + i + q];
          }
#pragma unroll
          for (int q = 0; q < K; ++q)
            if (i + q < n) acc[q & 3] += (TA)pc[(long long)(i + q) * nb] * ts[from + i + q];
        }
        return (acc[0] + acc[1]) + (acc[2] + acc[3]);
      };
      static_assert(AH == CC || AH % 4 == 0, "a column goes to the same sum wherever it is read from");
      TA s = piece(c0, cn, std::true_type());
      if constexpr (WIDE && S::COLS > 1) {
        ps[tid] = s;
        __syncthreads();
        if (tid < nb) {
#pragma unroll
          for (int q = 1; q < S::COLS; ++q) s += ps[q * S::RP + tid];
        }
      } else if constexpr (S::COLS > 1) {
#pragma unroll 1
        for (int q = 1; q < S::COLS; ++q)
          s += piece(q * CC, q * CC + CC <= nb ? CC : nb - q * CC, std::false_type());
      }
      if (tid < nb) {
        zs[tid] = (TV)s;
        z[boff + xf * EN + elem(step) * NN + xi] = (TV)s;
      }
      __syncthreads();
    }
  }
  wait_for_launch_before();
}

// The sweep over every line of elements along axis a, for every operating point.
template <int P, int NF, bool WIDE, class TV, class TS>
static cudaError_t launch_sweep_shape(const OpParams& prm, const void* binv, const TV* x, TV* z,
                                      const TV* upc, int batch, cudaStream_t stream, int a, int dir,
                                      int shared_blocks, bool beside) {
  using TA = typename std::conditional<sizeof(TS) == 8, double, float>::type;
  constexpr size_t bytes = SweepSmem<P, NF, WIDE, TV, TA>::bytes;
  auto kern = sweep_line_kernel<P, NF, WIDE, TV, TS>;
  static SmemAttr attr;
  cudaError_t e = raise_smem_limit(attr, kern, bytes);
  if (e != cudaSuccess) return e;
  const int lines = prm.ne[a == 0 ? 1 : 0] * prm.ne[a == 2 ? 1 : 2];
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)lines, (unsigned)batch);
  cfg.blockDim = dim3(SweepShape<P, NF, WIDE>::NT);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = stream;
  cfg.attrs = &early;
  cfg.numAttrs = beside ? 1 : 0;
  return launch_status(cudaLaunchKernelEx(&cfg, kern, prm, static_cast<const TS*>(binv), x, z, upc, a,
                                          dir, shared_blocks));
}
// Blocks of 192 rows and more (p = 3 with three fields, p = 4) take 768 threads wide,
// one line an SM. That is the faster chain, but more lines than SMs then wait for one
// another, each SM idle on memory during its line's face stages; with a thread per row two
// to four lines share an SM. 8 elements a line, p = 4, two fields, FP32 inverses and
// vectors: 80 lines 83 us wide and 108 so, 150 lines 114 and 115, 192 lines 182 and 147,
// 2,400 lines 1,570 and 1,153; FP64 vectors, whose face stages keep the FP64 pipe busy
// from one warp only, p = 3, three fields: 80 lines 134 and 108, 2,400 lines 2,060 and 732.
// Blocks of 128 rows take 256 threads wide, two lines an SM, and gain with FP64 vectors
// only: 300 lines 123 and 121, 2,400 lines 935 and 575 (FP32 vectors 220 and 319).
// Both shapes give the same bits.
constexpr int kSweepWideLines = 152;      // an SM each
template <int P, int NF, class TV, class TS>
static cudaError_t launch_sweep_typed(const OpParams& prm, const void* binv, const TV* x, TV* z,
                                      const TV* upc, int batch, cudaStream_t stream, int a, int dir,
                                      int shared_blocks, bool beside) {
  constexpr int rows = SweepShape<P, NF, true>::nb;
  if constexpr (rows > 128 || (rows == 128 && std::is_same<TV, double>::value)) {
    const long long lines = (long long)prm.ne[a == 0 ? 1 : 0] * prm.ne[a == 2 ? 1 : 2] * batch;
    if (lines > (rows > 128 ? 1 : 2) * kSweepWideLines)
      return launch_sweep_shape<P, NF, false, TV, TS>(prm, binv, x, z, upc, batch, stream, a, dir,
                                                      shared_blocks, beside);
  }
  return launch_sweep_shape<P, NF, true, TV, TS>(prm, binv, x, z, upc, batch, stream, a, dir,
                                                 shared_blocks, beside);
}
template <int P, int NF, class TV>
static cudaError_t launch_sweep_pn(const OpParams& prm, const void* binv, int storage, const TV* x,
                                   TV* z, const TV* upc, int batch, cudaStream_t s, int a, int dir,
                                   int shared_blocks, bool beside) {
  if (storage == 0) return launch_sweep_typed<P, NF, TV, double>(prm, binv, x, z, upc, batch, s, a, dir, shared_blocks, beside);
  if (storage == 1) return launch_sweep_typed<P, NF, TV, float>(prm, binv, x, z, upc, batch, s, a, dir, shared_blocks, beside);
  return launch_sweep_typed<P, NF, TV, __nv_bfloat16>(prm, binv, x, z, upc, batch, s, a, dir, shared_blocks, beside);
}

template <class TV>
cudaError_t launch_sweep(const OpParams& prm, const void* binv, int storage, const TV* x, TV* z,
                         const TV* upc, int batch, cudaStream_t s, int a, int dir,
                         int shared_blocks, bool beside) {
  if (prm.dim != 3 || storage < 0 || storage > 2 || (dir != 1 && dir != -1))
    return cudaErrorInvalidConfiguration;
#define ENP_SW(PP)                                                                                  \
  case PP:                                                                                          \
    if (prm.NF == 2)                                                                                \
      return launch_sweep_pn<PP, 2, TV>(prm, binv, storage, x, z, upc, batch, s, a, dir, shared_blocks, beside); \
    if (prm.NF == 3)                                                                                \
      return launch_sweep_pn<PP, 3, TV>(prm, binv, storage, x, z, upc, batch, s, a, dir, shared_blocks, beside); \
    return cudaErrorInvalidConfiguration;
  switch (prm.p) { ENP_SW(1) ENP_SW(2) ENP_SW(3) ENP_SW(4) }
#undef ENP_SW
  return cudaErrorInvalidConfiguration;
}

}  // namespace enp
