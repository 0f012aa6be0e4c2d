// R(u), J(u)v and J(u)^T w on quadrilaterals: two warps per element, one for the
// volume and one for its four faces, which need nothing of each other until the
// rows are formed; all stages pooled over fields, vectors and lines as in
// enp_tile3d.cuh. The faces are evaluated from this element's side in the same
// launch (a second launch would cost more than the other side's flux). Bound by
// latency on the meshes these
// problems have (8 x 8 elements, p = 2, residual and J v: 82 us with one array and
// face after the other, 35 pooled in one warp, 27 so), by the FP64 pipe on large ones.
#pragma once
#include "enp_launch.cuh"
#include "enp_tile3d.cuh"

namespace enp {

template <int P, int NF, int MODE>
struct Quad {
  using SL = Slots<P, NF, MODE>;
  static constexpr int N = P + 1, Q = P + 2, QP = Rows<P>::QP, AQ = Q * QP;
  static constexpr int NA = SL::NA, NG = SL::NG, NSL = SL::NSL, NTR = NA + NG;
  static constexpr int kV = NA * AQ;                 // values
  static constexpr int kG = 2 * NG * AQ;             // gradients, then fluxes; T1 before
  static constexpr int kT = NA * N * QP;             // after the x contraction
  static constexpr int kFL = 8 * NTR * N, kTR = 8 * NTR * Q, kFC = 4 * NSL * Q, kLC = 4 * NSL * N;
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  static constexpr int kA = kV, kB = mx(kG, kT), kC = mx(kFL, kFC), kD = mx(kTR, kLC);
  static constexpr int total = kA + kB + kC + kD;
};

// OP kBlockCol: column blockIdx.y of every element-diagonal block of J(u), the J v
// pass in the direction of the element's own basis function with the neighbours'
// direction zero, written to out[e][row][col].
template <int P, int NF, int OP, class R>
__global__ void __launch_bounds__(64)
quad2d_kernel(const OpParams prm, const R* __restrict__ u, const R* __restrict__ v,
              R* __restrict__ out) {
  constexpr bool kBlk = OP == kBlockCol;
  constexpr int MODE = kBlk ? (int)kJvp : OP;
  using S = Quad<P, NF, MODE>;
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, AQ = S::AQ, NN = N * N, FQ = Q * Q;
  constexpr int NA = S::NA, NG = S::NG, NTR = S::NTR, NSL = S::NSL;
  const PhysT<R>& ph = phys<R>(prm);
  extern __shared__ __align__(16) unsigned char tile_raw[];
  const int lane = threadIdx.x & 31;
  const bool faces = threadIdx.x >= 32;         // the second warp's part
  const int e = blockIdx.x;
  R* A = reinterpret_cast<R*>(tile_raw);
  R* B = A + S::kA;
  R* C = B + S::kB;
  R* D = C + S::kC;
  const int col = kBlk ? (int)blockIdx.y : -1, bidx = kBlk ? 0 : (int)blockIdx.y;
  const long long boff = (long long)bidx * prm.batch_stride, EN = (long long)prm.E * NN;
  const int idx[2] = {e % prm.ne[0], e / prm.ne[0]};
  // node i of array s of element en
  auto node = [&](int s, long long en, int i) -> R {
    if (kBlk && SL::vec(s)) return R(en == e && SL::field(s) * NN + i == col ? 1 : 0);
    return (SL::vec(s) ? v : u)[boff + SL::field(s) * EN + en * NN + i];
  };
  R lo[2], h[2], sc[2];
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    lo[a] = vertex<R>(prm, a, idx[a]);
    h[a] = elem_size<R>(prm, a, idx[a]);
    sc[a] = inv_scale<R>(prm, a, idx[a]);
  }
  auto bnd = [&](int a, int hi) { return hi ? idx[a] == prm.ne[a] - 1 : idx[a] == 0; };

  const bool has_val = MODE == kVjp || (MODE == kResidual && prm.src != nullptr);
  if (faces) {
    // layer values and physical normal derivatives along +axis of both sides (0
    // lower, 1 upper) of the four faces, their traces, fluxes and lifting
    for (int w = lane; w < 8 * N; w += 32) {
      const int fs_ = w / N, j = w - fs_ * N, s = fs_ >> 1, side = fs_ & 1, a = s >> 1, hi = s & 1;
      // hi face: this element is the lower one (side 0)
      const int step = hi == side ? (hi ? 1 : -1) : 0;
      if (step && bnd(a, hi)) continue;
      const long long en = e + step * (a == 0 ? 1 : prm.ne[0]);
      const int fs = a == 0 ? 1 : N, n0 = a == 0 ? N * j : j, lay = side == 0 ? P : 0;
      const R scn = inv_scale<R>(prm, a, (a == 0 ? idx[0] : idx[1]) + step);
      R dl[N];
#pragma unroll
      for (int k = 0; k < N; ++k) dl[k] = ctab<P, R>(TO::dL + (1 - side) * N + k);
      R* o = C + fs_ * (NTR * N) + j;
#pragma unroll
      for (int t = 0; t < NA; ++t) {
        o[t * N] = node(t, en, n0 + lay * fs);
        if (t < NG) {
          R d = dl[0] * node(t, en, n0);
#pragma unroll
          for (int k = 1; k < N; ++k) d = mad(dl[k], node(t, en, n0 + k * fs), d);
          o[(NA + t) * N] = scn * d;
        }
      }
    }
    __syncwarp();
    for (int w = lane; w < 8 * NTR; w += 32)
      line<P, TO::B, false, N, Q, R>(C + w * N, 1, D + w * Q, 1);
    __syncwarp();
    // face fluxes
    for (int w = lane; w < 4 * Q; w += 32) {
      const int s = w / Q, pt = w - s * Q, a = s >> 1, hi = s & 1;
      const R* t0 = D + 2 * s * (NTR * Q) + pt;
      R* c0 = C + s * (NSL * Q) + pt;
      auto tr = [&](int side, int t) -> R { return t0[(side * NTR + t) * Q]; };
      auto put = [&](int slot, R val) { c0[slot * Q] = val; };
      const R ha = a == 0 ? h[0] : h[1], hb = a == 0 ? h[1] : h[0], lb = a == 0 ? lo[1] : lo[0];
      const int ia = a == 0 ? idx[0] : idx[1];
      const R xb = lb + halfv((ctab<P, R>(TO::X + pt) + R(1)) * hb), xa = vertex<R>(prm, a, ia + hi);
      const R xp[3] = {a == 0 ? xa : xb, a == 0 ? xb : xa, R(0)};
      R uv[3];
      velocity(ph, xp, uv);
      const R ua = a == 0 ? uv[0] : uv[1], wt = ctab<P, R>(TO::W + pt) * halfv(hb), hh = hb * hb;
      if (!bnd(a, hi)) {
        const R hn = elem_size<R>(prm, a, ia + (hi ? 1 : -1));
        const R delta = ph.cip * R(P * P) / halfv(sqrtv(ha * ha + hh) + sqrtv(hn * hn + hh));
        face_interior_point<P, NF, MODE, R>(ph, ua, wt, delta, tr, put);
      } else {
        const int bface = prm.side_off[s] + (a == 0 ? idx[1] : idx[0]);
        face_boundary_point<P, NF, MODE, R>(prm, prm.btag[bface], bface, 1 - hi, ua, wt,
                                            ph.cip * R(P * P) / sqrtv(ha * ha + hh), xp, bidx, pt, tr,
                                            put);
      }
    }
    __syncwarp();
    for (int w = lane; w < 4 * NSL; w += 32)
      line<P, TO::B, true, Q, N, R>(C + w * Q, 1, D + w * N, 1);
  } else {
    for (int w = lane; w < NA * N; w += 32) {
      const int s = w / N, iy = w - s * N;
      R x[N];
#pragma unroll
      for (int k = 0; k < N; ++k) x[k] = node(s, e, iy * N + k);
      line_rows<P, TO::B, false, N, Q, R>(x, [&](int q, R val) { B[w * QP + q] = val; });
    }
    __syncwarp();
    for (int w = lane; w < NA * Q; w += 32) {
      const int s = w / Q, qx = w - s * Q;
      line<P, TO::B, false, N, Q, R>(B + s * (N * QP) + qx, QP, A + s * AQ + qx, QP);
    }
    __syncwarp();
    for (int w = lane; w < 2 * NG * Q; w += 32) {
      const int d = w >= NG * Q, t = w - d * (NG * Q), s = t / Q, r = t - s * Q;
      const int o = d ? r : r * QP, is = d ? QP : 1;
      line<P, TO::Dq, false, Q, Q, R>(A + s * AQ + o, is, B + (2 * s + d) * AQ + o, is);
    }
    __syncwarp();
    // point fluxes: x, y of field f over the gradients of slot f, the value
    // coefficient over the values
    for (int pt = lane; pt < FQ; pt += 32) {
      const int kx = pt % Q, ky = pt / Q, o = kx + QP * ky;
      const R w = ctab<P, R>(TO::W + kx) * ctab<P, R>(TO::W + ky);
      const R xp[3] = {lo[0] + halfv((ctab<P, R>(TO::X + kx) + R(1)) * h[0]),
                       lo[1] + halfv((ctab<P, R>(TO::X + ky) + R(1)) * h[1]), R(0)};
      R uv[3], s2[2], adv[2];
      velocity(ph, xp, uv);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const R s1 = w * halfv(h[1 - a]);
        s2[a] = s1 * sc[a];
        adv[a] = -(s1 * uv[a]);
      }
      point_flux<NF, MODE, R, 2>(ph, s2, adv, [&](int s) { return A[s * AQ + o]; },
                                 [&](int s, int a) { return B[(2 * s + a) * AQ + o]; },
                                 [&](int f, int a, R x) { B[(2 * f + a) * AQ + o] = x; },
                                 [&](int f, R x) { A[f * AQ + o] = x; });
      if (MODE == kResidual && has_val) {
        const R pw = w * (R(0.25) * h[0] * h[1]);
#pragma unroll
        for (int f = 0; f < NF; ++f)
          A[f * AQ + o] = -(pw * R(prm.src[((long long)f * prm.E + e) * FQ + pt]));
      }
    }
    __syncwarp();
    for (int w = lane; w < 2 * NF * Q; w += 32) {
      const int d = w >= NF * Q, t = w - d * (NF * Q), f = t / Q, r = t - f * Q;
      const int is = d ? QP : 1;
      R* p = B + (2 * f + d) * AQ + (d ? r : r * QP);
      line<P, TO::Dq, true, Q, Q, R>(p, is, p, is);
    }
    __syncwarp();
    for (int w = lane; w < NF * Q; w += 32) {
      const int f = w / Q, qx = w - f * Q;
      const R* hx = B + 2 * f * AQ + qx;
      R x[Q];
#pragma unroll
      for (int k = 0; k < Q; ++k) {
        x[k] = hx[k * QP] + hx[AQ + k * QP];
        if (MODE != kJvp && has_val) x[k] += A[f * AQ + qx + k * QP];
      }
      // over the line's own points of the values: no other line reads them
      line_rows<P, TO::B, true, Q, N, R>(x, [&](int n, R val) { A[f * AQ + n * QP + qx] = val; });
    }
  }
  __syncthreads();
  for (int w = threadIdx.x; w < NF * N; w += 64) {
    const int f = w / N, iy = w - f * N;
    R x[Q], acc[N];
#pragma unroll
    for (int k = 0; k < Q; ++k) x[k] = A[f * AQ + iy * QP + k];
    line_rows<P, TO::B, true, Q, N, R>(x, [&](int n, R val) { acc[n] = val; });
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int a = s >> 1, hi = s & 1;
      const R* L = D + s * (NSL * N);
      const R* Sp = L + (MODE == kVjp && !hi && f > 0 ? 2 * NF + f : f) * N;
      const R* Tp = L + (!hi && f == 0 ? 2 * NF : NF + f) * N;
      const bool neg = !hi && !(MODE == kVjp && f > 0);
      if (a == 0) {
        const R tv = sc[0] * Tp[iy], sv = neg ? -Sp[iy] : Sp[iy];
        acc[hi ? P : 0] += sv;
#pragma unroll
        for (int n = 0; n < N; ++n) acc[n] = mad(ctab<P, R>(TO::dL + hi * N + n), tv, acc[n]);
      } else {
        const R cf = ctab<P, R>(TO::dL + hi * N + iy) * sc[1];
#pragma unroll
        for (int n = 0; n < N; ++n) acc[n] = mad(cf, Tp[n], acc[n]);
        if (iy == (hi ? P : 0))
#pragma unroll
          for (int n = 0; n < N; ++n) acc[n] += neg ? -Sp[n] : Sp[n];
      }
    }
    if (kBlk) {
      const long long nb = NF * NN;
#pragma unroll
      for (int n = 0; n < N; ++n) out[((long long)e * nb + f * NN + iy * N + n) * nb + col] = acc[n];
    } else {
      R* o = out + boff + f * EN + (long long)e * NN + iy * N;
#pragma unroll
      for (int n = 0; n < N; ++n) o[n] = acc[n];
    }
  }
}

// grid.y: operating points, or the columns of the blocks.
template <int P, int NF, int MODE, class R>
static cudaError_t launch_quad(const OpParams& prm, const R* u, const R* v, R* out, int batch,
                               cudaStream_t stream) {
  constexpr size_t bytes = (size_t)Quad<P, NF, MODE == kBlockCol ? (int)kJvp : MODE>::total * sizeof(R);
  static_assert(bytes <= 200 * 1024, "quad kernel shared memory");
  auto k = quad2d_kernel<P, NF, MODE, R>;
  static SmemAttr attr;
  cudaError_t e = raise_smem_limit(attr, k, bytes);
  if (e != cudaSuccess) return e;
  k<<<dim3(prm.E, batch), 64, bytes, stream>>>(prm, u, v, out);
  return cudaGetLastError();
}

}  // namespace enp
