// R(u), J(u)v and J(u)^T w on hexahedra (Eq. NPDG / Eq. chargeDG, Sec. 3.3):
// one small group of warps per element, one warp per face (or two, three).
//
// Both kernels are bound by instruction issue, not by memory (30 flops per byte
// in FP64 accuracy, 12 instructions per multiply-add in double-float), so they
// are laid out to issue as few instructions per multiply-add as possible:
//  * a group is one to four warps, so that the stages of an element are short
//    and separated by a warp or a small block barrier;
//  * each stage is a pool of equal pencils (all arrays, all lines) dealt to the
//    group's lanes. A pencil loads its line into registers and forms all its
//    outputs with table entries at compile-time indices; its two addresses are
//    linear in the pool index (one small division per pencil);
//  * the x contraction reads the nodal lines straight from global memory, and
//    its transpose adds the face terms and stores the rows: no staging passes;
//  * only what the pointwise physics reads is formed. J v and J^T w need of the
//    state: the potential's gradient, the species' values, and on faces the
//    potential's normal derivative, but no species gradients or derivatives.
//  * pointwise, the reference gradients are kept unscaled and the two chain
//    factors and the weight are folded into one factor per direction.
//
// The face kernel runs first and leaves, per face, the lifted coefficients of
// the numerical flux. Conservation makes most of them common to both sides:
// slots [S_0..S_(NF-1), T_0..T_(NF-1), T_0 of the upper side (, S_1.. of the
// upper side for J^T w)], where a side's value coefficient is +S (lower) or -S
// (upper) and its derivative coefficient is T times the element's own 2/h:
// 2 NF + 1 (J^T w: 3 NF) arrays per face instead of 4 NF.
#pragma once
#include "enp_operator3d.cuh"

namespace enp {

// ------------------------------------------------------------ accumulators
// Sum of products: fused multiply-adds, or in double-float the leading parts by
// TwoSum with every error term gathered in one binary32, one
// renormalisation at the end.
template <class R>
struct Dot {
  R a;
  __device__ __forceinline__ Dot() {}
  __device__ __forceinline__ Dot(R x, R y) : a(x * y) {}
  __device__ __forceinline__ explicit Dot(R x) : a(x) {}
  __device__ __forceinline__ void fma(R x, R y) { a = mad(x, y, a); }
  __device__ __forceinline__ void add(R x) { a += x; }
  __device__ __forceinline__ R get() const { return a; }
};
template <>
struct Dot<df> {
  float s, t;
  __device__ __forceinline__ Dot() {}
  __device__ __forceinline__ Dot(df x, df y) {
    s = __fmul_rn(x.hi, y.hi);
    t = __fmaf_rn(x.hi, y.hi, -s);
    t = __fmaf_rn(x.hi, y.lo, t);
    t = __fmaf_rn(x.lo, y.hi, t);
  }
  __device__ __forceinline__ explicit Dot(df x) : s(x.hi), t(x.lo) {}
  __device__ __forceinline__ void fma(df x, df y) {
    const float p = __fmul_rn(x.hi, y.hi);
    float e = __fmaf_rn(x.hi, y.hi, -p);
    e = __fmaf_rn(x.hi, y.lo, e);
    e = __fmaf_rn(x.lo, y.hi, e);
    float s2, err;
    two_sum(s, p, s2, err);
    s = s2;
    t = __fadd_rn(t, __fadd_rn(err, e));
  }
  __device__ __forceinline__ void add(df x) {
    float s2, err;
    two_sum(s, x.hi, s2, err);
    s = s2;
    t = __fadd_rn(t, __fadd_rn(err, x.lo));
  }
  __device__ __forceinline__ df get() const { return fast_two_sum(s, t); }
};
// d = x y (the first term of an unrolled sum), or d += x y.
template <class R>
__device__ __forceinline__ void acc(Dot<R>& d, bool first, R x, R y) {
  if (first) d = Dot<R>(x, y);
  else d.fma(x, y);
}
__device__ __forceinline__ float halfv(float x) { return 0.5f * x; }
__device__ __forceinline__ double halfv(double x) { return 0.5 * x; }
__device__ __forceinline__ df halfv(df x) { return df(0.5f * x.hi, 0.5f * x.lo); }

// Size h of element i along axis a, and the reference-to-physical factor 2 / h.
template <class R> __device__ __forceinline__ R elem_size(const OpParams& p, int a, int i);
template <class R> __device__ __forceinline__ R inv_scale(const OpParams& p, int a, int i);
template <> __device__ __forceinline__ double elem_size<double>(const OpParams& p, int a, int i) { return p.xs[a][i].x; }
template <> __device__ __forceinline__ double inv_scale<double>(const OpParams& p, int a, int i) { return p.xs[a][i].y; }
template <> __device__ __forceinline__ float elem_size<float>(const OpParams& p, int a, int i) { return p.xsf[a][i].x; }
template <> __device__ __forceinline__ float inv_scale<float>(const OpParams& p, int a, int i) { return p.xsf[a][i].y; }
template <> __device__ __forceinline__ df elem_size<df>(const OpParams& p, int a, int i) {
  const float4 c = p.xsdf[a][i];
  return df(c.x, c.y);
}
template <> __device__ __forceinline__ df inv_scale<df>(const OpParams& p, int a, int i) {
  const float4 c = p.xsdf[a][i];
  return df(c.z, c.w);
}

// One line through a table: out[r] (r < ROWS) = sum_k M[r][k] x[k], with M at
// table offset TAB (B: Q x N, BD: Q x N, Dq: Q x Q) or its transpose.
template <int P, int TAB, bool TRANS, int COLS, class R>
__device__ __forceinline__ Dot<R> line_dot(const R (&x)[COLS], int r) {
  constexpr int W = TAB == TabOff<P>::Dq ? TabOff<P>::Q : TabOff<P>::N;  // row length of the table
  Dot<R> d(ctab<P, R>(TAB + (TRANS ? r : r * W)), x[0]);
#pragma unroll
  for (int k = 1; k < COLS; ++k) d.fma(ctab<P, R>(TAB + (TRANS ? k * W + r : r * W + k)), x[k]);
  return d;
}
template <int P, int TAB, bool TRANS, int COLS, int ROWS, class R>
__device__ __forceinline__ void line_dots(const R (&x)[COLS], Dot<R> (&d)[ROWS]) {
#pragma unroll
  for (int r = 0; r < ROWS; ++r) d[r] = line_dot<P, TAB, TRANS, COLS, R>(x, r);
}
template <int P, int TAB, bool TRANS, int COLS, int ROWS, class R, class ST>
__device__ __forceinline__ void line_rows(const R (&x)[COLS], ST store) {
#pragma unroll
  for (int r = 0; r < ROWS; ++r) store(r, line_dot<P, TAB, TRANS, COLS, R>(x, r).get());
}
template <int P, int TAB, bool TRANS, int COLS, int ROWS, class R>
__device__ __forceinline__ void line(const R* src, int is, R* dst, int os) {
  R x[COLS];
#pragma unroll
  for (int k = 0; k < COLS; ++k) x[k] = src[k * is];
  line_rows<P, TAB, TRANS, COLS, ROWS, R>(x, [&](int r, R v) { dst[r * os] = v; });
}

// ------------------------------------------------------------------ shapes
// Row length Q padded to odd: lines along x start in different banks.
template <int P> struct Rows { static constexpr int Q = P + 2, QP = Q % 2 ? Q : Q + 1; };

// Threads per group. FP32: see lane3d_kernel. FP64: one warp (the FP64 pipe
// bounds it, and more warps only add ragged pools), two at p = 4. Double-float:
// two warps from p = 3 on, whose 18 KB and more of shared memory per element
// leave too few warps resident otherwise.
template <int P, class R> __host__ __device__ constexpr int tile_threads() {
  if constexpr (std::is_same<R, float>::value) return P == 4 ? 128 : 32;
  else if constexpr (std::is_same<R, double>::value) return P == 4 ? 64 : 32;
  else return P >= 3 ? 64 : 32;
}
// Elements per group (FP32: lane3d_kernel; FP64 at p = 1: launch_3d_op).
template <int P, class R> __host__ __device__ constexpr int tile_elems() {
  if constexpr (std::is_same<R, double>::value) return P == 1 ? 3 : 1;
  return std::is_same<R, float>::value ? (P == 1 ? 3 : (P == 2 ? 2 : (P == 3 ? 1 : 3))) : 1;
}
// Faces per warp: as many as fill its lanes with face points (9, 16, 25, 36).
template <int P> __host__ __device__ constexpr int tile_faces() { return P == 1 ? 3 : (P == 2 ? 2 : 1); }
constexpr int kTileThreads = 128;   // largest block of either kernel

template <int P, int NF, int MODE>
struct Slots {
  static constexpr bool JAC = MODE == kJvp || MODE == kVjp;
  static constexpr int NA = MODE == kResidual ? NF : 2 * NF;   // arrays interpolated to the points
  static constexpr int NG = JAC ? NF + 1 : NA;                 // of them with gradients (listed first)
  // face coefficient arrays (none for <w, dR/dtheta>, kParam, which sums at the points)
  static constexpr int NSL = MODE == kParam ? 0 : (MODE == kVjp ? 3 * NF : 2 * NF + 1);
  static_assert(NSL <= 3 * NF, "the face buffer holds 3 NF arrays a face");
  // array s: vector (0 u, 1 v) and field
  __device__ static __forceinline__ int vec(int s) {
    return MODE == kParam ? s >= NF : (JAC && s >= 1 && s <= NF ? 1 : 0);
  }
  __device__ static __forceinline__ int field(int s) {
    if (MODE == kParam) return s < NF ? s : s - NF;
    return !JAC ? s : (s == 0 ? 0 : (s <= NF ? s - 1 : s - NF));
  }
};

template <int P, int NF, int MODE>
struct TileE {
  using SL = Slots<P, NF, MODE>;
  static constexpr int N = P + 1, Q = P + 2, QP = Rows<P>::QP;
  static constexpr int AQ = Q * Q * QP;              // one array of point values
  static constexpr int NA = SL::NA, NG = SL::NG;
  static constexpr int kT1 = NA * N * N * QP;        // after the x contraction
  static constexpr int kT2 = NA * N * Q * QP;        // after the y contraction
  // region A: values [NA], z gradients [NG] (over T1); region B: x, y gradients
  // [NG][2] (over T2). Transposed: T2 over A, T1 over B.
  static constexpr int kA0 = (NA + NG) * AQ, kB0 = 2 * NG * AQ;
  static constexpr int kA = kA0 > kT1 ? kA0 : kT1;
  static constexpr int kB = kB0 > kT2 ? kB0 : kT2;
  static constexpr int total = kA + kB;
};

// Whether the stages of a kernel are separated by a block barrier, also between
// groups that share no data. Double-float: its kernels are 50 to 60 KB of
// straight-line code, and warps that drift apart evict each other's instructions
// (channel of 64 x 32 x 16 elements, p = 3, J v: element kernel 0.70 ms with
// independent pairs of warps, 0.59 ms with two elements in step; face kernel 0.50
// and 0.47 ms). FP32 faces gain 3 %, its elements and FP64 nothing.
template <int P, class R> __host__ __device__ constexpr bool tile_lock() {
  return tile_threads<P, R>() > 32 || std::is_same<R, df>::value;
}
template <class R> __host__ __device__ constexpr bool face_lock() {
  return !std::is_same<R, double>::value;
}
template <bool LOCK>
__device__ __forceinline__ void group_sync() {
  if constexpr (!LOCK) __syncwarp();
  else __syncthreads();
}

// Resident face-kernel blocks per SM that the registers are sized for.
template <class R> struct FaceBlocks { static constexpr int value = std::is_same<R, float>::value ? 7 : 6; };

// ------------------------------------------------------------ point fluxes
// The fluxes of one volume point from values and unscaled reference gradients:
// val(s) and grad(s, a) of array s, putg(f, a, x) the coefficient of the
// reference derivative of field f's test function along a, putv(f, x) of its
// value (J^T w). s2[a] = w (2/h_a)^2 and adv[a] = -w (2/h_a) u_a carry the weight.
template <int NF, int MODE, class R, int DIM = 3, class VAL, class GRAD, class PUTG, class PUTV>
__device__ __forceinline__ void point_flux(const PhysT<R>& ph, const R* s2, const R* adv, VAL val,
                                           GRAD grad, PUTG putg, PUTV putv) {
  if constexpr (MODE == kResidual) {
    R c[NF - 1], m[NF - 1];
    Dot<R> kd;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      c[k] = val(k + 1);
      m[k] = ph.mig[k] * c[k];
      acc(kd, k == 0, ph.kcoef[k], c[k]);
    }
    const R kap = kd.get();
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      R g[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) g[f] = grad(f, a);
      Dot<R> f0(kap, g[0]);
#pragma unroll
      for (int k = 0; k < NF - 1; ++k) f0.fma(ph.acoef[k], g[k + 1]);
      putg(0, a, s2[a] * f0.get());
#pragma unroll
      for (int k = 0; k < NF - 1; ++k) {
        Dot<R> fk(ph.D[k], g[k + 1]);
        fk.fma(m[k], g[0]);
        Dot<R> t(s2[a], fk.get());
        t.fma(adv[a], c[k]);
        putg(k + 1, a, t.get());
      }
    }
  } else if constexpr (MODE == kJvp) {
    // state: potential gradient (array 0), species values (arrays NF + 1 + k);
    // tangent: gradients (arrays 1 + f), species values
    R m0[NF - 1], m1[NF - 1], c1[NF - 1];
    Dot<R> k0, k1;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const R c0 = val(NF + 1 + k);
      c1[k] = val(2 + k);
      acc(k0, k == 0, ph.kcoef[k], c0);
      acc(k1, k == 0, ph.kcoef[k], c1[k]);
      m0[k] = ph.mig[k] * c0;
      m1[k] = ph.mig[k] * c1[k];
    }
    const R kap0 = k0.get(), kap1 = k1.get();
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const R g0 = grad(0, a);
      R t1[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) t1[f] = grad(1 + f, a);
      Dot<R> f0(kap0, t1[0]);
      f0.fma(kap1, g0);
#pragma unroll
      for (int k = 0; k < NF - 1; ++k) f0.fma(ph.acoef[k], t1[k + 1]);
      putg(0, a, s2[a] * f0.get());
#pragma unroll
      for (int k = 0; k < NF - 1; ++k) {
        Dot<R> fk(ph.D[k], t1[k + 1]);
        fk.fma(m0[k], t1[0]);
        fk.fma(m1[k], g0);
        Dot<R> t(s2[a], fk.get());
        t.fma(adv[a], c1[k]);
        putg(k + 1, a, t.get());
      }
    }
  } else {
    // J^T w: test gradients (arrays 1 + f), state as above
    R m0[NF - 1];
    Dot<R> k0;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const R c0 = val(NF + 1 + k);
      acc(k0, k == 0, ph.kcoef[k], c0);
      m0[k] = ph.mig[k] * c0;
    }
    const R kap0 = k0.get();
    Dot<R> gw0, ch[NF - 1], cm[NF - 1];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      const R sg0 = s2[a] * grad(0, a);
      R W[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) W[f] = grad(1 + f, a);
      Dot<R> f0(kap0, W[0]);
      acc(gw0, a == 0, sg0, W[0]);
#pragma unroll
      for (int k = 0; k < NF - 1; ++k) {
        f0.fma(m0[k], W[k + 1]);
        acc(cm[k], a == 0, sg0, W[k + 1]);
        acc(ch[k], a == 0, adv[a], W[k + 1]);
        Dot<R> fk(ph.acoef[k], W[0]);
        fk.fma(ph.D[k], W[k + 1]);
        putg(k + 1, a, s2[a] * fk.get());
      }
      putg(0, a, s2[a] * f0.get());
    }
    const R g0 = gw0.get();
    putv(0, R(0));
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      ch[k].fma(ph.kcoef[k], g0);
      ch[k].fma(ph.mig[k], cm[k].get());
      putv(k + 1, ch[k].get());
    }
  }
}

// Element geometry, and the weight factors of one of its points. The direction
// factors start from the face areas, h_b h_c / 4, formed as the face kernel forms
// them, so that volume and face terms of a constant flux cancel to rounding.
template <int P, class R>
struct ElemGeo {
  int idx[3];
  R lo[3], h[3], sc[3], area[3];
  __device__ __forceinline__ ElemGeo(const OpParams& prm, int e) {
    idx[0] = e % prm.ne[0];
    idx[1] = (e / prm.ne[0]) % prm.ne[1];
    idx[2] = e / (prm.ne[0] * prm.ne[1]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = vertex<R>(prm, a, idx[a]);
      h[a] = elem_size<R>(prm, a, idx[a]);
      sc[a] = inv_scale<R>(prm, a, idx[a]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) area[a] = R(0.25f) * h[a == 0 ? 1 : 0] * h[a == 2 ? 1 : 2];
  }
  __device__ __forceinline__ R coord(int a, int k) const {
    return lo[a] + halfv((ctab<P, R>(TabOff<P>::X + k) + R(1)) * h[a]);
  }
  // w: reference weight of the point; uv: the velocity there
  __device__ __forceinline__ void factors(R w, const R* uv, R* s2, R* adv) const {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const R s1 = w * area[a];
      s2[a] = s1 * sc[a];
      adv[a] = -(s1 * uv[a]);
    }
  }
  // physical weight
  __device__ __forceinline__ R weight(R w) const { return w * (area[0] * halfv(h[0])); }
};

// A load of what the kernel before wrote while this one was already running: an
// ordinary (coherent) load, and not moved above wait_for_faces.
__device__ __forceinline__ float load_after_wait(const float* p) {
  float x;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ double load_after_wait(const double* p) {
  double x;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(x) : "l"(p));
  return x;
}
__device__ __forceinline__ df load_after_wait(const df* p) {
  float hi, lo;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(hi), "=f"(lo) : "l"(p));
  return df(hi, lo);
}

// The element kernel starts as soon as every block of the face kernel has (programmatic
// launch): its volume stages read u and v only. The face terms are there after this.
// One after the other, the face kernel's last wave and a launch stood between the two:
// double-float J v on 24 x 6 x 2 elements, p = 2, eight points 41.0 -> 36.9 us, FP32 on
// 61 x 15 x 5, p = 4, two points 82.0 -> 77.8 us, on 64 x 32 x 16, p = 3 192.6 -> 188.4 us.
__device__ __forceinline__ void wait_for_faces() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Adds the six face terms of field f to the row of N nodes r = iy + N iz, in
// side order, from the face kernel's coefficients.
template <int P, int NF, int MODE, class R>
__device__ __forceinline__ void add_face_terms(const OpParams& prm, const R* fb,
                                               const int* idx, const R* sc, int f, int r,
                                               Dot<R> (&acc)[P + 1]) {
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = P + 1, FN = N * N;
  const int iy = r % N, iz = r / N;
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int a = s >> 1, hi = s & 1;
    const int b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
    const long long gid = prm.foff[a] + (idx[a] + hi) +
                          (long long)(prm.ne[a] + 1) * (idx[b0] + (long long)prm.ne[b0] * idx[b1]);
    const R* F = fb + gid * (SL::NSL * FN);
    const R* Sp = F + (MODE == kVjp && !hi && f > 0 ? 2 * NF + f : f) * FN;
    const R* Tp = F + (!hi && f == 0 ? 2 * NF : NF + f) * FN;
    const bool neg = !hi && !(MODE == kVjp && f > 0);
    if (a == 0) {
      const R tv = sc[0] * load_after_wait(Tp + r);
      R sv = load_after_wait(Sp + r);
      if (neg) sv = -sv;
      acc[hi ? N - 1 : 0].add(sv);
#pragma unroll
      for (int n = 0; n < N; ++n) acc[n].fma(ctab<P, R>(TO::dL + hi * N + n), tv);
    } else {
      const int k = a == 1 ? iy : iz;
      const int j = N * (a == 1 ? iz : iy);
      const R cf = ctab<P, R>(TO::dL + hi * N + k) * sc[a];
#pragma unroll
      for (int n = 0; n < N; ++n) acc[n].fma(cf, load_after_wait(Tp + j + n));
      if (k == (hi ? N - 1 : 0)) {
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const R sv = load_after_wait(Sp + j + n);
          acc[n].add(neg ? -sv : sv);
        }
      }
    }
    // double-float: one renormalisation per side keeps the gathered error terms
    // at the size of one product's
#pragma unroll
    for (int n = 0; n < N; ++n) acc[n] = Dot<R>(acc[n].get());
  }
}

// Element (of EG in the group) of item w, n items an element; w becomes its own item.
template <int EG>
__device__ __forceinline__ int take_elem(int& w, int n) {
  if constexpr (EG == 1) return 0;
  const int el = w / n;
  w -= el * n;
  return el;
}

// The pooled stages from the nodal values of a group's EG elements to the values and
// reference gradients at their points: per element (regions total apart) region A
// [NA] values, [NG] z gradients; region B [NG][2] x and y gradients. Element el's nodes
// follow the first's by min(el, last) elements. Ends with a barrier of the group.
template <int P, int NF, int MODE, class R, int EG = 1>
__device__ __forceinline__ void tile_points(const io_t<R>* __restrict__ ue,
                                            const io_t<R>* __restrict__ ve, long long EN, R* A0,
                                            R* B0, int tid, int last = 0) {
  using S = TileE<P, NF, MODE>;
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, AQ = S::AQ, FN = N * N, FQ = Q * Q, NN = N * FN;
  constexpr int NA = S::NA, NG = S::NG, T = tile_threads<P, R>();
  // x: nodal lines from global memory
#pragma unroll 1
  for (int i = tid; i < EG * NA * FN; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NA * FN);
    const int s = w / FN, r = w - s * FN;
    const io_t<R>* src = (SL::vec(s) ? ve : ue) + SL::field(s) * EN + min(el, last) * NN + r * N;
    R x[N];
#pragma unroll
    for (int k = 0; k < N; ++k) x[k] = R(src[k]);
    R* dst = A0 + el * S::total + w * QP;
    line_rows<P, TO::B, false, N, Q, R>(x, [&](int q, R val) { dst[q] = val; });
  }
  group_sync<tile_lock<P, R>()>();
#pragma unroll 1
  for (int i = tid; i < EG * NA * N * Q; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NA * N * Q);
    const int g = w / Q, qx = w - g * Q;
    line<P, TO::B, false, N, Q, R>(A0 + el * S::total + g * (N * QP) + qx, QP,
                                   B0 + el * S::total + g * (Q * QP) + qx, QP);
  }
  group_sync<tile_lock<P, R>()>();
  // z: values of every array, then the z gradients (BD) of the first NG
#pragma unroll 1
  for (int i = tid; i < EG * NA * FQ; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NA * FQ);
    const int s = w / FQ, r = w - s * FQ, o = (r / Q) * QP + r % Q;
    line<P, TO::B, false, N, Q, R>(B0 + el * S::total + s * (N * Q * QP) + o, Q * QP,
                                   A0 + el * S::total + s * AQ + o, Q * QP);
  }
#pragma unroll 1
  for (int i = tid ^ (T > 32 ? 32 : 0); i < EG * NG * FQ; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NG * FQ);
    const int s = w / FQ, r = w - s * FQ, o = (r / Q) * QP + r % Q;
    line<P, TO::BD, false, N, Q, R>(B0 + el * S::total + s * (N * Q * QP) + o, Q * QP,
                                    A0 + el * S::total + (NA + s) * AQ + o, Q * QP);
  }
  group_sync<tile_lock<P, R>()>();
  // x and y gradients of the first NG arrays, one pool
#pragma unroll 1
  for (int i = tid; i < EG * 2 * NG * FQ; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, 2 * NG * FQ);
    const int d = w >= NG * FQ, t = w - d * (NG * FQ);
    const int s = t / FQ, r = t - s * FQ;
    const int o = d ? (r / Q) * (Q * QP) + r % Q : r * QP;
    const int is = d ? QP : 1;
    line<P, TO::Dq, false, Q, Q, R>(A0 + el * S::total + s * AQ + o, is,
                                    B0 + el * S::total + (2 * s + d) * AQ + o, is);
  }
  group_sync<tile_lock<P, R>()>();
}

// ------------------------------------------- element kernel, pooled pencils
// FP64 and double-float, whose pencils cost 100 to 300 issue slots: every stage
// is one pool, so that the lanes stay full (94 % at p = 3) at the price of one
// index computation per pencil.
template <int P, int NF, int MODE, class R, int EG = 1>
__global__ void __launch_bounds__(kTileThreads, 5)
tile3d_kernel(const OpParams prm, const io_t<R>* __restrict__ u, const io_t<R>* __restrict__ v,
              io_t<R>* __restrict__ out) {
  using S = TileE<P, NF, MODE>;
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, AQ = S::AQ, NN = N * N * N, FN = N * N, FQ = Q * Q;
  constexpr int NA = S::NA, T = tile_threads<P, R>();
  extern __shared__ __align__(16) unsigned char tile_raw[];
  const int grp = threadIdx.x / T, tid = threadIdx.x % T;
  const int eraw = (blockIdx.x * (blockDim.x / T) + grp) * EG;
  if (!tile_lock<P, R>() && eraw >= prm.E) return;
  const bool valid = eraw < prm.E;
  const int e0 = valid ? eraw : prm.E - 1;
  const int last = EG == 1 ? 0 : min(EG, prm.E - e0) - 1;   // elements beyond the mesh shadow it
  R* A0 = reinterpret_cast<R*>(tile_raw) + grp * (EG * S::total);
  R* B0 = A0 + S::kA;
  const int bidx = blockIdx.y;
  const long long boff = (long long)bidx * prm.batch_stride;
  const long long EN = (long long)prm.E * NN;
  const io_t<R>* ue = u + boff + (long long)e0 * NN;
  const io_t<R>* ve = SL::JAC ? v + boff + (long long)e0 * NN : nullptr;
  tile_points<P, NF, MODE, R, EG>(ue, ve, EN, A0, B0, tid, last);

  // point fluxes: those of field f replace x, y in region B slots 2f, 2f + 1, z
  // in region A slot NA + f; the value coefficient (R with sources, J^T w) in
  // region A slot f
  const ElemGeo<P, R> G0(prm, e0);     // of the only element (EG 1)
  const bool has_val = MODE == kVjp || (MODE == kResidual && prm.src != nullptr);
  {
    const PhysT<R>& ph = phys<R>(prm);
#pragma unroll 1
    for (int i = tid; i < EG * Q * FQ; i += T) {
      int pt = i;
      const int el = take_elem<EG>(pt, Q * FQ), e = e0 + min(el, last);
      const ElemGeo<P, R> G = EG == 1 ? G0 : ElemGeo<P, R>(prm, e);
      const int kx = pt % Q, ky = (pt / Q) % Q, kz = pt / FQ;
      const int o = kx + QP * (ky + Q * kz);
      const R w = ctab<P, R>(TO::W + kx) * ctab<P, R>(TO::W + ky) * ctab<P, R>(TO::W + kz);
      R s2[3], adv[3];
      {
        const R xp[3] = {G.coord(0, kx), G.coord(1, ky), G.coord(2, kz)};
        R uv[3];
        velocity(ph, xp, uv);
        G.factors(w, uv, s2, adv);
      }
      R* V = A0 + el * S::total + o;
      R* Gz = V + NA * AQ;
      R* Gxy = B0 + el * S::total + o;
      auto at = [&](int s, int a) -> R& { return a < 2 ? Gxy[(2 * s + a) * AQ] : Gz[s * AQ]; };
      point_flux<NF, MODE, R>(ph, s2, adv, [&](int s) { return V[s * AQ]; },
                              [&](int s, int a) { return at(s, a); },
                              [&](int f, int a, R x) { at(f, a) = x; },
                              [&](int f, R x) { V[f * AQ] = x; });
      if (MODE == kResidual && has_val) {
#pragma unroll
        for (int f = 0; f < NF; ++f)
          V[f * AQ] = -(G.weight(w) * R(prm.src[((long long)f * prm.E + e) * (Q * FQ) + pt]));
      }
    }
  }
  group_sync<tile_lock<P, R>()>();
  // transposed x and y derivatives, in place, one pool
#pragma unroll 1
  for (int i = tid; i < EG * 2 * NF * FQ; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, 2 * NF * FQ);
    const int d = w >= NF * FQ, t = w - d * (NF * FQ);
    const int f = t / FQ, r = t - f * FQ;
    const int o = d ? (r / Q) * (Q * QP) + r % Q : r * QP;
    const int is = d ? QP : 1;
    R* p = B0 + el * S::total + (2 * f + d) * AQ + o;
    line<P, TO::Dq, true, Q, Q, R>(p, is, p, is);
  }
  group_sync<tile_lock<P, R>()>();
  // z: values through B^T, z fluxes through BD^T, to the z nodes (over region A:
  // the line's own values and z fluxes are read before it writes slot f's first
  // N planes, which no other line reads)
#pragma unroll 1
  for (int i = tid; i < EG * NF * FQ; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NF * FQ);
    R* A = A0 + el * S::total;
    const int f = w / FQ, r = w - f * FQ, o = (r / Q) * QP + r % Q;
    R x[Q], y[Q];
    const R* hx = A + S::kA + 2 * f * AQ + o;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      x[k] = hx[k * Q * QP] + hx[AQ + k * Q * QP];
      y[k] = A[(NA + f) * AQ + o + k * Q * QP];
      if (MODE != kJvp && has_val) x[k] += A[f * AQ + o + k * Q * QP];
    }
    R* dst = A + f * AQ + o;
#pragma unroll
    for (int n = 0; n < N; ++n) {
      Dot<R> d(ctab<P, R>(TO::B + n), x[0]);
#pragma unroll
      for (int k = 1; k < Q; ++k) d.fma(ctab<P, R>(TO::B + k * N + n), x[k]);
      d = Dot<R>(d.get());
#pragma unroll
      for (int k = 0; k < Q; ++k) d.fma(ctab<P, R>(TO::BD + k * N + n), y[k]);
      dst[n * Q * QP] = d.get();
    }
  }
  group_sync<tile_lock<P, R>()>();
  // y^T into region B [NF][N z][N y][QP]
#pragma unroll 1
  for (int i = tid; i < EG * NF * N * Q; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NF * N * Q);
    const int g = w / Q, qx = w - g * Q;         // g = f * N + iz
    const int f = g / N, iz = g - f * N;
    line<P, TO::B, true, Q, N, R>(A0 + el * S::total + f * AQ + iz * (Q * QP) + qx, QP,
                                  B0 + el * S::total + g * (N * QP) + qx, QP);
  }
  group_sync<tile_lock<P, R>()>();
  wait_for_faces();
  // x^T: one row of N nodes per lane; the six face terms; store
  const R* fb = reinterpret_cast<const R*>(prm.fbuf) + (long long)bidx * prm.fbuf_stride;
#pragma unroll 1
  for (int i = tid; i < EG * NF * FN; i += T) {
    int w = i;
    const int el = take_elem<EG>(w, NF * FN), e = e0 + min(el, last);
    const ElemGeo<P, R> G = EG == 1 ? G0 : ElemGeo<P, R>(prm, e);
    const int f = w / FN, r = w - f * FN;        // r = iy + N * iz
    R x[Q];
    Dot<R> acc[N];
#pragma unroll
    for (int k = 0; k < Q; ++k) x[k] = B0[el * S::total + w * QP + k];
    line_dots<P, TO::B, true, Q, N, R>(x, acc);
    add_face_terms<P, NF, MODE, R>(prm, fb, G.idx, G.sc, f, r, acc);
    if (!valid || el > last) continue;
    io_t<R>* o = out + boff + f * EN + (long long)e * NN + r * N;
#pragma unroll
    for (int n = 0; n < N; ++n) o[n] = to_io(acc[n].get());
  }
}

// --------------------------------------------- element kernel, owned lines
// FP32, whose pencils cost 25 to 35 issue slots, so that an index computation
// each would double them: a lane owns one z line of points (kx, ky) of one
// element through the z contraction, the point fluxes and the transposed z
// contraction, holding species values, z gradients and z fluxes in registers;
// in the other stages it owns one line position and runs over the arrays, at
// compile-time offsets. A group holds as many elements as fill its lanes with z
// lines (27 of 32, 32 of 32, 25 of 32, 108 of 128 at p = 1..4).
template <int P> struct LaneGroup {
  static constexpr int E = tile_elems<P, float>(), T = tile_threads<P, float>();
};
template <int P, int NF, int MODE>
struct TileL {
  using SL = Slots<P, NF, MODE>;
  static constexpr int N = P + 1, Q = P + 2, QP = Rows<P>::QP, AQ = Q * Q * QP;
  static constexpr int kT1 = SL::NA * N * N * QP, kT2 = SL::NA * N * Q * QP;
  // region A: T1, then values [NG], then (transposed) T2; region B: T2, then x, y
  // gradients [NG][2], then (transposed) T1
  static constexpr int kA = SL::NG * AQ > kT1 ? SL::NG * AQ : kT1;
  static constexpr int kB = 2 * SL::NG * AQ > kT2 ? 2 * SL::NG * AQ : kT2;
  static constexpr int total = kA + kB;
};

// Runs f(s, l) for arrays s < CNT and line positions l < L of the lane's own
// element; K arrays at a time where the group's lanes allow it.
template <int L, int CNT, int E, int T, class F>
__device__ __forceinline__ void each_array(int tid, F f) {
  constexpr int K = T / (L * E) < 1 ? 1 : (T / (L * E) > CNT ? CNT : T / (L * E));
  const int el = tid / (L * K), t = tid % (L * K), sub = t / L, l = t % L;
  if (el < E) {
#pragma unroll
    for (int i = 0; i < CNT; i += K)
      if (CNT % K == 0 || i + sub < CNT) f(el, i + sub, l);
  }
}

template <int P, int NF, int MODE>
__global__ void __launch_bounds__(kTileThreads, 5)
lane3d_kernel(const OpParams prm, const float* __restrict__ u, const float* __restrict__ v,
              float* __restrict__ out) {
  using R = float;
  using S = TileL<P, NF, MODE>;
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, AQ = S::AQ, NN = N * N * N, FN = N * N, FQ = Q * Q;
  constexpr int NA = SL::NA, NG = SL::NG, NV = NF - 1;
  constexpr int T = LaneGroup<P>::T, EG = LaneGroup<P>::E;
  constexpr int ZS = Q * QP;    // plane stride of a point array
  extern __shared__ __align__(16) unsigned char tile_raw[];
  const int grp = threadIdx.x / T, tid = threadIdx.x % T;
  const int eraw = (blockIdx.x * (blockDim.x / T) + grp) * EG;
  if (!tile_lock<P, R>() && eraw >= prm.E) return;
  const int e0 = min(eraw, prm.E - 1);
  R* base = reinterpret_cast<R*>(tile_raw) + grp * (EG * S::total);
  const int bidx = blockIdx.y;
  const long long boff = (long long)bidx * prm.batch_stride;
  const long long EN = (long long)prm.E * NN;
  // elements beyond the mesh shadow the last one and store nothing
  auto elem = [&](int el) { return EG == 1 ? e0 : min(e0 + el, prm.E - 1); };

  each_array<FN, NA, EG, T>(tid, [&](int el, int s, int r) {
    const R* src = (SL::vec(s) ? v : u) + boff + SL::field(s) * EN + (long long)elem(el) * NN + r * N;
    R x[N];
#pragma unroll
    for (int k = 0; k < N; ++k) x[k] = src[k];
    R* dst = base + el * S::total + (s * FN + r) * QP;
    line_rows<P, TO::B, false, N, Q, R>(x, [&](int q, R val) { dst[q] = val; });
  });
  group_sync<tile_lock<P, R>()>();
  each_array<N * Q, NA, EG, T>(tid, [&](int el, int s, int l) {
    const int iz = l / Q, qx = l % Q;
    R* A = base + el * S::total;
    line<P, TO::B, false, N, Q, R>(A + (s * N + iz) * (N * QP) + qx, QP,
                                   A + S::kA + (s * N + iz) * (Q * QP) + qx, QP);
  });
  group_sync<tile_lock<P, R>()>();

  const int el = tid / FQ, l = tid % FQ, kx = l % Q, ky = l / Q;
  const bool own = el < EG;
  R* A = base + (own ? el : 0) * S::total;
  R* Bq = A + S::kA;
  const int o = ky * QP + kx;
  // z: values and z gradients of the lane's line; the values of the gradient
  // arrays also to region A for the x and y derivatives
  R gz[NG][Q];        // z gradients, then z fluxes
  R c0[NV][Q];        // state species, then (J^T w) value coefficients
  R c1[MODE == kJvp ? NV : 1][Q];   // tangent species
  if (own) {
#pragma unroll
    for (int s = 0; s < NA; ++s) {
      R x[N];
#pragma unroll
      for (int k = 0; k < N; ++k) x[k] = Bq[s * (N * ZS) + k * ZS + o];
      line_rows<P, TO::B, false, N, Q, R>(x, [&](int q, R val) {
        if (s < NG) A[s * AQ + q * ZS + o] = val;
        if (!SL::JAC && s > 0) c0[s - 1][q] = val;
        if (SL::JAC && s >= NG) c0[s - NG][q] = val;
        if (MODE == kJvp && s >= 2 && s < NG) c1[s - 2][q] = val;
      });
      if (s < NG) line_rows<P, TO::BD, false, N, Q, R>(x, [&](int q, R val) { gz[s][q] = val; });
    }
  }
  group_sync<tile_lock<P, R>()>();
  each_array<FQ, NG, EG, T>(tid, [&](int el_, int s, int r) {
    R* A_ = base + el_ * S::total;
    line<P, TO::Dq, false, Q, Q, R>(A_ + s * AQ + r * QP, 1, A_ + S::kA + 2 * s * AQ + r * QP, 1);
  });
  each_array<FQ, NG, EG, T>(tid, [&](int el_, int s, int r) {
    R* A_ = base + el_ * S::total;
    const int oy = (r / Q) * ZS + r % Q;
    line<P, TO::Dq, false, Q, Q, R>(A_ + s * AQ + oy, QP, A_ + S::kA + (2 * s + 1) * AQ + oy, QP);
  });
  group_sync<tile_lock<P, R>()>();
  const ElemGeo<P, R> G(prm, elem(own ? el : 0));
  const bool has_src = MODE == kResidual && prm.src != nullptr;
  R sv[MODE == kResidual ? NF : 1][Q];   // value coefficients of the sources
  if (own) {
    const PhysT<R>& ph = prm.pf;
    const R wxy = ctab<P, R>(TO::W + kx) * ctab<P, R>(TO::W + ky);
    const R xx = G.coord(0, kx), xy = G.coord(1, ky);
    R* Gxy = Bq + o;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const R w = wxy * ctab<P, R>(TO::W + q);
      R s2[3], adv[3];
      {
        const R xp[3] = {xx, xy, G.coord(2, q)};
        R uv[3];
        velocity(ph, xp, uv);
        G.factors(w, uv, s2, adv);
      }
      point_flux<NF, MODE, R>(
          ph, s2, adv,
          [&](int s) {
            return !SL::JAC ? c0[s - 1][q] : (s >= NG ? c0[s - NG][q] : c1[MODE == kJvp ? s - 2 : 0][q]);
          },
          [&](int s, int a) { return a < 2 ? Gxy[(2 * s + a) * AQ + q * ZS] : gz[s][q]; },
          [&](int f, int a, R x) {
            if (a < 2) Gxy[(2 * f + a) * AQ + q * ZS] = x;
            else gz[f][q] = x;
          },
          [&](int f, R x) { if (f > 0) c0[f - 1][q] = x; });
      if (MODE == kResidual && has_src) {
#pragma unroll
        for (int f = 0; f < NF; ++f)
          sv[MODE == kResidual ? f : 0][q] =
              -(G.weight(w) * R(prm.src[((long long)f * prm.E + elem(el)) * (Q * FQ) + l + FQ * q]));
      }
    }
  }
  group_sync<tile_lock<P, R>()>();
  each_array<FQ, NF, EG, T>(tid, [&](int el_, int f, int r) {
    R* p = base + el_ * S::total + S::kA + 2 * f * AQ + r * QP;
    line<P, TO::Dq, true, Q, Q, R>(p, 1, p, 1);
  });
  each_array<FQ, NF, EG, T>(tid, [&](int el_, int f, int r) {
    R* p = base + el_ * S::total + S::kA + (2 * f + 1) * AQ + (r / Q) * ZS + r % Q;
    line<P, TO::Dq, true, Q, Q, R>(p, QP, p, QP);
  });
  group_sync<tile_lock<P, R>()>();
  if (own) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      R x[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        x[q] = Bq[2 * f * AQ + q * ZS + o] + Bq[(2 * f + 1) * AQ + q * ZS + o];
        if (MODE == kVjp && f > 0) x[q] += c0[f > 0 ? f - 1 : 0][q];
        if (MODE == kResidual && has_src) x[q] += sv[MODE == kResidual ? f : 0][q];
      }
#pragma unroll
      for (int n = 0; n < N; ++n) {
        R d = ctab<P, R>(TO::B + n) * x[0];
#pragma unroll
        for (int q = 1; q < Q; ++q) d = mad(ctab<P, R>(TO::B + q * N + n), x[q], d);
#pragma unroll
        for (int q = 0; q < Q; ++q) d = mad(ctab<P, R>(TO::BD + q * N + n), gz[f][q], d);
        A[(f * N + n) * ZS + o] = d;
      }
    }
  }
  group_sync<tile_lock<P, R>()>();
  each_array<N * Q, NF, EG, T>(tid, [&](int el_, int f, int t) {
    const int iz = t / Q, qx = t % Q;
    R* A_ = base + el_ * S::total;
    line<P, TO::B, true, Q, N, R>(A_ + (f * N + iz) * ZS + qx, QP,
                                  A_ + S::kA + (f * N + iz) * (N * QP) + qx, QP);
  });
  group_sync<tile_lock<P, R>()>();
  wait_for_faces();
  const R* fb = reinterpret_cast<const R*>(prm.fbuf) + (long long)bidx * prm.fbuf_stride;
  // x^T: one row of N nodes per lane; the six face terms; store
  constexpr int KX = T / (FN * EG) < 1 ? 1 : (T / (FN * EG) > NF ? NF : T / (FN * EG));
  const int ex = tid / (FN * KX), fx = (tid % (FN * KX)) / FN, r = tid % FN;
  if (ex < EG && eraw + ex < prm.E) {
    const int e = e0 + ex;
    const int idx[3] = {e % prm.ne[0], (e / prm.ne[0]) % prm.ne[1], e / (prm.ne[0] * prm.ne[1])};
    const R sc[3] = {inv_scale<R>(prm, 0, idx[0]), inv_scale<R>(prm, 1, idx[1]),
                     inv_scale<R>(prm, 2, idx[2])};
    const R* Bx = base + ex * S::total + S::kA + r * QP;
#pragma unroll 1
    for (int f = fx; f < NF; f += KX) {
      R x[Q];
      Dot<R> acc[N];
#pragma unroll
      for (int k = 0; k < Q; ++k) x[k] = Bx[f * FN * QP + k];
      line_dots<P, TO::B, true, Q, N, R>(x, acc);
      add_face_terms<P, NF, MODE, R>(prm, fb, idx, sc, f, r, acc);
      R* op = out + boff + f * EN + (long long)e * NN + r * N;
#pragma unroll
      for (int n = 0; n < N; ++n) op[n] = acc[n].get();
    }
  }
}

// ------------------------------------------------------------- face kernel
template <int P, int NF, int MODE>
struct TileF {
  using SL = Slots<P, NF, MODE>;
  static constexpr int N = P + 1, Q = P + 2, QP = Rows<P>::QP;
  static constexpr int NX = N % 2 ? N : N + 1;
  static constexpr int FN = N * N, FQ = Q * Q, NF_ = tile_faces<P>();
  static constexpr int NTR = SL::NA + SL::NG;      // traces per side: values, then derivatives
  static constexpr int kFL = 2 * NTR * N * NX;
  static constexpr int kF1 = 2 * NTR * N * QP;
  static constexpr int kTR = 2 * NTR * Q * QP;
  static constexpr int kFC = SL::NSL * Q * QP;
  static constexpr int kG1 = SL::NSL * N * QP;
  static constexpr int max3(int a, int b, int c) { return a > b ? (a > c ? a : c) : (b > c ? b : c); }
  // region A: layer data, then traces, then the first transposed contraction;
  // region B: the first contraction, then the flux coefficients
  static constexpr int kA = NF_ * max3(kFL, kTR, kG1), kB = NF_ * (kF1 > kFC ? kF1 : kFC);
  static constexpr int total = kA + kB;
};

// Where face g lies: axis, plane, in-plane cell, and its two elements.
struct FaceAt {
  int a, ia, j0, j1, eL, eU;
  bool hasL, hasU;
};
__device__ __forceinline__ FaceAt face_at(const OpParams& prm, long long g) {
  FaceAt f;
  f.a = (g >= prm.foff[1]) + (g >= prm.foff[2]);
  // at most 2^30 elements, so at most 2^31 faces of one direction
  const unsigned fi = (unsigned)(g - (f.a == 0 ? 0 : (f.a == 1 ? prm.foff[1] : prm.foff[2])));
  const unsigned n0 = prm.ne[0], n1 = prm.ne[1];
  const unsigned na = f.a == 0 ? n0 : (f.a == 1 ? n1 : prm.ne[2]), nb = f.a == 0 ? n1 : n0;
  const unsigned rr = fi / (na + 1), ia = fi - rr * (na + 1);
  const unsigned j1 = rr / nb, j0 = rr - j1 * nb;
  f.ia = (int)ia;
  f.j0 = (int)j0;
  f.j1 = (int)j1;
  f.hasL = ia > 0;
  f.hasU = ia < na;
  const unsigned sa = f.a == 0 ? 1 : (f.a == 1 ? n0 : n0 * n1);
  const unsigned s0 = f.a == 0 ? n0 : 1, s1 = f.a == 2 ? n0 : n0 * n1;
  const unsigned eU = ia * sa + j0 * s0 + j1 * s1;
  f.eU = (int)eU;          // an element only when hasU
  f.eL = (int)(eU - sa);   // an element only when hasL
  return f;
}

// Sizes and position of a face: in-plane corner and lengths, plane coordinate,
// the two elements' lengths along the axis (1 where there is none).
template <class R>
struct FaceGeo {
  R lo0, lo1, h0, h1, xa, hL, hU;
  __device__ __forceinline__ void in_plane(const OpParams& prm, int a, int j0, int j1) {
    const int b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
    lo0 = vertex<R>(prm, b0, j0);
    lo1 = vertex<R>(prm, b1, j1);
    h0 = elem_size<R>(prm, b0, j0);
    h1 = elem_size<R>(prm, b1, j1);
  }
  __device__ __forceinline__ void along(const OpParams& prm, int a, int ia, bool hasL, bool hasU) {
    xa = vertex<R>(prm, a, ia);
    hL = hasL ? elem_size<R>(prm, a, ia - 1) : R(1);
    hU = hasU ? elem_size<R>(prm, a, ia) : R(1);
  }
};

// The flux coefficients at a point of an interior face: ua the velocity along
// +axis, w the weight, delta the penalty. tr(side, t): trace t (values of the NA
// arrays, then physical normal derivatives along +axis of the first NG) of the
// lower (0) or upper (1) side; put(slot, value).
template <int P, int NF, int MODE, class R, class TR, class PUT>
__device__ __forceinline__ void face_interior_point(const PhysT<R>& ph, R ua, R w, R delta, TR tr,
                                                    PUT put) {
  constexpr int NA = Slots<P, NF, MODE>::NA;
  const R hw = halfv(w);
  if constexpr (MODE == kResidual) {
    const R pm = tr(0, 0), pp = tr(1, 0), dm = tr(0, NA), dp = tr(1, NA);
    const R jphi = pm - pp;
    R kapm, kapp;
    Dot<R> t0, s0;
    Dot<R> km, kp;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const R cm = tr(0, k + 1), cp = tr(1, k + 1);
      const R jc = cm - cp, dd = tr(0, NA + k + 1) + tr(1, NA + k + 1);
      Dot<R> qmd(ua), qpd(ua);
      qmd.fma(-ph.mig[k], dm);
      qpd.fma(-ph.mig[k], dp);
      const R qm = qmd.get(), qp = qpd.get();
      const R qa = halfv(qm + qp);
      // 2 S = D (2 delta jc - dd) + cm qm + cp qp + |qa| jc
      Dot<R> x(delta + delta, jc);
      x.add(-dd);
      Dot<R> sk(ph.D[k], x.get());
      sk.fma(cm, qm);
      sk.fma(cp, qp);
      sk.fma(absv(qa), jc);
      put(k + 1, hw * sk.get());
      put(NF + k + 1, -(hw * (ph.D[k] * jc)));
      acc(km, k == 0, ph.kcoef[k], cm);
      acc(kp, k == 0, ph.kcoef[k], cp);
      acc(t0, k == 0, ph.acoef[k], jc);
      acc(s0, k == 0, ph.acoef[k], dd);
    }
    kapm = km.get(); kapp = kp.get();
    Dot<R> tL = t0, tU = t0;
    tL.fma(kapm, jphi);
    tU.fma(kapp, jphi);
    put(NF, -(hw * tL.get()));
    put(2 * NF, -(hw * tU.get()));
    s0.fma(kapm, dm);
    s0.fma(kapp, dp);
    s0.fma(-(delta * jphi), kapm + kapp);
    put(0, -(hw * s0.get()));
  } else if constexpr (MODE == kJvp) {
    const R jphi0 = tr(0, 0) - tr(1, 0), jphi1 = tr(0, 1) - tr(1, 1);
    const R d0m = tr(0, NA), d0p = tr(1, NA), d1m = tr(0, NA + 1), d1p = tr(1, NA + 1);
    const R e1 = halfv(d1m + d1p);
    Dot<R> t0, s0;
    Dot<R> k0m, k0p, k1m, k1p;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const R c0m = tr(0, NF + 1 + k), c0p = tr(1, NF + 1 + k);
      const R c1m = tr(0, 2 + k), c1p = tr(1, 2 + k);
      const R jc0 = c0m - c0p, jc1 = c1m - c1p;
      const R dd = tr(0, NA + 2 + k) + tr(1, NA + 2 + k);
      Dot<R> qmd(ua), qpd(ua);
      qmd.fma(-ph.mig[k], d0m);
      qpd.fma(-ph.mig[k], d0p);
      const R qm = qmd.get(), qp = qpd.get();
      const R qa = halfv(qm + qp);
      const R sg = qa > R(0) ? jc0 : (qa < R(0) ? -jc0 : R(0));
      // 2 S' = D (2 delta jc' - dd') + cm' qm + cp' qp + |qa| jc'
      //        - mig (cm dm' + cp dp' + sign(qa) jc (dm' + dp') / 2)
      Dot<R> x(delta + delta, jc1);
      x.add(-dd);
      Dot<R> y(c0m, d1m);
      y.fma(c0p, d1p);
      y.fma(sg, e1);
      Dot<R> sk(ph.D[k], x.get());
      sk.fma(c1m, qm);
      sk.fma(c1p, qp);
      sk.fma(absv(qa), jc1);
      sk.fma(-ph.mig[k], y.get());
      put(k + 1, hw * sk.get());
      put(NF + k + 1, -(hw * (ph.D[k] * jc1)));
      acc(k0m, k == 0, ph.kcoef[k], c0m);
      acc(k0p, k == 0, ph.kcoef[k], c0p);
      acc(k1m, k == 0, ph.kcoef[k], c1m);
      acc(k1p, k == 0, ph.kcoef[k], c1p);
      acc(t0, k == 0, ph.acoef[k], jc1);
      acc(s0, k == 0, ph.acoef[k], dd);
    }
    const R a0m = k0m.get(), a0p = k0p.get(), a1m = k1m.get(), a1p = k1p.get();
    Dot<R> tL = t0, tU = t0;
    tL.fma(a1m, jphi0);
    tL.fma(a0m, jphi1);
    tU.fma(a1p, jphi0);
    tU.fma(a0p, jphi1);
    put(NF, -(hw * tL.get()));
    put(2 * NF, -(hw * tU.get()));
    s0.fma(a1m, d0m);
    s0.fma(a0m, d1m);
    s0.fma(a1p, d0p);
    s0.fma(a0p, d1p);
    Dot<R> pen(a1m + a1p, jphi0);
    pen.fma(a0m + a0p, jphi1);
    s0.fma(-delta, pen.get());
    put(0, -(hw * s0.get()));
  } else {
    // adjoint: the functional S_f (wm_f - wp_f) + T_f (dwm_f + dwp_f) (the
    // potential's T with each side's own kappa), differentiated by both states
    const R jphi = tr(0, 0) - tr(1, 0), dm = tr(0, NA), dp = tr(1, NA);
    const R jw0 = tr(0, 1) - tr(1, 1), vm0 = tr(0, NA + 1), vp0 = tr(1, NA + 1);
    const R vs = vm0 + vp0;
    const R dj = delta * jphi;
    Dot<R> km, kp, am, ap;
#pragma unroll
    for (int k = 0; k < NF - 1; ++k) {
      const R cm = tr(0, NF + 1 + k), cp = tr(1, NF + 1 + k), jc = cm - cp;
      const R jw = tr(0, 2 + k) - tr(1, 2 + k), vw = tr(0, NA + 2 + k) + tr(1, NA + 2 + k);
      Dot<R> qmd(ua), qpd(ua);
      qmd.fma(-ph.mig[k], dm);
      qpd.fma(-ph.mig[k], dp);
      const R qm = qmd.get(), qp = qpd.get();
      const R qa = halfv(qm + qp), aq = absv(qa);
      const R sg = qa > R(0) ? jc : (qa < R(0) ? -jc : R(0));
      const R dj2 = ph.D[k] * (delta + delta);
      // 2 x (derivatives with respect to cm, cp)
      Dot<R> xm(dj2 + qm + aq, jw), xp_(-dj2 + qp - aq, jw);
      Dot<R> dv(ph.D[k], vw);
      dv.fma(ph.acoef[k], vs);
      const R dvv = dv.get();
      Dot<R> ym(dj - dm, jw0), yp(dj - dp, jw0);
      ym.fma(-jphi, vm0);
      yp.fma(-jphi, vp0);
      xm.add(-dvv);
      xm.fma(ph.kcoef[k], ym.get());
      xp_.add(dvv);
      xp_.fma(ph.kcoef[k], yp.get());
      put(k + 1, hw * xm.get());
      put(2 * NF + k + 1, hw * xp_.get());
      Dot<R> tk(ph.D[k], jw);
      tk.fma(ph.acoef[k], jw0);
      put(NF + k + 1, -(hw * tk.get()));
      const R mj = ph.mig[k] * jw, hs = halfv(sg);
      acc(am, k == 0, mj, cm + hs);
      acc(ap, k == 0, mj, cp + hs);
      acc(km, k == 0, ph.kcoef[k], cm);
      acc(kp, k == 0, ph.kcoef[k], cp);
    }
    const R kapm = km.get(), kapp = kp.get();
    Dot<R> x0(kapm, vm0);
    x0.fma(kapp, vp0);
    x0.fma(-(delta * jw0), kapm + kapp);
    put(0, -(hw * x0.get()));
    am.fma(kapm, jw0);
    ap.fma(kapp, jw0);
    put(NF, -(hw * am.get()));
    put(2 * NF, -(hw * ap.get()));
  }
}

// The same at a point pt of a boundary face of the element on `side`: tag and
// index of the face, ua the velocity along +axis at xp.
template <int P, int NF, int MODE, class R, class TR, class PUT>
__device__ __forceinline__ void face_boundary_point(const OpParams& prm, int tag, int bface, int side,
                                                    R ua, R w, R delta, const R* xp, int bidx, int pt,
                                                    TR tr, PUT put) {
  using SL = Slots<P, NF, MODE>;
  constexpr int NA = SL::NA;
  const PhysT<R>& ph = phys<R>(prm);
  const R nrm = side == 0 ? R(1) : R(-1);
  R oS[NF], oT[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) { oS[f] = R(0); oT[f] = R(0); }
  if (!(tag == kWall || (tag == kInlet && MODE != kResidual))) {
    const R phiapp = (tag >= kElectrode0)
        ? (prm.phiapp_batch ? R(prm.phiapp_batch[bidx * 4 + (tag - kElectrode0)])
                            : ph.phiapp[tag - kElectrode0])
        : R(0);
    const R un = ua * nrm;
    R c[NF], d[NF], g[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      // the state's species derivatives enter neither J v nor J^T w
      c[f] = tr(side, !SL::JAC || f == 0 ? f : NF + f);
      d[f] = !SL::JAC || f == 0 ? tr(side, NA + f) * nrm : R(0);
      g[f] = (tag == kDirichlet && prm.dirv)
                 ? R(prm.dirv[((long long)f * prm.NBF + bface) * prm.Nfq + pt]) : R(0);
    }
    if constexpr (MODE == kResidual) {
      face_boundary_flux<NF, R, R>(ph, tag, c, d, g, un, delta, xp, phiapp, oS, oT);
    } else {
      R c1[NF], d1[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) { c1[f] = tr(side, 1 + f); d1[f] = tr(side, NA + 1 + f) * nrm; }
      if constexpr (MODE == kJvp) {
        Tan<R> tm[NF], td[NF], Sf[NF], Tf[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) { tm[f] = Tan<R>(c[f], c1[f]); td[f] = Tan<R>(d[f], d1[f]); }
        face_boundary_flux<NF, Tan<R>, R>(ph, tag, tm, td, g, un, delta, xp, phiapp, Sf, Tf);
#pragma unroll
        for (int f = 0; f < NF; ++f) { oS[f] = Sf[f].d; oT[f] = Tf[f].d; }
      } else {
        face_boundary_adjoint<NF, R>(ph, tag, c, d, g, un, delta, xp, phiapp, c1, d1, oS, oT);
      }
    }
  }
  // value coefficients carry the side's sign, derivative coefficients +axis
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const R s = w * oS[f], t = w * (side == 0 ? oT[f] : -oT[f]);
    if (MODE == kVjp && f > 0) {
      put(f, s);
      put(2 * NF + f, s);
    } else {
      put(f, side == 0 ? s : -s);
    }
    put(NF + f, t);
    if (f == 0) put(2 * NF, t);
  }
}

// The flux coefficients of one face point (tr and put as above).
template <int P, int NF, int MODE, class R, class TR, class PUT>
__device__ __forceinline__ void face_point(const OpParams& prm, const FaceAt& F,
                                           const FaceGeo<R>& G, int bidx, int pt, TR tr, PUT put) {
  using TO = TabOff<P>;
  constexpr int Q = P + 2;
  const PhysT<R>& ph = phys<R>(prm);
  const int a = F.a, b0 = a == 0 ? 1 : 0;
  const int k1 = pt % Q, k2 = pt / Q;
  const R h0 = G.h0, h1 = G.h1, xa = G.xa, hL = G.hL, hU = G.hU;
  const R hh = h0 * h0 + h1 * h1;
  R xp[3], uv[3];
  {
    const R xb0 = G.lo0 + halfv((ctab<P, R>(TO::X + k1) + R(1)) * h0);
    const R xb1 = G.lo1 + halfv((ctab<P, R>(TO::X + k2) + R(1)) * h1);
#pragma unroll
    for (int c = 0; c < 3; ++c) xp[c] = c == a ? xa : (c == b0 ? xb0 : xb1);
  }
  velocity(ph, xp, uv);
  const R ua = pick3(uv, a);
  const R w = ctab<P, R>(TO::W + k1) * ctab<P, R>(TO::W + k2) * (R(0.25f) * h0 * h1);
  if (F.hasL && F.hasU) {
    const R delta = ph.cip * R(P * P) / halfv(sqrtv(hL * hL + hh) + sqrtv(hU * hU + hh));
    face_interior_point<P, NF, MODE, R>(ph, ua, w, delta, tr, put);
    return;
  }
  const int side = F.hasL ? 0 : 1;
  const int bface = prm.side_off[2 * a + (side == 0 ? 1 : 0)] + F.j0 + pick3(prm.ne, b0) * F.j1;
  const R hs = side == 0 ? hL : hU;
  face_boundary_point<P, NF, MODE, R>(prm, prm.btag[bface], bface, side, ua, w,
                                      ph.cip * R(P * P) / sqrtv(hs * hs + hh), xp, bidx, pt, tr, put);
}

// The stages from both elements' nodal values to the traces at the points of
// the warp's nw faces (from face g0): region A [face][side][NTR][Q][QP], values
// of the NA arrays, then physical normal derivatives along +axis of the first NG.
// B: scratch. Ends with a barrier.
template <int P, int NF, int MODE, class R>
__device__ __forceinline__ void face_traces(const OpParams& prm, const io_t<R>* __restrict__ u,
                                            const io_t<R>* __restrict__ v, long long boff,
                                            long long g0, int nw, const FaceAt& F0, int lane, R* A,
                                            R* B) {
  using S = TileF<P, NF, MODE>;
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, NX = S::NX, FN = S::FN, NN = N * N * N;
  constexpr int NA = SL::NA, NG = SL::NG, NTR = S::NTR, FW = S::NF_;
  const long long EN = (long long)prm.E * NN;
  // layer values, and physical normal derivatives along +axis, of both elements
  // (node (k along a, (j1, j2) in the face) at base(j1, j2) + k * fs); a side
  // that does not exist is skipped, and its traces are never used
#pragma unroll 1
  for (int w = lane; w < nw * 2 * FN; w += 32) {
    const int fs_ = w / FN, j = w - fs_ * FN;
    const int side = fs_ & 1;
    const FaceAt F = FW == 1 ? F0 : face_at(prm, g0 + (fs_ >> 1));
    if (side == 0 ? !F.hasL : !F.hasU) continue;
    const int j1 = j % N, j2 = j / N;
    const int fs = F.a == 0 ? 1 : (F.a == 1 ? N : FN);
    const int nb = F.a == 0 ? N * j : (F.a == 1 ? j1 + FN * j2 : j);
    const int lay = side == 0 ? P : 0;
    const R sc = inv_scale<R>(prm, F.a, side == 0 ? F.ia - 1 : F.ia);
    const long long eo = boff + (long long)(side == 0 ? F.eL : F.eU) * NN + nb;
    R* o = A + fs_ * (NTR * N * NX) + j1 + NX * j2;
    io_t<R> x[NG][N], y[NA - NG + 1];
#pragma unroll
    for (int s = 0; s < NA; ++s) {
      const io_t<R>* src = (SL::vec(s) ? v : u) + eo + SL::field(s) * EN;
      if (s < NG) {
#pragma unroll
        for (int k = 0; k < N; ++k) x[s][k] = src[k * fs];
      } else {
        y[s - NG] = src[lay * fs];
      }
    }
    R dl[N];   // the side's end derivatives (run-time side: no divergence)
#pragma unroll
    for (int k = 0; k < N; ++k) dl[k] = ctab<P, R>(TO::dL + (1 - side) * N + k);
#pragma unroll
    for (int s = 0; s < NA; ++s) {
      if (s < NG) {
        Dot<R> d(dl[0], R(x[s][0]));
#pragma unroll
        for (int k = 1; k < N; ++k) d.fma(dl[k], R(x[s][k]));
        o[s * (N * NX)] = R(side == 0 ? x[s][P] : x[s][0]);
        o[(NA + s) * (N * NX)] = sc * d.get();
      } else {
        o[s * (N * NX)] = R(y[s - NG]);
      }
    }
  }
  group_sync<face_lock<R>()>();
#pragma unroll 1
  for (int w = lane; w < nw * 2 * NTR * N; w += 32)
    line<P, TO::B, false, N, Q, R>(A + w * NX, 1, B + w * QP, 1);
  group_sync<face_lock<R>()>();
  // lane (sub, k1): line k1 of every K-th array
  constexpr int K = 32 / Q;
  const int sub = lane / Q, k1 = lane - sub * Q;
  if (sub < K) {
#pragma unroll 1
    for (int g = sub; g < nw * 2 * NTR; g += K)
      line<P, TO::B, false, N, Q, R>(B + g * (N * QP) + k1, QP, A + g * (Q * QP) + k1, QP);
  }
  group_sync<face_lock<R>()>();
}

template <int P, int NF, int MODE, class R>
__global__ void __launch_bounds__(kTileThreads, FaceBlocks<R>::value)
tileface3d_kernel(const OpParams prm, const io_t<R>* __restrict__ u, const io_t<R>* __restrict__ v) {
  using S = TileF<P, NF, MODE>;
  using SL = Slots<P, NF, MODE>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, FN = S::FN, FQ = S::FQ;
  constexpr int NTR = S::NTR, NSL = SL::NSL, FW = S::NF_;
  extern __shared__ __align__(16) unsigned char tile_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  R* A = reinterpret_cast<R*>(tile_raw) + warp * S::total;
  R* B = A + S::kA;
  asm volatile("griddepcontrol.launch_dependents;");   // see wait_for_faces
  const long long nf = prm.foff[3];
  const long long g0 = ((long long)blockIdx.x * (blockDim.x >> 5) + warp) * FW;
  if (!face_lock<R>() && g0 >= nf) return;
  const int nw = g0 >= nf ? 0 : (int)(nf - g0 < FW ? nf - g0 : FW);   // faces of this warp
  const int bidx = blockIdx.y;
  const long long boff = (long long)bidx * prm.batch_stride;

  const FaceAt F0 = face_at(prm, g0);
  face_traces<P, NF, MODE, R>(prm, u, v, boff, g0, nw, F0, lane, A, B);
#pragma unroll 1
  for (int w = lane; w < nw * FQ; w += 32) {
    const int fi = w / FQ, pt = w - fi * FQ;
    const int o = (pt / Q) * QP + pt % Q;
    const R* t0 = A + fi * 2 * NTR * (Q * QP) + o;
    R* c0 = B + fi * NSL * (Q * QP) + o;
    const FaceAt F = FW == 1 ? F0 : face_at(prm, g0 + fi);
    FaceGeo<R> G;
    G.in_plane(prm, F.a, F.j0, F.j1);
    G.along(prm, F.a, F.ia, F.hasL, F.hasU);
    face_point<P, NF, MODE, R>(
        prm, F, G, bidx, pt, [&](int side, int t) -> R { return t0[(side * NTR + t) * (Q * QP)]; },
        [&](int slot, R val) { c0[slot * (Q * QP)] = val; });
  }
  group_sync<face_lock<R>()>();
  // lane (sub, k1): line k1 of every K-th array
  constexpr int K = 32 / Q;
  const int sub = lane / Q, k1 = lane - sub * Q;
  if (sub < K) {
#pragma unroll 1
    for (int g = sub; g < nw * NSL; g += K)
      line<P, TO::B, true, Q, N, R>(B + g * (Q * QP) + k1, QP, A + g * (N * QP) + k1, QP);
  }
  group_sync<face_lock<R>()>();
  R* fb = reinterpret_cast<R*>(prm.fbuf) + (long long)bidx * prm.fbuf_stride + g0 * (NSL * FN);
#pragma unroll 1
  for (int w = lane; w < nw * NSL * N; w += 32)
    line<P, TO::B, true, Q, N, R>(A + w * QP, 1, fb + w * N, 1);
}

}  // namespace enp
