// Hexahedra, thread-per-pencil layout (sm_103a): the basis tables, the pencil
// contractions, and the parameter Jacobian dR/dtheta of Eq. NPDG / Eq. chargeDG (R, J v and J^T w:
// enp_tile3d.cuh; the element blocks: enp_assemble.cuh).
//  * every 1D contraction is done by one thread per pencil: it loads the
//    pencil into registers and forms all outputs with the basis table in
//    __constant__ memory at compile-time indices (the table entries become
//    FMA operands, no loads);
//  * each stage runs over all fields and vectors of the element at once, so a
//    stage costs one __syncthreads;
//  * the pointwise physics (volume and faces) is that of enp_operator.cuh.
#pragma once
#include <type_traits>

#include "enp_operator.cuh"

namespace enp {

constexpr int kTabSz = 128;  // per degree: B (Q*N), Dq (Q*Q), dL (2N), wq (Q), xq (Q), BD (Q*N)
// One struct per degree, so that a table set is one copy (there is one set per
// translation unit with hexahedral kernels).
struct ConstTab {
  double d[kTabSz];
  float2 df[kTabSz];   // (hi, lo) double-float pairs
  float f[kTabSz];
};
static __constant__ ConstTab c_tab[kMaxP + 1];

// Upload the tables of degree p to this translation unit's constant banks on
// the current device.
static inline cudaError_t upload_const_tables(int p, const Tables& t) {
  const int n = p + 1, q = p + 2;
  ConstTab c{};
  double* d = c.d;
  int o = 0;
  for (int i = 0; i < q * n; ++i) d[o++] = t.B[i];
  for (int i = 0; i < q * q; ++i) d[o++] = t.Dq[i];
  for (int i = 0; i < 2 * n; ++i) d[o++] = t.dL[i];
  for (int i = 0; i < q; ++i) d[o++] = t.wq[i];
  for (int i = 0; i < q; ++i) d[o++] = t.xq[i];
  // BD = Dq B: the derivative of each basis function at the Gauss points, as the
  // operator forms gradients (collocation derivative of the interpolant)
  for (int a = 0; a < q; ++a)
    for (int i = 0; i < n; ++i) {
      double sacc = 0.0;
      for (int b = 0; b < q; ++b) sacc += t.Dq[a * q + b] * t.B[b * n + i];
      d[o++] = sacc;
    }
  for (int i = 0; i < kTabSz; ++i) {
    c.f[i] = (float)d[i];
    const df x(d[i]);
    c.df[i] = make_float2(x.hi, x.lo);
  }
  return cudaMemcpyToSymbol(c_tab, &c, sizeof(c), sizeof(c) * p);
}

template <int P, class R>
__device__ __forceinline__ R ctab(int i) {
  if constexpr (std::is_same<R, double>::value) return c_tab[P].d[i];
  else if constexpr (std::is_same<R, df>::value) return df(c_tab[P].df[i].x, c_tab[P].df[i].y);
  else return c_tab[P].f[i];
}
template <int P> struct TabOff {
  static constexpr int N = P + 1, Q = P + 2;
  static constexpr int B = 0, Dq = Q * N, dL = Q * N + Q * Q, W = dL + 2 * N, X = W + Q;
  static constexpr int BD = X + Q;
  static_assert(BD + Q * N <= kTabSz, "table block too small");
};

// The outputs of one pencil: dst[r * os] = sum_k M[r][k] src[k * is] (+ dst[r * os]
// when ACC), r < ROWS, k < COLS, with M the B table (TAB 0, Q x N, or its
// transpose) or the Dq table (TAB 1, Q x Q); table entries at compile-time
// indices.
template <int P, int TAB, bool TRANS, bool ACC, int COLS, int ROWS, class R>
__device__ __forceinline__ void pencil_rows(const R* __restrict__ src, int is, R* __restrict__ dst,
                                            int os) {
  using T = TabOff<P>;
  R x[COLS];
#pragma unroll
  for (int k = 0; k < COLS; ++k) x[k] = src[k * is];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    R acc = ACC ? dst[r * os] : R(0);
#pragma unroll
    for (int k = 0; k < COLS; ++k) {
      int idx;
      if (TAB == 0) idx = T::B + (TRANS ? k * T::N + r : r * T::N + k);
      else idx = T::Dq + (TRANS ? k * T::Q + r : r * T::Q + k);
      acc = mad(ctab<P, R>(idx), x[k], acc);
    }
    dst[r * os] = acc;
  }
}

// One thread per pencil: out = M in along direction DIR of a 3D array with
// input extents (E0, E1, E2); M is the B table (TAB 0, ROWS x COLS = Q x N, or
// its transpose) or the Dq table (TAB 1, Q x Q). CNT arrays (stride IN_ST in
// the input, OUT_ST in the output) are processed, pencils shared over the
// NT threads of the element.
template <int P, int E0, int E1, int E2, int DIR, int TAB, bool TRANS, bool ACC, int CNT,
          int IN_ST, int OUT_ST, class R, int IX = E0, int OX = -1>
__device__ __forceinline__ void pencil(const R* __restrict__ in, R* __restrict__ out, int tid,
                                       int NT) {
  // IX: input row stride along dimension 0 (>= E0, padded arrays); OX: output row
  // stride (default: the output extent of dimension 0).
  using T = TabOff<P>;
  constexpr int COLS = DIR == 0 ? E0 : (DIR == 1 ? E1 : E2);
  constexpr int ROWS = TAB == 0 ? (TRANS ? T::N : T::Q) : T::Q;
  constexpr int O0 = DIR == 0 ? ROWS : E0, O1 = DIR == 1 ? ROWS : E1, O2 = DIR == 2 ? ROWS : E2;
  constexpr int OXX = OX < 0 ? O0 : OX;
  constexpr int IS = DIR == 0 ? 1 : (DIR == 1 ? IX : IX * E1);
  constexpr int OS = DIR == 0 ? 1 : (DIR == 1 ? OXX : OXX * O1);
  constexpr int PA = DIR == 0 ? O1 : O0;          // pencil index ranges over the other dims
  constexpr int PB = DIR == 2 ? O1 : O2;
  constexpr int NP = PA * PB;
  // work item w = c * NP + pp; (c, pp) advance by constant steps (no division
  // per item), and the pencil's position is recomputed only when pp moves
  int c = tid / NP, pp = tid % NP;
  const int dc = NT / NP, dp = NT % NP;
#pragma unroll 1
  for (int w = tid; w < NP * CNT; w += NT) {
    const int ia = pp % PA, ib = pp / PA;
    int ibase, obase;
    if (DIR == 0) { ibase = IX * (ia + E1 * ib); obase = OXX * (ia + O1 * ib); }
    else if (DIR == 1) { ibase = ia + IX * E1 * ib; obase = ia + OXX * O1 * ib; }
    else { ibase = ia + IX * ib; obase = ia + OXX * ib; }
    pencil_rows<P, TAB, TRANS, ACC, COLS, ROWS, R>(in + c * IN_ST + ibase, IS,
                                                    out + c * OUT_ST + obase, OS);
    c += dc;
    pp += dp;
    if (pp >= NP) { pp -= NP; ++c; }
  }
}

// The three reference derivatives at the Q^3 points in one pass: for each of
// CNT arrays (stride ST) of point values V, the arrays V + d Q^3 (d = 1, 2, 3)
// receive Dq V along x, y and z. Work items run over (direction, array,
// pencil), so the three directions share the passes of the block's threads.
template <int P, int CNT, int ST, class R>
__device__ __forceinline__ void pencil_grad3(R* V, int tid, int NT) {
  constexpr int Q = P + 2, NQ = Q * Q * Q, NP = Q * Q, PER = NP * CNT;
#pragma unroll 1
  for (int w = tid; w < 3 * PER; w += NT) {
    const int d = w / PER, r = w - d * PER;
    const int c = r / NP, pp = r - c * NP;
    const int ia = pp % Q, ib = pp / Q;
    // pencil along d: the other two coordinates are (ia, ib) in increasing order
    const int is = d == 0 ? 1 : (d == 1 ? Q : Q * Q);
    const int base = d == 0 ? Q * (ia + Q * ib) : (d == 1 ? ia + Q * Q * ib : ia + Q * ib);
    const R* src = V + c * ST + base;
    pencil_rows<P, 1, false, false, Q, Q, R>(src, is, V + c * ST + (1 + d) * NQ + base, is);
  }
}

// Nodal arrays are stored with the x row padded to an odd length, so that
// threads working on neighbouring x-pencils hit different shared-memory banks.
template <int N> struct Pad { static constexpr int X = (N % 2 == 0) ? N + 1 : N; };
template <int N>
__device__ __forceinline__ int padded_node(int i) {  // lexicographic node -> padded offset
  const int ix = i % N, iyz = i / N;
  return ix + Pad<N>::X * iyz;
}
template <int N>
__device__ __forceinline__ int face_node_pad(int a, int k, int j1, int j2) {
  constexpr int X = Pad<N>::X;
  if (a == 0) return k + X * (j1 + N * j2);
  if (a == 1) return j1 + X * (k + N * j2);
  return j1 + X * (j2 + N * k);
}

// The coefficients as forward tangents seeded on parameter j of
// theta = (D_1..D_m, c_in_1..c_in_{m-1}, phi_app_0..phi_app_3).
template <class R>
__device__ PhysT<Tan<R>> seed_phys(const PhysT<R>& p, int m, int j) {
  PhysT<Tan<R>> q;
  for (int k = 0; k < kMaxSpecies; ++k) {
    q.D[k] = Tan<R>(p.D[k]); q.cin[k] = Tan<R>(p.cin[k]); q.mig[k] = Tan<R>(p.mig[k]);
    q.acoef[k] = Tan<R>(p.acoef[k]); q.kcoef[k] = Tan<R>(p.kcoef[k]); q.z[k] = Tan<R>(p.z[k]);
    q.zratio[k] = Tan<R>(p.zratio[k]);
    q.dmig[k] = Tan<R>(p.dmig[k]); q.da[k] = Tan<R>(p.da[k]);
    q.dkc_own[k] = Tan<R>(p.dkc_own[k]); q.dkc_m[k] = Tan<R>(p.dkc_m[k]);
  }
  q.neg_inv_zm = Tan<R>(p.neg_inv_zm);
  for (int i = 0; i < 8; ++i) q.vp[i] = Tan<R>(p.vp[i]);
  q.vel_coef = Tan<R>(p.vel_coef);
  q.J0 = Tan<R>(p.J0); q.e1 = Tan<R>(p.e1); q.e2 = Tan<R>(p.e2);
  q.gam = Tan<R>(p.gam); q.gam1 = Tan<R>(p.gam1); q.inv_cref = Tan<R>(p.inv_cref);
  q.ox_species_scale = Tan<R>(p.ox_species_scale); q.ox_charge_scale = Tan<R>(p.ox_charge_scale);
  for (int i = 0; i < 4; ++i) q.phiapp[i] = Tan<R>(p.phiapp[i]);
  q.J0lo = Tan<R>(p.J0lo); q.J0half = Tan<R>(p.J0half); q.J0inv_half = Tan<R>(p.J0inv_half);
  q.cip = Tan<R>(p.cip);
  q.vel_kind = p.vel_kind; q.velA = p.velA; q.velN = p.velN; q.bv_ox = p.bv_ox; q.J0axis = p.J0axis;
  if (j < m) {                        // D_j: D, z_j mu_j F, the a_k and kappa coefficients
    if (j < m - 1) { q.D[j].d = R(1); q.mig[j].d = p.dmig[j]; }
    for (int k = 0; k < m - 1; ++k) {
      q.acoef[k].d = (k == j ? p.da[k] : R(0)) - (j == m - 1 ? p.da[k] : R(0));
      q.kcoef[k].d = (k == j ? p.dkc_own[k] : R(0)) + (j == m - 1 ? p.dkc_m[k] : R(0));
    }
  } else if (j < 2 * m - 1) {         // c_in of species j - m
    q.cin[j - m].d = R(1);
  } else {                            // phi_app of electrode j - (2m - 1)
    q.phiapp[j - (2 * m - 1)].d = R(1);
  }
  return q;
}

// Threads per element of param3d_kernel: Q x Q, one per pencil (the FP64 pipe bounds it).
template <int P>
__host__ __device__ constexpr int tpe3d() { return (P + 2) * (P + 2); }

template <int P, int NF, int NT>
struct Smem3 {
  static constexpr int N = P + 1, Q = P + 2;
  static constexpr int NX = Pad<N>::X;                   // padded x row of nodal arrays
  static constexpr int NN = N * N * N, NQ = Q * Q * Q, FN = N * N, FQ = Q * Q;
  static constexpr int NNP = NX * N * N;                 // padded nodal array
  static constexpr int FNP = NX * N;                     // padded face-node array
  static constexpr int NA = NF;                          // arrays carried through the volume
  static constexpr int kX = NA * NNP;                    // element data
  static constexpr int kOut = NF * NNP;                  // rows
  static constexpr int kT1 = NA * Q * N * N;             // after the x contraction
  static constexpr int kT2 = NA * Q * Q * N;             // after the y contraction
  static constexpr int kPts = NA * 4 * NQ;               // values + 3 gradients
  static constexpr int kFace = NA * NNP              // neighbour data
                               + 2 * NA * 2 * FNP         // layer values + normal derivatives
                               + 2 * NA * 2 * Q * N       // after the first face contraction
                               + 2 * NA * 2 * FQ          // traces at face points
                               + 2 * NF * FQ              // face coefficients
                               + 2 * NF * Q * N           // transposed, first stage
                               + 2 * NF * FNP;            // transposed, at face nodes
  // T1 is dead once T2 is formed, so it shares space with the point arrays
  static constexpr int kVol = kT2 + (kPts > kT1 ? kPts : kT1);
  static constexpr int kWork = kVol > kFace ? kVol : kFace;
  static constexpr int raw = kX + kOut + kWork;
  // stride between element regions: congruent to the element's thread count
  // modulo the bank count (32 words), so that a warp spanning two elements
  // keeps consecutive threads on consecutive banks
  static constexpr int kBankWords = 32;
  static constexpr int total = raw + ((NT - raw % kBankWords) % kBankWords + kBankWords) % kBankWords;
  static constexpr int kPrefetch = (NA * NN + NT - 1) / NT;  // neighbour values per thread
};

// Largest thread block of the hexahedral kernel; the elements per block (EB,
// chosen at launch by the autotuner) satisfy EB * tpe3d <= this.
constexpr int kMaxThreads3D = 256;
// dR/dtheta_j for every parameter j (grid.y: operating points x parameters).
template <int P, int NF, class R>
__global__ void __launch_bounds__(kMaxThreads3D)
param3d_kernel(const OpParams prm, const R* __restrict__ u, R* __restrict__ out) {
  using S = Smem3<P, NF, tpe3d<P>()>;
  using TO = TabOff<P>;
  constexpr int N = S::N, Q = S::Q, NN = S::NN, NQ = S::NQ, FN = S::FN, FQ = S::FQ;
  constexpr int NX = S::NX, NNP = S::NNP, FNP = S::FNP;
  constexpr int NA = S::NA, NT = tpe3d<P>(), PF = S::kPrefetch;
  const PhysT<R>& ph = phys<R>(prm);
  extern __shared__ __align__(16) unsigned char smem3_raw[];
  const int es = threadIdx.x / NT, tid = threadIdx.x % NT;
  R* base = reinterpret_cast<R*>(smem3_raw) + es * S::total;
  R* XA = base;                 // [NA][NNP] padded nodal arrays
  R* RO = XA + S::kX;           // [NF][NNP]
  R* WK = RO + S::kOut;
  const int EB = blockDim.x / NT;   // elements per block, chosen at launch
  const int e = blockIdx.x * EB + es;
  const bool valid = e < prm.E;
  const int ee = valid ? e : prm.E - 1;   // invalid slots shadow a valid element, write nothing
  const int bidx = (int)blockIdx.y / prm.n_theta;
  const int theta_j = (int)blockIdx.y % prm.n_theta;
  const long long boff = (long long)bidx * prm.batch_stride;
  const long long ooff = ((long long)theta_j * prm.batch + bidx) * prm.batch_stride;
  const long long EN = (long long)prm.E * NN;

  int idx[3];
  idx[0] = ee % prm.ne[0];
  idx[1] = (ee / prm.ne[0]) % prm.ne[1];
  idx[2] = ee / (prm.ne[0] * prm.ne[1]);
  R lo[3], h[3], sc[3];
  R diag2 = R(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = vertex<R>(prm, a, idx[a]);
    h[a] = vertex<R>(prm, a, idx[a] + 1) - lo[a];
    sc[a] = R(2) / h[a];
    diag2 += h[a] * h[a];
  }
  const R diag = sqrtv(diag2);
  const R detJ = R(0.125) * h[0] * h[1] * h[2];

  for (int t = tid; t < NF * NN; t += NT) {
    const int f = t / NN, i = t % NN;
    const long long gi = boff + f * EN + (long long)ee * NN + i;
    const int pi = f * NNP + padded_node<N>(i);
    XA[pi] = u[gi];
  }
  // neighbour data of a face, fetched into registers one face ahead so that the
  // global loads overlap the computation of the previous stage
  const int stride[3] = {1, prm.ne[0], prm.ne[0] * prm.ne[1]};
  R pf[PF];
  auto prefetch = [&](int s) {
    const int a = s >> 1, hi = s & 1;
    const bool bnd = hi ? (idx[a] == prm.ne[a] - 1) : (idx[a] == 0);
    if (bnd) return;
    const int en = ee + (hi ? stride[a] : -stride[a]);
#pragma unroll
    for (int k = 0; k < PF; ++k) {
      const int t = tid + k * NT;
      if (t < NA * NN) {
        const int f = t / NN, i = t % NN;
        pf[k] = u[boff + f * EN + (long long)en * NN + i];
      }
    }
  };
  prefetch(0);
  __syncthreads();

  // ---------------------------------------------------------------- volume
  R* T2 = WK;                   // [NA][N][Q][Q]
  R* PT = T2 + S::kT2;          // [NA][4][NQ]
  R* T1 = PT;                   // [NA][N][N][Q], dead before PT is written
  pencil<P, N, N, N, 0, 0, false, false, NA, NNP, Q * N * N, R, NX>(XA, T1, tid, NT);
  __syncthreads();
  pencil<P, Q, N, N, 1, 0, false, false, NA, Q * N * N, Q * Q * N>(T1, T2, tid, NT);
  __syncthreads();
  pencil<P, Q, Q, N, 2, 0, false, false, NA, Q * Q * N, 4 * NQ>(T2, PT, tid, NT);
  __syncthreads();
  pencil_grad3<P, NA, 4 * NQ>(PT, tid, NT);
  __syncthreads();

  {
    // points pt = tid, tid + NT, ...: with NT = Q^2 one thread runs down the z
    // line of its (kx, ky), and the x-y weight and coordinates are hoisted
    constexpr bool kLine = NT == Q * Q;
    const int kx0 = tid % Q, ky0 = (tid / Q) % Q;
    const R wxy0 = ctab<P, R>(TO::W + kx0) * ctab<P, R>(TO::W + ky0) * detJ;
    const R xp00 = lo[0] + R(0.5) * (ctab<P, R>(TO::X + kx0) + R(1)) * h[0];
    const R xp01 = lo[1] + R(0.5) * (ctab<P, R>(TO::X + ky0) + R(1)) * h[1];
#pragma unroll 1
    for (int pt = tid; pt < NQ; pt += NT) {
      const int kx = kLine ? kx0 : pt % Q, ky = kLine ? ky0 : (pt / Q) % Q, kz = pt / (Q * Q);
      const R wxy = kLine ? wxy0 : ctab<P, R>(TO::W + kx) * ctab<P, R>(TO::W + ky) * detJ;
      R xp[3];
      xp[0] = kLine ? xp00 : lo[0] + R(0.5) * (ctab<P, R>(TO::X + kx) + R(1)) * h[0];
      xp[1] = kLine ? xp01 : lo[1] + R(0.5) * (ctab<P, R>(TO::X + ky) + R(1)) * h[1];
      xp[2] = lo[2] + R(0.5) * (ctab<P, R>(TO::X + kz) + R(1)) * h[2];
      R uv[3];
      velocity(ph, xp, uv);
      const R w = wxy * ctab<P, R>(TO::W + kz);
      R c0[NF], g0[NF][3];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        const R* V = PT + f * 4 * NQ;
        c0[f] = V[pt];
#pragma unroll
        for (int a = 0; a < 3; ++a) g0[f][a] = V[(1 + a) * NQ + pt] * sc[a];
      }
      R oS[NF], oG[NF][3];
      {
        const PhysT<Tan<R>> pt = seed_phys<R>(ph, NF, theta_j);
        Tan<R> ct[NF], gt[NF][3], Sf[NF], Gf[NF][3];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          ct[f] = Tan<R>(c0[f]);
#pragma unroll
          for (int a = 0; a < 3; ++a) gt[f][a] = Tan<R>(g0[f][a]);
        }
        volume_flux<NF, 3, Tan<R>, R, Tan<R>>(pt, ct, gt, uv, Sf, Gf);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          oS[f] = Sf[f].d;
#pragma unroll
          for (int a = 0; a < 3; ++a) oG[f][a] = Gf[f][a].d;
        }
      }
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        R* V = PT + f * 4 * NQ;
        V[pt] = w * oS[f];
#pragma unroll
        for (int a = 0; a < 3; ++a) V[(1 + a) * NQ + pt] = w * sc[a] * oG[f][a];
      }
    }
  }
  __syncthreads();
  R* PO = PT;   // the NF output point arrays
  pencil<P, Q, Q, Q, 0, 1, true, true, NF, 4 * NQ, 4 * NQ>(PO + NQ, PO, tid, NT);
  __syncthreads();
  pencil<P, Q, Q, Q, 1, 1, true, true, NF, 4 * NQ, 4 * NQ>(PO + 2 * NQ, PO, tid, NT);
  __syncthreads();
  pencil<P, Q, Q, Q, 2, 1, true, true, NF, 4 * NQ, 4 * NQ>(PO + 3 * NQ, PO, tid, NT);
  __syncthreads();
  pencil<P, Q, Q, Q, 2, 0, true, false, NF, 4 * NQ, Q * Q * N>(PO, T2, tid, NT);
  __syncthreads();
  R* T1b = PT;  // the point arrays are dead once T2 holds the z-transposed values
  pencil<P, Q, Q, N, 1, 0, true, false, NF, Q * Q * N, Q * N * N>(T2, T1b, tid, NT);
  __syncthreads();
  pencil<P, Q, N, N, 0, 0, true, false, NF, Q * N * N, NNP, R, Q, NX>(T1b, RO, tid, NT);
  __syncthreads();

  // ---------------------------------------------------------------- faces
  R* XN = WK;                                  // [NA][NNP] neighbour data
  R* FL = XN + NA * NNP;                       // [2 sides][NA][2][FNP] layer values, derivatives
  R* F1 = FL + 2 * NA * 2 * FNP;               // [2][NA][2][Q][N]
  R* TR = F1 + 2 * NA * 2 * Q * N;             // [2][NA][2][FQ]
  R* FC = TR + 2 * NA * 2 * FQ;                // [2][NF][FQ]: S then T coefficients
  R* G1 = FC + 2 * NF * FQ;                    // [2][NF][N][Q]
  R* G2 = G1 + 2 * NF * Q * N;                 // [2][NF][FNP]
#pragma unroll 1
  for (int s = 0; s < 6; ++s) {
    const int a = s >> 1, hi = s & 1;
    const int b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
    const R nrm = hi ? R(1) : R(-1);
    const bool boundary = hi ? (idx[a] == prm.ne[a] - 1) : (idx[a] == 0);
    int tag = kInterior, bface = -1;
    R hn = h[a], diagn = diag;
    if (boundary) {
      const int loc = idx[b0] + prm.ne[b0] * idx[b1];
      bface = prm.side_off[s] + loc;
      tag = prm.btag[bface];
    } else {
      int in3[3] = {idx[0], idx[1], idx[2]};
      in3[a] += hi ? 1 : -1;
      R d2 = R(0);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const R hc = vertex<R>(prm, c, in3[c] + 1) - vertex<R>(prm, c, in3[c]);
        d2 += hc * hc;
        if (c == a) hn = hc;
      }
      diagn = sqrtv(d2);
#pragma unroll
      for (int k = 0; k < PF; ++k) {
        const int t = tid + k * NT;
        if (t < NA * NN) {
          const int arr = t / NN, i = t % NN;
          XN[arr * NNP + padded_node<N>(i)] = pf[k];
        }
      }
    }
    if (s < 5) prefetch(s + 1);
    const bool active = tag != kWall;
    __syncthreads();
    // layer values and reference normal derivatives at the face nodes
    const int lay = hi ? N - 1 : 0, layo = hi ? 0 : N - 1;
    const int nsides = boundary ? 1 : 2;
    for (int w = tid; w < nsides * NA * FN; w += NT) {
      const int side = w / (NA * FN), r = w % (NA * FN), arr = r / FN, j = r % FN;
      const int j1 = j % N, j2 = j / N;
      const R* X = (side == 0 ? XA : XN) + arr * NNP;
      const int L = side == 0 ? lay : layo;
      const int dsel = side == 0 ? hi : 1 - hi;
      R d = R(0);
#pragma unroll
      for (int k = 0; k < N; ++k)
        d = mad(ctab<P, R>(TO::dL + dsel * N + k), X[face_node_pad<N>(a, k, j1, j2)], d);
      R* o = FL + ((side * NA + arr) * 2) * FNP;
      const int jp = j1 + NX * j2;
      o[jp] = X[face_node_pad<N>(a, L, j1, j2)];
      o[FNP + jp] = d;
    }
    __syncthreads();
    // 2D interpolation to the face Gauss points: along b0, then b1. Both sides
    // are always processed so that every thread reaches every barrier; on a
    // boundary face the second side holds stale values that are never read.
    pencil<P, N, N, 1, 0, 0, false, false, 4 * NA, FNP, Q * N, R, NX>(FL, F1, tid, NT);
    __syncthreads();
    pencil<P, Q, N, 1, 1, 0, false, false, 4 * NA, Q * N, FQ>(F1, TR, tid, NT);
    __syncthreads();
    // pointwise face fluxes, one thread per face point
    {
      const R area = R(0.25) * h[b0] * h[b1];
      const R delta = ph.cip * R(P * P) / (boundary ? diag : R(0.5) * (diag + diagn));
      const R sca = sc[a] * nrm;
      const R scn = R(2) / hn * nrm;
      const R phiapp = (tag >= kElectrode0)
          ? (prm.phiapp_batch ? R(prm.phiapp_batch[bidx * 4 + (tag - kElectrode0)])
                              : ph.phiapp[tag - kElectrode0])
          : R(0);
#pragma unroll 1
      for (int pt = tid; pt < FQ; pt += NT) {
      const int k1 = pt % Q, k2 = pt / Q;
      R xp[3];
      xp[a] = hi ? lo[a] + h[a] : lo[a];
      xp[b0] = lo[b0] + R(0.5) * (ctab<P, R>(TO::X + k1) + R(1)) * h[b0];
      xp[b1] = lo[b1] + R(0.5) * (ctab<P, R>(TO::X + k2) + R(1)) * h[b1];
      R uv[3];
      velocity(ph, xp, uv);
      const R un = uv[a] * nrm;
      const R w = ctab<P, R>(TO::W + k1) * ctab<P, R>(TO::W + k2) * area;
      auto trv = [&](int side, int f, int comp) -> R {
        return TR[((side * NA + f) * 2 + comp) * FQ + pt];
      };
      R cm[NF], dm[NF], cp[NF], dp[NF], g[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        cm[f] = trv(0, f, 0);
        dm[f] = trv(0, f, 1) * sca;
        cp[f] = boundary ? R(0) : trv(1, f, 0);
        dp[f] = boundary ? R(0) : trv(1, f, 1) * scn;
        g[f] = (tag == kDirichlet && prm.dirv)
                   ? R(prm.dirv[((long long)f * prm.NBF + bface) * prm.Nfq + pt]) : R(0);
      }
      R oS[NF], oT[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) { oS[f] = R(0); oT[f] = R(0); }
      if (active) {
        {
          const PhysT<Tan<R>> pt = seed_phys<R>(ph, NF, theta_j);
          const Tan<R> phit(phiapp, (tag >= kElectrode0 && theta_j == 2 * NF - 1 + tag - kElectrode0)
                                        ? R(1) : R(0));
          Tan<R> tm[NF], tdm[NF], tp[NF], tdp[NF], Sf[NF], Tf[NF];
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            tm[f] = Tan<R>(cm[f]); tdm[f] = Tan<R>(dm[f]);
            tp[f] = Tan<R>(cp[f]); tdp[f] = Tan<R>(dp[f]);
          }
          if (boundary)
            face_boundary_flux<NF, Tan<R>, R, Tan<R>>(pt, tag, tm, tdm, g, un, delta, xp, phit, Sf, Tf);
          else
            face_interior_flux<NF, Tan<R>, R, Tan<R>>(pt, tm, tdm, tp, tdp, un, delta, Sf, Tf);
#pragma unroll
          for (int f = 0; f < NF; ++f) { oS[f] = Sf[f].d; oT[f] = Tf[f].d; }
        }
      }
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        FC[f * FQ + pt] = w * oS[f];
        FC[(NF + f) * FQ + pt] = w * sca * oT[f];
      }
      }
    }
    __syncthreads();
    // transposed 2D contraction back to the face nodes, then into the rows
    pencil<P, Q, Q, 1, 1, 0, true, false, 2 * NF, FQ, Q * N>(FC, G1, tid, NT);
    __syncthreads();
    pencil<P, Q, N, 1, 0, 0, true, false, 2 * NF, Q * N, FNP, R, Q, NX>(G1, G2, tid, NT);
    __syncthreads();
    for (int w = tid; w < NF * FN; w += NT) {
      const int f = w / FN, j = w % FN, j1 = j % N, j2 = j / N;
      R* Rf = RO + f * NNP;
      const int jp = j1 + NX * j2;
      const R sv = G2[f * FNP + jp], tv = G2[(NF + f) * FNP + jp];
      if (active) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
          R add = ctab<P, R>(TO::dL + hi * N + k) * tv;
          if (k == lay) add += sv;
          Rf[face_node_pad<N>(a, k, j1, j2)] += add;
        }
      }
    }
    __syncthreads();
  }

  if (valid) {
    for (int t = tid; t < NF * NN; t += NT) {
      const int f = t / NN, i = t % NN;
      out[ooff + f * EN + (long long)e * NN + i] = RO[f * NNP + padded_node<N>(i)];
    }
  }
}

}  // namespace enp
