// Element-diagonal blocks of J(u) on hexahedra (the "element-wise Jacobi" blocks
// of Sec. 4.2: volume terms and the element's own side of every face term, all
// fields coupled), assembled as matrices by sum factorisation.
//
// Entry (test phi_i, trial phi_j) of the block of fields (f, g) is a sum over the
// points of a coefficient times a product of 1D factors in i and j. By Eq. NPDG
// and Eq. chargeDG the volume needs few coefficient fields whatever the columns:
//   (0,0): sum_k kappa_k M_k       (k,0): mig_k M_k
//   (0,k): a_k K + kappa_k G       (k,k): D_k K + mig_k G - Gu
//   (k,l), k != l: zero,
// M_k = int c_k grad phi_i . grad phi_j, K = int grad . grad (closed form),
// G = int phi_j grad Phi . grad phi_i, Gu the same with the velocity. Each is
// contracted in z, then y, then x over pairs (i_a, j_a). The face terms are mass
// matrices on the face points (the fields listed at FaceFld), contracted over the
// higher in-face axis first, and enter where i or j lies on the face's layer (a
// value) or anywhere (a normal derivative); those of the y and z faces join the
// volume's x contraction. About 9 times fewer multiply-adds than one J v pass per
// column, and no barrier per column: on 64 x 32 x 16 elements, p = 3, three fields
// (192 columns, FP32) 48 ms with the columns of an element formed one after the
// other, 1.8 ms so.
//
// One thread block per element; in the last stage a thread owns one (i_y, j_y,
// i_z, j_z) and forms the n x n entries over (i_x, j_x) of every field pair, with
// the products of the 1D tables in constant memory at compile-time indices.
// Bound by instruction issue, then by the store of the blocks. At p = 4 the entries' stage
// does not fit its registers (spilled stores a thread: FP32 640 to 950 bytes, FP64 380 to 730).
#pragma once
#include "enp_launch.cuh"
#include "enp_tile3d.cuh"

namespace enp {

// Products of the 1D tables of degree p, [q][i][j]: BB, DD (both derivatives), DB
// (derivative of the test function i), then the 1D mass and stiffness [i][j].
constexpr int kPairSz = 512;
template <int P> struct PairOff {
  static constexpr int N = P + 1, Q = P + 2, L = Q * N * N;
  static constexpr int BB = 0, DD = L, DB = 2 * L, M = 3 * L, K = M + N * N;
  static_assert(K + N * N <= kPairSz, "pair table too small");
};
template <class R> struct PairTable;   // one type per translation unit (ENP_ASSEMBLE_TYPE)
#define ENP_ASSEMBLE_TYPE(R, NAME)                                                          \
  namespace enp {                                                                           \
  static __constant__ R NAME[kMaxP + 1][kPairSz];                                           \
  template <> struct PairTable<R> {                                                         \
    static __device__ __forceinline__ R at(int p, int i) { return NAME[p][i]; }             \
    static cudaError_t set(int p, const R* t) {                                             \
      return cudaMemcpyToSymbol(NAME, t, sizeof(NAME[0]), sizeof(NAME[0]) * p);             \
    }                                                                                       \
  };                                                                                        \
  }

template <class R>
static cudaError_t upload_pair_table(int p, const Tables& t) {
  const int n = p + 1, q = p + 2, L = q * n * n;
  double v[kPairSz] = {0};
  for (int a = 0; a < q; ++a) {
    double bd[kMaxN];
    for (int i = 0; i < n; ++i) {
      bd[i] = 0.0;
      for (int b = 0; b < q; ++b) bd[i] += t.Dq[a * q + b] * t.B[b * n + i];
    }
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        const double bi = t.B[a * n + i], bj = t.B[a * n + j];
        const int o = (a * n + i) * n + j;
        v[o] = bi * bj;
        v[L + o] = bd[i] * bd[j];
        v[2 * L + o] = bd[i] * bj;
        v[3 * L + i * n + j] += t.wq[a] * bi * bj;
        v[3 * L + n * n + i * n + j] += t.wq[a] * bd[i] * bd[j];
      }
  }
  R s[kPairSz];
  for (int i = 0; i < kPairSz; ++i) s[i] = (R)v[i];
  return PairTable<R>::set(p, s);
}

// Coefficient fields of a face's own-side linearisation (<- c, p, d: with respect
// to the own value of the species, of the potential, the own normal derivative):
// per species k: S_k <- c_k, S_k <- d_0, S_k <- p, S_0 <- c_k, T_0 <- c_k; then
// S_0 <- p and S_0 <- d_0 (= T_0 <- p). S_k <- d_k = T_k <- c_k and S_0 <- d_k
// are constants.
template <int NF> struct FaceFld {
  static constexpr int NK = NF - 1, A = 0, C = NK, B = 2 * NK, E = 3 * NK, T = 4 * NK, P = 5 * NK,
                       K = 5 * NK + 1, count = 5 * NK + 2;
};

template <int P, int NF>
struct AsmS {
  static constexpr int N = P + 1, Q = P + 2, QP = Rows<P>::QP, NX = N % 2 ? N : N + 1;
  static constexpr int NN = N * N * N, FN = N * N, FQ = Q * Q, PR = N * N, AQ = Q * Q * QP;
  static constexpr int NK = NF - 1, nb = NF * NN;
  static constexpr int NT = P == 1 ? 32 : (P == 2 ? 96 : (P == 3 ? 256 : 320));
  static constexpr int NZ = 2 * NK + 6;              // z-contracted arrays [pair][line]
  static constexpr int FL = FaceFld<NF>::count;
  static constexpr int kZ = NZ * PR * FQ, kH = 6 * FL * PR * Q;
  // scratch: the interpolation of u to the points [NF values, 3 gradients of Phi,
  // 3 advection fields], and of both sides' traces to the face points
  static constexpr int NTR = NF + 1;                 // values, derivative of Phi
  static constexpr int kT1 = NF * N * N * QP, kT2 = NF * N * Q * QP, kPt = (NF + 6) * AQ;
  static constexpr int kFL = 12 * NTR * N * NX, kF1 = 12 * NTR * N * QP, kTR = 12 * NTR * Q * QP;
  static constexpr int mx(int a, int b) { return a > b ? a : b; }
  // volume: T1 then points at 0, T2 behind; faces: behind the points
  static constexpr int oT2 = mx(kT1, kPt), oFA = oT2, oFB = oFA + mx(kFL, mx(kTR, kT2));
  static constexpr int kScratch = oFB + mx(kF1, 6 * FL * FQ);
  static constexpr int total = kScratch + kZ + kH;
};

template <int P, int NF, class R>
__global__ void __launch_bounds__(AsmS<P, NF>::NT)
assemble3d_kernel(const OpParams prm, const io_t<R>* __restrict__ u, io_t<R>* __restrict__ out,
                  int vec_ok) {
  using S = AsmS<P, NF>;
  using TO = TabOff<P>;
  using PO = PairOff<P>;
  using FF = FaceFld<NF>;
  using PT_ = PairTable<R>;
  constexpr int N = S::N, Q = S::Q, QP = S::QP, NX = S::NX, NN = S::NN, FN = S::FN, FQ = S::FQ;
  constexpr int PR = S::PR, AQ = S::AQ, NK = S::NK, NT = S::NT, FL = S::FL, NTR = S::NTR, nb = S::nb;
  const PhysT<R>& ph = phys<R>(prm);
  extern __shared__ __align__(16) unsigned char asm_raw[];
  R* W = reinterpret_cast<R*>(asm_raw);
  R* PT = W;                       // [NF + 6][AQ]
  R* T2 = W + S::oT2;
  R* FA = W + S::oFA;
  R* FB = W + S::oFB;
  R* Z = W + S::kScratch;          // [NZ][PR][FQ]
  R* H = Z + S::kZ;                // [6][FL][PR][Q]
  const int tid = threadIdx.x;
  const int e = blockIdx.x;
  const long long EN = (long long)prm.E * NN;
  const ElemGeo<P, R> G(prm, e);
  const int st[3] = {1, prm.ne[0], prm.ne[0] * prm.ne[1]};

  // ------------------------------------------------ the state at the points
  for (int w = tid; w < NF * FN; w += NT) {
    const int f = w / FN, r = w - f * FN;
    const io_t<R>* src = u + f * EN + (long long)e * NN + r * N;
    R x[N];
#pragma unroll
    for (int k = 0; k < N; ++k) x[k] = R(src[k]);
    line_rows<P, TO::B, false, N, Q, R>(x, [&](int q, R v) { PT[w * QP + q] = v; });
  }
  __syncthreads();
  for (int w = tid; w < NF * N * Q; w += NT) {
    const int g = w / Q, qx = w - g * Q;
    line<P, TO::B, false, N, Q, R>(PT + g * (N * QP) + qx, QP, T2 + g * (Q * QP) + qx, QP);
  }
  __syncthreads();
  for (int w = tid; w < NF * FQ; w += NT) {
    const int f = w / FQ, r = w - f * FQ, o = (r / Q) * QP + r % Q;
    line<P, TO::B, false, N, Q, R>(T2 + f * (N * Q * QP) + o, Q * QP, PT + f * AQ + o, Q * QP);
  }
  for (int r = tid; r < FQ; r += NT) {
    const int o = (r / Q) * QP + r % Q;
    line<P, TO::BD, false, N, Q, R>(T2 + o, Q * QP, PT + (NF + 2) * AQ + o, Q * QP);
  }
  __syncthreads();
  for (int w = tid; w < 2 * FQ; w += NT) {
    const int d = w >= FQ, r = w - d * FQ;
    const int o = d ? (r / Q) * (Q * QP) + r % Q : r * QP, is = d ? QP : 1;
    line<P, TO::Dq, false, Q, Q, R>(PT + o, is, PT + (NF + d) * AQ + o, is);
  }
  // layer values and physical normal derivatives of Phi along +axis, both sides
  // (0 own, 1 neighbour) of the six faces (T2 is dead: the barrier above)
  for (int w = tid; w < 12 * FN; w += NT) {
    const int sd = w / FN, j = w - sd * FN, s = sd >> 1, nbr = sd & 1;
    const int a = s >> 1, hi = s & 1;
    const int ia = pick3(G.idx, a);
    const bool bnd = hi ? ia == pick3(prm.ne, a) - 1 : ia == 0;
    if (nbr && bnd) continue;
    const int step = nbr ? (hi ? 1 : -1) : 0;
    const int low = hi != nbr;      // this element touches the face with its upper end
    const int j1 = j % N, j2 = j / N;
    const int fs = a == 0 ? 1 : (a == 1 ? N : FN);
    const int n0 = a == 0 ? N * j : (a == 1 ? j1 + FN * j2 : j);
    const io_t<R>* src = u + (long long)(e + step * pick3(st, a)) * NN + n0;
    R* o = FA + sd * (NTR * N * NX) + j1 + NX * j2;
    Dot<R> d(ctab<P, R>(TO::dL + low * N), R(src[0]));
#pragma unroll
    for (int k = 1; k < N; ++k) d.fma(ctab<P, R>(TO::dL + low * N + k), R(src[k * fs]));
#pragma unroll
    for (int f = 0; f < NF; ++f) o[f * (N * NX)] = R(src[f * EN + (low ? P : 0) * fs]);
    o[NF * (N * NX)] = inv_scale<R>(prm, a, ia + step) * d.get();
  }
  __syncthreads();
  for (int w = tid; w < 12 * NTR * N; w += NT)
    line<P, TO::B, false, N, Q, R>(FA + w * NX, 1, FB + w * QP, 1);
  // the volume's coefficient fields, weighted
  for (int pt = tid; pt < Q * FQ; pt += NT) {
    const int kx = pt % Q, ky = (pt / Q) % Q, kz = pt / FQ;
    const int o = kx + QP * (ky + Q * kz);
    const R w = ctab<P, R>(TO::W + kx) * ctab<P, R>(TO::W + ky) * ctab<P, R>(TO::W + kz);
    const R xp[3] = {G.coord(0, kx), G.coord(1, ky), G.coord(2, kz)};
    R uv[3];
    velocity(ph, xp, uv);
#pragma unroll
    for (int k = 0; k < NK; ++k) PT[(k + 1) * AQ + o] = w * PT[(k + 1) * AQ + o];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const R s1 = w * G.area[a];
      PT[(NF + a) * AQ + o] = s1 * G.sc[a] * PT[(NF + a) * AQ + o];
      PT[(NF + 3 + a) * AQ + o] = s1 * uv[a];
    }
  }
  __syncthreads();
  for (int w = tid; w < 12 * NTR * Q; w += NT) {
    const int g = w / Q, k1 = w - g * Q;
    line<P, TO::B, false, N, Q, R>(FB + g * (N * QP) + k1, QP, FA + g * (Q * QP) + k1, QP);
  }
  // z contraction of the volume fields: c_k with BB and DD, the x and y components
  // of grad Phi and u with BB, the z components with DB
  for (int w = tid; w < (NK + 6) * FQ; w += NT) {
    const int src = w / FQ, r = w - src * FQ, o = (r / Q) * QP + r % Q;
    R x[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) x[k] = PT[(src < NK ? src + 1 : src - NK + NF) * AQ + o + k * Q * QP];
    auto put = [&](int tab, int arr) {
      R* z = Z + arr * (PR * FQ) + r;
#pragma unroll
      for (int p = 0; p < PR; ++p) {
        R v = PT_::at(P, tab + p) * x[0];
#pragma unroll
        for (int k = 1; k < Q; ++k) v = mad(PT_::at(P, tab + k * PR + p), x[k], v);
        z[p * FQ] = v;
      }
    };
    if (src < NK) {
      put(PO::BB, 2 * src);
      put(PO::DD, 2 * src + 1);
    } else if ((src - NK) % 3 < 2) {
      put(PO::BB, NK + src);
    } else {
      put(PO::DB, NK + src);
    }
  }
  __syncthreads();
  // face coefficients at the points (FB: [6][FL][FQ])
  for (int w = tid; w < 6 * FQ; w += NT) {
    const int s = w / FQ, pt = w - s * FQ, k1 = pt % Q, k2 = pt / Q;
    const int a = s >> 1, hi = s & 1, b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
    const int ia = pick3(G.idx, a);
    const bool bnd = hi ? ia == pick3(prm.ne, a) - 1 : ia == 0;
    const R nrm = hi ? R(1) : R(-1);
    const R h0 = pick3(G.h, b0), h1 = pick3(G.h, b1), ha = pick3(G.h, a);
    const R hh = h0 * h0 + h1 * h1;
    const R xb0 = pick3(G.lo, b0) + halfv((ctab<P, R>(TO::X + k1) + R(1)) * h0);
    const R xb1 = pick3(G.lo, b1) + halfv((ctab<P, R>(TO::X + k2) + R(1)) * h1);
    const R xa = vertex<R>(prm, a, ia + hi);
    R xp[3], uv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) xp[c] = c == a ? xa : (c == b0 ? xb0 : xb1);
    velocity(ph, xp, uv);
    const R un = pick3(uv, a) * nrm;
    const R wt = ctab<P, R>(TO::W + k1) * ctab<P, R>(TO::W + k2) * (R(0.25f) * h0 * h1);
    const R* tr = FA + 2 * s * NTR * (Q * QP) + k2 * QP + k1;
    auto own = [&](int t) -> R { return tr[t * (Q * QP)]; };
    auto nbr = [&](int t) -> R { return tr[(NTR + t) * (Q * QP)]; };
    R* c = FB + s * (FL * FQ) + pt;
    auto put = [&](int fld, R v) { c[fld * FQ] = wt * v; };
    const R dm = own(NF) * nrm;
    const int tag = bnd ? prm.btag[prm.side_off[s] + pick3(G.idx, b0) + pick3(prm.ne, b0) * pick3(G.idx, b1)]
                        : (int)kInterior;
    if (!bnd) {
      const R hn = elem_size<R>(prm, a, ia + (hi ? 1 : -1));
      const R delta = ph.cip * R(P * P) / halfv(sqrtv(ha * ha + hh) + sqrtv(hn * hn + hh));
      const R dp = nbr(NF) * nrm, jphi = own(0) - nbr(0);
      R km = R(0), kp = R(0);
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        const R cm = own(k + 1), cp = nbr(k + 1), jc = cm - cp;
        const R qm = un - ph.mig[k] * dm, qp = un - ph.mig[k] * dp, qa = halfv(qm + qp);
        const R sg = qa > R(0) ? jc : (qa < R(0) ? -jc : R(0));
        put(FF::A + k, ph.D[k] * delta + halfv(qm + absv(qa)));
        put(FF::C + k, -(halfv(ph.mig[k]) * (cm + halfv(sg))));
        put(FF::B + k, R(0));
        put(FF::E + k, halfv(ph.kcoef[k]) * (delta * jphi - dm));
        put(FF::T + k, -halfv(ph.acoef[k] + ph.kcoef[k] * jphi));
        km += ph.kcoef[k] * cm;
        kp += ph.kcoef[k] * cp;
      }
      put(FF::P, halfv(delta) * (km + kp));
      put(FF::K, -halfv(km));
    } else if (tag == kDirichlet) {
      const R delta = ph.cip * R(P * P) / sqrtv(ha * ha + hh);
      const int bface = prm.side_off[s] + pick3(G.idx, b0) + pick3(prm.ne, b0) * pick3(G.idx, b1);
      auto gv = [&](int f) -> R {
        return prm.dirv ? R(prm.dirv[((long long)f * prm.NBF + bface) * prm.Nfq + pt]) : R(0);
      };
      const R jphi = own(0) - gv(0);
      R km = R(0);
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        const R cm = own(k + 1), g = gv(k + 1), jc = cm - g, qn = un - ph.mig[k] * dm;
        const R sg = qn > R(0) ? jc : (qn < R(0) ? -jc : R(0));
        put(FF::A + k, ph.D[k] * delta + halfv(qn + absv(qn)));
        put(FF::C + k, -(ph.mig[k] * halfv(cm + g + sg)));
        put(FF::B + k, R(0));
        put(FF::E + k, ph.kcoef[k] * (delta * jphi - dm));
        put(FF::T + k, -(ph.acoef[k] + ph.kcoef[k] * jphi));
        km += ph.kcoef[k] * cm;
      }
      put(FF::P, delta * km);
      put(FF::K, -km);
    } else {
#pragma unroll
      for (int q = 0; q < FL; ++q) c[q * FQ] = R(0);
      if (tag == kOutlet) {
#pragma unroll
        for (int k = 0; k < NK; ++k) {
          put(FF::A + k, un - ph.mig[k] * dm);
          put(FF::C + k, -(ph.mig[k] * own(k + 1)));
        }
      } else if (tag >= kElectrode0 && ph.bv_ox >= 0) {
        const R phiapp = prm.phiapp_batch ? R(prm.phiapp_batch[tag - kElectrode0])
                                          : ph.phiapp[tag - kElectrode0];
        R cs[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) cs[f] = own(f);
        const R co = oxidant_conc<NF, R, R>(ph, cs);
        const R eta = phiapp - cs[0];
        const R E1 = expv(ph.e1 * eta), E2 = expv((-ph.e2) * eta);
        R r = ph.inv_cref * co, drdc = ph.inv_cref;
        if (ph.gam != R(1)) {
          const R rb = r;
          r = powv(rb, ph.gam);
          drdc = ph.gam * powv(rb, ph.gam1) * ph.inv_cref;
        }
        const R J0 = exchange_current(ph, xp);
        const R dJp = -(J0 * (ph.e1 * E1 + r * (ph.e2 * E2))), dJc = -(J0 * E2 * drdc);
        put(FF::P, ph.ox_charge_scale * dJp);
#pragma unroll
        for (int k = 0; k < NK; ++k) {
          const bool ox = k == ph.bv_ox;
          if (ox) {
            put(FF::A + k, ph.ox_species_scale * dJc);
            put(FF::B + k, ph.ox_species_scale * dJp);
          }
          if (ox || ph.bv_ox >= NK)
            put(FF::E + k, ph.ox_charge_scale * dJc * (ox ? R(1) : ph.zratio[k]));
        }
      }
    }
  }
  __syncthreads();
  // contraction of the face fields over the higher in-face axis, lines along the
  // lower: H[s][field][pair][line]
  for (int w = tid; w < 6 * FL * Q; w += NT) {
    const int g = w / Q, l = w - g * Q;
    R x[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) x[k] = FB[g * FQ + k * Q + l];
    R* z = H + g * (PR * Q) + l;
#pragma unroll
    for (int p = 0; p < PR; ++p) {
      R v = PT_::at(P, PO::BB + p) * x[0];
#pragma unroll
      for (int k = 1; k < Q; ++k) v = mad(PT_::at(P, PO::BB + k * PR + p), x[k], v);
      z[p * Q] = v;
    }
  }
  __syncthreads();

  // ------------------------------------------------ the entries
  // constant face coefficients: interior faces half, Dirichlet faces whole, none
  // on the others
  R half6[6];
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    const int a = s >> 1, hi = s & 1, b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
    const bool bnd = hi ? G.idx[a] == prm.ne[a] - 1 : G.idx[a] == 0;
    R c = R(0.5f);
    if (bnd)
      c = prm.btag[prm.side_off[s] + G.idx[b0] + prm.ne[b0] * G.idx[b1]] == kDirichlet ? R(1) : R(0);
    // times the area and the outward factor 2/h of the derivative
    half6[s] = -(c * G.area[a] * (hi ? G.sc[a] : -G.sc[a]));
  }
  const R e2[3] = {G.area[0] * G.sc[0], G.area[1] * G.sc[1], G.area[2] * G.sc[2]};
  io_t<R>* blk = out + (long long)e * nb * nb;
#pragma unroll 1
  for (int w = tid; w < PR * PR; w += NT) {
    // j_y fastest, then j_z, i_y, i_z: a warp's stores run along the columns
    const int jy = w % N, jz = (w / N) % N, iy = (w / (N * N)) % N, iz = w / (N * N * N);
    const int py = iy * N + jy, pz = iz * N + jz;
    R bby[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) bby[q] = PT_::at(P, PO::BB + q * PR + py);
    const R my = PT_::at(P, PO::M + py), ky = PT_::at(P, PO::K + py);
    const R mz = PT_::at(P, PO::M + pz), kz = PT_::at(P, PO::K + pz);
    const R kx_c = e2[0] * my * mz, mx_c = e2[1] * ky * mz + e2[2] * my * kz;
    const long long row0 = N * (iy + N * iz), col0 = N * (jy + N * jz);
    // contraction in y of three z-contracted arrays: U[x] = sum_y t1(y) z1 + bb z2,
    // V[x] = sum_y bb z3
    auto y_sum = [&](int tab1, int a1, int a2, int a3, R s1, R s2, R s3, R* U, R* V) {
      R t1[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) t1[q] = s1 * PT_::at(P, tab1 + q * PR + py);
      const R *z1 = Z + (a1 * PR + pz) * FQ, *z2 = Z + (a2 * PR + pz) * FQ, *z3 = Z + (a3 * PR + pz) * FQ;
#pragma unroll
      for (int x = 0; x < Q; ++x) {
        R us = R(0), vs = R(0), ub = R(0);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          us = mad(t1[q], z1[q * Q + x], us);
          ub = mad(bby[q], z2[q * Q + x], ub);
          vs = mad(bby[q], z3[q * Q + x], vs);
        }
        U[x] = mad(s2, ub, us);
        V[x] = s3 * vs;
      }
    };
    // one field pair: x contraction of U with BB and V with DD or DB, the closed
    // form of K times kc, and the face terms: value-value field ll, value-
    // derivative ld, derivative-value dl (-1: none), constant cd in the place of
    // ld and (if both) of dl
    auto emit = [&](int f, int g, R* U, const R* V, int vtab, R kc, int ll, int ld, int dl, R cd,
                    bool both) {
#pragma unroll
      for (int s = 2; s < 6; ++s) {      // y and z faces: into U
        const int a = s >> 1, hi = s & 1, lay = hi ? P : 0;
        const int i = a == 1 ? iy : iz, j = a == 1 ? jy : jz, po = a == 1 ? pz : py;
        const bool il = i == lay, jl = j == lay;
        if (!il && !jl) continue;
        const R sca = hi ? G.sc[a] : -G.sc[a];
        const R di = ctab<P, R>(TO::dL + hi * N + i), dj = ctab<P, R>(TO::dL + hi * N + j);
        const R* h = H + s * (FL * PR * Q) + po * Q;
        const R cll = il && jl ? R(1) : R(0), cld = il ? sca * dj : R(0), cdl = jl ? sca * di : R(0);
        const R cc = half6[s] * cd * (a == 1 ? mz : my) *
                     ((il ? dj : R(0)) + (both && jl ? di : R(0)));
#pragma unroll
        for (int x = 0; x < Q; ++x) {
          R t = cc * ctab<P, R>(TO::W + x);
          if (ll >= 0) t = mad(cll, h[ll * (PR * Q) + x], t);
          if (ld >= 0) t = mad(cld, h[ld * (PR * Q) + x], t);
          if (dl >= 0) t = mad(cdl, h[dl * (PR * Q) + x], t);
          U[x] += t;
        }
      }
      R fl[2][3];                        // x faces: ll, ld, dl at this (i_y, j_y, i_z, j_z)
#pragma unroll
      for (int hi = 0; hi < 2; ++hi) {
        const R* h = H + hi * (FL * PR * Q) + pz * Q;
        const R sca = hi ? G.sc[0] : -G.sc[0];
        auto sum = [&](int fld) {
          R v = bby[0] * h[fld * (PR * Q)];
#pragma unroll
          for (int q = 1; q < Q; ++q) v = mad(bby[q], h[fld * (PR * Q) + q], v);
          return v;
        };
        const R cc = half6[hi] * cd * my * mz;
        fl[hi][0] = ll >= 0 ? sum(ll) : R(0);
        fl[hi][1] = ld >= 0 ? sca * sum(ld) : cc;
        fl[hi][2] = dl >= 0 ? (dl == ld ? fl[hi][1] : sca * sum(dl)) : (both ? cc : R(0));
      }
#pragma unroll
      for (int ix = 0; ix < N; ++ix) {
        io_t<R> o[N];
#pragma unroll
        for (int jx = 0; jx < N; ++jx) {
          const int px = ix * N + jx;
          R v = kc * mad(PT_::at(P, PO::K + px), kx_c, PT_::at(P, PO::M + px) * mx_c);
#pragma unroll
          for (int x = 0; x < Q; ++x) {
            v = mad(PT_::at(P, PO::BB + x * PR + px), U[x], v);
            v = mad(PT_::at(P, vtab + x * PR + px), V[x], v);
          }
#pragma unroll
          for (int hi = 0; hi < 2; ++hi) {
            const int lay = hi ? P : 0;
            if (ix == lay && jx == lay) v += fl[hi][0];
            if (ix == lay) v = mad(ctab<P, R>(TO::dL + hi * N + jx), fl[hi][1], v);
            if (jx == lay) v = mad(ctab<P, R>(TO::dL + hi * N + ix), fl[hi][2], v);
          }
          o[jx] = to_io(v);
        }
        io_t<R>* d = blk + (f * NN + row0 + ix) * nb + g * NN + col0;
        if constexpr (std::is_same<R, float>::value && N == 4) {
          if (vec_ok) *reinterpret_cast<float4*>(d) = make_float4(o[0], o[1], o[2], o[3]);
          else {
#pragma unroll
            for (int jx = 0; jx < N; ++jx) d[jx] = o[jx];
          }
        } else {
#pragma unroll
          for (int jx = 0; jx < N; ++jx) d[jx] = o[jx];
        }
      }
    };
    R U00[Q], V00[Q];
#pragma unroll
    for (int k = 0; k < NK; ++k) {       // M_k: (k,0), and into (0,0)
      R U[Q], V[Q];
      y_sum(PO::DD, 2 * k, 2 * k + 1, 2 * k, e2[1], e2[2], e2[0], U, V);
#pragma unroll
      for (int x = 0; x < Q; ++x) {
        U00[x] = k ? mad(ph.kcoef[k], U[x], U00[x]) : ph.kcoef[k] * U[x];
        V00[x] = k ? mad(ph.kcoef[k], V[x], V00[x]) : ph.kcoef[k] * V[x];
        U[x] = ph.mig[k] * U[x];
        V[x] = ph.mig[k] * V[x];
      }
      emit(k + 1, 0, U, V, PO::DD, R(0), FF::B + k, FF::C + k, -1, R(0), false);
    }
    emit(0, 0, U00, V00, PO::DD, R(0), FF::P, FF::K, FF::K, R(0), false);
    R UG[Q], VG[Q], Uu[Q], Vu[Q];
    y_sum(PO::DB, 2 * NK + 1, 2 * NK + 2, 2 * NK, R(1), R(1), R(1), UG, VG);
    y_sum(PO::DB, 2 * NK + 4, 2 * NK + 5, 2 * NK + 3, R(1), R(1), R(1), Uu, Vu);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      R U[Q], V[Q];
#pragma unroll
      for (int x = 0; x < Q; ++x) { U[x] = ph.kcoef[k] * UG[x]; V[x] = ph.kcoef[k] * VG[x]; }
      emit(0, k + 1, U, V, PO::DB, ph.acoef[k], FF::E + k, -1, FF::T + k, ph.acoef[k], false);
#pragma unroll
      for (int x = 0; x < Q; ++x) {
        U[x] = mad(ph.mig[k], UG[x], -Uu[x]);
        V[x] = mad(ph.mig[k], VG[x], -Vu[x]);
      }
      emit(k + 1, k + 1, U, V, PO::DB, ph.D[k], FF::A + k, -1, -1, ph.D[k], true);
      // the other species' columns
#pragma unroll
      for (int l = 0; l < NK; ++l)
        if (l != k)
#pragma unroll
          for (int ix = 0; ix < N; ++ix) {
            io_t<R>* d = blk + ((k + 1) * NN + row0 + ix) * nb + (l + 1) * NN + col0;
#pragma unroll
            for (int jx = 0; jx < N; ++jx) d[jx] = io_t<R>(0);
          }
    }
  }
}

template <int P, int NF, class R>
static cudaError_t launch_assemble_pn(const OpParams& prm, const io_t<R>* u, io_t<R>* out,
                                      cudaStream_t stream) {
  using S = AsmS<P, NF>;
  constexpr size_t smem = (size_t)S::total * sizeof(R);
  static_assert(smem <= 227 * 1024, "block assembly shared memory");
  auto k = assemble3d_kernel<P, NF, R>;
  static SmemAttr attr;
  cudaError_t e = raise_smem_limit(attr, k, smem);
  if (e != cudaSuccess) return e;
  const int vec = reinterpret_cast<uintptr_t>(out) % 16 == 0;   // rows of nb = 4 x values then too
  k<<<prm.E, S::NT, smem, stream>>>(prm, u, out, vec);
  return cudaGetLastError();
}

template <class R>
cudaError_t launch_assemble(const OpParams& prm, const io_t<R>* u, io_t<R>* blocks, cudaStream_t s) {
  if (prm.dim != 3) return cudaErrorInvalidConfiguration;
#define ENP_AS(PP)                                                              \
  case PP:                                                                      \
    if (prm.NF == 2) return launch_assemble_pn<PP, 2, R>(prm, u, blocks, s);    \
    if (prm.NF == 3) return launch_assemble_pn<PP, 3, R>(prm, u, blocks, s);    \
    return cudaErrorInvalidConfiguration;
  switch (prm.p) { ENP_AS(1) ENP_AS(2) ENP_AS(3) ENP_AS(4) }
#undef ENP_AS
  return cudaErrorInvalidConfiguration;
}
template <class R>
cudaError_t upload_tables_assemble(int p, const Tables& t) {
  cudaError_t e = upload_const_tables(p, t);
  return e == cudaSuccess ? upload_pair_table<R>(p, t) : e;
}

}  // namespace enp
