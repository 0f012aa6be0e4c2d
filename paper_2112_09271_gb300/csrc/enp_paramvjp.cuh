// <w, dR/dtheta> on hexahedra without forming dR/dtheta (theta = the
// diffusivities, inlet concentrations and applied potentials; FP64).
//
// R is linear in the coefficients D_k, mig_k = z_k mu_k F, a_k and kappa_k that
// the diffusivities enter through (Eq. NE, Eq. charge2), so for each species k
// four sums over the volume and face points are enough, whatever m is:
//   A_k (a_k), B_k (D_k), C_k (mig_k), E_k (kappa_k),
// plus one per inlet concentration and one per electrode. A pass costs the
// interpolation of u and w to the points and a few products there: no seeded
// tangents per parameter, no transposed contraction, no [n_theta][n] array and
// no dot products over it (cube of 24^3 elements, p = 2, two fields, forward and
// backward of the residual in double-float: 6.4 ms with the former product, 0.98 now).
// Bound by the FP64 pipe. Warps run over elements (faces) by a fixed stride and
// keep their sums in registers; a fixed grid and order make results reproducible
// and independent of the batch.
#pragma once
#include "enp_launch.cuh"
#include "enp_reduce.cuh"
#include "enp_tile3d.cuh"

namespace enp {

constexpr int kPvjpBlocks = 608;   // at most: 4 per SM on 152 SMs
// Sums per operating point: A, B, C, E and c_in per unknown species, 4 electrodes.
template <int NF> struct PvjpAcc {
  static constexpr int NK = NF - 1, A = 0, B = NK, C = 2 * NK, E = 3 * NK, CIN = 4 * NK, PHI = 5 * NK;
  static constexpr int count = 5 * NK + 4;
  static_assert(2 * kPvjpBlocks * count <= kPvjpPartials, "workspace of the parameter adjoint");
};

// part[(b * count + i) * nparts + first + block] = the block's sum of acc[i].
template <int COUNT>
__device__ __forceinline__ void pvjp_block_sums(const double (&acc)[COUNT], double* __restrict__ part,
                                                int nparts, int slot) {
  __shared__ double red[kTileThreads / 32][COUNT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < COUNT; ++i) {
    const double s = warp_sum(acc[i]);
    if (lane == 0) red[warp][i] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < COUNT; i += blockDim.x) {
    double s = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) s += red[w][i];
    part[((long long)blockIdx.y * COUNT + i) * nparts + slot] = s;
  }
}

template <int P, int NF>
__global__ void __launch_bounds__(kTileThreads, 3)
pvjp_elem_kernel(const OpParams prm, const double* __restrict__ u, const double* __restrict__ w,
                 double* __restrict__ part, int nparts) {
  using R = double;
  using S = TileE<P, NF, kParam>;
  using TO = TabOff<P>;
  using AC = PvjpAcc<NF>;
  constexpr int Q = S::Q, QP = S::QP, AQ = S::AQ, NN = S::N * S::N * S::N, FQ = Q * Q;
  constexpr int NA = S::NA, T = tile_threads<P, R>();
  extern __shared__ __align__(16) unsigned char tile_raw[];
  const int grp = threadIdx.x / T, tid = threadIdx.x % T, ng = blockDim.x / T;
  R* A = reinterpret_cast<R*>(tile_raw) + grp * S::total;
  R* Bq = A + S::kA;
  const long long boff = (long long)blockIdx.y * prm.batch_stride, EN = (long long)prm.E * NN;
  double acc[AC::count] = {};
  const int step = gridDim.x * ng;
  // all groups of a block take the same number of turns (barriers); a turn
  // beyond the mesh adds nothing
  for (int first = blockIdx.x * ng; first < prm.E; first += step) {
    const bool valid = first + grp < prm.E;
    const int e = valid ? first + grp : prm.E - 1;
    const long long eo = boff + (long long)e * NN;
    tile_points<P, NF, kParam, R>(u + eo, w + eo, EN, A, Bq, tid);
    const ElemGeo<P, R> G(prm, e);
#pragma unroll 1
    for (int pt = tid; pt < Q * FQ && valid; pt += T) {
      const int kx = pt % Q, ky = (pt / Q) % Q, kz = pt / FQ;
      const int o = kx + QP * (ky + Q * kz);
      const R wt = ctab<P, R>(TO::W + kx) * ctab<P, R>(TO::W + ky) * ctab<P, R>(TO::W + kz);
      const R uv[3] = {0.0, 0.0, 0.0};
      R s2[3], adv[3];
      G.factors(wt, uv, s2, adv);
      auto grad = [&](int s, int a) -> R {
        return a < 2 ? Bq[(2 * s + a) * AQ + o] : A[(NA + s) * AQ + o];
      };
      R q0[NF] = {};                 // weighted grad Phi . grad w_f
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const R g0 = s2[a] * grad(0, a), W0 = grad(NF, a);
        q0[0] = fma(g0, W0, q0[0]);
#pragma unroll
        for (int k = 0; k < AC::NK; ++k) {
          const R gk = s2[a] * grad(k + 1, a), Wk = grad(NF + k + 1, a);
          q0[k + 1] = fma(g0, Wk, q0[k + 1]);
          acc[AC::A + k] = fma(gk, W0, acc[AC::A + k]);
          acc[AC::B + k] = fma(gk, Wk, acc[AC::B + k]);
        }
      }
#pragma unroll
      for (int k = 0; k < AC::NK; ++k) {
        const R c = A[(k + 1) * AQ + o];
        acc[AC::C + k] = fma(c, q0[k + 1], acc[AC::C + k]);
        acc[AC::E + k] = fma(c, q0[0], acc[AC::E + k]);
      }
    }
    group_sync<(T > 32)>();   // before the next element's nodes overwrite the points
  }
  pvjp_block_sums<AC::count>(acc, part, nparts, blockIdx.x);
}

template <int P, int NF>
__global__ void __launch_bounds__(kTileThreads, 4)
pvjp_face_kernel(const OpParams prm, const double* __restrict__ u, const double* __restrict__ w,
                 double* __restrict__ part, int nparts, int first_part) {
  using R = double;
  using S = TileF<P, NF, kParam>;
  using TO = TabOff<P>;
  using AC = PvjpAcc<NF>;
  constexpr int Q = S::Q, QP = S::QP, FQ = S::FQ, NTR = S::NTR, FW = S::NF_, NA = 2 * NF;
  extern __shared__ __align__(16) unsigned char tile_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
  R* Ar = reinterpret_cast<R*>(tile_raw) + warp * S::total;
  R* Br = Ar + S::kA;
  const PhysT<R>& ph = prm.pd;
  const int bidx = blockIdx.y;
  const long long boff = (long long)bidx * prm.batch_stride, nf = prm.foff[3];
  double acc[AC::count] = {};
  for (long long g0 = ((long long)blockIdx.x * nwarp + warp) * FW; g0 < nf;
       g0 += (long long)gridDim.x * nwarp * FW) {
    const int nw = (int)(nf - g0 < FW ? nf - g0 : FW);
    const FaceAt F0 = face_at(prm, g0);
    face_traces<P, NF, kParam, R>(prm, u, w, boff, g0, nw, F0, lane, Ar, Br);
#pragma unroll 1
    for (int it = lane; it < nw * FQ; it += 32) {
      const int fi = it / FQ, pt = it - fi * FQ;
      const R* t0 = Ar + fi * 2 * NTR * (Q * QP) + (pt / Q) * QP + pt % Q;
      // trace t of side s: u values, w values, u derivatives, w derivatives
      auto tr = [&](int s, int t) -> R { return t0[(s * NTR + t) * (Q * QP)]; };
      const FaceAt F = FW == 1 ? F0 : face_at(prm, g0 + fi);
      const int a = F.a, b0 = a == 0 ? 1 : 0, b1 = a == 2 ? 1 : 2;
      const int k1 = pt % Q, k2 = pt / Q;
      const R lo0 = vertex<R>(prm, b0, F.j0), lo1 = vertex<R>(prm, b1, F.j1);
      const R h0 = elem_size<R>(prm, b0, F.j0), h1 = elem_size<R>(prm, b1, F.j1);
      const R xa = vertex<R>(prm, a, F.ia);
      const R hL = F.hasL ? elem_size<R>(prm, a, F.ia - 1) : R(1);
      const R hU = F.hasU ? elem_size<R>(prm, a, F.ia) : R(1);
      const R hh = h0 * h0 + h1 * h1;
      R xp[3], uv[3];
      {
        const R xb0 = lo0 + halfv((ctab<P, R>(TO::X + k1) + R(1)) * h0);
        const R xb1 = lo1 + halfv((ctab<P, R>(TO::X + k2) + R(1)) * h1);
#pragma unroll
        for (int c = 0; c < 3; ++c) xp[c] = c == a ? xa : (c == b0 ? xb0 : xb1);
      }
      velocity(ph, xp, uv);
      const R ua = pick3(uv, a);
      const R wt = ctab<P, R>(TO::W + k1) * ctab<P, R>(TO::W + k2) * (R(0.25) * h0 * h1);
      if (F.hasL && F.hasU) {
        const R delta = ph.cip * R(P * P) / halfv(sqrtv(hL * hL + hh) + sqrtv(hU * hU + hh));
        const R jphi = tr(0, 0) - tr(1, 0), dm = tr(0, NA), dp = tr(1, NA), ds = dm + dp;
        const R hw = halfv(wt);
        const R jw0 = hw * (tr(0, NF) - tr(1, NF));
        const R vm0 = hw * tr(0, NA + NF), vp0 = hw * tr(1, NA + NF), vs = vm0 + vp0;
        const R dj = delta * jphi;
#pragma unroll
        for (int k = 0; k < AC::NK; ++k) {
          const R cm = tr(0, k + 1), cp = tr(1, k + 1), jc = cm - cp;
          const R dd = tr(0, NA + k + 1) + tr(1, NA + k + 1);
          const R jw = hw * (tr(0, NF + k + 1) - tr(1, NF + k + 1));
          const R vw = hw * (tr(0, NA + NF + k + 1) + tr(1, NA + NF + k + 1));
          const R qa = halfv((ua - ph.mig[k] * dm) + (ua - ph.mig[k] * dp));
          const R sg = qa > R(0) ? jc : (qa < R(0) ? -jc : R(0));
          acc[AC::A + k] -= fma(dd, jw0, jc * vs);
          acc[AC::B + k] += fma(fma(R(2) * delta, jc, -dd), jw, -jc * vw);
          acc[AC::C + k] -= fma(cm, dm, fma(cp, dp, halfv(sg) * ds)) * jw;
          acc[AC::E + k] += fma(fma(dj, cm + cp, -fma(cm, dm, cp * dp)), jw0,
                                -jphi * fma(cm, vm0, cp * vp0));
        }
      } else {
        const int side = F.hasL ? 0 : 1;
        const R nrm = side == 0 ? R(1) : R(-1);
        const int bface = prm.side_off[2 * a + (side == 0 ? 1 : 0)] + F.j0 + pick3(prm.ne, b0) * F.j1;
        const int tag = prm.btag[bface];
        const R un = ua * nrm, d0 = tr(side, NA) * nrm;
        if (tag == kInlet) {
#pragma unroll
          for (int k = 0; k < AC::NK; ++k)
            acc[AC::CIN + k] = fma(wt * un, tr(side, NF + k + 1), acc[AC::CIN + k]);
        } else if (tag == kOutlet) {
#pragma unroll
          for (int k = 0; k < AC::NK; ++k)
            acc[AC::C + k] -= wt * d0 * tr(side, k + 1) * tr(side, NF + k + 1);
        } else if (tag >= kElectrode0) {
          if (ph.bv_ox >= 0) {
            R c[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) c[f] = tr(side, f);
            const R phiapp = prm.phiapp_batch ? prm.phiapp_batch[bidx * 4 + (tag - kElectrode0)]
                                              : ph.phiapp[tag - kElectrode0];
            const R eta = phiapp - c[0];
            R r = ph.inv_cref * oxidant_conc<NF, R, R>(ph, c);
            if (ph.gam != R(1)) r = powv(r, ph.gam);
            const R dJ = exchange_current(ph, xp) *
                         (ph.e1 * expv(ph.e1 * eta) + r * (ph.e2 * expv((-ph.e2) * eta)));
            R Jh = ph.ox_charge_scale * tr(side, NF);
#pragma unroll
            for (int k = 0; k < AC::NK; ++k)
              if (k == ph.bv_ox) Jh += ph.ox_species_scale * tr(side, NF + k + 1);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j == tag - kElectrode0) acc[AC::PHI + j] += wt * dJ * Jh;
          }
        } else if (tag == kDirichlet) {
          const R hs = side == 0 ? hL : hU;
          const R delta = ph.cip * R(P * P) / sqrtv(hs * hs + hh);
          auto gv = [&](int f) -> R {
            return prm.dirv ? prm.dirv[((long long)f * prm.NBF + bface) * prm.Nfq + pt] : R(0);
          };
          const R jphi = tr(side, 0) - gv(0);
          const R w0 = wt * tr(side, NF), v0 = wt * tr(side, NA + NF) * nrm;
#pragma unroll
          for (int k = 0; k < AC::NK; ++k) {
            const R c = tr(side, k + 1), g = gv(k + 1), jc = c - g, dk = tr(side, NA + k + 1) * nrm;
            const R wk = wt * tr(side, NF + k + 1), vk = wt * tr(side, NA + NF + k + 1) * nrm;
            const R qn = un - ph.mig[k] * d0;
            const R sg = qn > R(0) ? jc : (qn < R(0) ? -jc : R(0));
            acc[AC::A + k] -= fma(jc, v0, dk * w0);
            acc[AC::B + k] += fma(fma(delta, jc, -dk), wk, -jc * vk);
            acc[AC::C + k] -= d0 * halfv(c + g + sg) * wk;
            acc[AC::E + k] += c * fma(fma(delta, jphi, -d0), w0, -jphi * v0);
          }
        }
      }
    }
    __syncwarp();
  }
  pvjp_block_sums<AC::count>(acc, part, nparts, first_part + blockIdx.x);
}

// dtheta[b][j] from the block sums, in block order; one block per point.
template <int NF>
__global__ void pvjp_finish_kernel(const OpParams prm, const double* __restrict__ part, int nparts,
                                   double* __restrict__ dtheta) {
  using AC = PvjpAcc<NF>;
  __shared__ double s[AC::count];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x;
  for (int i = warp; i < AC::count; i += blockDim.x >> 5) {
    double v = 0.0;
    for (int k = lane; k < nparts; k += 32) v += part[((long long)b * AC::count + i) * nparts + k];
    v = warp_sum(v);
    if (lane == 0) s[i] = v;
  }
  __syncthreads();
  const PhysT<double>& ph = prm.pd;
  constexpr int m = NF;
  for (int j = threadIdx.x; j < prm.n_theta; j += blockDim.x) {
    double v = 0.0;
    if (j < m - 1) {
      v = s[AC::B + j] + ph.dmig[j] * s[AC::C + j] + ph.da[j] * s[AC::A + j] + ph.dkc_own[j] * s[AC::E + j];
    } else if (j == m - 1) {
      for (int k = 0; k < m - 1; ++k) v += ph.dkc_m[k] * s[AC::E + k] - ph.da[k] * s[AC::A + k];
    } else if (j < 2 * m - 1) {
      v = s[AC::CIN + j - m];
    } else {
      v = s[AC::PHI + j - (2 * m - 1)];
    }
    dtheta[(long long)b * prm.n_theta + j] = v;
  }
}

// Blocks of the two passes: a function of the mesh alone.
template <int P, int NF>
static void pvjp_blocks(const OpParams& prm, int* elem, int* face) {
  constexpr int ng = kTileThreads / tile_threads<P, double>(), nfw = kTileThreads / 32 * tile_faces<P>();
  const long long ne = ((long long)prm.E + ng - 1) / ng, nf = (prm.foff[3] + nfw - 1) / nfw;
  *elem = (int)(ne < kPvjpBlocks ? ne : kPvjpBlocks);
  *face = (int)(nf < kPvjpBlocks ? nf : kPvjpBlocks);
}

template <int P, int NF>
static cudaError_t launch_pvjp_pn(const OpParams& prm, const double* u, const double* w, double* part,
                                  double* dtheta, int batch, cudaStream_t s) {
  int be, bf;
  pvjp_blocks<P, NF>(prm, &be, &bf);
  constexpr size_t se = (size_t)TileE<P, NF, kParam>::total * sizeof(double) *
                        (kTileThreads / tile_threads<P, double>());
  constexpr size_t sf = (size_t)TileF<P, NF, kParam>::total * sizeof(double) * (kTileThreads / 32);
  static_assert(se <= 200 * 1024 && sf <= 200 * 1024, "parameter adjoint shared memory");
  static SmemAttr ae, af;
  cudaError_t e = raise_smem_limit(ae, pvjp_elem_kernel<P, NF>, se);
  if (e == cudaSuccess) e = raise_smem_limit(af, pvjp_face_kernel<P, NF>, sf);
  if (e != cudaSuccess) return e;
  pvjp_elem_kernel<P, NF><<<dim3(be, batch), kTileThreads, se, s>>>(prm, u, w, part, be + bf);
  pvjp_face_kernel<P, NF><<<dim3(bf, batch), kTileThreads, sf, s>>>(prm, u, w, part, be + bf, be);
  pvjp_finish_kernel<NF><<<batch, 256, 0, s>>>(prm, part, be + bf, dtheta);
  return cudaGetLastError();
}

}  // namespace enp
