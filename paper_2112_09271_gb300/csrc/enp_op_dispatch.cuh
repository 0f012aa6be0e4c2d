// Run-time dispatch from (dim, p, fields, mode) to a compiled operator kernel.
// For kBlockCol (quads), `batch` is the number of block columns (NF * Np): grid.y
// runs over the columns.
#pragma once
#include "enp_internal.h"
#include "enp_launch.cuh"
#include "enp_operator.cuh"
#include "enp_operator3d.cuh"
#include "enp_quad2d.cuh"
#include "enp_tile3d.cuh"

namespace enp {

// Elements per block of the hexahedral kernel, per (p, fields, mode) and
// arithmetic type; 0 = the default. One table per
// type for the whole library (the double-float kernels span several
// translation units).
template <class R>
inline int (&eb3d_table())[kMaxP + 1][4][5] {
  static int t[kMaxP + 1][4][5] = {};
  return t;
}
// Faces per block of the face kernel (modes R, J v, J^T w), the same way.
template <class R>
inline int (&fpb3d_table())[kMaxP + 1][4][3] {
  static int t[kMaxP + 1][4][3] = {};
  return t;
}

// Shared memory of one element's group and of one warp of the face kernel.
template <int P, int NF, int MODE, class R>
static constexpr size_t elem_bytes() {
  if constexpr (MODE <= kVjp && std::is_same<R, float>::value) return (size_t)TileL<P, NF, MODE>::total * sizeof(R);
  else if constexpr (MODE <= kVjp) return (size_t)TileE<P, NF, MODE>::total * sizeof(R);
  else return (size_t)Smem3<P, NF, tpe3d<P>()>::total * sizeof(R);
}
template <int P, int NF, int MODE, class R>
static constexpr size_t face_bytes() {
  return (size_t)TileF<P, NF, MODE>::total * sizeof(R);
}
// Faces per block: as many warps as the block may hold, each tile_faces faces
// (the warps of a block share nothing, so more only saves block launches).
template <int P, int NF, int MODE, class R>
static int max_fpb() { return tile_faces<P>() * (kTileThreads / 32); }
template <int P, int NF, int MODE, class R>
static int default_fpb() {
  return (face_lock<R>() ? 4 : 2) * tile_faces<P>();
}

// Elements per block: groups that share nothing; two by default.
template <int P, int NF, int MODE, class R>
static int max_eb() {
  if constexpr (MODE <= kVjp) {
    return kTileThreads / tile_threads<P, R>() * tile_elems<P, R>();
  } else {
    int eb = kMaxThreads3D / tpe3d<P>();
    while (eb > 1 && (size_t)eb * elem_bytes<P, NF, MODE, R>() > 200 * 1024) --eb;
    return eb < 1 ? 1 : eb;
  }
}
template <int P, int NF, int MODE, class R>
static int default_eb() {
  if constexpr (MODE <= kVjp) {
    return (tile_threads<P, R>() * 2 > kTileThreads ? 1 : 2) * tile_elems<P, R>();
  } else {  // shared memory near 96 KB
    int eb = (int)((96 * 1024) / elem_bytes<P, NF, MODE, R>());
    eb = eb < 1 ? 1 : eb;
    while (eb > 1 && eb * tpe3d<P>() > kMaxThreads3D) --eb;
    return eb;
  }
}

// FP64 at p = 1: the stages of one element fill 8 to 27 of a warp's 32 lanes, and the FP64
// pipe takes as long for a part of a warp. Three elements a warp take a third fewer
// instructions an element, but a longer chain; below this many elements (of all points)
// there are too few of those to go round. R (J v), two fields: 24 elements 14 us with one
// and 20 with three, 5,760 elements 125 and 118 (145 and 147), 14,400 283 and 241 (327 and
// 297), 196,608 3,676 and 3,019; three fields: 7,680 elements 185 and 191 (225 and 224),
// 14,400 340 and 320 (414 and 403). The same bits.
constexpr long long kFewElements = 8192;

// Hexahedra: R, J v, J^T w and dR/dtheta (the blocks: enp_assemble.cuh).
template <int P, int NF, int MODE, class R>
static cudaError_t launch_3d_op(const OpParams& prm, const io_t<R>* u, const io_t<R>* v,
                                io_t<R>* out, int batch, cudaStream_t stream) {
  constexpr size_t per_el = elem_bytes<P, NF, MODE, R>();
  int eb = eb3d_table<R>()[P][NF][MODE];
  if (eb <= 0) eb = default_eb<P, NF, MODE, R>();
  static SmemAttr attr;
  if constexpr (MODE <= kVjp) {
    // the faces first: each face once, both sides' terms into the face buffer
    constexpr size_t per_warp = face_bytes<P, NF, MODE, R>();
    constexpr int FW = tile_faces<P>();
    int fpb = fpb3d_table<R>()[P][NF][MODE];
    if (fpb <= 0) fpb = default_fpb<P, NF, MODE, R>();
    const int warps = (fpb + FW - 1) / FW;
    auto fk = tileface3d_kernel<P, NF, MODE, R>;
    static SmemAttr fattr;
    cudaError_t e = raise_smem_limit(fattr, fk, (size_t)(kTileThreads / 32) * per_warp);
    if (e != cudaSuccess) return e;
    const long long nf = prm.foff[3], per_block = (long long)warps * FW;
    const dim3 fgrid((unsigned)((nf + per_block - 1) / per_block), batch);
    fk<<<fgrid, warps * 32, warps * per_warp, stream>>>(prm, u, v);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    constexpr int EG = tile_elems<P, R>();
    const int groups = (eb + EG - 1) / EG;
    // FP64 at p = 1: one element a warp while warps are few
    constexpr bool kFew = EG > 1 && std::is_same<R, double>::value;
    const bool few = kFew && (long long)prm.E * batch < kFewElements;
    const int per_group = few ? 1 : EG;
    const dim3 grid((prm.E + groups * per_group - 1) / (groups * per_group), batch);
    auto kern = [&] {
      if constexpr (std::is_same<R, float>::value) return lane3d_kernel<P, NF, MODE>;
      else if constexpr (kFew) return few ? tile3d_kernel<P, NF, MODE, R, 1> : tile3d_kernel<P, NF, MODE, R, EG>;
      else return tile3d_kernel<P, NF, MODE, R, EG>;
    }();
    static SmemAttr few_attr;
    e = raise_smem_limit(few ? few_attr : attr, kern, (size_t)max_eb<P, NF, MODE, R>() * per_el);
    if (e != cudaSuccess) return e;
    // beside the face kernel: its volume stages need nothing of the faces
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(groups * tile_threads<P, R>());
    cfg.dynamicSmemBytes = groups * per_group * per_el;
    cfg.stream = stream;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    return launch_status(cudaLaunchKernelEx(&cfg, kern, prm, u, v, out));
  } else {
    auto kern = param3d_kernel<P, NF, R>;
    cudaError_t e = raise_smem_limit(attr, kern, (size_t)max_eb<P, NF, MODE, R>() * per_el);
    if (e != cudaSuccess) return e;
    const dim3 grid((prm.E + eb - 1) / eb, batch);
    kern<<<grid, eb * tpe3d<P>(), eb * per_el, stream>>>(prm, u, out);
  }
  return cudaGetLastError();
}

template <int DIM, int P, int NF, int MODE, class R>
static cudaError_t launch_one(const OpParams& prm, const io_t<R>* u,
                              const io_t<R>* v, io_t<R>* out, int batch, cudaStream_t stream) {
  if constexpr (DIM == 3) {
    return launch_3d_op<P, NF, MODE, R>(prm, u, v, out, batch, stream);
  } else {
    return launch_quad<P, NF, MODE, R>(prm, u, v, out, batch, stream);
  }
}

template <int DIM, int P, int NF, class R>
static cudaError_t launch_mode(int mode, const OpParams& prm, const io_t<R>* u,
                               const io_t<R>* v, io_t<R>* out, int batch, cudaStream_t s) {
  if constexpr (std::is_same<R, df>::value) {
    // double-float: the residual, J v and J^T w (the element blocks and dR/dtheta
    // stay with the FP64 kernels)
    switch (mode) {
      case kResidual: return launch_one<DIM, P, NF, kResidual, R>(prm, u, v, out, batch, s);
      case kJvp: return launch_one<DIM, P, NF, kJvp, R>(prm, u, v, out, batch, s);
      case kVjp: return launch_one<DIM, P, NF, kVjp, R>(prm, u, v, out, batch, s);
    }
    return cudaErrorNotSupported;
  } else {
    switch (mode) {
      case kResidual: return launch_one<DIM, P, NF, kResidual, R>(prm, u, v, out, batch, s);
      case kJvp: return launch_one<DIM, P, NF, kJvp, R>(prm, u, v, out, batch, s);
      case kVjp: return launch_one<DIM, P, NF, kVjp, R>(prm, u, v, out, batch, s);
      case kBlockCol:
        if constexpr (DIM == 2) return launch_one<DIM, P, NF, kBlockCol, R>(prm, u, v, out, batch, s);
        return cudaErrorNotSupported;
      case kParam:
        if constexpr (DIM == 3 && std::is_same<R, double>::value)
          return launch_one<DIM, P, NF, kParam, R>(prm, u, v, out, batch, s);
        return cudaErrorNotSupported;
    }
    return cudaErrorInvalidValue;
  }
}

template <int DIM, int P, class R>
static cudaError_t launch_nf(int mode, const OpParams& prm, const io_t<R>* u,
                             const io_t<R>* v, io_t<R>* out, int batch, cudaStream_t s) {
  if (prm.NF == 2) return launch_mode<DIM, P, 2, R>(mode, prm, u, v, out, batch, s);
  if (prm.NF == 3) return launch_mode<DIM, P, 3, R>(mode, prm, u, v, out, batch, s);
  return cudaErrorInvalidConfiguration;
}

// Elements-per-block of the hexahedral kernel: the largest feasible value for
// (p, fields, mode), and setting the value launches use (0 = default).
template <class R>
int eb3d_step(int p) {
  return p == 1 ? tile_elems<1, R>() : (p == 2 ? tile_elems<2, R>() : (p == 3 ? tile_elems<3, R>() : tile_elems<4, R>()));
}
template <class R>
int eb3d_max(int p, int nf, int mode) {
#define ENP_EBM(PP, NFF, MM) \
  if (p == PP && nf == NFF && mode == MM && (MM != kParam || std::is_same<R, double>::value)) return max_eb<PP, NFF, MM, R>();
#define ENP_EBM_P(PP) ENP_EBM(PP, 2, 0) ENP_EBM(PP, 2, 1) ENP_EBM(PP, 2, 2) ENP_EBM(PP, 2, 4) \
  ENP_EBM(PP, 3, 0) ENP_EBM(PP, 3, 1) ENP_EBM(PP, 3, 2) ENP_EBM(PP, 3, 4)
  ENP_EBM_P(1) ENP_EBM_P(2) ENP_EBM_P(3) ENP_EBM_P(4)
#undef ENP_EBM_P
#undef ENP_EBM
  return 1;
}

// Faces per block of the face kernel (modes 0..2), as above.
template <class R>
int fpb3d_max(int p, int nf, int mode) {
#define ENP_FBM(PP, NFF, MM) if (p == PP && nf == NFF && mode == MM) return max_fpb<PP, NFF, MM, R>();
#define ENP_FBM_P(PP) ENP_FBM(PP, 2, 0) ENP_FBM(PP, 2, 1) ENP_FBM(PP, 2, 2) \
  ENP_FBM(PP, 3, 0) ENP_FBM(PP, 3, 1) ENP_FBM(PP, 3, 2)
  ENP_FBM_P(1) ENP_FBM_P(2) ENP_FBM_P(3) ENP_FBM_P(4)
#undef ENP_FBM_P
#undef ENP_FBM
  return 1;
}

template <class R>
void fpb3d_set(int p, int nf, int mode, int fpb) {
  if (p >= 1 && p <= kMaxP && nf >= 2 && nf <= 3 && mode >= 0 && mode <= 2) fpb3d_table<R>()[p][nf][mode] = fpb;
}

template <class R>
int fpb3d_get(int p, int nf, int mode) {
  if (p >= 1 && p <= kMaxP && nf >= 2 && nf <= 3 && mode >= 0 && mode <= 2) return fpb3d_table<R>()[p][nf][mode];
  return 0;
}

template <class R>
void eb3d_set(int p, int nf, int mode, int eb) {
  if (p >= 1 && p <= kMaxP && nf >= 2 && nf <= 3 && mode >= 0 && mode <= 4) eb3d_table<R>()[p][nf][mode] = eb;
}

template <class R>
int eb3d_get(int p, int nf, int mode) {
  if (p >= 1 && p <= kMaxP && nf >= 2 && nf <= 3 && mode >= 0 && mode <= 4) return eb3d_table<R>()[p][nf][mode];
  return 0;
}

// Upload the degree-p tables to this translation unit's constant memory on
// the current device (idempotent: the tables depend on p only).
template <class R>
cudaError_t prepare_tables(int p, const Tables& t) {
  return upload_const_tables(p, t);
}

template <class R>
cudaError_t launch_op(int mode, const OpParams& prm, const io_t<R>* u,
                      const io_t<R>* v, io_t<R>* out, int batch, cudaStream_t s) {
  if constexpr (std::is_same<R, double>::value) {
    // R, J v and J^T w in double-float arithmetic on hexahedra
    if (prm.arith == kArithDF && prm.dim == 3 && mode <= kVjp)
      return launch_op_df(mode, prm, u, v, out, batch, s);
  }
  if (prm.dim == 3) {
    switch (prm.p) {
      case 1: return launch_nf<3, 1, R>(mode, prm, u, v, out, batch, s);
      case 2: return launch_nf<3, 2, R>(mode, prm, u, v, out, batch, s);
      case 3: return launch_nf<3, 3, R>(mode, prm, u, v, out, batch, s);
      case 4: return launch_nf<3, 4, R>(mode, prm, u, v, out, batch, s);
    }
  }
  if (prm.dim == 2) {
    switch (prm.p) {
      case 1: return launch_nf<2, 1, R>(mode, prm, u, v, out, batch, s);
      case 2: return launch_nf<2, 2, R>(mode, prm, u, v, out, batch, s);
      case 3: return launch_nf<2, 3, R>(mode, prm, u, v, out, batch, s);
    }
  }
  return cudaErrorInvalidConfiguration;
}

}  // namespace enp

// The double-float hexahedral kernels of one degree PP (op_df_pPP.cu): the
// launcher and the upload of that translation unit's constant tables.
#define ENP_DF_DEGREE(PP)                                                                    \
  cudaError_t enp::launch_df_p##PP(int mode, const OpParams& prm, const double* u,             \
                                   const double* v, double* out, int batch, cudaStream_t s) { \
    if (prm.dim != 3) return cudaErrorInvalidConfiguration;                                   \
    return launch_nf<3, PP, df>(mode, prm, u, v, out, batch, s);                              \
  }                                                                                           \
  cudaError_t enp::upload_tables_df_p##PP(const Tables& t) { return upload_const_tables(PP, t); }
