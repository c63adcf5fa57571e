// Kernels of two-dimensional boxes (one periodic z cell), plain forms:
// instantiations and launchers of one precision.  Included once by each
// per-precision translation unit, which defines:
//   MHD_UNIT_PREC      P_FP64, P_MIXED or P_FP32
//   MHD_UNIT_FN(name)  name##_fp64, name##_mixed or name##_fp32
//   MHD_TILES(X)       the tiles of the plain kernels, X(TX, TY)
#include "stage_impl.cuh"

namespace mhd {

namespace {

template <int TX, int TY>
constexpr size_t flat_bytes() {
  using R = Prec<MHD_UNIT_PREC>::R;
  using S = Prec<MHD_UNIT_PREC>::S;
  return Tile<TX, TY, ring_xo<MHD_UNIT_PREC, FM_PLAIN, BOX_2D>(), true>::template bytes<
      R, S, slopes_in_smem<MHD_UNIT_PREC, FM_PLAIN, TX, TY>()>();
}

template <int STAGE, int TX, int TY>
cudaError_t launch_2d(unsigned nblocks, cudaStream_t st, const Geo& g, const StageArgs& args) {
  stage_kernel_2d<MHD_UNIT_PREC, STAGE, TX, TY>
      <<<nblocks, stage_threads<MHD_UNIT_PREC, TX, TY>(), flat_bytes<TX, TY>(), st>>>(g, args);
  return cudaGetLastError();
}

template <int STAGE, int TX, int TY>
cudaError_t set_smem_2d() {
  return cudaFuncSetAttribute(stage_kernel_2d<MHD_UNIT_PREC, STAGE, TX, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)flat_bytes<TX, TY>());
}

}  // namespace

cudaError_t MHD_UNIT_FN(launch_stage_2d)(int stage, int tx, int ty, unsigned nblocks, cudaStream_t st, const Geo& g,
                                         const StageArgs& args) {
  if (stage >= ST_RK3_1) {   // SSP-RK3 runs on the 16 x 8 tile only
    if (tx != 16 || ty != 8) return cudaErrorInvalidValue;
    if (stage == ST_RK3_1) return launch_2d<ST_RK3_1, 16, 8>(nblocks, st, g, args);
    if (stage == ST_RK3_2) return launch_2d<ST_RK3_2, 16, 8>(nblocks, st, g, args);
    return launch_2d<ST_RK3_3, 16, 8>(nblocks, st, g, args);
  }
#define X(TXv, TYv)                                                                    \
  if (tx == TXv && ty == TYv)                                                          \
    return stage == 1 ? launch_2d<1, TXv, TYv>(nblocks, st, g, args) : launch_2d<2, TXv, TYv>(nblocks, st, g, args);
  MHD_TILES(X)
#undef X
  return cudaErrorInvalidValue;
}

cudaError_t MHD_UNIT_FN(set_smem_2d)(int tx, int ty, bool rk3) {
  cudaError_t e = cudaErrorInvalidValue;
  if (rk3) {
    if (tx != 16 || ty != 8) return e;
    e = set_smem_2d<ST_RK3_1, 16, 8>();
    if (e == cudaSuccess) e = set_smem_2d<ST_RK3_2, 16, 8>();
    if (e == cudaSuccess) e = set_smem_2d<ST_RK3_3, 16, 8>();
    return e;
  }
#define X(TXv, TYv)                                  \
  if (tx == TXv && ty == TYv) {                      \
    e = set_smem_2d<1, TXv, TYv>();                  \
    if (e == cudaSuccess) e = set_smem_2d<2, TXv, TYv>(); \
  }
  MHD_TILES(X)
#undef X
  return e;
}

}  // namespace mhd
