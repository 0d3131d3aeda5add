// dc_backproject_rows.cu -- the staged cone-beam backprojection for filtered
// projections whose rows TMA cannot address (a row of W elements that is not a
// multiple of 16 bytes, or a base that is not 16-byte aligned): each view's
// footprint is copied row by row with asynchronous copies, two views ahead,
// instead of by one tiled load.  Everything after the copy is bp_box's.
//
// 128 x 512 x 512 voxels from 400 views of 480 x 620 BF16 pixels (rows of 1240
// bytes) with compensated sums: 36.1 ms by bounds-checked gathers from global
// memory (k_bp3d), 13.8 ms here.
#include "dc_bp_box.cuh"

namespace {

template <typename T, bool KAHAN, int NZ, int LD>
__global__ void __launch_bounds__(TB_TX *TB_TY, 2) k_bp3d_rows(BPArgs a) {
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ dc::BPView sv[TB_VCH];
  __shared__ int4 vtab[TB_VCH];
  bp_layer_box<T, KAHAN, NZ, LD>(a, nullptr, nullptr, nullptr, dsm, nullptr, sv, vtab);
}

template <typename T, bool KAHAN, int LD>
__global__ void __launch_bounds__(TB_TX *TB_TY, 2) k_bp3d_rows_split(BPArgs a, int split) {
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ dc::BPView sv[TB_VCH];
  __shared__ int4 vtab[TB_VCH];
  __shared__ int good;
  bp_split_box<T, KAHAN, 16, LD>(a, nullptr, nullptr, nullptr, split, dsm, nullptr, sv, vtab, &good);
}

template <typename T, bool KAHAN, int NZ, int LD>
int launch(const BPArgs &a, int split, cudaStream_t st) {
  const size_t sm = bp_smem<T, LD>();
  dim3 grid((a.nx + TB_TX - 1) / TB_TX, (a.ny + TB_TY - 1) / TB_TY,
            ((a.z_end - a.z_begin + NZ - 1) / NZ) * a.B);
  if (split > 1 && NZ == 16) {
    auto kernel = k_bp3d_rows_split<T, KAHAN, LD>;
    DC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    DC_CUDA(launch_split(kernel, grid, sm, st, split, a, split));
    DC_CHECK_LAUNCH("k_bp3d_rows_split");
    return DC_OK;
  }
  DC_CUDA(cudaFuncSetAttribute(k_bp3d_rows<T, KAHAN, NZ, LD>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_bp3d_rows<T, KAHAN, NZ, LD><<<grid, dim3(TB_TX, TB_TY), sm, st>>>(a);
  DC_CHECK_LAUNCH("k_bp3d_rows");
  return DC_OK;
}

template <typename T, int LD>
int launch_any(const BPArgs &a, bool kahan, int nz, int split, cudaStream_t st) {
  if (kahan)
    return nz == 16 ? launch<T, true, 16, LD>(a, split, st) : launch<T, true, 32, LD>(a, split, st);
  return nz == 16 ? launch<T, false, 16, LD>(a, split, st) : launch<T, false, 32, LD>(a, split, st);
}

}  // namespace

namespace dc {

int backproject_rows(const dc_geometry *g, int B, const void *gF, int dtype,
                     const float *gF_scale, float *vol, unsigned flags, int z_begin, int z_end,
                     cudaStream_t st, bool *used) {
  BPArgs a = bp_args(g, B, gF, dtype, gF_scale, vol, flags);
  a.z_begin = z_begin;
  a.z_end = z_end;
  const bool kahan = (flags & DC_KAHAN) != 0;
  const uintptr_t base = (uintptr_t)gF;
  // 16-bit rows that start on 4-byte units can be copied as they are
  const bool units = (a.W & 1) == 0 && (base & 3) == 0;
  *used = false;
  if ((dtype == DC_F32X2 && (base & 7)) || (dtype == DC_F32 && (base & 3)) || (base & 1))
    return DC_OK;
  *used = true;
  switch (dtype) {
    case DC_F32: return launch_any<float, LD_UNITS>(a, kahan, g->bp_nz, g->bp_split, st);
    case DC_F32X2: return launch_any<float2, LD_UNITS>(a, kahan, g->bp_nz, g->bp_split, st);
    case DC_BF16:
      return units ? launch_any<__nv_bfloat16, LD_UNITS>(a, kahan, g->bp_nz, g->bp_split, st)
                   : launch_any<__nv_bfloat16, LD_SHIFT>(a, kahan, g->bp_nz, g->bp_split, st);
    default:
      return units ? launch_any<__half, LD_UNITS>(a, kahan, g->bp_nz, g->bp_split, st)
                   : launch_any<__half, LD_SHIFT>(a, kahan, g->bp_nz, g->bp_split, st);
  }
}

}  // namespace dc
