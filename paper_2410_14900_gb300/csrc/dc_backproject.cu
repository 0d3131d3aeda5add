// dc_backproject.cu -- voxel-driven cone-beam backprojection A3d^T of the
// filtered projections (Ye et al., DRACO, Eq. 5 and the last layer of
// Eq. 12), optional ReLU (Sec. 2.3), and the batched reconstruction.
//
//   f(X) = sum_i bilinear(g^F_i, P_i X) / |X - a_i|^2
//
// Each thread owns a column of NZ voxels along z (register blocking); the
// projection of the column is affine in z before the perspective divide, so
// a voxel costs one reciprocal for the depth and one for the distance
// weight.  Coordinates are taken relative to the volume centre and to the
// principal point so that FP32 keeps ~1e-5 pixel accuracy.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "dc_async.cuh"
#include "dc_bp_box.cuh"
#include "dc_common.cuh"

namespace {

template <typename T, bool KAHAN>
__global__ void __launch_bounds__(BP_TX *BP_TY) k_bp3d(BPArgs a) {
  __shared__ dc::BPView sv[BP_VCHUNK];
  const int ix = blockIdx.x * BP_TX + threadIdx.x;
  const int iy = blockIdx.y * BP_TY + threadIdx.y;
  const int zblocks = (a.nz + BP_NZ - 1) / BP_NZ;
  const int b = blockIdx.z / zblocks;
  const int z0 = (blockIdx.z % zblocks) * BP_NZ;
  const int tid = threadIdx.y * BP_TX + threadIdx.x;
  const float xo = ((float)ix - 0.5f * (float)(a.nx - 1)) * a.dx;
  const float yo = ((float)iy - 0.5f * (float)(a.ny - 1)) * a.dy;
  const float zo = ((float)z0 - 0.5f * (float)(a.nz - 1)) * a.dz;
  const size_t np = (size_t)a.H * a.W;
  const T *gbase = (const T *)a.gF + (size_t)b * a.V * np;

  float acc[BP_NZ], cmp[BP_NZ];
#pragma unroll
  for (int k = 0; k < BP_NZ; ++k) acc[k] = cmp[k] = 0.0f;

  for (int i0 = 0; i0 < a.V; i0 += BP_VCHUNK) {
    int nvc = min(BP_VCHUNK, a.V - i0);
    __syncthreads();
    if (tid < nvc) sv[tid] = a.views[i0 + tid];
    __syncthreads();
    for (int ii = 0; ii < nvc; ++ii) {
      const dc::BPView w = sv[ii];
      const int i = i0 + ii;
      const T *img = gbase + (size_t)i * np;
      float sc = 1.0f;
      if (a.scale) sc = a.scale[(size_t)b * a.V + i];
      float U0 = fmaf(w.r0.x, xo, fmaf(w.r0.y, yo, fmaf(w.r0.z, zo, w.r0.w)));
      float V0 = fmaf(w.r1.x, xo, fmaf(w.r1.y, yo, fmaf(w.r1.z, zo, w.r1.w)));
      float W0 = fmaf(w.r2.x, xo, fmaf(w.r2.y, yo, fmaf(w.r2.z, zo, w.r2.w)));
      float dU = w.r0.z * a.dz, dV = w.r1.z * a.dz, dW = w.r2.z * a.dz;
      float ex = w.ca.x + xo, ey = w.ca.y + yo, ez0 = w.ca.z + zo;
      float rho2 = fmaf(ex, ex, ey * ey);
#pragma unroll
      for (int k = 0; k < BP_NZ; ++k) {
        float kf = (float)k;
        float dep = fmaf(kf, dW, W0);
        if (!(dep > 0.0f)) continue;
        float rw = __frcp_rn(dep);
        float u = fmaf(fmaf(kf, dU, U0), rw, w.pp.x);
        float v = fmaf(fmaf(kf, dV, V0), rw, w.pp.y);
        float val = bilinear<T>(img, a.H, a.W, u, v) * sc;
        float ez = fmaf(kf, a.dz, ez0);
        float wt = __frcp_rn(fmaf(ez, ez, rho2));
        float term = val * wt;
        if (KAHAN) {
          float y = term - cmp[k];
          float t = acc[k] + y;
          cmp[k] = (t - acc[k]) - y;
          acc[k] = t;
        } else {
          acc[k] += term;
        }
      }
    }
  }
  if (ix >= a.nx || iy >= a.ny) return;
  const size_t nvox = (size_t)a.nx * a.ny * a.nz;
#pragma unroll
  for (int k = 0; k < BP_NZ; ++k) {
    int iz = z0 + k;
    if (iz >= a.nz) break;
    size_t o = (size_t)b * nvox + ((size_t)iz * a.ny + iy) * a.nx + ix;
    float f = acc[k];
    if (a.flags & DC_ACCUM) f += a.vol[o];
    if ((a.flags & DC_RELU) && f < 0.0f) f = 0.0f;
    a.vol[o] = f;
  }
}

template <typename T, bool KAHAN, int NZ>
__global__ void __launch_bounds__(TB_TX *TB_TY, 2) k_bp3d_tma(BPArgs a, unsigned *err,
                                                             const __grid_constant__ CUtensorMap tmn,
                                                             const __grid_constant__ CUtensorMap tmw) {
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ uint64_t full[TB_NS];
  __shared__ dc::BPView sv[TB_VCH];
  __shared__ int4 vtab[TB_VCH];
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    for (int q = 0; q < TB_NS; ++q) dc::mbar_init(&full[q], 1);
    dc::fence_barrier_init();
  }
  __syncthreads();
  if (!bp_layer_box<T, KAHAN, NZ, LD_TMA>(a, &tmn, &tmw, err, dsm, full, sv, vtab)) {
    for (int q = 0; q < TB_NS; ++q) dc::mbar_wait_bounded(&full[q], 0, nullptr);
  }
}

// views split over the CTAs of a cluster (bp_split_box); 16-deep boxes
template <typename T, bool KAHAN>
__global__ void __launch_bounds__(TB_TX *TB_TY, 2)
    k_bp3d_split(BPArgs a, unsigned *err, int split, const __grid_constant__ CUtensorMap tmn,
                 const __grid_constant__ CUtensorMap tmw) {
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ uint64_t full[TB_NS];
  __shared__ dc::BPView sv[TB_VCH];
  __shared__ int4 vtab[TB_VCH];
  __shared__ int good;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    for (int q = 0; q < TB_NS; ++q) dc::mbar_init(&full[q], 1);
    dc::fence_barrier_init();
  }
  __syncthreads();
  bp_split_box<T, KAHAN, 16, LD_TMA>(a, &tmn, &tmw, err, split, dsm, full, sv, vtab, &good);
}

// Persistent backprojection of a batch of problems (orbits of uneven view
// counts, detectors and volumes): CTAs take (problem, box) items from a
// device counter until all are done.  Items are ordered by problem, largest
// view count first, so the long boxes start early.
constexpr int DC_MAX_BATCH = 32;
struct BatchProblem {
  BPArgs a;               // a.vol is unused: the output comes with the run
  const CUtensorMap *tmn; // global-memory tensor maps over the problem's g^F
  const CUtensorMap *tmw;
  int bx, by, bz;         // boxes per dimension (bz includes the batch)
  int nz;                 // voxels per thread along z (box depth) of this problem: 16 or 32
  long long first;        // first work item of this problem
};
struct BatchRun {
  float *vol[DC_MAX_BATCH];
};

template <typename T, bool KAHAN>
__global__ void __launch_bounds__(TB_TX *TB_TY, 2) k_bp3d_batched(const BatchProblem *probs,
                                                                 int nprob, long long total,
                                                                 unsigned long long *counter,
                                                                 unsigned *err, BatchRun run) {
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ uint64_t full[TB_NS];
  __shared__ dc::BPView sv[TB_VCH];
  __shared__ int4 vtab[TB_VCH];
  __shared__ long long item;
  const int tid = threadIdx.y * TB_TX + threadIdx.x;
  if (tid == 0) {
    for (int q = 0; q < TB_NS; ++q) dc::mbar_init(&full[q], 1);
    dc::fence_barrier_init();
  }
  unsigned it = 0;
  for (;;) {
    __syncthreads();
    if (tid == 0) item = (long long)atomicAdd(counter, 1ull);
    __syncthreads();
    const long long w = item;
    if (w >= total) break;
    int p = 0;
    while (p + 1 < nprob && probs[p + 1].first <= w) ++p;
    const BatchProblem &P = probs[p];
    long long lw = w - P.first;
    int bxi = (int)(lw % P.bx);
    long long rest = lw / P.bx;
    int byi = (int)(rest % P.by);
    int bzi = (int)(rest / P.by);
    // each problem has its own box depth (the autotuner's choice for its
    // detector-to-voxel scale); the CTA-uniform branch picks the instance
    const bool done = (P.nz == 16)
                          ? bp_box<T, KAHAN, 16>(P.a, run.vol[p], P.tmn, P.tmw, err, bxi, byi, bzi,
                                                 dsm, full, sv, vtab, it)
                          : bp_box<T, KAHAN, 32>(P.a, run.vol[p], P.tmn, P.tmw, err, bxi, byi, bzi,
                                                 dsm, full, sv, vtab, it);
    if (!done) {
      for (int q = 0; q < TB_NS; ++q) dc::mbar_wait_bounded(&full[q], 0, nullptr);
      return;
    }
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

// bytes per g^F pixel of a storage form
int pixel_bytes(int dtype) { return dtype == DC_F32 ? 4 : dtype == DC_F32X2 ? 8 : 2; }

// 3-D map over g^F viewed as [B*V][H][W] with a box of bw x TB_BH x 1 (a
// DC_F32X2 pair is one 8-byte element: the copy moves its bits)
bool make_map(CUtensorMap *m, const void *base, int dtype, int W, int H, long long nimg,
              int bw) {
  auto fn = encode_fn();
  if (!fn) return false;
  int es = pixel_bytes(dtype);
  CUtensorMapDataType t = (dtype == DC_F32)     ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                          : (dtype == DC_F32X2) ? CU_TENSOR_MAP_DATA_TYPE_UINT64
                          : (dtype == DC_BF16)  ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)nimg};
  cuuint64_t strides[2] = {(cuuint64_t)W * es, (cuuint64_t)W * H * es};
  cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)TB_BH, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, t, 3, const_cast<void *>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

template <typename T, int NZ>
int launch_bp_tma_nz(const dc_geometry *g, BPArgs &a, bool kahan, cudaStream_t st,
                     const CUtensorMap &mn, const CUtensorMap &mw) {
  if (g->bp_split > 1 && NZ == 16) {
    auto kernel = kahan ? k_bp3d_split<T, true> : k_bp3d_split<T, false>;
    DC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)bp_smem<T>()));
    dim3 grid((a.nx + TB_TX - 1) / TB_TX, (a.ny + TB_TY - 1) / TB_TY,
              ((a.z_end - a.z_begin + 15) / 16) * a.B);
    DC_CUDA(launch_split(kernel, grid, bp_smem<T>(), st, g->bp_split, a, g->w_flags, g->bp_split,
                         mn, mw));
    return DC_OK;
  }
  dim3 blk(TB_TX, TB_TY);
  dim3 grid((a.nx + TB_TX - 1) / TB_TX, (a.ny + TB_TY - 1) / TB_TY,
            ((a.z_end - a.z_begin + NZ - 1) / NZ) * a.B);
  const size_t sm = bp_smem<T>();
  if (kahan) {
    DC_CUDA(cudaFuncSetAttribute(k_bp3d_tma<T, true, NZ>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_bp3d_tma<T, true, NZ><<<grid, blk, sm, st>>>(a, g->w_flags, mn, mw);
  } else {
    DC_CUDA(cudaFuncSetAttribute(k_bp3d_tma<T, false, NZ>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_bp3d_tma<T, false, NZ><<<grid, blk, sm, st>>>(a, g->w_flags, mn, mw);
  }
  return DC_OK;
}

bool tma_ok(const void *base, int W, int dtype) {
  int es = pixel_bytes(dtype);
  return ((size_t)W * es) % 16 == 0 && ((uintptr_t)base & 15) == 0 && encode_fn() != nullptr;
}

template <typename T>
int launch_bp_tma(const dc_geometry *g, BPArgs &a, int dtype, bool kahan, cudaStream_t st,
                  bool *used) {
  *used = false;
  if (!tma_ok(a.gF, a.W, dtype)) return DC_OK;
  CUtensorMap mn, mw;
  long long nimg = (long long)a.B * a.V;
  if (!make_map(&mn, a.gF, dtype, a.W, a.H, nimg, TileShape<T>::BWN) ||
      !make_map(&mw, a.gF, dtype, a.W, a.H, nimg, TileShape<T>::BWW))
    return DC_OK;
  int rc = (g->bp_nz == 16) ? launch_bp_tma_nz<T, 16>(g, a, kahan, st, mn, mw)
                            : launch_bp_tma_nz<T, 32>(g, a, kahan, st, mn, mw);
  if (rc) return rc;
  *used = true;
  return DC_OK;
}

int check_bp(const dc_geometry *g, int B, const char *who) {
  if (!g) return dc::fail(DC_ERR_ARG, std::string(who) + ": NULL geometry");
  if (B < 1) return dc::fail(DC_ERR_ARG, std::string(who) + ": batch must be >= 1");
  int dev = -1;
  cudaGetDevice(&dev);
  if (dev != g->device)
    return dc::fail(DC_ERR_ARG, std::string(who) + ": geometry belongs to another device");
  return DC_OK;
}

}  // namespace

namespace dc {

bool encode_map_f32(CUtensorMap *m, const void *base, size_t d0, size_t d1, size_t d2, int b0,
                    int b1) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {d0, d1, d2};
  cuuint64_t strides[2] = {d0 * sizeof(float), d0 * d1 * sizeof(float)};
  cuuint32_t box[3] = {(cuuint32_t)b0, (cuuint32_t)b1, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void *>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int backproject_check(const dc_geometry *g, int B, const void *gF, int dtype,
                      const float *gF_scale, const float *vol, unsigned flags, const char *who) {
  int rc = check_bp(g, B, who);
  if (rc) return rc;
  if (!gF || !vol) return fail(DC_ERR_ARG, std::string(who) + ": NULL gF or vol");
  if (flags & ~(DC_ACCUM | DC_KAHAN | DC_RELU))
    return fail(DC_ERR_ARG, std::string(who) + ": unknown flag");
  if (dtype != DC_F32 && dtype != DC_BF16 && dtype != DC_F16 && dtype != DC_F32X2)
    return fail(DC_ERR_ARG, std::string(who) + ": unknown dtype");
  if (dtype == DC_F16 && !gF_scale)
    return fail(DC_ERR_ARG, std::string(who) + ": DC_F16 needs gF_scale");
  return DC_OK;
}

int backproject_slab(const dc_geometry *g, int B, const void *gF, int dtype,
                     const float *gF_scale, float *vol, unsigned flags, int z_begin, int z_end,
                     cudaStream_t st, bool *used) {
  *used = false;
  if (getenv("DC_BP_NO_TMA")) return DC_OK;
  // A launch takes at most 65535 CTAs along z: layers of boxes times batch
  // items times the CTAs that share a box's views.  More go in several
  // launches, whole items each (a result does not depend on where they part).
  const dc_geometry_desc &d = g->d;
  const int nz = g->bp_nz, share = nz == 16 ? g->bp_split : 1, most = 65535 / share;
  const int layers = bp_layers(z_begin, z_end, nz);
  if (layers > most) {
    const int zm = z_begin + most * nz;
    int rc = backproject_slab(g, B, gF, dtype, gF_scale, vol, flags, z_begin, zm, st, used);
    if (rc || !*used) return rc;
    return backproject_slab(g, B, gF, dtype, gF_scale, vol, flags, zm, z_end, st, used);
  }
  const size_t item = (size_t)d.n_views * d.det_rows * d.det_cols * pixel_bytes(dtype);
  const size_t nvox = (size_t)d.vol_x * d.vol_y * d.vol_z;
  const int per = std::min(B, most / layers);
  for (int b = 0; b < B; b += per) {
    const int n = std::min(per, B - b);
    const void *p = (const char *)gF + b * item;
    const float *sc = gF_scale ? gF_scale + (size_t)b * d.n_views : nullptr;
    float *v = vol + b * nvox;
    BPArgs a = bp_args(g, n, p, dtype, sc, v, flags);
    a.z_begin = z_begin;
    a.z_end = z_end;
    // the staged kernel compensates the sums over TB_VCH views (and those of a
    // cluster's CTAs): a single one needs none (8 views of 512 x 512 in BF16,
    // 128^3 voxels: 33 us with it, 22 without; the same bits)
    const bool kahan = (flags & DC_KAHAN) != 0 && (d.n_views > TB_VCH || share > 1);
    ProfScope ps(KID_BP3D, st);
    int rc;
    switch (dtype) {
      case DC_F32: rc = launch_bp_tma<float>(g, a, dtype, kahan, st, used); break;
      case DC_F32X2: rc = launch_bp_tma<float2>(g, a, dtype, kahan, st, used); break;
      case DC_BF16: rc = launch_bp_tma<__nv_bfloat16>(g, a, dtype, kahan, st, used); break;
      default: rc = launch_bp_tma<__half>(g, a, dtype, kahan, st, used); break;
    }
    if (rc) return rc;
    if (*used) DC_CHECK_LAUNCH("k_bp3d_tma");
    else if ((rc = backproject_rows(g, n, p, dtype, sc, v, flags, z_begin, z_end, st, used))) return rc;
    if (!*used) return DC_OK;  // the layout that neither reads: true of every item
  }
  return DC_OK;
}

// Box depth: 32 voxels per thread, or 16 where the projections of 32-deep
// boxes do not fit the staged tile (their views would take the bounds-checked
// global path: 64^3 voxels of 2 mm on 2 mm pixels, 1.6 pixels per voxel, 557 us
// with 32 and 31 us with 16) or where 32-deep boxes are fewer than the SMs.
// Judged on the boxes at the volume's centre and at its four lateral sides.
void bp_plan(dc_geometry *g) {
  const dc_geometry_desc &d = g->d;
  const double dx = d.voxel[0], dy = d.voxel[1], dz = d.voxel[2];
  const double off[5][2] = {{0, 0}, {1, 0}, {-1, 0}, {0, 1}, {0, -1}};
  const double ex = std::max(0.0, 0.5 * dx * (d.vol_x - TB_TX)),
               ey = std::max(0.0, 0.5 * dy * (d.vol_y - TB_TY));
  long fit = 0, all = 0;
  for (int i = 0; i < d.n_views; ++i) {
    const double *v = g->host_geo + (size_t)DC_VIEW_GEO_N * i;  // a, lx, ly, lz, D
    for (int o = 0; o < 5; ++o) {
      double vmin = 1e30, vmax = -1e30;
      bool front = true;
      for (int c = 0; c < 8; ++c) {
        const double X[3] = {
            d.vol_center[0] + off[o][0] * ex + ((c & 1) ? 0.5 : -0.5) * dx * (TB_TX - 1),
            d.vol_center[1] + off[o][1] * ey + ((c & 2) ? 0.5 : -0.5) * dy * (TB_TY - 1),
            d.vol_center[2] + ((c & 4) ? 0.5 : -0.5) * dz * (TB_NZ - 1)};
        double pv = 0.0, dep = 0.0;
        for (int t = 0; t < 3; ++t) {
          pv += v[6 + t] * (X[t] - v[t]);
          dep -= v[9 + t] * (X[t] - v[t]);
        }
        if (!(dep > 1.0)) front = false;
        else {
          vmin = std::min(vmin, pv / dep * v[12] / d.pitch);
          vmax = std::max(vmax, pv / dep * v[12] / d.pitch);
        }
      }
      ++all;
      if (front && vmax - vmin + 5.0 <= TB_BH) ++fit;
    }
  }
  {  // pixels per voxel at the volume's centre, in the middle view
    const double *v = g->host_geo + (size_t)DC_VIEW_GEO_N * (d.n_views / 2);
    double dep = 0.0;
    for (int t = 0; t < 3; ++t) dep -= v[9 + t] * (d.vol_center[t] - v[t]);
    g->bp_px = std::cbrt(dx * dy * dz) * v[12] / (dep * d.pitch);
  }
  const long boxes = (long)((d.vol_x + TB_TX - 1) / TB_TX) * ((d.vol_y + TB_TY - 1) / TB_TY) *
                     ((d.vol_z + TB_NZ - 1) / TB_NZ);
  g->bp_fit32 = fit >= all * 0.95;
  g->bp_nz = (!g->bp_fit32 || boxes < g->sms) ? 16 : 32;
  // views split over clusters where 16-deep boxes are fewer than the SMs: as
  // many CTAs as two per SM hold, at least 8 views each (64 boxes, 64 views:
  // 57 us unsplit, 33 us split by four)
  const long boxes16 = (long)((d.vol_x + TB_TX - 1) / TB_TX) * ((d.vol_y + TB_TY - 1) / TB_TY) *
                       ((d.vol_z + 15) / 16);
  g->bp_split = 1;
  while (g->bp_split < 8 && g->bp_split * boxes16 <= g->sms && d.n_views >= 16 * g->bp_split)
    g->bp_split *= 2;
}

}  // namespace dc

extern "C" {

int dc_backproject(const dc_geometry *g, int B, const void *gF, int dtype,
                   const float *gF_scale, float *vol, unsigned flags, void *stream) {
  int rc = check_bp(g, B, "dc_backproject");
  if (rc) return rc;
  if (!gF || !vol) return dc::fail(DC_ERR_ARG, "dc_backproject: NULL gF or vol");
  if (flags & ~(DC_ACCUM | DC_KAHAN | DC_RELU))
    return dc::fail(DC_ERR_ARG, "dc_backproject: unknown flag");
  if (dtype == DC_F16 && !gF_scale)
    return dc::fail(DC_ERR_ARG, "dc_backproject: DC_F16 needs gF_scale");
  if (dtype != DC_F32 && dtype != DC_BF16 && dtype != DC_F16 && dtype != DC_F32X2)
    return dc::fail(DC_ERR_ARG, "dc_backproject: unknown dtype");
  const dc_geometry_desc &d = g->d;
  cudaStream_t st = (cudaStream_t)stream;
  bool used = false;
  rc = dc::backproject_slab(g, B, gF, dtype, gF_scale, vol, flags, 0, d.vol_z, st, &used);
  if (rc || used) return rc;
  // g^F of a layout that neither staged kernel reads (pairs off their 8 bytes)
  BPArgs a = bp_args(g, B, gF, dtype, gF_scale, vol, flags);
  dim3 blk(BP_TX, BP_TY);
  dim3 grid((d.vol_x + BP_TX - 1) / BP_TX, (d.vol_y + BP_TY - 1) / BP_TY,
            ((d.vol_z + BP_NZ - 1) / BP_NZ) * B);
  bool kahan = (flags & DC_KAHAN) != 0;
  dc::ProfScope ps(dc::KID_BP3D, st);
  switch (dtype) {
    case DC_F32:
      if (kahan) k_bp3d<float, true><<<grid, blk, 0, st>>>(a);
      else k_bp3d<float, false><<<grid, blk, 0, st>>>(a);
      break;
    case DC_F32X2:
      if (kahan) k_bp3d<float2, true><<<grid, blk, 0, st>>>(a);
      else k_bp3d<float2, false><<<grid, blk, 0, st>>>(a);
      break;
    case DC_BF16:
      if (kahan) k_bp3d<__nv_bfloat16, true><<<grid, blk, 0, st>>>(a);
      else k_bp3d<__nv_bfloat16, false><<<grid, blk, 0, st>>>(a);
      break;
    case DC_F16:
      if (kahan) k_bp3d<__half, true><<<grid, blk, 0, st>>>(a);
      else k_bp3d<__half, false><<<grid, blk, 0, st>>>(a);
      break;
    default:
      return dc::fail(DC_ERR_ARG, "dc_backproject: unknown dtype");
  }
  DC_CHECK_LAUNCH("k_bp3d");
  return DC_OK;
}

}  // extern "C"

// ------------------------------------------------------------------------
// Batched reconstruction: the filter of every problem (its chunked launches,
// or with DC_PERSISTENT_FILTER one persistent kernel over the (problem,
// view) images of all problems), then one persistent backprojection over all
// problems' voxel boxes.  Everything a run needs is allocated by
// dc_batch_create, so dc_batch_run allocates nothing and can be captured in
// a CUDA graph.
struct dc_batch {
  int n;
  int dtype;
  unsigned flags;
  int nz;                         // 16 / 32 for every problem, 0: each geometry's own bp_nz
  int grid;
  long long total;
  int order[DC_MAX_BATCH];        // table position -> problem index
  dc_geometry *geoms[DC_MAX_BATCH];
  void *gF[DC_MAX_BATCH];         // owned filtered projections [V][H][W]
  float *scale[DC_MAX_BATCH];     // owned FP16 scales [V]
  BatchProblem *d_probs;
  CUtensorMap *d_maps;
  unsigned long long *d_counter;
  dc::BatchFilterPlan *fplan;     // persistent filter of every problem (NULL: per-problem calls)
};

namespace {

void free_batch(dc_batch *b) {
  if (!b) return;
  for (int i = 0; i < b->n; ++i) {
    cudaFree(b->gF[i]);
    cudaFree(b->scale[i]);
  }
  cudaFree(b->d_probs);
  cudaFree(b->d_maps);
  cudaFree(b->d_counter);
  dc::batch_filter_destroy(b->fplan);
  delete b;
}

int build_batch_tables(dc_batch *b) {
  std::vector<BatchProblem> probs(b->n);
  std::vector<CUtensorMap> maps(2 * b->n);
  long long first = 0;
  for (int t = 0; t < b->n; ++t) {
    int i = b->order[t];
    const dc_geometry *g = b->geoms[i];
    const dc_geometry_desc &d = g->d;
    BatchProblem &P = probs[t];
    memset(&P, 0, sizeof(P));
    P.a.gF = b->gF[i];
    P.a.scale = (b->dtype == DC_F16) ? b->scale[i] : nullptr;
    P.a.views = g->bpv;
    P.a.vol = nullptr;
    P.a.flags = b->flags & DC_RELU;
    P.a.V = d.n_views;
    P.a.H = d.det_rows;
    P.a.W = d.det_cols;
    P.a.nx = d.vol_x;
    P.a.ny = d.vol_y;
    P.a.nz = d.vol_z;
    P.a.z_begin = 0;
    P.a.z_end = d.vol_z;
    P.a.B = 1;
    P.a.dx = (float)d.voxel[0];
    P.a.dy = (float)d.voxel[1];
    P.a.dz = (float)d.voxel[2];
    const bool pairs = (b->dtype == DC_F32X2);
    if (!make_map(&maps[2 * t], b->gF[i], b->dtype, d.det_cols, d.det_rows, d.n_views,
                  pairs ? TB_PBWN : TB_BWN) ||
        !make_map(&maps[2 * t + 1], b->gF[i], b->dtype, d.det_cols, d.det_rows, d.n_views,
                  pairs ? TB_PBWW : TB_BWW))
      return dc::fail(DC_ERR_CUDA, "dc_batch: tensor map encoding failed");
    P.tmn = b->d_maps + 2 * t;
    P.tmw = b->d_maps + 2 * t + 1;
    P.bx = (d.vol_x + TB_TX - 1) / TB_TX;
    P.by = (d.vol_y + TB_TY - 1) / TB_TY;
    P.nz = b->nz ? b->nz : g->bp_nz;
    P.bz = (d.vol_z + P.nz - 1) / P.nz;
    P.first = first;
    first += (long long)P.bx * P.by * P.bz;
  }
  b->total = first;
  DC_CUDA(cudaMemcpy(b->d_maps, maps.data(), sizeof(CUtensorMap) * maps.size(),
                     cudaMemcpyHostToDevice));
  DC_CUDA(cudaMemcpy(b->d_probs, probs.data(), sizeof(BatchProblem) * probs.size(),
                     cudaMemcpyHostToDevice));
  return DC_OK;
}

template <typename T, bool KAHAN>
int launch_batched(dc_batch *b, BatchRun &run, cudaStream_t st) {
  const size_t sm = bp_smem<T>();
  DC_CUDA(cudaFuncSetAttribute(k_bp3d_batched<T, KAHAN>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_bp3d_batched<T, KAHAN><<<b->grid, dim3(TB_TX, TB_TY), sm, st>>>(
      b->d_probs, b->n, b->total, b->d_counter, b->geoms[0]->w_flags, run);
  return DC_OK;
}

template <typename T>
int launch_batched_t(dc_batch *b, BatchRun &run, cudaStream_t st) {
  return (b->flags & DC_KAHAN) ? launch_batched<T, true>(b, run, st)
                               : launch_batched<T, false>(b, run, st);
}

}  // namespace

extern "C" {

int dc_batch_create(int n, dc_geometry *const *geoms, int dtype, unsigned flags,
                    dc_batch **out) {
  if (!out || !geoms) return dc::fail(DC_ERR_ARG, "dc_batch_create: NULL argument");
  *out = nullptr;
  if (n < 1 || n > DC_MAX_BATCH)
    return dc::fail(DC_ERR_ARG, "dc_batch_create: 1 <= n <= " + std::to_string(DC_MAX_BATCH));
  if (dtype != DC_F32 && dtype != DC_BF16 && dtype != DC_F16 && dtype != DC_F32X2)
    return dc::fail(DC_ERR_ARG, "dc_batch_create: unknown dtype");
  if (flags & ~(DC_KAHAN | DC_RELU | DC_PERSISTENT_FILTER))
    return dc::fail(DC_ERR_ARG,
                    "dc_batch_create: flags may be DC_KAHAN | DC_RELU | DC_PERSISTENT_FILTER");
  if (!encode_fn()) return dc::fail(DC_ERR_UNSUPPORTED, "dc_batch_create: no TMA encoder");
  int dev = -1;
  cudaGetDevice(&dev);
  int es = pixel_bytes(dtype);
  for (int i = 0; i < n; ++i) {
    if (!geoms[i]) return dc::fail(DC_ERR_ARG, "dc_batch_create: NULL geometry");
    if (geoms[i]->device != dev)
      return dc::fail(DC_ERR_ARG, "dc_batch_create: geometry on another device");
    if (((size_t)geoms[i]->d.det_cols * es) % 16 != 0)
      return dc::fail(DC_ERR_UNSUPPORTED,
                      "dc_batch_create: detector rows must be a multiple of 16 bytes");
  }
  dc_batch *b = new dc_batch();
  memset((void *)b, 0, sizeof(dc_batch));
  b->n = n;
  b->dtype = dtype;
  b->flags = flags;
  b->nz = 0;  // each problem's box depth from its geometry (dc_geometry_set_tuning)
  for (int i = 0; i < n; ++i) b->geoms[i] = geoms[i];
  // largest view count first
  for (int i = 0; i < n; ++i) b->order[i] = i;
  std::sort(b->order, b->order + n, [&](int x, int y) {
    return geoms[x]->d.n_views > geoms[y]->d.n_views;
  });
  auto bail = [&](int code) {
    free_batch(b);
    return code;
  };
  for (int i = 0; i < n; ++i) {
    const dc_geometry_desc &d = geoms[i]->d;
    size_t bytes = (size_t)d.n_views * d.det_rows * d.det_cols * es;
    cudaError_t e = dc::dmalloc(&b->gF[i], bytes);
    if (e != cudaSuccess) return bail(dc::cuda_fail(e, "dc_batch_create: g^F"));
    if (dtype == DC_F16) {
      e = dc::dmalloc((void **)&b->scale[i], sizeof(float) * d.n_views);
      if (e != cudaSuccess) return bail(dc::cuda_fail(e, "dc_batch_create: scales"));
    }
  }
  cudaError_t e = dc::dmalloc((void **)&b->d_probs, sizeof(BatchProblem) * n);
  if (e == cudaSuccess) e = dc::dmalloc((void **)&b->d_maps, sizeof(CUtensorMap) * 2 * n);
  if (e == cudaSuccess) e = dc::dmalloc((void **)&b->d_counter, sizeof(unsigned long long));
  if (e != cudaSuccess) return bail(dc::cuda_fail(e, "dc_batch_create: tables"));
  int rc = build_batch_tables(b);
  if (rc) return bail(rc);
  // optionally one persistent launch filters every problem; problems whose
  // rows do not fit its shared memory keep the per-problem filter calls
  if (flags & DC_PERSISTENT_FILTER) {
    rc = dc::batch_filter_create(n, b->geoms, dtype, b->gF, b->scale, &b->fplan);
    if (rc == DC_ERR_UNSUPPORTED) {
      b->fplan = nullptr;
    } else if (rc) {
      return bail(rc);
    }
  }
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  b->grid = std::max(1, sms) * 2;
  *out = b;
  return DC_OK;
}

int dc_batch_set_bp_nz(dc_batch *b, int nz) {
  if (!b || (nz != 0 && nz != 16 && nz != 32))
    return dc::fail(DC_ERR_ARG, "dc_batch_set_bp_nz: nz must be 16, 32 or 0 (per geometry)");
  b->nz = nz;
  return build_batch_tables(b);
}

int dc_batch_run(dc_batch *b, const float *const *g, const float *const *W, float *const *vol,
                 void *stream) {
  if (!b || !g || !vol) return dc::fail(DC_ERR_ARG, "dc_batch_run: NULL argument");
  for (int i = 0; i < b->n; ++i)
    if (!g[i] || !vol[i]) return dc::fail(DC_ERR_ARG, "dc_batch_run: NULL g or vol");
  cudaStream_t st = (cudaStream_t)stream;
  if (b->fplan) {
    int rc = dc::batch_filter_run(b->fplan, g, W, st);
    if (rc) return rc;
  } else {
    for (int i = 0; i < b->n; ++i) {
      int rc = dc_filter(b->geoms[i], 1, g[i], W ? W[i] : nullptr, b->gF[i], b->dtype,
                         b->scale[i], stream);
      if (rc) return rc;
    }
  }
  BatchRun run;
  memset(&run, 0, sizeof(run));
  for (int t = 0; t < b->n; ++t) run.vol[t] = vol[b->order[t]];
  DC_CUDA(cudaMemsetAsync(b->d_counter, 0, sizeof(unsigned long long), st));
  dc::ProfScope ps(dc::KID_BP3D, st);
  int rc = DC_OK;
  switch (b->dtype) {
    case DC_F32: rc = launch_batched_t<float>(b, run, st); break;
    case DC_F32X2: rc = launch_batched_t<float2>(b, run, st); break;
    case DC_BF16: rc = launch_batched_t<__nv_bfloat16>(b, run, st); break;
    default: rc = launch_batched_t<__half>(b, run, st); break;
  }
  if (rc) return rc;
  DC_CHECK_LAUNCH("k_bp3d_batched");
  return DC_OK;
}

void dc_batch_destroy(dc_batch *b) { free_batch(b); }

int dc_geometry_set_tuning(dc_geometry *g, int chunk_images, int bp_nz) {
  if (!g) return dc::fail(DC_ERR_ARG, "dc_geometry_set_tuning: NULL geometry");
  if (chunk_images < 0 || chunk_images > g->chunk_capacity)
    return dc::fail(DC_ERR_ARG, "dc_geometry_set_tuning: chunk_images must be in [1, " +
                                    std::to_string(g->chunk_capacity) + "] (0 keeps it)");
  if (bp_nz != 0 && bp_nz != 16 && bp_nz != 32)
    return dc::fail(DC_ERR_ARG, "dc_geometry_set_tuning: bp_nz must be 16 or 32 (0 keeps it)");
  if (chunk_images > 0) g->chunk_images = chunk_images;
  if (bp_nz > 0) g->bp_nz = bp_nz;
  return DC_OK;
}

int dc_geometry_get_tuning(const dc_geometry *g, int *chunk_images, int *chunk_capacity,
                           int *bp_nz) {
  if (!g) return dc::fail(DC_ERR_ARG, "dc_geometry_get_tuning: NULL geometry");
  if (chunk_images) *chunk_images = g->chunk_images;
  if (chunk_capacity) *chunk_capacity = g->chunk_capacity;
  if (bp_nz) *bp_nz = g->bp_nz;
  return DC_OK;
}

}  // extern "C"
