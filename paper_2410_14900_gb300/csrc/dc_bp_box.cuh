// dc_bp_box.cuh -- one box of the shared-memory staged cone-beam
// backprojection, shared by the kernels that stage footprints by TMA
// (dc_backproject.cu) and by rows (dc_backproject_rows.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cstring>
#include <type_traits>

#include "dc_async.cuh"
#include "dc_common.cuh"

namespace {

constexpr int BP_TX = 16, BP_TY = 16;
constexpr int BP_NZ = 16;      // voxels per thread along z
constexpr int BP_VCHUNK = 32;  // views staged in shared memory at a time

struct BPArgs {
  const void *gF;
  const float *scale;  // [B][V] for F16
  const dc::BPView *views;
  float *vol;
  unsigned flags;
  int V, H, W, nx, ny, nz, B;
  float dx, dy, dz;
  int z_begin, z_end;  // voxel planes [z_begin, z_end) of the staged kernels
};

template <typename T>
__device__ __forceinline__ float ld(const T *p);
template <>
__device__ __forceinline__ float ld<float>(const float *p) { return __ldg(p); }
template <>
__device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16 *p) {
  return __bfloat162float(__ldg(p));
}
template <>
__device__ __forceinline__ float ld<__half>(const __half *p) { return __half2float(__ldg(p)); }
// DC_F32X2: the value is the first half of the (g, right difference) pair
template <>
__device__ __forceinline__ float ld<float2>(const float2 *p) {
  return __ldg(reinterpret_cast<const float *>(p));
}

// bilinear interpolation with zero outside the detector
template <typename T>
__device__ __forceinline__ float bilinear(const T *img, int H, int W, float u, float v) {
  u = fminf(fmaxf(u, -2.0f), (float)W + 1.0f);
  v = fminf(fmaxf(v, -2.0f), (float)H + 1.0f);
  float fu, fv;
  int j = dc::floor_frac(u, fu), r = dc::floor_frac(v, fv);
  bool j0 = (j >= 0 && j < W), j1 = (j + 1 >= 0 && j + 1 < W);
  bool r0 = (r >= 0 && r < H), r1 = (r + 1 >= 0 && r + 1 < H);
  const T *p = img + (ptrdiff_t)r * W + j;
  float g00 = (r0 && j0) ? ld(p) : 0.0f;
  float g01 = (r0 && j1) ? ld(p + 1) : 0.0f;
  float g10 = (r1 && j0) ? ld(p + W) : 0.0f;
  float g11 = (r1 && j1) ? ld(p + W + 1) : 0.0f;
  float a = fmaf(fu, g01 - g00, g00);
  float b = fmaf(fu, g11 - g10, g10);
  return fmaf(fv, b - a, a);
}

// ------------------------------------------------------------------------
// Shared-memory staged backprojection.  A CTA owns a 16 x 16 x 32 voxel box.
// For every view the box's eight corners are projected; the bounding box of
// the projections (plus a one-pixel margin) is the footprint of every voxel
// of the box on the detector.  A tiled TMA load copies that footprint
// (a 32x48 or 64x48 box, zero outside the detector) into shared memory
// through a three-stage mbarrier pipeline, and the voxels interpolate from
// shared memory without bounds checks.  Footprints are computed for 32 views
// at a time, one corner per thread.  Views whose footprint does not fit (or
// whose box reaches behind the source) fall back to bounds-checked global
// loads; views whose footprint misses the detector are skipped.
constexpr int TB_TX = 16, TB_TY = 16, TB_NZ = 32;
constexpr int TB_BWN = 32, TB_BWW = 64, TB_BH = 48;
constexpr int TB_NS = 3;
constexpr int TB_VCH = 32;
enum { FP_GLOBAL = 0, FP_NARROW = 1, FP_WIDE = 2, FP_SKIP = 3 };

// How a view's footprint reaches the raw stage:
//   LD_TMA    one tiled TMA load (rows of a multiple of 16 bytes)
//   LD_UNITS  the CTA's threads copy it row by row with asynchronous copies of
//             one FP32 value, one FP32 pair or two aligned 16-bit values, zeros
//             outside the detector: the same stage as the TMA's
//   LD_SHIFT  16-bit rows of any alignment: copies of the 4-byte units that
//             hold the row, one element late where the row starts at an odd
//             half, sorted out (and masked) by the conversion to pairs
enum { LD_TMA = 0, LD_UNITS = 1, LD_SHIFT = 2 };

// With DC_F32X2 storage g^F already holds the (g, right difference) pairs
// of the work tile, so the TMA box itself is the tile, read in place: boxes
// of 40 or 72 pairs give a row stride of 8 mod 16 pairs (the bank spread of
// the converted tile below), and every staged column is usable.
constexpr int TB_PBWN = 40, TB_PBWW = 72;
template <typename T>
struct TileShape {
  static constexpr bool PAIRS = false;
  static constexpr int BWN = TB_BWN, BWW = TB_BWW;
};
template <>
struct TileShape<float2> {
  static constexpr bool PAIRS = true;
  static constexpr int BWN = TB_PBWN, BWW = TB_PBWW;
};

template <typename T>
__device__ __forceinline__ float sld(const T *p);
template <>
__device__ __forceinline__ float sld<float>(const float *p) { return *p; }
template <>
__device__ __forceinline__ float sld<__nv_bfloat16>(const __nv_bfloat16 *p) {
  return __bfloat162float(*p);
}
template <>
__device__ __forceinline__ float sld<__half>(const __half *p) { return __half2float(*p); }

// Shared memory of k_bp3d_tma (dynamic): NS raw TMA stages, then two FP32
// work tiles of tap pairs (g[r][j], g[r][j+1] - g[r][j]) with a row stride
// of TB_S2 float2 (8 mod 16): adjacent rows put one column on different
// banks, a row's linear interpolation is one 64-bit load and one FMA.
// DC_F32X2 storage needs only the stages (the pairs come from g^F).
constexpr int TB_S2 = TB_BWW + 8;
// elements of a raw stage row (LD_SHIFT: one more unit)
template <typename T, int LD>
__host__ __device__ constexpr int bp_raw_pitch(int bw) {
  return LD == LD_SHIFT ? bw + 2 : bw;
}
template <typename T, int LD>
__host__ __device__ constexpr size_t bp_stage_bytes() {
  return (size_t)TB_BH * bp_raw_pitch<T, LD>(TileShape<T>::BWW) * sizeof(T);
}
template <typename T, int LD = LD_TMA>
constexpr size_t bp_smem() {
  return TB_NS * bp_stage_bytes<T, LD>() +
         (TileShape<T>::PAIRS ? 0 : 2 * (size_t)TB_BH * TB_S2 * sizeof(float2));
}

// asynchronous copy of BYTES (4 or 8) or, if !ok, of as many zeros
template <int BYTES>
__device__ __forceinline__ void cp_async_or_zero(void *dst, const void *src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dc::smem_addr(dst)), "l"(src),
               "n"(BYTES), "r"(ok ? BYTES : 0)
               : "memory");
}

// Tap addressing without integer conversions: x + kM rounded toward -inf is
// floor(x) + kM (unit spacing below 2^24), and taking kM off again leaves
// floor(x) as a float.  Byte offsets are then summed as subnormal floats: an
// integer below 2^23 and the float with its bits (the integer times 2^-149)
// are the same number in other units, and an FMA of small integers times such
// strides is exact, so one packed FMA gives the offsets of two voxels.
constexpr float kM = 12582912.0f;  // 1.5 * 2^23

__device__ __forceinline__ float as_subnormal(unsigned bytes) { return __uint_as_float(bytes); }

__device__ __forceinline__ float2 ldpair(const char *sb, unsigned off) {
  return *reinterpret_cast<const float2 *>(sb + off);
}

// packed (two-lane) floor (as a float) and fraction f = x - floor(x), exact
__device__ __forceinline__ void floor_frac2(float2 x, float2 &t, float2 &f) {
  t = __fadd2_rn(__fadd2_rd(x, make_float2(kM, kM)), make_float2(-kM, -kM));
  f = __ffma2_rn(t, make_float2(-1.0f, -1.0f), x);
}

// What bounds it: per update two 8-byte tap pairs (8 updates per clock and SM
// at most: 26.4 ms for 512^3 voxels and 496 views, 73 % of them circle views)
// and about 15.5 instructions.  That volume from FP32 pairs: 38.0 ms when every
// pair of voxels was clamped into its tile (21 instructions per update), 36.3
// without clamps, 34.1 with addresses from packed subnormal FMAs (35.9 with
// integer multiply-adds) and immediate step constants; shared-memory pipe
// 75 %, issue 63 %, FMA pipe 61 %.
//
// One CTA backprojects one box of 16 x 16 x NZ voxels (box indices bxi, byi
// and bzi = batch item * z-blocks + z-block) over every view.  `it` is the
// CTA's running view counter (mbarrier stage and parity), carried across
// boxes by the persistent kernel.  Returns false if a bounded wait gave up.
//
// SPLIT: the CTA takes the views [v_begin, v_end) and leaves its sums in `part`
// ([NZ][threads], shared memory of the staged views, free by then) instead of
// storing voxels.
template <typename T, bool KAHAN, int NZ, int LD = LD_TMA, bool SPLIT = false>
__device__ __forceinline__ bool bp_box(const BPArgs &a, float *vol, const CUtensorMap *tmn,
                                       const CUtensorMap *tmw, unsigned *err, int bxi, int byi,
                                       int bzi, unsigned char *dsm, uint64_t *full,
                                       dc::BPView *sv, int4 *vtab, unsigned &it, int v_begin = 0,
                                       int v_end = 0, float *part = nullptr) {
  if (!SPLIT) v_end = a.V;
  constexpr bool PAIRS = TileShape<T>::PAIRS;
  constexpr int BWN = TileShape<T>::BWN, BWW = TileShape<T>::BWW;
  constexpr size_t STAGE_BYTES = bp_stage_bytes<T, LD>();
  float2 *wtile0 = (float2 *)(dsm + TB_NS * STAGE_BYTES);  // converted tiles (not PAIRS)
  const char *sb = reinterpret_cast<const char *>(dsm);

  const int tid = threadIdx.y * TB_TX + threadIdx.x;
  // each half-warp (the lanes of one 64-bit shared-memory wavefront) takes a
  // 4 x 4 patch of voxel columns: its taps span a few columns and at most two
  // rows of the pair tile, which the row stride maps to distinct banks
  static_assert(TB_TX == 16 && TB_TY == 16, "4 x 4 patches of a 16 x 16 box");
  const int hw = tid >> 4, l16 = tid & 15;
  // A box at the volume's end is moved back inside and stores only the voxels
  // that are its own, so that every box is full (where the volume holds one):
  // its footprint, of the whole box, then holds the taps of every voxel that
  // a thread computes (the projection is a convex image of the box) and no
  // position needs a clamp.
  const int zblocks = (a.z_end - a.z_begin + NZ - 1) / NZ;
  const int b = bzi / zblocks;
  const int x_own = bxi * TB_TX, y_own = byi * TB_TY, z_own = a.z_begin + (bzi % zblocks) * NZ;
  const int x0b = max(min(x_own, a.nx - TB_TX), 0), y0b = max(min(y_own, a.ny - TB_TY), 0);
  const int z0 = max(min(z_own, a.nz - NZ), 0);
  const int ix = x0b + ((hw & 3) << 2) + (l16 & 3);
  const int iy = y0b + ((hw >> 2) << 2) + (l16 >> 2);
  const float cx = 0.5f * (float)(a.nx - 1), cy = 0.5f * (float)(a.ny - 1),
              cz = 0.5f * (float)(a.nz - 1);
  const float xo = ((float)ix - cx) * a.dx;
  const float yo = ((float)iy - cy) * a.dy;
  const float zo = ((float)z0 - cz) * a.dz;
  // extremal voxel centres of this CTA's box
  const float bx0 = ((float)x0b - cx) * a.dx, bx1 = ((float)(x0b + TB_TX - 1) - cx) * a.dx;
  const float by0 = ((float)y0b - cy) * a.dy, by1 = ((float)(y0b + TB_TY - 1) - cy) * a.dy;
  const float bz0 = zo, bz1 = ((float)(z0 + NZ - 1) - cz) * a.dz;
  const size_t np = (size_t)a.H * a.W;
  const T *gbase = (const T *)a.gF + (size_t)b * a.V * np;

  // The column's voxels in pairs: element h of acc2 holds voxels h and
  // h + NH, so that two voxels' positions, floors, weights and sums take one
  // packed FP32x2 operation each (sm_100+; each half rounded as the scalar
  // operation would round it).
  // With KAHAN each view chunk's terms are summed in plain FP32 into acc2,
  // and the chunk sums are added to tot with Kahan compensation (cmp), so
  // the compensated sum runs over the V / TB_VCH chunk sums rather than
  // every view: the FP32 error is that of a TB_VCH-term sum, at 1/TB_VCH of
  // the per-view compensation cost.  The total and its compensation are
  // touched once per chunk, in a rolled loop, and so live in local memory
  // (in registers beside the chunk sum they cost a quarter of the time).
  // Footprints staged by rows (LD != LD_TMA) compensate every view's term, as
  // the kernel for such rows always did; neg2 is the negative of the running
  // compensation (13.8 ms for 128 x 512 x 512 voxels and 400 views of BF16
  // rows, 13.4 with chunk sums).  Without KAHAN terms go to acc2.
  constexpr bool PER_VIEW = KAHAN && LD != LD_TMA, CHUNKED = KAHAN && !PER_VIEW;
  constexpr int NH = NZ / 2;
  float2 acc2[NH], neg2[PER_VIEW ? NH : 1];
  float tot[CHUNKED ? NZ : 1], cmp[CHUNKED ? NZ : 1], prt[CHUNKED ? NZ : 1];
#pragma unroll
  for (int h = 0; h < NH; ++h) acc2[h] = make_float2(0.0f, 0.0f);
  if constexpr (PER_VIEW) {
#pragma unroll
    for (int h = 0; h < NH; ++h) neg2[h] = make_float2(0.0f, 0.0f);
  }
  if (CHUNKED) {
#pragma unroll 1
    for (int k = 0; k < NZ; ++k) tot[k] = cmp[k] = 0.0f;
  }
  // a pair of terms val * wt into voxels (h, h + NH); one term into voxel k
  auto add2 = [&](int h, float2 val, float2 wt) {
    if constexpr (PER_VIEW) {
      const float2 m1 = make_float2(-1.0f, -1.0f);
      const float2 y = __ffma2_rn(val, wt, neg2[h]), t = __fadd2_rn(acc2[h], y);
      neg2[h] = __ffma2_rn(__ffma2_rn(acc2[h], m1, t), m1, y);
      acc2[h] = t;
    } else {
      acc2[h] = __ffma2_rn(val, wt, acc2[h]);
    }
  };
  auto add1 = [&](int k, float term) {
    const int h = k < NH ? k : k - NH;
    float &c = k < NH ? acc2[h].x : acc2[h].y;
    if constexpr (PER_VIEW) {
      float &n = k < NH ? neg2[h].x : neg2[h].y;
      const float y = term + n, t = c + y;
      n = y - (t - c);
      c = t;
    } else {
      c += term;
    }
  };

  bool ok = true;
  for (int c0 = v_begin; c0 < v_end && ok; c0 += TB_VCH) {
    const int nvc = min(TB_VCH, v_end - c0);
    __syncthreads();
    {  // footprints of this chunk: thread = (view, corner)
      const int vi = tid >> 3, cr = tid & 7;
      float umin = 0.0f, umax = 0.0f, vmin = 0.0f, vmax = 0.0f;
      int good = 1;
      if (vi < nvc) {
        const dc::BPView w = a.views[c0 + vi];
        if (cr == 0) sv[vi] = w;
        float X = (cr & 1) ? bx1 : bx0, Y = (cr & 2) ? by1 : by0, Z = (cr & 4) ? bz1 : bz0;
        float U = fmaf(w.r0.x, X, fmaf(w.r0.y, Y, fmaf(w.r0.z, Z, w.r0.w)));
        float Vv = fmaf(w.r1.x, X, fmaf(w.r1.y, Y, fmaf(w.r1.z, Z, w.r1.w)));
        float Wd = fmaf(w.r2.x, X, fmaf(w.r2.y, Y, fmaf(w.r2.z, Z, w.r2.w)));
        good = (Wd > 1.0f);
        float u = good ? U / Wd + w.pp.x : 0.0f, v = good ? Vv / Wd + w.pp.y : 0.0f;
        umin = umax = u;
        vmin = vmax = v;
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        umin = fminf(umin, __shfl_xor_sync(0xffffffffu, umin, o));
        umax = fmaxf(umax, __shfl_xor_sync(0xffffffffu, umax, o));
        vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        good &= __shfl_xor_sync(0xffffffffu, good, o);
      }
      if (vi < nvc && cr == 0) {
        int4 t = make_int4(0, 0, FP_GLOBAL, BWW);
        if (good && fabsf(umin) < 1e6f && fabsf(umax) < 1e6f && fabsf(vmin) < 1e6f &&
            fabsf(vmax) < 1e6f) {
          constexpr int ALIGN = 16 / (int)sizeof(T);  // TMA x offset: 16-byte multiple
          int j0 = (int)floorf(umin) - 1, j1 = (int)floorf(umax) + 2;
          int r0 = (int)floorf(vmin) - 1, r1 = (int)floorf(vmax) + 2;
          int x0 = j0 & ~(ALIGN - 1);
          int ncol = j1 - x0 + 1, nrow = r1 - r0 + 1;
          if (j1 < 0 || x0 >= a.W || r1 < 0 || r0 >= a.H) {
            t = make_int4(x0, r0, FP_SKIP, BWW);
          } else if (nrow <= TB_BH && ncol <= BWN) {
            t = make_int4(x0, r0, FP_NARROW | nrow << 8, BWN);
          } else if (nrow <= TB_BH && ncol <= BWW) {
            t = make_int4(x0, r0, FP_WIDE | nrow << 8, BWW);
          }
        }
        vtab[vi] = t;
      }
    }
    __syncthreads();
    auto issue = [&](int vi, unsigned s) {
      const int4 t = vtab[vi];
      unsigned char *dst = dsm + s * STAGE_BYTES;
      const int type = t.z & 255, nrow = t.z >> 8;
      if constexpr (LD == LD_TMA) {
        dc::fence_proxy_async();
        if (type == FP_NARROW) {
          dc::mbar_arrive_expect_tx(&full[s], BWN * TB_BH * sizeof(T));
          dc::tma_load_3d(dst, tmn, t.x, t.y, b * a.V + c0 + vi, &full[s]);
        } else if (type == FP_WIDE) {
          dc::mbar_arrive_expect_tx(&full[s], BWW * TB_BH * sizeof(T));
          dc::tma_load_3d(dst, tmw, t.x, t.y, b * a.V + c0 + vi, &full[s]);
        } else {
          dc::mbar_arrive(&full[s]);
        }
      } else {
        // a warp copies every eighth row; one group per view, also an empty one
        if (type == FP_NARROW || type == FP_WIDE) {
          const T *img = gbase + (size_t)(c0 + vi) * np;
          const int lane = tid & 31;
          for (int r = tid >> 5; r < nrow; r += (TB_TX * TB_TY) >> 5) {
            const int row = t.y + r;
            const bool rok = row >= 0 && row < a.H;
            const T *src = img + ((ptrdiff_t)row * a.W + t.x);
            if constexpr (LD == LD_UNITS) {
              constexpr int UE = sizeof(T) == 2 ? 2 : 1;  // W and x0 are even for 16-bit units
              for (int c = lane * UE; c < t.w; c += 32 * UE) {
                const bool okc = rok && t.x + c >= 0 && t.x + c < a.W;
                cp_async_or_zero<UE * sizeof(T)>((T *)dst + r * t.w + c, okc ? src + c : gbase, okc);
              }
            } else if (rok) {
              const int sh = (int)(((uintptr_t)src >> 1) & 1);  // 1: the row starts in mid-unit
              unsigned *d = (unsigned *)(dst + (size_t)r * bp_raw_pitch<T, LD>(BWW) * sizeof(T));
              const T *gend = (const T *)a.gF + (size_t)a.B * a.V * np;
              for (int c = lane; c <= t.w >> 1; c += 32) {
                const T *u = src - sh + 2 * c;
                const int col = t.x - sh + 2 * c;
                if (col + 1 < 0 || col >= a.W) continue;  // masked by the conversion
                if (u >= (const T *)a.gF && u + 1 < gend) dc::cp_async4(d + c, u);
                else  // a unit that sticks out of the array
                  for (int q = 0; q < 2; ++q)
                    if (u + q >= (const T *)a.gF && u + q < gend) ((T *)(d + c))[q] = u[q];
              }
            }
          }
        }
        dc::cp_async_commit();
      }
    };
    if (LD != LD_TMA || tid == 0)
      for (int q = 0; q < TB_NS - 1; ++q) {
        if (q < nvc) issue(q, (it + q) % TB_NS);
        else if (LD != LD_TMA) dc::cp_async_commit();
      }

    for (int vi = 0; vi < nvc; ++vi, ++it) {
      const unsigned s = it % TB_NS;
      const int4 t = vtab[vi];
      const int i = c0 + vi;
      float sc = 1.0f;
      if (a.scale) sc = a.scale[(size_t)b * a.V + i];
      bool w_ok = true;
      if constexpr (LD == LD_TMA) {
        w_ok = dc::mbar_wait_bounded(&full[s], (it / TB_NS) & 1, err);
      } else {
        dc::cp_async_wait<TB_NS - 2>();  // this view's group is the oldest but TB_NS - 2
        __syncthreads();
      }
      const int type = t.z & 255, nrow = t.z >> 8;
      float2 *wt = wtile0 + (size_t)(it & 1) * TB_BH * TB_S2;
      // the pair tile (bytes from dsm) and its row stride: the converted tile,
      // or with PAIRS the TMA stage itself (row stride = box width)
      const unsigned wt_off = PAIRS ? s * (unsigned)STAGE_BYTES
                                    : (unsigned)((const unsigned char *)wt - dsm);
      const bool staged = (type == FP_NARROW || type == FP_WIDE);
      if (!PAIRS && w_ok && staged) {
        // raw box -> FP32 pair tile (times the FP16 scale)
        const T *raw = (const T *)(dsm + s * STAGE_BYTES);
        const int bw = t.w;
        if constexpr (sizeof(T) == 4) {
          // four pairs per thread and step: one 16-byte load (+ the next
          // element) and two 16-byte stores
          const int lg = (bw == TB_BWN) ? 3 : 4;  // log2 of the groups per row
          for (int e = tid; e < (nrow * bw) >> 2; e += TB_TX * TB_TY) {
            int r = e >> lg, j4 = (e - (r << lg)) << 2;
            const float *src = (const float *)raw + r * bw + j4;
            float4 v = *(const float4 *)src;
            float nx = (j4 + 4 < bw) ? src[4] : 0.0f;
            float4 *dst = (float4 *)(wt + r * TB_S2 + j4);
            dst[0] = make_float4(v.x, v.y - v.x, v.y, v.z - v.y);
            dst[1] = make_float4(v.z, v.w - v.z, v.w, nx - v.w);
          }
        } else if constexpr (sizeof(T) == 2) {
          // 16-bit storage: four values per 8-byte load, converted (and
          // scaled) to FP32 pairs with two 16-byte stores.  A BF16 value is
          // the upper half of the FP32 with the same bits, so its conversion
          // is a shift or a mask (exact), and BF16 storage has no scale.
          constexpr bool BF = std::is_same<T, __nv_bfloat16>::value;
          const int lg = (bw == TB_BWN) ? 3 : 4;
          for (int e = tid; e < (nrow * bw) >> 2; e += TB_TX * TB_TY) {
            int r = e >> lg, j4 = (e - (r << lg)) << 2;
            const T *src = raw + r * bw + j4;
            float v0, v1, v2, v3, nx;
            if constexpr (LD == LD_SHIFT) {
              const int row = t.y + r, c = t.x + j4;
              const bool rok = row >= 0 && row < a.H;
              const T *g = gbase + (size_t)i * np + ((ptrdiff_t)row * a.W + t.x);
              const T *h = raw + r * bp_raw_pitch<T, LD>(BWW) + (int)(((uintptr_t)g >> 1) & 1) + j4;
              float m[5];
#pragma unroll
              for (int q = 0; q < 5; ++q)
                m[q] = (rok && c + q >= 0 && c + q < a.W && j4 + q < bw) ? sld(h + q) * sc : 0.0f;
              v0 = m[0];
              v1 = m[1];
              v2 = m[2];
              v3 = m[3];
              nx = m[4];
            } else if (BF) {
              const uint2 pk = *(const uint2 *)src;
              v0 = __uint_as_float(pk.x << 16);
              v1 = __uint_as_float(pk.x & 0xffff0000u);
              v2 = __uint_as_float(pk.y << 16);
              v3 = __uint_as_float(pk.y & 0xffff0000u);
              nx = (j4 + 4 < bw)
                       ? __uint_as_float((unsigned)*reinterpret_cast<const unsigned short *>(src + 4)
                                         << 16)
                       : 0.0f;
            } else {
              const uint2 pk = *(const uint2 *)src;
              T h[4];
              memcpy(h, &pk, sizeof(pk));
              v0 = sld(&h[0]) * sc;
              v1 = sld(&h[1]) * sc;
              v2 = sld(&h[2]) * sc;
              v3 = sld(&h[3]) * sc;
              nx = (j4 + 4 < bw) ? sld(src + 4) * sc : 0.0f;
            }
            float4 *dst = (float4 *)(wt + r * TB_S2 + j4);
            dst[0] = make_float4(v0, v1 - v0, v1, v2 - v1);
            dst[1] = make_float4(v2, v3 - v2, v3, nx - v3);
          }
        }
      }
      if constexpr (PAIRS) {
        // the pair left of column 0 (fill zero from the copy) is (0, g[r][0]):
        // its difference is the first column's value, which the tile holds
        // whenever it reaches left of the detector (x0 < 0)
        if (w_ok && staged && t.x < 0 && tid < nrow) {
          float2 *row = reinterpret_cast<float2 *>(dsm + wt_off) + (size_t)tid * t.w;
          row[-1 - t.x].y = row[-t.x].x;
          dc::fence_proxy_async();  // before a later copy into this stage
        }
      }
      if (__syncthreads_or(!w_ok)) {
        ok = false;
        break;
      }
      if (LD != LD_TMA || tid == 0) {
        if (vi + TB_NS - 1 < nvc) issue(vi + TB_NS - 1, (it + TB_NS - 1) % TB_NS);
        else if (LD != LD_TMA) dc::cp_async_commit();
      }
      const dc::BPView w = sv[vi];
      float U0 = fmaf(w.r0.x, xo, fmaf(w.r0.y, yo, fmaf(w.r0.z, zo, w.r0.w)));
      float V0 = fmaf(w.r1.x, xo, fmaf(w.r1.y, yo, fmaf(w.r1.z, zo, w.r1.w)));
      float W0 = fmaf(w.r2.x, xo, fmaf(w.r2.y, yo, fmaf(w.r2.z, zo, w.r2.w)));
      float dU = w.r0.z * a.dz, dV = w.r1.z * a.dz, dW = w.r2.z * a.dz;
      float ex = w.ca.x + xo, ey = w.ca.y + yo, ez0 = w.ca.z + zo;
      float rho2 = fmaf(ex, ex, ey * ey);
      // a staged view, with the tile's row stride RS (bytes) a constant: the
      // second row's taps are an immediate offset from the first's
      auto staged_view = [&](auto rs_const) {
        constexpr unsigned RS = decltype(rs_const)::value;
        const float cul = w.pp.x - (float)t.x, cvl = w.pp.y - (float)t.y;
        const float2 rho22 = make_float2(rho2, rho2), m12 = make_float2(-1.0f, -1.0f);
        const float2 rs2 = make_float2(as_subnormal(RS), as_subnormal(RS));
        // rows' interpolations x0 + fv (x1 - x0) of the two voxels, weighted
        auto sum2 = [&](int h, float2 fu, float2 fv, float2 ad, float2 r2) {
          const unsigned oa = __float_as_uint(ad.x), ob = __float_as_uint(ad.y);
          const float2 a0 = ldpair(sb, oa), a1 = ldpair(sb, oa + RS);
          const float2 b0 = ldpair(sb, ob), b1 = ldpair(sb, ob + RS);
          const float2 x0 = make_float2(fmaf(fu.x, a0.y, a0.x), fmaf(fu.y, b0.y, b0.x));
          const float2 x1 = make_float2(fmaf(fu.x, a1.y, a1.x), fmaf(fu.y, b1.y, b1.x));
          const float2 val = __ffma2_rn(fv, __ffma2_rn(x0, m12, x1), x0);
          add2(h, val, make_float2(dc::rcp_approx(r2.x), dc::rcp_approx(r2.y)));
        };
        // b + k d of voxels k = h and h + NH: scalar FMAs with immediate k (a
        // packed one would need its pair of constants in registers)
        auto at = [](int h, float d, float b) {
          return make_float2(fmaf((float)h, d, b), fmaf((float)(h + NH), d, b));
        };
        if (w.ca.w != 0.0f) {
          // circle view: u and the depth do not change along the column
          const float rw = dc::rcp_approx(W0);
          float fu;
          const int j = dc::floor_frac(fmaf(U0, rw, cul), fu);
          const float2 fu2 = make_float2(fu, fu);
          const float cj = as_subnormal(wt_off + (unsigned)j * 8u);
          const float2 cj2 = make_float2(cj, cj);
          const float vb = fmaf(V0, rw, cvl), dv = dV * rw;
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            const float2 v = at(h, dv, vb), ez = at(h, a.dz, ez0);
            float2 tv, fv;
            floor_frac2(v, tv, fv);
            sum2(h, fu2, fv, __ffma2_rn(tv, rs2, cj2), __ffma2_rn(ez, ez, rho22));
          }
        } else {
          const float2 cul2 = make_float2(cul, cul), cvl2 = make_float2(cvl, cvl);
          const float2 s82 = make_float2(as_subnormal(8u), as_subnormal(8u));
          const float2 cg2 = make_float2(as_subnormal(wt_off), as_subnormal(wt_off));
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            const float2 dep = at(h, dW, W0);
            const float2 rw = make_float2(dc::rcp_approx(dep.x), dc::rcp_approx(dep.y));
            const float2 u = __ffma2_rn(at(h, dU, U0), rw, cul2);
            const float2 v = __ffma2_rn(at(h, dV, V0), rw, cvl2);
            float2 tu, fu, tv, fv;
            floor_frac2(u, tu, fu);
            floor_frac2(v, tv, fv);
            const float2 ez = at(h, a.dz, ez0);
            sum2(h, fu, fv, __ffma2_rn(tv, rs2, __ffma2_rn(tu, s82, cg2)),
                 __ffma2_rn(ez, ez, rho22));
          }
        }
      };
      if (staged) {
        if constexpr (PAIRS) {
          if (t.w == BWN) staged_view(std::integral_constant<unsigned, BWN * 8u>());
          else staged_view(std::integral_constant<unsigned, BWW * 8u>());
        } else {
          staged_view(std::integral_constant<unsigned, TB_S2 * 8u>());
        }
      } else if (type == FP_GLOBAL) {
        const T *img = gbase + (size_t)i * np;
#pragma unroll
        for (int k = 0; k < NZ; ++k) {
          float kf = (float)k;
          float dep = fmaf(kf, dW, W0);
          if (!(dep > 0.0f)) continue;
          float rw = __frcp_rn(dep);
          float u = fmaf(fmaf(kf, dU, U0), rw, w.pp.x);
          float v = fmaf(fmaf(kf, dV, V0), rw, w.pp.y);
          float val = bilinear<T>(img, a.H, a.W, u, v) * sc;
          float ez = fmaf(kf, a.dz, ez0);
          add1(k, val * __frcp_rn(fmaf(ez, ez, rho2)));
        }
      }
    }
    if (CHUNKED && ok) {
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        prt[h] = acc2[h].x;
        prt[h + NH] = acc2[h].y;
        acc2[h] = make_float2(0.0f, 0.0f);
      }
#pragma unroll 1
      for (int k = 0; k < NZ; ++k) {
        const float y = prt[k] - cmp[k];
        const float t = tot[k] + y;
        cmp[k] = (t - tot[k]) - y;
        tot[k] = t;
      }
    }
  }
  if (SPLIT) {
    if constexpr (LD != LD_TMA) dc::cp_async_wait<0>();
    __syncthreads();  // every thread is done with the stages
#pragma unroll
    for (int k = 0; k < NZ; ++k)
      part[k * (TB_TX * TB_TY) + tid] = CHUNKED ? tot[k] : (k < NH) ? acc2[k].x : acc2[k - NH].y;
    return ok;
  }
  if (!ok) return false;
  if (ix < x_own || ix >= a.nx || iy < y_own || iy >= a.ny) return true;
  const size_t nvox = (size_t)a.nx * a.ny * a.nz;
#pragma unroll
  for (int k = 0; k < NZ; ++k) {
    const int iz = z0 + k;
    if (iz < z_own || iz >= a.z_end) continue;
    size_t o = (size_t)b * nvox + ((size_t)iz * a.ny + iy) * a.nx + ix;
    float f = CHUNKED ? tot[k] : (k < NH) ? acc2[k].x : acc2[k - NH].y;
    if (a.flags & DC_ACCUM) f += vol[o];
    if ((a.flags & DC_RELU) && f < 0.0f) f = 0.0f;
    vol[o] = f;
  }
  return true;
}

// The box of a CTA of a whole-volume launch: blockIdx.z = batch item * layers +
// layer.  With 32-deep boxes, a last layer of at most 16 planes takes 16-deep
// ones (half the work, and a footprint of its own size).
__host__ __device__ inline int bp_layers(int z_begin, int z_end, int nz) {
  return (z_end - z_begin + nz - 1) / nz;
}
template <typename T, bool KAHAN, int NZ, int LD>
__device__ __forceinline__ bool bp_layer_box(BPArgs &a, const CUtensorMap *tmn,
                                             const CUtensorMap *tmw, unsigned *err,
                                             unsigned char *dsm, uint64_t *full, dc::BPView *sv,
                                             int4 *vtab) {
  unsigned it = 0;
  if constexpr (NZ == 32) {
    const int layers = bp_layers(a.z_begin, a.z_end, NZ), tail = (a.z_end - a.z_begin) % NZ;
    if (tail > 0 && tail <= 16 && (int)blockIdx.z % layers == layers - 1) {
      a.z_begin = a.z_end - tail;  // one layer per batch item
      return bp_box<T, KAHAN, 16, LD>(a, a.vol, tmn, tmw, err, blockIdx.x, blockIdx.y,
                                      blockIdx.z / layers, dsm, full, sv, vtab, it);
    }
  }
  return bp_box<T, KAHAN, NZ, LD>(a, a.vol, tmn, tmw, err, blockIdx.x, blockIdx.y, blockIdx.z, dsm,
                                  full, sv, vtab, it);
}

// ------------------------------------------------------------------------
// Volumes of few boxes (64^3: 64 of them for 152 SMs) have their views split
// over the CTAs of a cluster: each sums its share of the views into shared
// memory, and after a cluster barrier the first adds the others' sums, in rank
// order (compensated with KAHAN), and stores.  The split is a property of the
// geometry, so that a result does not depend on batch or slab.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// the float at shared address `addr` of CTA `rank` of this cluster
__device__ __forceinline__ float ld_cluster(unsigned addr, unsigned rank) {
  unsigned r;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(r) : "memory");
  return v;
}

// The cluster's part of a split box: blockIdx.z = box * split + rank.
template <typename T, bool KAHAN, int NZ, int LD>
__device__ __forceinline__ void bp_split_box(const BPArgs &a, const CUtensorMap *tmn,
                                             const CUtensorMap *tmw, unsigned *err, int split,
                                             unsigned char *dsm, uint64_t *full, dc::BPView *sv,
                                             int4 *vtab, int *good) {
  static_assert(NZ * TB_TX * TB_TY * sizeof(float) <= TB_NS * bp_stage_bytes<T, LD>() +
                                                          (TileShape<T>::PAIRS ? 0 : 2 * TB_BH * TB_S2 * 8),
                "the partial sums reuse the staged views' memory");
  const int rank = blockIdx.z % split, bzi = blockIdx.z / split;
  const int tid = threadIdx.y * TB_TX + threadIdx.x;
  float *part = reinterpret_cast<float *>(dsm);
  unsigned it = 0;
  const bool ok = bp_box<T, KAHAN, NZ, LD, true>(
      a, a.vol, tmn, tmw, err, blockIdx.x, blockIdx.y, bzi, dsm, full, sv, vtab, it,
      (int)((long long)a.V * rank / split), (int)((long long)a.V * (rank + 1) / split), part);
  if (tid == 0) *good = ok;
  if (LD == LD_TMA && !ok)
    for (int q = 0; q < TB_NS; ++q) dc::mbar_wait_bounded(&full[q], 0, nullptr);
  cluster_sync();
  if (rank == 0) {
    int all = 1;
    for (int r = 0; r < split; ++r)
      all &= __float_as_int(ld_cluster(dc::smem_addr(good), (unsigned)r));
    const int hw = tid >> 4, l16 = tid & 15;
    const int zblocks = (a.z_end - a.z_begin + NZ - 1) / NZ, b = bzi / zblocks;
    const int x_own = blockIdx.x * TB_TX, y_own = blockIdx.y * TB_TY,
              z_own = a.z_begin + (bzi % zblocks) * NZ;
    const int ix = max(min(x_own, a.nx - TB_TX), 0) + ((hw & 3) << 2) + (l16 & 3);
    const int iy = max(min(y_own, a.ny - TB_TY), 0) + ((hw >> 2) << 2) + (l16 >> 2);
    const int z0 = max(min(z_own, a.nz - NZ), 0);
    if (all && ix >= x_own && ix < a.nx && iy >= y_own && iy < a.ny) {
      for (int k = 0; k < NZ; ++k) {
        const int iz = z0 + k;
        if (iz < z_own || iz >= a.z_end) continue;
        const unsigned ad = dc::smem_addr(part + k * (TB_TX * TB_TY) + tid);
        float f = ld_cluster(ad, 0), cmp = 0.0f;
        for (int r = 1; r < split; ++r) {
          const float y = ld_cluster(ad, (unsigned)r) - cmp, t = f + y;
          if (KAHAN) cmp = (t - f) - y;
          f = t;
        }
        const size_t o = (size_t)b * a.nx * a.ny * a.nz + ((size_t)iz * a.ny + iy) * a.nx + ix;
        if (a.flags & DC_ACCUM) f += a.vol[o];
        if ((a.flags & DC_RELU) && f < 0.0f) f = 0.0f;
        a.vol[o] = f;
      }
    }
  }
  cluster_sync();  // no CTA ends while its sums are read
}

// launch of a split kernel: grid.z boxes times `split` CTAs, `split` per cluster
template <typename... KArgs, typename... Args>
inline cudaError_t launch_split(void (*kernel)(KArgs...), dim3 grid, size_t smem, cudaStream_t st,
                                int split, Args... args) {
  cudaLaunchConfig_t c = {};
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = at.val.clusterDim.y = 1;
  at.val.clusterDim.z = split;
  grid.z *= split;
  c.gridDim = grid;
  c.blockDim = dim3(TB_TX, TB_TY);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

inline BPArgs bp_args(const dc_geometry *g, int B, const void *gF, int dtype, const float *gF_scale,
               float *vol, unsigned flags) {
  const dc_geometry_desc &d = g->d;
  BPArgs a;
  a.gF = gF;
  a.scale = (dtype == DC_F16) ? gF_scale : nullptr;
  a.views = g->bpv;
  a.vol = vol;
  a.flags = flags;
  a.V = d.n_views;
  a.H = d.det_rows;
  a.W = d.det_cols;
  a.nx = d.vol_x;
  a.ny = d.vol_y;
  a.nz = d.vol_z;
  a.z_begin = 0;
  a.z_end = d.vol_z;
  a.B = B;
  a.dx = (float)d.voxel[0];
  a.dy = (float)d.voxel[1];
  a.dz = (float)d.voxel[2];
  return a;
}

}  // namespace
