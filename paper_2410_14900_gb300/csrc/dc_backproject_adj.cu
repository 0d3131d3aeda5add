// dc_backproject_adj.cu -- the transpose of the voxel-driven cone-beam
// backprojection (Ye et al., DRACO, Sec. 2.3: the reverse mode of Eq. 5).
#include <algorithm>
#include <cstdlib>
#include <string>

#include "dc_bp_box.cuh"

namespace {

struct BPAdjArgs {
  const float *grad_vol;
  const float *relu_vol;
  const dc::BPView *views;
  float *grad_gF;
  int V, H, W, nx, ny, nz, B;
  float dx, dy, dz;
};

// transpose: every voxel scatters its weighted gradient onto the four taps
__global__ void __launch_bounds__(BP_TX *BP_TY) k_bp3d_adj(BPAdjArgs a) {
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
  const size_t nvox = (size_t)a.nx * a.ny * a.nz;
  const bool inside = (ix < a.nx && iy < a.ny);
  float gv[BP_NZ];
#pragma unroll
  for (int k = 0; k < BP_NZ; ++k) {
    int iz = z0 + k;
    gv[k] = 0.0f;
    if (inside && iz < a.nz) {
      size_t o = (size_t)b * nvox + ((size_t)iz * a.ny + iy) * a.nx + ix;
      float g = a.grad_vol[o];
      if (a.relu_vol && !(a.relu_vol[o] > 0.0f)) g = 0.0f;
      gv[k] = g;
    }
  }
  float *gbase = a.grad_gF + (size_t)b * a.V * np;
  for (int i0 = 0; i0 < a.V; i0 += BP_VCHUNK) {
    int nvc = min(BP_VCHUNK, a.V - i0);
    __syncthreads();
    if (tid < nvc) sv[tid] = a.views[i0 + tid];
    __syncthreads();
    if (!inside) continue;
    for (int ii = 0; ii < nvc; ++ii) {
      const dc::BPView w = sv[ii];
      float *img = gbase + (size_t)(i0 + ii) * np;
      float U0 = fmaf(w.r0.x, xo, fmaf(w.r0.y, yo, fmaf(w.r0.z, zo, w.r0.w)));
      float V0 = fmaf(w.r1.x, xo, fmaf(w.r1.y, yo, fmaf(w.r1.z, zo, w.r1.w)));
      float W0 = fmaf(w.r2.x, xo, fmaf(w.r2.y, yo, fmaf(w.r2.z, zo, w.r2.w)));
      float dU = w.r0.z * a.dz, dV = w.r1.z * a.dz, dW = w.r2.z * a.dz;
      float ex = w.ca.x + xo, ey = w.ca.y + yo, ez0 = w.ca.z + zo;
      float rho2 = fmaf(ex, ex, ey * ey);
#pragma unroll
      for (int k = 0; k < BP_NZ; ++k) {
        if (gv[k] == 0.0f) continue;
        float kf = (float)k;
        float dep = fmaf(kf, dW, W0);
        if (!(dep > 0.0f)) continue;
        float rw = __frcp_rn(dep);
        float u = fmaf(fmaf(kf, dU, U0), rw, w.pp.x);
        float v = fmaf(fmaf(kf, dV, V0), rw, w.pp.y);
        float ez = fmaf(kf, a.dz, ez0);
        float g = gv[k] * __frcp_rn(fmaf(ez, ez, rho2));
        u = fminf(fmaxf(u, -2.0f), (float)a.W + 1.0f);
        v = fminf(fmaxf(v, -2.0f), (float)a.H + 1.0f);
        float fu, fv;
        int j = dc::floor_frac(u, fu), r = dc::floor_frac(v, fv);
        bool j0 = (j >= 0 && j < a.W), j1 = (j + 1 >= 0 && j + 1 < a.W);
        bool r0 = (r >= 0 && r < a.H), r1 = (r + 1 >= 0 && r + 1 < a.H);
        float *p = img + (ptrdiff_t)r * a.W + j;
        if (r0 && j0) atomicAdd(p, g * (1.0f - fu) * (1.0f - fv));
        if (r0 && j1) atomicAdd(p + 1, g * fu * (1.0f - fv));
        if (r1 && j0) atomicAdd(p + a.W, g * (1.0f - fu) * fv);
        if (r1 && j1) atomicAdd(p + a.W + 1, g * fu * fv);
      }
    }
  }
}

// ------------------------------------------------------------------------
// Transpose of the staged backprojection.  Same CTA boxes and footprints as
// the forward kernel; for every view the CTA's voxels scatter their weighted
// gradients into a shared-memory footprint tile, which is then added to g^F's
// gradient with one global atomic per four pixels (or per pixel where rows are
// not 16-byte multiples).  Two tiles alternate: a view's tile is flushed while
// the next view scatters into the other, one barrier per view.
//
// The tile accumulates in 32-bit fixed point, because integer shared-memory
// atomics are native while floating-point ones are not.  The unit is chosen
// per (box, view) from a rigorous bound on any pixel sum: every voxel's four
// bilinear weights sum to one, so a pixel gets at most the box's total,
// sum_box |g| / d_min^2, with d_min the source's distance to the box (centre
// distance minus half-diagonal).  That bound maps to 2^30, so the sums cannot
// overflow; each contribution is rounded to the nearest unit.
//
// Bound by the shared atomics: a bare loop of four per voxel runs at 8.1e11
// voxels/s, 29.8 ms for 4 x 256^3 voxels and 360 views.  With 55 instructions
// per voxel that took 44.9 ms; two voxels of a column stepped together in packed
// FP32x2, without clamps (full boxes, as in the forward kernel), take 30
// instructions; with float4 atomics into g^F's gradient (scalar ones: 5 ms
// more) and three CTAs per SM (two: 0.5 to 1 ms more) 32.2 ms, and without the
// atomics of zero gradients (half of the voxels there, behind the ReLU) 30.1 ms.
// Merging a column's consecutive voxels, which mostly share a detector row,
// saves up to half of the atomics but wants the others predicated: 43 to 52 ms.
//
// Boxes are 32 deep, or 16 where 32-deep ones mostly do not fit the tile and
// would scatter into global memory (214^2 x 178 voxels of 1.4 pixels, 86 views:
// 5.2 ms, here 1.3).
//
// Three CTAs per SM take 80 registers and spill; two take 128 and do not.  For
// voxels finer than 0.75 pixels, whose atomics meet in the same pixels, the
// third CTA does not pay for that: 128^3 voxels, 200 views of 256 x 256, dense
// gradient, three CTAs 1921, 1013 and 833 us at 0.1, 0.3 and 0.7 pixels per
// voxel, two 1872, 952 and 783; behind a mask 1216, 784 and 749 against 1135,
// 732 and 687.  At 1 pixel two cost 0.6 % behind a mask; where three hold every box
// at once (100 x 100 x 33 voxels, 0.5 pixels: 322 us) two cost 25 %.
constexpr double TA_FINE = 0.75;
constexpr int TA_S = 68;  // row stride: 16-byte rows (69: 34.0 ms)
static_assert(TA_S >= TB_BWW + 3, "a tile row holds the widest footprint from an aligned column");

// four taps: pixel pairs at addr and one tile row below
__device__ __forceinline__ void red_add4(unsigned addr, int i00, int i01, int i10, int i11) {
  asm volatile(
      "red.shared.add.s32 [%0], %1;\n\t"
      "red.shared.add.s32 [%0+4], %2;\n\t"
      "red.shared.add.s32 [%0+%5], %3;\n\t"
      "red.shared.add.s32 [%0+%6], %4;" ::"r"(addr),
      "r"(i00), "r"(i01), "r"(i10), "r"(i11), "n"(4 * TA_S), "n"(4 * TA_S + 4)
      : "memory");
}

template <bool VEC4, int NZ, int CTAS>
__global__ void __launch_bounds__(TB_TX *TB_TY, CTAS) k_bp3d_adj_tile(BPAdjArgs a, int split) {
  constexpr int NH = NZ / 2;  // a step takes voxels NH apart
  __shared__ __align__(16) int tiles[2][TB_BH * TA_S];
  __shared__ dc::BPView sv[TB_VCH];
  __shared__ int4 vtab[TB_VCH];
  __shared__ float wsum[TB_TX * TB_TY / 32];
  __shared__ float wmax[TB_TX * TB_TY / 32];
  const int tid = threadIdx.y * TB_TX + threadIdx.x;
  const int zblocks = (a.nz + NZ - 1) / NZ;
  // blockIdx.z = box * split + share of the views
  const int bz = blockIdx.z / split, part = blockIdx.z % split, b = bz / zblocks;
  const int v_begin = (int)((long long)a.V * part / split),
            v_end = (int)((long long)a.V * (part + 1) / split);
  // full boxes: one at the volume's end is moved back inside and takes the
  // gradients of its own voxels only (see bp_box)
  const int x_own = blockIdx.x * TB_TX, y_own = blockIdx.y * TB_TY;
  const int z_own = (bz % zblocks) * NZ;
  const int x0b = max(min(x_own, a.nx - TB_TX), 0), y0b = max(min(y_own, a.ny - TB_TY), 0);
  const int z0 = max(min(z_own, a.nz - NZ), 0);
  const int ix = x0b + threadIdx.x, iy = y0b + threadIdx.y;
  const float cx = 0.5f * (float)(a.nx - 1), cy = 0.5f * (float)(a.ny - 1),
              cz = 0.5f * (float)(a.nz - 1);
  const float xo = ((float)ix - cx) * a.dx;
  const float yo = ((float)iy - cy) * a.dy;
  const float zo = ((float)z0 - cz) * a.dz;
  const float bx0 = ((float)x0b - cx) * a.dx, bx1 = ((float)(x0b + TB_TX - 1) - cx) * a.dx;
  const float by0 = ((float)y0b - cy) * a.dy, by1 = ((float)(y0b + TB_TY - 1) - cy) * a.dy;
  const float bz0 = zo, bz1 = ((float)(z0 + NZ - 1) - cz) * a.dz;
  // box centre and half-diagonal (for the distance bound)
  const float bcx = 0.5f * (bx0 + bx1), bcy = 0.5f * (by0 + by1), bcz = 0.5f * (bz0 + bz1);
  const float bhd = 0.5f * sqrtf((bx1 - bx0) * (bx1 - bx0) + (by1 - by0) * (by1 - by0) +
                                 (bz1 - bz0) * (bz1 - bz0)) + 0.5f * (a.dx + a.dy + a.dz);
  const size_t np = (size_t)a.H * a.W;
  const size_t nvox = (size_t)a.nx * a.ny * a.nz;
  const bool own = ix >= x_own && ix < a.nx && iy >= y_own && iy < a.ny;
  // Step k takes the column's voxels kz and kz + NH with kz = (k + lane) mod NH,
  // every second NH lanes in the other order: at each step NZ neighbouring lanes
  // are at NZ different depths, so lanes whose columns project to the same
  // detector column (columns lined up with the view direction) hit different
  // detector rows.  The fixed-point sums are exact, so the order does not
  // change the result.
  const int rot = tid & (NH - 1), off = tid & NH;
  const float flip = off ? -(float)NH : (float)NH;
  float2 gv[NH];
  float gs = 0.0f, gm = 0.0f;
#pragma unroll
  for (int k = 0; k < NH; ++k) {
    const int kz = ((k + rot) & (NH - 1)) + off;
    float g[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int iz = z0 + (kz ^ (NH * h));
      g[h] = 0.0f;
      if (own && iz >= z_own && iz < a.nz) {
        const size_t o = (size_t)b * nvox + ((size_t)iz * a.ny + iy) * a.nx + ix;
        g[h] = a.grad_vol[o];
        if (a.relu_vol && !(a.relu_vol[o] > 0.0f)) g[h] = 0.0f;
      }
      gs += fabsf(g[h]);
      gm = fmaxf(gm, fabsf(g[h]));
    }
    gv[k] = make_float2(g[0], g[1]);
  }
  const bool any = __any_sync(0xffffffffu, gs > 0.0f);
  for (int o = 16; o > 0; o >>= 1) {
    gs += __shfl_xor_sync(0xffffffffu, gs, o);
    gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
  }
  if ((tid & 31) == 0) {
    wsum[tid >> 5] = gs;
    wmax[tid >> 5] = gm;
  }
  for (int e = tid; e < 2 * TB_BH * TA_S; e += TB_TX * TB_TY) (&tiles[0][0])[e] = 0;
  __syncthreads();
  float gsum = 0.0f, gmax = 0.0f;
  for (int q = 0; q < TB_TX * TB_TY / 32; ++q) {
    gsum += wsum[q];
    gmax = fmaxf(gmax, wmax[q]);
  }
  gsum *= 1.0001f;  // headroom for the rounding of this sum
  if (!(gsum > 0.0f)) return;  // nothing to scatter from this box (CTA-uniform)
  // One contribution is at most gmax / d^2 <= gmax / dmin^2, i.e. at most
  // 2^30 gmax / gsum units.  When the box's gradient is spread over at least
  // 512 voxels' worth of its largest value, every contribution stays below
  // 2^21 units and is rounded to an integer by adding 1.5 * 2^23 (the sum
  // has unit spacing, and round-to-nearest-even is the same rounding as
  // __float2int_rn) instead of a conversion instruction.  CTA-uniform.
  const bool magic_round = gsum >= 512.0f * gmax;
  float *gbase = a.grad_gF + (size_t)b * a.V * np;

  // The pending tile: the last scattered view's, flushed while the next view
  // scatters into the other tile.  Its footprint rectangle (columns pt.w &
  // 255, rows pt.w >> 8) holds every tap of the view (one pixel of margin on
  // each side of the projected box), so flushing it clears the whole tile.
  int cur = 0;
  bool pending = false;
  int4 pt = make_int4(0, 0, 0, 0);
  float p_from_fix = 0.0f;
  float *p_img = nullptr;
  auto flush_pending = [&]() {
    int *T = tiles[cur ^ 1];
    const int nc = pt.w & 255, nr = pt.w >> 8;
    if (VEC4) {  // pt.x and W are multiples of 4: a quad is inside or outside as a whole
      const int nq = (nc + 3) >> 2, lg = nq <= 8 ? 3 : nq <= 16 ? 4 : 5;
      const int c = tid & ((1 << lg) - 1);
      const int jj = pt.x + 4 * c;
      if (c >= nq) return;
      for (int r = tid >> lg; r < nr; r += (TB_TX * TB_TY) >> lg) {
        int4 *t4 = reinterpret_cast<int4 *>(T + r * TA_S + 4 * c);
        const int4 q = *t4;
        if ((q.x | q.y | q.z | q.w) == 0) continue;
        *t4 = make_int4(0, 0, 0, 0);
        const int rr = pt.y + r;
        if (jj >= 0 && jj < a.W && rr >= 0 && rr < a.H)
          atomicAdd(reinterpret_cast<float4 *>(p_img + (size_t)rr * a.W + jj),
                    make_float4((float)q.x * p_from_fix, (float)q.y * p_from_fix,
                                (float)q.z * p_from_fix, (float)q.w * p_from_fix));
      }
      return;
    }
    for (int c = tid & 31; c < nc; c += 32) {
      const int jj = pt.x + c;
      for (int r = tid >> 5; r < nr; r += (TB_TX * TB_TY) >> 5) {
        const int q = T[r * TA_S + c];
        if (q != 0) {
          T[r * TA_S + c] = 0;
          const int rr = pt.y + r;
          if (jj >= 0 && jj < a.W && rr >= 0 && rr < a.H)
            atomicAdd(p_img + (size_t)rr * a.W + jj, (float)q * p_from_fix);
        }
      }
    }
  };

  for (int c0 = v_begin; c0 < v_end; c0 += TB_VCH) {
    const int nvc = min(TB_VCH, v_end - c0);
    __syncthreads();
    {  // footprints: thread = (view, corner), as in the forward kernel
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
        int4 t = make_int4(0, 0, FP_GLOBAL, TB_BWW);
        if (good && fabsf(umin) < 1e6f && fabsf(umax) < 1e6f && fabsf(vmin) < 1e6f &&
            fabsf(vmax) < 1e6f) {
          int x0 = (int)floorf(umin) - 1, x1 = (int)floorf(umax) + 2;
          int r0 = (int)floorf(vmin) - 1, r1 = (int)floorf(vmax) + 2;
          const bool fits = r1 - r0 + 1 <= TB_BH && x1 - x0 + 1 <= TB_BWW;
          if (VEC4) x0 &= ~3;
          if (x1 < 0 || x0 >= a.W || r1 < 0 || r0 >= a.H)
            t = make_int4(x0, r0, FP_SKIP, 0);
          else if (fits)
            t = make_int4(x0, r0, FP_WIDE, (x1 - x0 + 1) | ((r1 - r0 + 1) << 8));
        }
        vtab[vi] = t;
      }
    }
    __syncthreads();
    for (int vi = 0; vi < nvc; ++vi) {
      int4 t = vtab[vi];
      if (t.z == FP_SKIP) continue;
      const dc::BPView w = sv[vi];
      float *img = gbase + (size_t)(c0 + vi) * np;
      const float U0 = fmaf(w.r0.x, xo, fmaf(w.r0.y, yo, fmaf(w.r0.z, zo, w.r0.w)));
      const float V0 = fmaf(w.r1.x, xo, fmaf(w.r1.y, yo, fmaf(w.r1.z, zo, w.r1.w)));
      const float W0 = fmaf(w.r2.x, xo, fmaf(w.r2.y, yo, fmaf(w.r2.z, zo, w.r2.w)));
      const float dU = w.r0.z * a.dz, dV = w.r1.z * a.dz, dW = w.r2.z * a.dz;
      const float ex = w.ca.x + xo, ey = w.ca.y + yo, ez0 = w.ca.z + zo;
      const float rho2 = fmaf(ex, ex, ey * ey);
      // fixed-point unit of this (box, view); CTA-uniform
      const float dcx = w.ca.x + bcx, dcy = w.ca.y + bcy, dcz = w.ca.z + bcz;
      const float dmin = sqrtf(dcx * dcx + dcy * dcy + dcz * dcz) - bhd;
      if (t.z == FP_WIDE && !(dmin > 1.0f)) t.z = FP_GLOBAL;
      if (t.z == FP_WIDE) {
        const float bound = gsum / (dmin * dmin);             // >= any pixel sum
        const float to_fix = 1073741824.0f / bound;            // bound -> 2^30
        const float from_fix = bound * (1.0f / 1073741824.0f);
        const unsigned tb = dc::smem_addr(tiles[cur]);
        const float2 m12 = make_float2(-1.0f, -1.0f), M2 = make_float2(kM, kM);
        const float2 cul2 = make_float2(w.pp.x - (float)t.x, w.pp.x - (float)t.x);
        const float2 cvl2 = make_float2(w.pp.y - (float)t.y, w.pp.y - (float)t.y);
        const float2 U02 = make_float2(U0, U0), dU2 = make_float2(dU, dU);
        const float2 V02 = make_float2(V0, V0), dV2 = make_float2(dV, dV);
        const float2 W02 = make_float2(W0, W0), dW2 = make_float2(dW, dW);
        const float2 ez02 = make_float2(ez0, ez0), dz2 = make_float2(a.dz, a.dz);
        const float2 rho22 = make_float2(rho2, rho2), fix2 = make_float2(to_fix, to_fix);
        const float2 rs2 = make_float2(as_subnormal(4u * TA_S), as_subnormal(4u * TA_S));
        const float2 s42 = make_float2(as_subnormal(4u), as_subnormal(4u));
        const float2 tb2 = make_float2(as_subnormal(tb), as_subnormal(tb));
        auto scatter = [&](auto magic) {
          float kf = (float)(rot + off);
#pragma unroll
          for (int k = 0; k < NH; ++k) {
            const float2 kf2 = make_float2(kf, kf + flip);  // voxels kz, kz ^ NH
            kf += 1.0f;
            if (((k + 1 + rot) & (NH - 1)) == 0) kf -= (float)NH;
            const float2 dep = __ffma2_rn(kf2, dW2, W02);
            const float2 rw = make_float2(dc::rcp_approx(dep.x), dc::rcp_approx(dep.y));
            const float2 u = __ffma2_rn(__ffma2_rn(kf2, dU2, U02), rw, cul2);
            const float2 v = __ffma2_rn(__ffma2_rn(kf2, dV2, V02), rw, cvl2);
            float2 tu, fu, tv, fv;
            floor_frac2(u, tu, fu);
            floor_frac2(v, tv, fv);
            const float2 ad = __ffma2_rn(tv, rs2, __ffma2_rn(tu, s42, tb2));
            const float2 ez = __ffma2_rn(kf2, dz2, ez02);
            const float2 r2 = __ffma2_rn(ez, ez, rho22);
            const float2 wt = make_float2(dc::rcp_approx(r2.x), dc::rcp_approx(r2.y));
            const float2 g = __fmul2_rn(__fmul2_rn(gv[k], wt), fix2);
            const float2 g1 = __fmul2_rn(g, fv), g0 = __ffma2_rn(g1, m12, g);
            const float2 g01 = __fmul2_rn(g0, fu), g11 = __fmul2_rn(g1, fu);
            const float2 g00 = __ffma2_rn(g01, m12, g0), g10 = __ffma2_rn(g11, m12, g1);
            int i00[2], i01[2], i10[2], i11[2];
            if constexpr (decltype(magic)::value) {
              auto bits = [&](float2 x, int *o) {  // |x| < 2^22
                const float2 y = __fadd2_rn(x, M2);
                o[0] = __float_as_int(y.x) - 0x4B400000;
                o[1] = __float_as_int(y.y) - 0x4B400000;
              };
              bits(g00, i00);
              bits(g01, i01);
              bits(g10, i10);
              bits(g11, i11);
            } else {
              i00[0] = __float2int_rn(g00.x), i00[1] = __float2int_rn(g00.y);
              i01[0] = __float2int_rn(g01.x), i01[1] = __float2int_rn(g01.y);
              i10[0] = __float2int_rn(g10.x), i10[1] = __float2int_rn(g10.y);
              i11[0] = __float2int_rn(g11.x), i11[1] = __float2int_rn(g11.y);
            }
            // a masked voxel's zeros would only take atomics (and collide)
            if (gv[k].x != 0.0f)
              red_add4(__float_as_uint(ad.x), i00[0], i01[0], i10[0], i11[0]);
            if (gv[k].y != 0.0f)
              red_add4(__float_as_uint(ad.y), i00[1], i01[1], i10[1], i11[1]);
          }
        };
        if (any) {
          if (magic_round) scatter(std::true_type());
          else scatter(std::false_type());
        }
        // the previous view's tile (complete since the last barrier) to g^F's
        // gradient, cleared for the view after this one
        if (pending) flush_pending();
        __syncthreads();
        pending = true;
        pt = t;
        p_from_fix = from_fix;
        p_img = img;
        cur ^= 1;
      } else if (any) {
#pragma unroll
        for (int k = 0; k < NZ; ++k) {
          const float gk = (k & NH) ? gv[k & (NH - 1)].y : gv[k & (NH - 1)].x;
          if (gk == 0.0f) continue;
          const float kf = (float)((((k & (NH - 1)) + rot) & (NH - 1)) + (off ^ (k & NH)));
          float dep = fmaf(kf, dW, W0);
          if (!(dep > 0.0f)) continue;
          float rw = __frcp_rn(dep);
          float u = fmaf(fmaf(kf, dU, U0), rw, w.pp.x);
          float v = fmaf(fmaf(kf, dV, V0), rw, w.pp.y);
          float ez = fmaf(kf, a.dz, ez0);
          float g = gk * __frcp_rn(fmaf(ez, ez, rho2));
          u = fminf(fmaxf(u, -2.0f), (float)a.W + 1.0f);
          v = fminf(fmaxf(v, -2.0f), (float)a.H + 1.0f);
          float fu, fv;
          int j = dc::floor_frac(u, fu), r = dc::floor_frac(v, fv);
          bool j0 = (j >= 0 && j < a.W), j1 = (j + 1 >= 0 && j + 1 < a.W);
          bool r0 = (r >= 0 && r < a.H), r1 = (r + 1 >= 0 && r + 1 < a.H);
          float *p = img + (ptrdiff_t)r * a.W + j;
          if (r0 && j0) atomicAdd(p, g * (1.0f - fu) * (1.0f - fv));
          if (r0 && j1) atomicAdd(p + 1, g * fu * (1.0f - fv));
          if (r1 && j0) atomicAdd(p + a.W, g * (1.0f - fu) * fv);
          if (r1 && j1) atomicAdd(p + a.W + 1, g * fu * fv);
        }
      }
    }
  }
  if (pending) flush_pending();  // its scatter ended at the last barrier
}

}  // namespace

extern "C" int dc_backproject_adjoint(const dc_geometry *g, int B, const float *grad_vol,
                                      const float *relu_vol, float *grad_gF, void *stream) {
  if (!g) return dc::fail(DC_ERR_ARG, "dc_backproject_adjoint: NULL geometry");
  if (B < 1) return dc::fail(DC_ERR_ARG, "dc_backproject_adjoint: batch must be >= 1");
  int dev = -1;
  cudaGetDevice(&dev);
  if (dev != g->device)
    return dc::fail(DC_ERR_ARG, "dc_backproject_adjoint: geometry belongs to another device");
  if (!grad_vol || !grad_gF)
    return dc::fail(DC_ERR_ARG, "dc_backproject_adjoint: NULL grad_vol or grad_gF");
  const dc_geometry_desc &d = g->d;
  cudaStream_t st = (cudaStream_t)stream;
  DC_CUDA(cudaMemsetAsync(grad_gF, 0,
                          sizeof(float) * (size_t)B * d.n_views * d.det_rows * d.det_cols, st));
  BPAdjArgs a;
  a.grad_vol = grad_vol;
  a.relu_vol = relu_vol;
  a.views = g->bpv;
  a.grad_gF = grad_gF;
  a.V = d.n_views;
  a.H = d.det_rows;
  a.W = d.det_cols;
  a.nx = d.vol_x;
  a.ny = d.vol_y;
  a.nz = d.vol_z;
  a.B = B;
  a.dx = (float)d.voxel[0];
  a.dy = (float)d.voxel[1];
  a.dz = (float)d.voxel[2];
  dim3 blk(BP_TX, BP_TY);
  dim3 grid((d.vol_x + BP_TX - 1) / BP_TX, (d.vol_y + BP_TY - 1) / BP_TY,
            ((d.vol_z + BP_NZ - 1) / BP_NZ) * B);
  dc::ProfScope ps(dc::KID_BP3D_ADJ, st);
  if (getenv("DC_BP_ADJ_GLOBAL")) {
    k_bp3d_adj<<<grid, blk, 0, st>>>(a);
  } else {
    // 16-deep boxes where 32-deep ones mostly do not fit the tile (and would
    // scatter into global memory): bp_plan's judgement
    const int nz = g->bp_fit32 || d.vol_z > 16 * 65535 ? 32 : 16;
    const int layers = (d.vol_z + nz - 1) / nz;
    dim3 gridt((d.vol_x + TB_TX - 1) / TB_TX, (d.vol_y + TB_TY - 1) / TB_TY);
    // few boxes share their views among CTAs (a view's gradient is summed by
    // atomics anyway), up to the three CTAs that an SM holds and down to 8
    // views each
    const long boxes = (long)gridt.x * gridt.y * layers * B;
    int split = 1;
    while (split < 16 && 2 * split * boxes <= 3 * g->sms && d.n_views >= 16 * split) split *= 2;
    // float4 atomics need 16-byte pixel quads
    const bool vec = (a.W & 3) == 0 && ((uintptr_t)grad_gF & 15) == 0;
    const bool fine = g->bp_px < TA_FINE && split * boxes > 3 * g->sms;
    auto pick = [&](auto k32, auto k32f, auto k16, auto k16f) {
      return nz == 32 ? (fine ? k32f : k32) : (fine ? k16f : k16);
    };
    auto kernel = vec ? pick(k_bp3d_adj_tile<true, 32, 3>, k_bp3d_adj_tile<true, 32, 2>,
                             k_bp3d_adj_tile<true, 16, 3>, k_bp3d_adj_tile<true, 16, 2>)
                      : pick(k_bp3d_adj_tile<false, 32, 3>, k_bp3d_adj_tile<false, 32, 2>,
                             k_bp3d_adj_tile<false, 16, 3>, k_bp3d_adj_tile<false, 16, 2>);
    // whole items per launch, at most 65535 CTAs along z
    const int per = std::min(B, std::max(1, 65535 / (layers * split)));
    const size_t np = (size_t)d.n_views * d.det_rows * d.det_cols,
                 nvox = (size_t)d.vol_x * d.vol_y * d.vol_z;
    for (int b = 0; b < B; b += per) {
      BPAdjArgs c = a;
      c.grad_vol += b * nvox;
      if (c.relu_vol) c.relu_vol += b * nvox;
      c.grad_gF += b * np;
      c.B = std::min(per, B - b);
      gridt.z = layers * c.B * split;
      kernel<<<gridt, blk, 0, st>>>(c, split);
    }
  }
  DC_CHECK_LAUNCH("k_bp3d_adj");
  return DC_OK;
}
