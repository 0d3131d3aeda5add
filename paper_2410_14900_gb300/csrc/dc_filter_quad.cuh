// dc_filter_quad.cuh -- the line sums and the 2-D backprojection of four
// detector images at once (part of dc_filter.cu: uses its argument structs
// and epilogue helpers).
//
// A Joseph line depends on the angle, the s-bin and the principal point
// only, so images that share the principal point (the views of one scanner,
// the items of a batch) share every sample position.  Four such images are
// interleaved as float4 samples: one position, floor and address serve four
// steps, and what remains is the shared-memory traffic (two taps, 8 bytes per
// step and lane).
//
// Bank conflicts are what the per-image kernel is left with: neighbouring
// lines are 1 to 1.41 samples apart, so in any layout with the sample as the
// fastest index some lanes of a wavefront meet in a bank.  Here a band of 8
// steps is staged as [sample][step] (128 bytes per sample, the step fastest)
// and at loop index t lane l takes step t ^ (l & 7): the 8 lanes of a 16-byte
// wavefront read 8 distinct steps, i.e. 8 distinct 16-byte banks, whatever
// samples their lines meet.  The bare step then runs at 15.6 steps per clock
// and SM (128 B / 8 B = 16 at most) where the per-image kernel's form gives
// 7.9.
#pragma once

// 19 warps over the tasks and one that issues the copies: 640 threads, 5 warps
// per scheduler at 96 registers.  Line sums of 496 images of 384 x 512, 720 x
// 512 lines: 37.1 ms with the per-image kernel (7.0 steps per clock and SM);
// here 22.3 ms with 16 warps and a CTA barrier per band (data pipe 65 %, waits
// for shared memory: too few warps), 20.7 ms with this split, 21.2 with 24
// warps (80 registers), 21.6 with 16 (128), all before the groups were planned
// by waves; now 20.3 ms, 12.8 steps per clock and SM.
constexpr int L4_WARPS = 19;
constexpr int L4_THREADS = 32 * L4_WARPS + 32;
constexpr int L4_T = 6;                  // tasks (angle, 32 lines) per warp
constexpr int L4_TASKS = L4_WARPS * L4_T;
constexpr int L4_MAX_MG = 32;            // angles per group
constexpr int L4_RB = 8;                 // steps per band
// a line that meets the detector in a band moves at most 7 samples in it:
// taps lie in [-8, len + 8]
constexpr int L4_PJ = 9;
constexpr int L4_SMEM_BUDGET = 222 * 1024;  // beside 4 KB of static tables

// staging of one band: nbox TMA boxes of boxh samples x 8 steps x 4 images
struct L4Shape {
  int nbox[2], boxh[2];  // by branch (samples: columns for 0, rows for 1)
  int stage_bytes;
  int nbands;            // bands of the longer branch (row length of the table)
};

inline L4Shape l4_shape(int H, int W) {
  L4Shape s;
  for (int br = 0; br < 2; ++br) {
    const int n = (br ? H : W) + 2 * L4_PJ;
    s.nbox[br] = (n + 255) / 256;
    s.boxh[br] = (n + s.nbox[br] - 1) / s.nbox[br];
  }
  s.stage_bytes = 128 * std::max(s.nbox[0] * s.boxh[0], s.nbox[1] * s.boxh[1]);
  s.nbands = (std::max(H, W) + L4_RB - 1) / L4_RB;
  return s;
}

// dynamic shared memory: two stages (reused as the epilogue's [mg][NSp] quads),
// then the per-(angle, band) anchors and the four exchange rows
inline size_t l4_smem(const L4Shape &s, int mg, int NSp) {
  const size_t front = std::max((size_t)2 * s.stage_bytes, (size_t)mg * NSp * 16);
  return front + (size_t)mg * s.nbands * 16 + 4 * (L4_TASKS + 1) * 16;
}

// weighted copy of four images at a time into quads: [grp][H][W][4] for the
// column-stepping branch and its transpose [grp][W][H][4] for the other.
// Missing images of the last group are zeros.
__global__ void __launch_bounds__(256) k_prep4(PrepArgs a, float4 *__restrict__ rows,
                                               float4 *__restrict__ cols) {
  __shared__ float4 tile[32][33];
  const int grp = blockIdx.z;
  const int j = blockIdx.x * 32 + threadIdx.x, rb = blockIdx.y * 32 + threadIdx.y;
  float val[4][4];  // [row rb + 8 p][image], all loads in flight together
  const float *src[4];
  dc::FView f[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = min(4 * grp + i, a.n_img - 1), v = a.v0 + n / a.B, b = a.b0 + n % a.B;
    src[i] = a.src + ((size_t)b * a.V + v) * a.H * a.W + j;
    f[i] = a.fv[v];
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int i = 0; i < 4; ++i)
      val[p][i] = (4 * grp + i < a.n_img && rb + 8 * p < a.H && j < a.W)
                      ? src[i][(size_t)(rb + 8 * p) * a.W]
                      : 0.0f;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int r = rb + 8 * p;
    if (r >= a.H || j >= a.W) continue;
    if (a.weight != WT_NONE) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float x = (j - f[i].cu) * a.pitch, y = (r - f[i].cv) * a.pitch;
        const float l2 = fmaf(x, x, fmaf(y, y, f[i].D * f[i].D));
        val[p][i] *= (a.weight == WT_COS) ? f[i].D * rsqrtf(l2) : l2;
      }
    }
    const float4 v4 = make_float4(val[p][0], val[p][1], val[p][2], val[p][3]);
    tile[threadIdx.y + 8 * p][threadIdx.x] = v4;
    rows[((size_t)grp * a.H + r) * a.W + j] = v4;
  }
  __syncthreads();
  const int r = blockIdx.y * 32 + threadIdx.x;
  if (r >= a.H) return;
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int c = blockIdx.x * 32 + q;
    if (c < a.W) cols[((size_t)grp * a.W + c) * a.H + r] = tile[threadIdx.x][q];
  }
}

__device__ __forceinline__ float4 lds128(unsigned addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr));
  return v;
}

// Line sums of angle group blockIdx.x for images 4 blockIdx.y .. + 3.  A task
// is 32 neighbouring lines of one angle (lane = line); a warp owns the same
// tasks in every band and keeps their sums in registers.  Differences of
// neighbouring lines are taken per band (never between two large sums): by
// shuffle inside a task, and for its last lane from the next task's first
// lane, whose band sum is read one band later.  The band anchors are the
// exact splits of the per-image kernel: line part + band part, each an
// integer and a fraction.
template <int MODE>
__global__ void __launch_bounds__(L4_THREADS, 1)
    k_linesum4(LineArgs a, L4Shape sh, const __grid_constant__ CUtensorMap tm_cols,
               const __grid_constant__ CUtensorMap tm_rows) {
  constexpr bool DIFF = (MODE != M_RAW);
  extern __shared__ __align__(1024) unsigned char dyn[];
  __shared__ LineMu lmu[L4_MAX_MG];
  __shared__ dc::MuRec lcs[L4_MAX_MG];
  __shared__ int lm[L4_MAX_MG];
  __shared__ dc::FView fvs[4];
  __shared__ uint64_t full[2], empty[2];

  const dc::MuGroup G = a.groups[blockIdx.x];
  const int grp = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows = G.branch ? a.W : a.H;  // steps along a line
  const int len = G.branch ? a.H : a.W;   // samples across a line
  const int nbands = (rows + L4_RB - 1) / L4_RB;
  const int nch = (a.n_s + 31) >> 5;
  const int ntask = G.count * nch;
  const size_t front = max((size_t)2 * sh.stage_bytes, (size_t)a.mg * a.NSp * 16);
  float4 *ep = reinterpret_cast<float4 *>(dyn);                 // [mg][NSp], after the bands
  float4 *bt = reinterpret_cast<float4 *>(dyn + front);         // [mg][nbands]
  float4 *xch = bt + (size_t)a.mg * sh.nbands;                  // [4][L4_TASKS + 1]
  const CUtensorMap *tm = G.branch ? &tm_rows : &tm_cols;
  const int nbox = G.branch ? sh.nbox[1] : sh.nbox[0];
  const int boxh = G.branch ? sh.boxh[1] : sh.boxh[0];
  const float M = 12582912.0f;  // 1.5 * 2^23: x + M rounded down holds floor(x)

  auto issue = [&](int band) {
    uint64_t *bar = &full[band & 1];
    unsigned char *dst = dyn + (size_t)(band & 1) * sh.stage_bytes;
    dc::fence_proxy_async();
    dc::mbar_arrive_expect_tx(bar, (unsigned)(nbox * boxh * 128));
    for (int q = 0; q < nbox; ++q)
      dc::tma_load_3d(dst + (size_t)q * boxh * 128, tm, band * (4 * L4_RB), q * boxh - L4_PJ, grp,
                      bar);
  };
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      dc::mbar_init(&full[q], 1);
      dc::mbar_init(&empty[q], L4_WARPS);
    }
    dc::fence_barrier_init();
  }
  if (tid < 4) {
    const int n = min(4 * grp + tid, a.n_img - 1);
    fvs[tid] = a.fv[a.v0 + n / a.B];
  }
  if (tid < G.count) {
    const int m = a.mu_order[G.first + tid];
    const dc::MuRec R = a.mu[m];
    const dc::VMu Q = a.vmu[m];  // the principal point is the same for every view
    LineMu L;
    L.b0i = Q.b0i;
    L.b0f = Q.b0f;
    L.a_hi = R.a_hi;
    L.a_lo = R.a_lo;
    L.d_hi = R.d_hi;
    L.d_lo = R.d_lo;
    L.dxi = R.dxi;
    L.jscale = R.jscale;
    lmu[tid] = L;
    lcs[tid] = R;
    lm[tid] = m;
  }
  for (int i = tid; i < 4 * (L4_TASKS + 1); i += L4_THREADS) xch[i] = make_float4(0, 0, 0, 0);
  __syncthreads();
  // band part of the anchor: r0 * slope, exactly split
  for (int i = tid; i < G.count * nbands; i += L4_THREADS) {
    const LineMu &L = lmu[i / nbands];
    const float r0f = (float)((i % nbands) * L4_RB);
    const float th = r0f * L.d_hi, thi = floorf(th);
    bt[(i / nbands) * sh.nbands + i % nbands] =
        make_float4(thi, fmaf(r0f, L.d_lo, th - thi), L.dxi, 0.0f);
  }
  // line part of the anchor of each of this warp's tasks, and the row of its angle
  const float kc = 0.5f * (float)(a.n_s - 1);
  // tasks of this warp (may be <= 0; the copying warp has none)
  const int nt = warp < L4_WARPS ? (ntask - warp + L4_WARPS - 1) / L4_WARPS : 0;
  float Jt[L4_T], ft[L4_T];
  int br[L4_T];
  float2 acc[L4_T][2];
#pragma unroll
  for (int i = 0; i < L4_T; ++i) {
    Jt[i] = ft[i] = 0.0f;
    br[i] = 0;
    acc[i][0] = acc[i][1] = make_float2(0.0f, 0.0f);
    if (i < nt) {
      const int t = warp + i * L4_WARPS, ml = t / nch;
      const LineMu &L = lmu[ml];
      const float kk = (float)min((t - ml * nch) * 32 + lane, a.n_s - 1) - kc;
      const float t1 = kk * L.a_hi, t1i = floorf(t1);
      Jt[i] = L.b0i + t1i;
      ft[i] = L.b0f + (t1 - t1i) + kk * L.a_lo;
      br[i] = ml * sh.nbands;
    }
  }
  float2 qf[L4_RB];
#pragma unroll
  for (int t = 0; t < L4_RB; ++t) {
    const float q = (float)(t ^ (lane & 7));
    qf[t] = make_float2(q, q);
  }
  const float2 M2 = make_float2(M, M), mM2 = make_float2(-M, -M), m12 = make_float2(-1.0f, -1.0f);
  const float2 one2 = make_float2(1.0f, 1.0f), zero2 = make_float2(0.0f, 0.0f);
  const float lenf = (float)len;
  // shared address of sample 0's step l & 7 in stage 0, minus the exponent
  // bits of the two rounded-down floats whose bits are added into an address
  const unsigned cb0 = dc::smem_addr(dyn) + L4_PJ * 128u + (unsigned)(lane & 7) * 16u -
                       2u * 128u * 0x4B400000u;
  __syncthreads();

  bool ok = true;
  if (warp == L4_WARPS) {
    if (lane == 0) {
      int issued = 0;
      for (; issued < nbands && ok; ++issued) {
        if (issued >= 2 && !dc::mbar_wait_bounded(&empty[issued & 1], ((issued >> 1) - 1) & 1, a.err)) {
          ok = false;
          break;
        }
        issue(issued);
      }
      // nothing may be in flight when the CTA ends (the last two bands; in the
      // ordinary case the waits below have seen the earlier ones land)
      for (int q = max(0, issued - 2); q < issued; ++q)
        if (!dc::mbar_wait_bounded(&full[q & 1], (q >> 1) & 1, a.err)) ok = false;
    }
  } else {
    for (int band = 0; band < nbands; ++band) {
      if (!dc::mbar_wait_bounded(&full[band & 1], (band >> 1) & 1, a.err)) {
        ok = false;
        break;
      }
      const unsigned cbs = cb0 + (unsigned)((band & 1) * sh.stage_bytes);
      float4 *xw = xch + (band & 3) * (L4_TASKS + 1);
      const float4 *xr = xch + ((band + 2) & 3) * (L4_TASKS + 1);
#pragma unroll
      for (int i = 0; i < L4_T; ++i) {
        if (i < nt) {
          const int t = warp + i * L4_WARPS;
          const float4 bp = bt[br[i] + band];
          const float fr = ft[i] + bp.y;
          const float fri = __fadd_rd(fr, M) - M;
          float J = Jt[i] + bp.x + fri, fb = fr - fri, dxi = bp.z;
          // the lane's samples lie in [-1, len] somewhere in the band, or
          // nowhere: such a lane reads the zeros left of the detector
          const float xb = fmaf((float)(L4_RB - 1), dxi, fb);
          const bool outside = (fmaxf(fb, xb) <= -1.0f - J) || (fminf(fb, xb) >= lenf - J);
          float2 s0 = zero2, s1 = zero2;
          if (!__all_sync(0xffffffffu, outside)) {
            J = outside ? (float)-L4_PJ : J;
            fb = outside ? 0.0f : fb;
            dxi = outside ? 0.0f : dxi;
            const unsigned cb = cbs + __float_as_uint(J + M) * 128u;
            const float2 fb2 = make_float2(fb, fb), dx2 = make_float2(dxi, dxi);
#pragma unroll
            for (int q = 0; q < L4_RB; ++q) {
              const float2 x = __ffma2_rn(qf[q], dx2, fb2);
              const float2 tt = __fadd2_rd(x, M2);
              const float2 f = __ffma2_rn(__fadd2_rn(tt, mM2), m12, x);
              const float2 w = __ffma2_rn(f, m12, one2);
              const unsigned ad = (__float_as_uint(tt.x) * 128u + cb) ^ (16u * q);
              const float4 g0 = lds128(ad), g1 = lds128(ad + 128u);
              s0 = __ffma2_rn(w, make_float2(g0.x, g0.y), s0);
              s1 = __ffma2_rn(w, make_float2(g0.z, g0.w), s1);
              s0 = __ffma2_rn(f, make_float2(g1.x, g1.y), s0);
              s1 = __ffma2_rn(f, make_float2(g1.z, g1.w), s1);
            }
          }
          if (DIFF) {
            float2 n0, n1;
            n0.x = __shfl_down_sync(0xffffffffu, s0.x, 1);
            n0.y = __shfl_down_sync(0xffffffffu, s0.y, 1);
            n1.x = __shfl_down_sync(0xffffffffu, s1.x, 1);
            n1.y = __shfl_down_sync(0xffffffffu, s1.y, 1);
            if (lane == 31) {  // the next task's first line, its sum of band - 2
              const float4 p = xr[t + 1];
              n0 = make_float2(p.x, p.y);
              n1 = make_float2(p.z, p.w);
            }
            if (lane == 0) xw[t] = make_float4(s0.x, s0.y, s1.x, s1.y);
            acc[i][0] = __fadd2_rn(acc[i][0], __ffma2_rn(s0, m12, n0));
            acc[i][1] = __fadd2_rn(acc[i][1], __ffma2_rn(s1, m12, n1));
          } else {
            acc[i][0] = __fadd2_rn(acc[i][0], s0);
            acc[i][1] = __fadd2_rn(acc[i][1], s1);
          }
        }
      }
      __syncwarp();
      if (lane == 0) dc::mbar_arrive(&empty[band & 1]);
    }
  }
  if (__syncthreads_or(!ok)) return;  // a copy never landed

  // line sums (RAW) or differences R_{k+1}-R_k (DIFF), times the Joseph scale
  {
    const int kmax = DIFF ? a.n_s - 2 : a.n_s - 1;
#pragma unroll
    for (int i = 0; i < L4_T; ++i) {
      if (i < nt) {
        const int t = warp + i * L4_WARPS, ml = t / nch, k = (t - ml * nch) * 32 + lane;
        if (DIFF && lane == 31) {  // the next task's first line, its last two bands
          for (int q = nbands; q < nbands + 2; ++q) {
            const float4 p = xch[((q + 2) & 3) * (L4_TASKS + 1) + t + 1];
            acc[i][0] = __fadd2_rn(acc[i][0], make_float2(p.x, p.y));
            acc[i][1] = __fadd2_rn(acc[i][1], make_float2(p.z, p.w));
          }
        }
        const float js = (k <= kmax) ? lmu[ml].jscale : 0.0f;
        if (k < a.NSp)
          ep[ml * a.NSp + k] = (k <= kmax) ? make_float4(acc[i][0].x * js, acc[i][0].y * js,
                                                         acc[i][1].x * js, acc[i][1].y * js)
                                           : make_float4(0, 0, 0, 0);
      }
    }
  }
  __syncthreads();

  // epilogues, as in linesum_body, a thread's four images at a time (their
  // loads in flight together)
  const int total = G.count * a.NSp;
  const int nv = min(4, a.n_img - 4 * grp);
  size_t vm[4], bvm[4];  // rows (v, 0) of W and (b, v, 0) of a user sinogram
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = min(4 * grp + i, a.n_img - 1), v = a.v0 + n / a.B, b = a.b0 + n % a.B;
    vm[i] = (size_t)v * a.n_mu;
    bvm[i] = ((size_t)b * a.V + v) * a.n_mu;
  }
  bool bad_w = false;
  for (int idx = tid; idx < total; idx += L4_THREADS) {
    const int ml = idx / a.NSp, k = idx - ml * a.NSp;
    const int m = lm[ml];
    const float4 e4 = ep[idx];
    const float e[4] = {e4.x, e4.y, e4.z, e4.w};
    if (MODE == M_RAW) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nv && k < a.n_s) a.out[(bvm[i] + m) * a.n_s + k] = e[i];
      continue;
    }
    const float sh2 = s_half_of(k, a.n_s, a.ds);
    if (MODE == M_GRANGEAT) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float D2 = fvs[i].D * fvs[i].D;
        if (i < nv && k < a.n_s)
          a.out[(bvm[i] + m) * a.n_s + k] =
              (k <= a.n_s - 2) ? e[i] * (fmaf(sh2, sh2, D2) / D2) / a.ds : 0.0f;
      }
      continue;
    }
    float4 *sA = reinterpret_cast<float4 *>(a.sinoA) + ((size_t)grp * a.n_mu + m) * a.NSp + k;
    if (MODE == M_DIFFSTORE) {
      *sA = e4;
      continue;
    }
    const bool on = k <= a.n_s - 2;
    float w[4], y[4], tW[4];
    const float4 t4 = (MODE == M_ADJ) ? *sA : make_float4(0, 0, 0, 0);
    const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = (on && a.Wred) ? a.Wred[(vm[i] + m) * a.n_s + k] : 0.5f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const dc::FView &fv = fvs[i];
      const float D2 = fv.D * fv.D, wsino = fmaf(sh2, sh2, D2) / D2;
      const float Kv = redundancy_k(lcs[ml], fv, sh2);
      bad_w |= !isfinite(w[i]);
      y[i] = 0.0f;
      if (MODE == M_FILTER) {
        if (on) y[i] = w[i] * Kv * wsino * e[i] / a.ds;
        // Grangeat's S (Eq. 7), kept for a reverse mode that reuses it
        if (a.Sout && i < nv && k < a.n_s)
          a.Sout[(bvm[i] + m) * a.n_s + k] = on ? e[i] * wsino / a.ds : 0.0f;
      } else {  // M_ADJ: as in linesum_body
        tW[i] = 0.0f;
        if (on) {
          const float Qg = -a.cT * t[i] / a.ds;  // D_b^T of dL/dP
          tW[i] = Kv * (wsino * e[i] / a.ds) * Qg;
          y[i] = wsino * w[i] * Kv * Qg;
        }
      }
    }
    if (MODE == M_ADJ) *sA = make_float4(tW[0], tW[1], tW[2], tW[3]);
    ep[idx] = make_float4(y[0], y[1], y[2], y[3]);
  }
  if (MODE == M_RAW || MODE == M_GRANGEAT || MODE == M_DIFFSTORE) return;
  if (bad_w) atomicOr(a.err, DC_FLAG_NONFINITE_W);
  __syncthreads();
  // FILTER: P = D_b Q times the A2d^T scale; ADJ: dL/dR = D_f^T y; both times
  // the Joseph scale for the transpose gather
  for (int idx = tid; idx < total; idx += L4_THREADS) {
    const int ml = idx / a.NSp, k = idx - ml * a.NSp;
    const int m = lm[ml];
    const float js = lmu[ml].jscale;
    const float4 c4 = ep[idx], p4 = (k > 0) ? ep[idx - 1] : make_float4(0, 0, 0, 0);
    const float c[4] = {c4.x, c4.y, c4.z, c4.w}, p[4] = {p4.x, p4.y, p4.z, p4.w};
    float val[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      val[i] = (MODE == M_FILTER) ? (c[i] - p[i]) / a.ds * a.cT * js : (p[i] - c[i]) / a.ds * js;
      if (k >= a.n_s) val[i] = 0.0f;
    }
    reinterpret_cast<float4 *>(MODE == M_FILTER ? a.out : a.sinoB)[((size_t)grp * a.n_mu + m) *
                                                                       a.NSp + k] =
        make_float4(val[0], val[1], val[2], val[3]);
  }
}

// the last step of the filter's reverse mode from a kept S (k_adj_from_s) on
// quad sinograms: a CTA takes AS4_ROWS angles of four images
constexpr int AS4_ROWS = 2;
__global__ void __launch_bounds__(256) k_adj_from_s4(LineArgs a, const float *__restrict__ S) {
  extern __shared__ __align__(16) float4 ys4[];  // [AS4_ROWS][NSp]
  const int grp = blockIdx.y, m0 = blockIdx.x * AS4_ROWS;
  const int total = min(AS4_ROWS, a.n_mu - m0) * a.NSp;
  float4 *sA = reinterpret_cast<float4 *>(a.sinoA) + ((size_t)grp * a.n_mu + m0) * a.NSp;
  float4 *sB = reinterpret_cast<float4 *>(a.sinoB) + ((size_t)grp * a.n_mu + m0) * a.NSp;
  bool bad_w = false;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int m = m0 + idx / a.NSp, k = idx % a.NSp;
    const bool on = k <= a.n_s - 2;
    const float4 t4 = sA[idx];
    const float t[4] = {t4.x, t4.y, t4.z, t4.w};
    const float sh = s_half_of(k, a.n_s, a.ds);
    float y[4], tW[4], w[4], Sv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = min(4 * grp + i, a.n_img - 1), v = a.v0 + n / a.B, b = a.b0 + n % a.B;
      w[i] = (on && a.Wred) ? a.Wred[((size_t)v * a.n_mu + m) * a.n_s + k] : 0.5f;
      Sv[i] = on ? S[(((size_t)b * a.V + v) * a.n_mu + m) * a.n_s + k] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = min(4 * grp + i, a.n_img - 1);
      const dc::FView fv = a.fv[a.v0 + n / a.B];
      const float D2 = fv.D * fv.D;
      y[i] = tW[i] = 0.0f;
      if (on) {
        const float wsino = fmaf(sh, sh, D2) / D2;
        const float Qg = -a.cT * t[i] / a.ds;  // D_b^T of dL/dP
        const float Kv = redundancy_k(a.mu[m], fv, sh);
        bad_w |= !isfinite(w[i]);
        tW[i] = Kv * Sv[i] * Qg;
        y[i] = wsino * w[i] * Kv * Qg;
      }
    }
    sA[idx] = make_float4(tW[0], tW[1], tW[2], tW[3]);
    ys4[idx] = make_float4(y[0], y[1], y[2], y[3]);
  }
  if (bad_w) atomicOr(a.err, DC_FLAG_NONFINITE_W);
  __syncthreads();
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int k = idx % a.NSp;
    float4 val = make_float4(0, 0, 0, 0);
    if (k < a.n_s) {
      const float js = a.mu[m0 + idx / a.NSp].jscale;
      const float4 ym = (k > 0) ? ys4[idx - 1] : make_float4(0, 0, 0, 0);
      const float4 y0 = ys4[idx];  // 0 at k = n_s - 1
      val = make_float4((ym.x - y0.x) / a.ds * js, (ym.y - y0.y) / a.ds * js,
                        (ym.z - y0.z) / a.ds * js, (ym.w - y0.w) / a.ds * js);
    }
    sB[idx] = val;
  }
}

// k_sino_in for four images: user sinograms into quads, times the Joseph scale
__global__ void k_sino_in4(const float *__restrict__ R, const dc::MuRec *__restrict__ mu, int n_mu,
                           int n_s, int NSp, int V, int B, int v0, int b0, int n_img,
                           float4 *__restrict__ dst) {
  const int grp = blockIdx.y;
  const size_t total = (size_t)n_mu * NSp;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(i / NSp), k = (int)(i % NSp);
    float val[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = 4 * grp + q, v = v0 + n / B, b = b0 + n % B;
      val[q] = (k < n_s && n < n_img) ? R[(((size_t)b * V + v) * n_mu + m) * n_s + k] * mu[m].jscale
                                      : 0.0f;
    }
    dst[(size_t)grp * total + i] = make_float4(val[0], val[1], val[2], val[3]);
  }
}

// -------------------------------------------- 2-D backprojection, four images
// As for the line sums: position, floor, hat weights and address of a
// (pixel, angle) pair once for four images, their taps one 16-byte load each.
// The bare pair then runs at 15.8 pairs per clock and SM (128 B / 8 B = 16 at
// most); the per-image kernel reaches 9.3, bound by instructions.
//
// A CTA takes a tile of 2048 (or, for grids too small to fill the GPU, 512)
// pixels: 8 warps of 32 columns x RY rows, nwx warps side by side.  Only the
// s-window that a tile meets is staged, per angle: TMA boxes of the quad
// sinogram, zeros outside [0, NSp), so no position is clamped.  A thread holds
// RY pixels x 4 images.
constexpr int B4_THREADS = 256;
constexpr int B4_MC = 16;  // angles per stage
struct B4Shape {
  int nwx;       // warps side by side
  int lwb, nb;   // boxes of lwb bins (multiple of 8, at most 64), nb of them per angle
};

struct B4Mu {
  float F00, Bc, Bs, winv;
  float w1c;
  unsigned cbase;  // byte offset of bin I00 in its stage row, minus the floor's exponent bits
  unsigned pad0, pad1;
};

// two stages of a tile's window
inline size_t b4_smem(const B4Shape &s) { return (size_t)2 * B4_MC * s.lwb * s.nb * 16; }

// taps per pixel and angle: the hat's half-width is at most pitch / ds bins
template <int NT>
constexpr int b4_left() { return NT / 2 - 1; }

inline int b4_taps(double pitch, double ds) {
  return ds >= pitch * (1.0 - 1e-12) ? 2 : 2.0 * ds >= pitch * (1.0 - 1e-12) ? 4 : 6;
}

// Dynamic shared memory up to which two CTAs share an SM (228 KB, 1 KB of it
// the system's per CTA, beside 2 KB of static tables), and the most that any
// launch asks for, whatever its geometry.
constexpr int B4_SMEM_TWO = 111 * 1024;
constexpr int B4_SMEM_MAX = 224 * 1024;

// the arrangement of nwx warps side by side and the window of its tile
inline B4Shape b4_arrange(int nwx, double pitch, double ds, int RY) {
  B4Shape s;
  s.nwx = nwx;
  const int tx = 32 * nwx, ty = RY * (8 / nwx), nt = b4_taps(pitch, ds);
  const double span = std::sqrt((tx - 1.0) * (tx - 1.0) + (ty - 1.0) * (ty - 1.0)) * pitch / ds;
  const int need = (int)(span + 0.1) + 3 + nt;
  s.nb = (need + 63) / 64;
  s.lwb = (((need + s.nb - 1) / s.nb) + 7) & ~7;
  return s;
}

inline long b4_tiles(int H, int W, const B4Shape &s, int RY, int images) {
  const int tx = 32 * s.nwx, ty = RY * (8 / s.nwx);
  return (long)((W + tx - 1) / tx) * ((H + ty - 1) / ty) * ((images + 3) / 4);
}

// What an SM's share of the tiles of `items` batch items of all views takes, in
// chunks of `chunk` images: two CTAs together 2 units, one alone, or at a time
// because two do not fit, 1.28 (two taps) or 1.13 (more).
inline double b4_rounds(int H, int W, const B4Shape &s, int taps, int views, int items, int chunk,
                        int sms) {
  const double alone = taps == 2 ? 1.28 : 1.13;
  const int bc = std::min(items, chunk), cv = std::min(views, std::max(1, chunk / bc));
  auto time = [&](int v) {
    const long n = (b4_tiles(H, W, s, 8, v * bc) + sms - 1) / sms;
    return b4_smem(s) <= (size_t)B4_SMEM_TWO ? 2.0 * (n / 2) + alone * (n % 2) : alone * n;
  };
  return (views / cv) * time(cv) + (views % cv ? time(views % cv) : 0.0);
}

// The warps' arrangement with the least time among those whose stages an SM
// holds (the squarest of equals: the smallest window) and no wider than the one
// with the fewest pixels outside the detector: a position is rounded at its
// distance from the tile's first column, so width costs accuracy (filter of 256
// images of 58 x 80: 1.5e-6 relative L2 from FP64 with 64 x 32 tiles, 1.1e-6 with
// 32 x 64), which is paid for fewer pixels only.  At ds >= pitch / 3 the two
// narrow ones always fit (112 KB); 256 x 8 tiles want 140 KB at ds = pitch, 288 at
// pitch / 2.  With 8 rows per thread the time is b4_rounds per item, over batches
// of one to four items, fewer items counting more: 96 images, 180 angles, ds =
// pitch: 360 x 512 974 us in 15 rounds of 256 x 8 tiles, one CTA per SM, 775 in
// 128 x 16 tiles; at 0.8 pitch 200 x 256 590 us in 4 rounds of 256 x 8, 655 in 5 of
// 128 x 16.  (Judged by one item alone, 30 views of 300 x 400 take 4 % longer with
// three.)  With 2 rows (grids of less than a wave) it is the pixels computed,
// those outside the detector too.
inline B4Shape b4_shape(int H, int W, double pitch, double ds, int RY, int views, int chunk,
                        int sms) {
  const int order[4] = {2, 1, 4, 8}, taps = b4_taps(pitch, ds);
  long fewest = -1;
  int widest = 0;
  for (int nwx : order) {
    const long tiles = b4_tiles(H, W, b4_arrange(nwx, pitch, ds, RY), RY, 4);
    if (fewest < 0 || tiles < fewest) {
      fewest = tiles;
      widest = nwx;
    }
  }
  B4Shape best = {};
  double least = -1.0;
  for (int nwx : order) {
    const B4Shape s = b4_arrange(nwx, pitch, ds, RY);
    if (nwx > widest || (nwx > 2 && b4_smem(s) > (size_t)B4_SMEM_MAX)) continue;
    double cost = 0.0;
    if (RY == 2) cost = (double)b4_tiles(H, W, s, RY, 4);
    else
      for (int b = 1; b <= 4; ++b) cost += b4_rounds(H, W, s, taps, views, b, chunk, sms) / (b * b);
    if (least < 0.0 || cost < least) {
      least = cost;
      best = s;
    }
  }
  return best;
}

// Rows per thread: 8, unless the 2048-pixel tiles of the views at hand leave
// SMs without a CTA, then 2 (64 views of 64 x 64, 32 tiles: 35 us against 70;
// 90 views of 128 x 128, 184 tiles: 168 against 158).  A property of the
// geometry, so that an image's result does not depend on the chunk or batch
// that it comes in.
inline int b4_rows(int H, int W, double pitch, double ds, int views, int chunk, int sms) {
  const B4Shape s = b4_shape(H, W, pitch, ds, 8, views, chunk, sms);
  return b4_tiles(H, W, s, 8, std::min(views, chunk)) < sms ? 2 : 8;
}

// 8 rows per thread want the registers of two CTAs per SM (496 images of 384 x
// 512 and 720 angles: 22.1 ms with the per-image kernel, 16.2 with three CTAs
// at 80 registers, waiting for shared memory; 15.1 with two: 14.8 pairs per
// clock and SM)
template <int NT, int RY>
__global__ void __launch_bounds__(B4_THREADS, RY == 8 ? 2 : 4)
    k_bp2d4(BP2Args a, B4Shape sh, const __grid_constant__ CUtensorMap tm) {
  extern __shared__ __align__(1024) unsigned char dyn[];
  __shared__ uint64_t full[2];
  __shared__ __align__(16) B4Mu bmu[2][B4_MC];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.z;
  const int tx = 32 * sh.nwx, ty = RY * (8 / sh.nwx);
  const int j0 = blockIdx.x * tx, r0 = blockIdx.y * ty;
  const int row_bytes = sh.lwb * sh.nb * 16;
  const int nchunk = (a.n_mu + B4_MC - 1) / B4_MC;
  constexpr int TL = b4_left<NT>();

  // constants of chunk c's angles for this tile (exact float splits of the
  // origin, as in the per-image kernel) and the copies of their s-windows:
  // one thread per angle
  auto stage = [&](int c) {
    const int st = c & 1, nm = min(B4_MC, a.n_mu - c * B4_MC);
    dc::fence_proxy_async();
    if (tid == 0) dc::mbar_arrive_expect_tx(&full[st], (unsigned)(nm * row_bytes));
    __syncwarp();
    if (tid < nm) {
      const int m = c * B4_MC + tid;
      const dc::MuRec R = a.mu[m];
      const dc::VMu Q = a.vmu[m];  // the principal point is the same for every view
      const float fj0 = (float)j0, fr0 = (float)r0;
      const float t = fj0 * R.bc_hi + fr0 * R.bs_hi;  // exact
      const float ti = floorf(t);
      const float F = Q.xof + (t - ti) + fmaf(fj0, R.bc_lo, fr0 * R.bs_lo);
      const float Fi = floorf(F);
      const int I00 = (int)(Q.xoi + ti + Fi);
      B4Mu M;
      M.F00 = F - Fi;
      M.Bc = R.bc_hi + R.bc_lo;
      M.Bs = R.bs_hi + R.bs_lo;
      M.winv = R.winv;
      M.w1c = 1.0f - R.winv;
      const float ex = (float)(tx - 1) * M.Bc, ey = (float)(ty - 1) * M.Bs;
      // first bin of the window relative to I00, with a margin for the
      // rounding of the positions
      const int kw = (int)floorf(M.F00 + fminf(ex, 0.0f) + fminf(ey, 0.0f) - 0.01f) - TL;
      M.cbase = (unsigned)(st * B4_MC * row_bytes + tid * row_bytes - kw * 16) - 16u * 0x4B400000u;
      M.pad0 = M.pad1 = 0u;
      bmu[st][tid] = M;
      unsigned char *dst = dyn + (size_t)(st * B4_MC + tid) * row_bytes;
      for (int q = 0; q < sh.nb; ++q)
        dc::tma_load_3d(dst + q * sh.lwb * 16, &tm, (I00 + kw + q * sh.lwb) * 4, m, grp, &full[st]);
    }
  };
  if (tid == 0) {
    dc::mbar_init(&full[0], 1);
    dc::mbar_init(&full[1], 1);
    dc::fence_barrier_init();
  }
  __syncthreads();
  if (warp == 0) {
    stage(0);
    if (nchunk > 1) stage(1);
  }
  __syncthreads();

  float2 acc[RY][2];
#pragma unroll
  for (int r = 0; r < RY; ++r) acc[r][0] = acc[r][1] = make_float2(0.0f, 0.0f);
  const int jl = (warp & (sh.nwx - 1)) * 32 + lane, rl = (warp / sh.nwx) * RY;
  const float jlf = (float)jl;
  float2 rlf[RY / 2];  // tile rows of the thread's pixels in pairs
#pragma unroll
  for (int r = 0; r < RY / 2; ++r) rlf[r] = make_float2((float)(rl + 2 * r), (float)(rl + 2 * r + 1));
  const float2 M2 = make_float2(12582912.0f, 12582912.0f);
  const float2 mM2 = make_float2(-12582912.0f, -12582912.0f), m12 = make_float2(-1.0f, -1.0f);
  const unsigned sbase = dc::smem_addr(dyn);

  bool ok = true;
  int c = 0;
  for (; c < nchunk; ++c) {
    if (!dc::mbar_wait_bounded(&full[c & 1], (c >> 1) & 1, a.err)) ok = false;
    const int nm = min(B4_MC, a.n_mu - c * B4_MC);
    // few pixels per thread: several angles in flight hide the chain from an
    // angle's constants to its taps
#pragma unroll(RY == 2 ? 4 : 2)
    for (int mi = 0; mi < nm; ++mi) {
      const B4Mu M = bmu[c & 1][mi];
      const unsigned cb = M.cbase + sbase;
      const float base = fmaf(jlf, M.Bc, M.F00);
      const float2 base2 = make_float2(base, base), Bs2 = make_float2(M.Bs, M.Bs);
#pragma unroll
      for (int r = 0; r < RY / 2; ++r) {
        const float2 x = __ffma2_rn(rlf[r], Bs2, base2);
        const float2 t = __fadd2_rd(x, M2);  // exact floor and fraction
        const float2 f = __ffma2_rn(__fadd2_rn(t, mM2), m12, x);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float fh = h ? f.y : f.x;
          const unsigned ad = __float_as_uint(h ? t.y : t.x) * 16u + cb;
          float2 &a0 = acc[2 * r + h][0], &a1 = acc[2 * r + h][1];
#pragma unroll
          for (int q = 0; q < NT; ++q) {
            // tap floor(x) + q - TL at distance |f + TL - q|: for ds >= pitch
            // (winv >= 1) the hat never exceeds 1 and the clamp at 0 is a
            // saturation
            float w;
            if (NT == 2)
              w = __saturatef(q == 0 ? fmaf(-fh, M.winv, 1.0f) : fmaf(fh, M.winv, M.w1c));
            else
              w = fmaxf(0.0f, fmaf(-fabsf(fh + (float)(TL - q)), M.winv, 1.0f));
            const float2 w2 = make_float2(w, w);
            const float4 p = lds128(ad + (unsigned)(16 * (q - TL)));
            a0 = __ffma2_rn(w2, make_float2(p.x, p.y), a0);
            a1 = __ffma2_rn(w2, make_float2(p.z, p.w), a1);
          }
        }
      }
    }
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    if (warp == 0 && c + 2 < nchunk) stage(c + 2);
  }
  if (!ok) {  // a copy never landed: nothing may be in flight when the CTA ends
    dc::mbar_wait_bounded(&full[c & 1], (c >> 1) & 1, nullptr);
    if (c + 1 < nchunk) dc::mbar_wait_bounded(&full[(c + 1) & 1], ((c + 1) >> 1) & 1, nullptr);
    return;
  }

  const int j = j0 + jl;
  float lmax[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (j < a.W) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = 4 * grp + i;
      if (n >= a.n_img) break;
      const int v = a.v0 + n / a.B, b = a.b0 + n % a.B;
      const dc::FView fv = a.fv[v];
      const float xx = (j - fv.cu) * a.pitch;
#pragma unroll
      for (int r = 0; r < RY; ++r) {
        const int rr = r0 + rl + r;
        if (rr >= a.H) break;
        float val = (i & 1) ? acc[r][i >> 1].y : acc[r][i >> 1].x;
        if (a.weight != WT_NONE) {
          const float yy = (rr - fv.cv) * a.pitch;
          const float l2 = fmaf(xx, xx, fmaf(yy, yy, fv.D * fv.D));
          val *= (a.weight == WT_D) ? l2 : fv.D * rsqrtf(l2);
        }
        if (a.out_kind == OUT_F32_ABSMAX || a.out_kind == OUT_F32_SLOT) {
          ((float *)a.out)[((size_t)n * a.H + rr) * a.Wp + j] = val;
          lmax[i] = fmaxf(lmax[i], fabsf(val));
        } else {
          const size_t o = (((size_t)b * a.V + v) * a.H + rr) * a.W + j;
          if (a.out_kind == OUT_BF16) ((__nv_bfloat16 *)a.out)[o] = __float2bfloat16_rn(val);
          else ((float *)a.out)[o] = val;
        }
      }
    }
  }
  if (a.out_kind == OUT_F32_ABSMAX) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float l = lmax[i];
      for (int o = 16; o > 0; o >>= 1) l = fmaxf(l, __shfl_xor_sync(0xffffffffu, l, o));
      if (lane == 0 && 4 * grp + i < a.n_img) atomicMax(&a.absmax[4 * grp + i], __float_as_uint(l));
    }
  }
}
