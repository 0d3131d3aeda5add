// dc_filter_quad.cuh -- the line sums of four detector images at once (part
// of dc_filter.cu: uses its LineArgs and epilogue helpers).
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
// warps (80 registers), 21.6 with 16 (128).  12.1 steps per clock and SM.
constexpr int L4_WARPS = 19;
constexpr int L4_THREADS = 32 * L4_WARPS + 32;
constexpr int L4_T = 6;                  // tasks (angle, 32 lines) per warp
constexpr int L4_TASKS = L4_WARPS * L4_T;
constexpr int L4_RB = 8;                 // steps per band
// a line that meets the detector in a band moves at most 7 samples in it:
// taps lie in [-8, len + 8]
constexpr int L4_PJ = 9;
constexpr int L4_SMEM_BUDGET = 225 * 1024;

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
  const int j = blockIdx.x * 32 + threadIdx.x;
  for (int q = threadIdx.y; q < 32; q += 8) {
    const int r = blockIdx.y * 32 + q;
    if (r >= a.H || j >= a.W) continue;
    float val[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = 4 * grp + i;
      val[i] = 0.0f;
      if (n < a.n_img) {
        const int v = a.v0 + n / a.B, b = a.b0 + n % a.B;
        val[i] = a.src[(((size_t)b * a.V + v) * a.H + r) * a.W + j];
        if (a.weight != WT_NONE) {
          const dc::FView f = a.fv[v];
          const float x = (j - f.cu) * a.pitch, y = (r - f.cv) * a.pitch;
          const float l2 = fmaf(x, x, fmaf(y, y, f.D * f.D));
          val[i] *= (a.weight == WT_COS) ? f.D * rsqrtf(l2) : l2;
        }
      }
    }
    const float4 v4 = make_float4(val[0], val[1], val[2], val[3]);
    tile[q][threadIdx.x] = v4;
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
  __shared__ LineMu lmu[dc::DC_LS_MAX_MG];
  __shared__ dc::MuRec lcs[dc::DC_LS_MAX_MG];
  __shared__ int lm[dc::DC_LS_MAX_MG];
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
    if (MODE == M_DIFFSTORE) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (i < nv) a.sinoA[((size_t)(4 * grp + i) * a.n_mu + m) * a.NSp + k] = e[i];
      continue;
    }
    const bool on = k <= a.n_s - 2;
    float w[4], t[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = (on && a.Wred) ? a.Wred[(vm[i] + m) * a.n_s + k] : 0.5f;
      t[i] = (MODE == M_ADJ && on && i < nv)
                 ? a.sinoA[((size_t)(4 * grp + i) * a.n_mu + m) * a.NSp + k]
                 : 0.0f;
    }
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
        float tW = 0.0f;
        if (on) {
          const float Qg = -a.cT * t[i] / a.ds;  // D_b^T of dL/dP
          tW = Kv * (wsino * e[i] / a.ds) * Qg;
          y[i] = wsino * w[i] * Kv * Qg;
        }
        if (i < nv) a.sinoA[((size_t)(4 * grp + i) * a.n_mu + m) * a.NSp + k] = tW;
      }
    }
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
    float *dst = (MODE == M_FILTER) ? a.out : a.sinoB;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float val = (MODE == M_FILTER) ? (c[i] - p[i]) / a.ds * a.cT * js : (p[i] - c[i]) / a.ds * js;
      if (k >= a.n_s) val = 0.0f;
      if (i < nv) dst[((size_t)(4 * grp + i) * a.n_mu + m) * a.NSp + k] = val;
    }
  }
}
