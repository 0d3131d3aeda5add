// dc_filter.cu -- the filtering part of the Defrise-Clack network
// (Ye et al., DRACO, Sec. 2.3, Eqs. 7, 8, 10, 11):
//
//   S   = w_sino D_f A2d w_cos g                (Grangeat's function, Eq. 7)
//   g^F = w_d A2d^T D_b (W K) S                 (shift-variant filter, Eq. 11)
//
// and its reverse mode.  Views are processed in chunks of images (view x
// batch item); where every view has the same principal point an image set is
// four images interleaved (dc_filter_quad.cuh), otherwise one:
//
//   k_prep      weight (w_cos or w_d) and write the image with padded rows
//   k_linesum   Joseph line sums of every (mu, s) line of an image, streamed
//               band by band (32, 16 or 8 detector rows or columns) through
//               shared memory by asynchronous copies, each band stored with
//               the band step as the fastest index; neighbouring lines of a
//               warp take the s-difference by shuffle so that D_f never
//               subtracts two large sums; the epilogue applies w_sino, K, W
//               and D_b (or the adjoint chain)
//   k_bp2d      pixel-driven A2d^T: each pixel gathers the two sinogram taps
//               of every angle (the exact transpose of the Joseph weights),
//               angles streamed through shared memory with bulk copies; the
//               epilogue applies w_d (forward) or w_cos (adjoint)
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "dc_async.cuh"
#include "dc_common.cuh"

namespace {

constexpr float kPi = 3.14159265358979323846f;
constexpr int PADL = 4;  // zero floats left of every shared-memory row (16 B)
constexpr int PADR = 4;  // zero floats right of every shared-memory row

// ------------------------------------------------------------------ prep
enum { WT_NONE = 0, WT_COS = 1, WT_D = 2 };

struct PrepArgs {
  const float *src;  // [B][V][H][W]
  float *img;        // [n][H][Wp]
  const dc::FView *fv;
  int H, W, Wp, V, B, v0, n_img;  // B = batch items in this chunk
  int b0, Bt;                     // first item of the chunk, total batch
  float pitch;
  int weight;
};

// weighted copy into rows padded to Wp (the pads are written as zeros)
__global__ void __launch_bounds__(256) k_prep(PrepArgs a) {
  int n = blockIdx.z;
  int v = a.v0 + n / a.B, b = a.b0 + n % a.B;
  const dc::FView f = a.fv[v];
  const float *src = a.src + ((size_t)b * a.V + v) * a.H * a.W;
  int j = blockIdx.x * 32 + threadIdx.x;
  if (j >= a.Wp) return;
  for (int q = threadIdx.y; q < 32; q += 8) {
    int r = blockIdx.y * 32 + q;
    if (r >= a.H) break;
    float val = 0.0f;
    if (j < a.W) {
      val = src[(size_t)r * a.W + j];
      if (a.weight != WT_NONE) {
        float x = (j - f.cu) * a.pitch, y = (r - f.cv) * a.pitch;
        float l2 = fmaf(x, x, fmaf(y, y, f.D * f.D));
        val *= (a.weight == WT_COS) ? f.D * rsqrtf(l2) : l2;
      }
    }
    a.img[((size_t)n * a.H + r) * a.Wp + j] = val;
  }
}

// ------------------------------------------------------------- line sums
enum { M_RAW = 0, M_GRANGEAT = 1, M_FILTER = 2, M_DIFFSTORE = 3, M_ADJ = 4 };

constexpr int LS_THREADS = 640;  // one CTA per SM: 20 warps at 96 registers
// A band of RB detector rows (32, or 16 / 8 when long detector rows would
// not fit) is staged with RB + 1 floats per sample: odd, so lanes at distinct
// samples hit distinct banks.  RB + 1 zero samples pad each side: a line that
// meets the detector anywhere in a band moves less than RB samples (slope at
// most 1) over the band, so its taps never leave the stage and need no clamp.
constexpr int LS_SMEM_BUDGET = 225 * 1024;  // one CTA per SM

struct LineArgs {
  const float *img;   // [n][H][Wp]
  int H, W, Wp;
  int n_mu, n_s, NSp;
  int V, B, v0, n_img;  // B = batch items in this chunk
  int b0;               // first batch item of the chunk
  float pitch, ds, cT;  // cT = (pi/n_mu) ds / pitch^2
  const dc::MuRec *mu;
  const dc::VMu *vmu;   // [V][n_mu]
  const int *mu_order;
  const dc::MuGroup *groups;
  const dc::FView *fv;
  const float *Wred;   // [V][n_mu][n_s] or NULL (= 1/2)
  float *out;          // RAW/GRANGEAT: user [B][V][n_mu][n_s]; else scratch [n][n_mu][NSp]
  float *sinoA;        // DIFFSTORE out / ADJ in-out (scratch)
  float *sinoB;        // ADJ out (scratch)
  float *Sout;         // FILTER: optional copy of S, user [B][V][n_mu][n_s]
  unsigned *err;
  int mg;              // max angles per group
};

// per-angle constants of one CTA (from the set-up tables)
struct LineMu {
  float b0i, b0f;    // c_col + c_row sn/cs  = b0i (integer) + b0f
  float a_hi, a_lo;  // (ds/p)/cs  (hi has 12 fractional bits)
  float d_hi, d_lo;  // -sn/cs     (slope per row)
  float dxi;         // -sn/cs as a float
  float jscale;      // p / |cs|
};

// half-grid abscissa s_{k+1/2} and the weight K = -(1/4pi^2)|v.theta| / (s^2 +
// D^2) of Eq. 10 on it (theta unnormalised: the norm is folded into the
// denominator); shared by the line-sum epilogues and the cached-S adjoint so
// that both give the same FP32 values
__device__ __forceinline__ float s_half_of(int k, int n_s, float ds) {
  return ((float)k - 0.5f * (float)(n_s - 1) + 0.5f) * ds;
}
__device__ __forceinline__ float redundancy_k(const dc::MuRec &r, const dc::FView &fv, float sh) {
  const float D = fv.D, D2 = D * D;
  const float inv4pi2 = 1.0f / (4.0f * kPi * kPi);
  const float vt = fmaf(sh, fv.az, D * fmaf(r.c, fv.ax, r.s * fv.ay));
  return -fabsf(vt) * inv4pi2 / fmaf(sh, sh, D2);
}

// Joseph sum of one line over the nr steps of a staged band: the sample at
// step q sits at fb + q*dxi samples from the band anchor and is interpolated
// linearly between its two neighbours (zero pads outside the detector).  The
// anchor's byte offset in shared memory is folded with the floor's exponent
// bits into cb, so one integer multiply-add turns the rounded-down position
// into the address; NR = RB unrolls the band so that the step offset 4q is an
// immediate (NR = 0 takes nr at run time).
template <int RB, int NR>
__device__ __forceinline__ float band_sum(const char *sb, unsigned cb, int nr, float fb,
                                          float dxi) {
  const float M = 12582912.0f;  // 1.5 * 2^23: x + M rounded down holds floor(x)
  constexpr int SQ = RB + 1;
  // even and odd steps in two sums: half the length of the dependent chain
  float sum[2] = {0.0f, 0.0f};
#pragma unroll
  for (int q = 0; q < (NR ? NR : RB); ++q) {
    if (!NR && q >= nr) break;
    const float x = fmaf((float)q, dxi, fb);
    const float t = __fadd_rd(x, M);
    const float f = x - (t - M);
    const unsigned off = __float_as_uint(t) * (unsigned)(SQ * 4) + cb + 4u * q;
    const float g0 = *reinterpret_cast<const float *>(sb + off);
    const float g1 = *reinterpret_cast<const float *>(sb + off + SQ * 4);
    sum[q & 1] += fmaf(f, g1 - g0, g0);
  }
  return sum[0] + sum[1];
}

// The line sums of angle group `gi` of image n (view a.v0 + n / a.B, item
// a.b0 + n % a.B) by a CTA of NT threads (a 1-D block).  The image is read
// from work-area slot `slot` of a.img and the scratch sinograms are written
// to slot `slot` of a.out / a.sinoA / a.sinoB (the chunked launches use
// slot = n).  Uses `smem` (dynamic, linesum_smem_for bytes), lmu and ttab;
// the CTA must synchronise before calling it again.
template <int MODE, int RB, int NT>
__device__ __forceinline__ void linesum_body(const LineArgs &a, int gi, int n, int slot,
                                             float *smem, LineMu *lmu, short2 *ttab) {
  constexpr bool DIFF = (MODE != M_RAW);
  constexpr int LS_RB = RB, LS_SQ = RB + 1, LS_PJ = RB + 1;
  constexpr int LS_THREADS = NT, LS_WARPS = NT / 32;
  static_assert(LS_THREADS % RB == 0 && RB <= 32, "band copy mapping");
    constexpr int STRIDE_L = DIFF ? 31 : 32;  // lines per task (diff: one overlap)

  const dc::MuGroup G = a.groups[gi];
  const int v = a.v0 + n / a.B, b = a.b0 + n % a.B;
  const dc::FView fv = a.fv[v];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // branch 0 steps over detector rows and samples along a row; branch 1
  // steps over detector columns and samples along a column.  Either way a
  // band of LS_RB steps is staged as [sample][LS_SQ]: the band position q is
  // the fastest index, so inside the unrolled band loop it is an immediate.
  const int rows = G.branch ? a.W : a.H;  // steps along a line
  const int len = G.branch ? a.H : a.W;   // samples across a line
  const float *src = a.img + (size_t)slot * a.H * a.Wp;
  const int stage_sz = (len + 2 * LS_PJ) * LS_SQ;
  float *stage0 = smem;
  float *stage1 = smem + stage_sz;
  float *ep = smem + 2 * stage_sz;  // [mg][NSp] epilogue buffer
  const char *sb = reinterpret_cast<const char *>(smem);

  if (threadIdx.x < G.count) {
    int m = a.mu_order[G.first + threadIdx.x];
    const dc::MuRec R = a.mu[m];
    const dc::VMu Q = a.vmu[(size_t)v * a.n_mu + m];
    LineMu L;
    L.b0i = Q.b0i;
    L.b0f = Q.b0f;
    L.a_hi = R.a_hi;
    L.a_lo = R.a_lo;
    L.d_hi = R.d_hi;
    L.d_lo = R.d_lo;
    L.dxi = R.dxi;
    L.jscale = R.jscale;
    lmu[threadIdx.x] = L;
  }
  // zero the sample pads of both stages (never written by the copies)
  for (int i = threadIdx.x; i < 2 * 2 * LS_PJ * LS_SQ; i += LS_THREADS) {
    int st = i / (2 * LS_PJ * LS_SQ), r = i % (2 * LS_PJ * LS_SQ);
    int jj = r / LS_SQ, q = r % LS_SQ;
    int row = jj < LS_PJ ? jj : len + jj;  // samples -PJ..-1 and len..len+PJ-1
    smem[(size_t)st * stage_sz + (size_t)row * LS_SQ + q] = 0.0f;
  }
  __syncthreads();

  // asynchronous 4-byte copies into the interleaved layout (coalesced reads)
  const int nbands = (rows + LS_RB - 1) / LS_RB;
  auto stage = [&](int band) {
    float *st = ((band & 1) ? stage1 : stage0) + LS_PJ * LS_SQ;
    const int r0 = band * LS_RB;
    const int nr = min(LS_RB, rows - r0);
    if (!G.branch) {
      for (int q = 0; q < nr; ++q) {
        const float *s = src + (size_t)(r0 + q) * a.Wp;
        for (int jj = threadIdx.x; jj < len; jj += LS_THREADS) dc::cp_async4(st + jj * LS_SQ + q, s + jj);
      }
    } else {
      const int q = threadIdx.x % LS_RB;
      if (q < nr)
        for (int jj = threadIdx.x / LS_RB; jj < len; jj += LS_THREADS / LS_RB)
          dc::cp_async4(st + jj * LS_SQ + q, src + (size_t)jj * a.Wp + r0 + q);
    }
    dc::cp_async_commit();
  };
  stage(0);

  // tasks: (angle of the group, chunk of STRIDE_L lines); lane = line in
  // chunk.  Each line accumulates straight into its epilogue slot ep[ml][k]
  // (a lane owns one slot per task), so the task loop needs no registers per
  // task and stays rolled.
  const int nch = (a.n_s - (DIFF ? 1 : 0) + STRIDE_L - 1) / STRIDE_L;
  const int ntask = G.count * nch;
  for (int t = threadIdx.x; t < ntask; t += LS_THREADS)
    ttab[t] = make_short2((short)(t / nch), (short)((t % nch) * STRIDE_L));
  for (int i = threadIdx.x; i < G.count * a.NSp; i += LS_THREADS) ep[i] = 0.0f;
  const float kc = 0.5f * (float)(a.n_s - 1);

  for (int band = 0; band < nbands; ++band) {
    if (band + 1 < nbands) {
      stage(band + 1);
      dc::cp_async_wait<1>();
    } else {
      dc::cp_async_wait<0>();
    }
    __syncthreads();
    // byte offset of sample 0 of this band's stage
    const int st_off = ((band & 1) ? stage_sz : 0) * 4 + LS_PJ * LS_SQ * 4;
    const int r0 = band * LS_RB;
    const int nr = min(LS_RB, rows - r0);
    const float r0f = (float)r0;
    for (int t = warp; t < ntask; t += LS_WARPS) {
      const short2 tk = ttab[t];
      const LineMu &L = lmu[tk.x];
      const int k = min(tk.y + lane, a.n_s - 1);
      // anchor xi(r0) = b0 + kk*A + r0*d = J + fb, exactly split: kk*a_hi and
      // r0*d_hi are exact products, the low parts add below 2^-12
      const float kk = (float)k - kc;  // half-integer or integer
      const float t1 = kk * L.a_hi, th = r0f * L.d_hi;
      const float t1i = floorf(t1), thi = floorf(th);
      const float fr = L.b0f + (t1 - t1i) + (th - thi) + fmaf(kk, L.a_lo, r0f * L.d_lo);
      const float fri = floorf(fr);
      const int J = (int)L.b0i + (int)t1i + (int)thi + (int)fri;
      const float fb = fr - fri;
      const float dxi = L.dxi;
      // the lane's samples lie in [-1, len] somewhere in the band, or nowhere
      const float lo = (float)(-1 - J), hi = (float)(len - J);
      const float xa = fb, xb = fmaf((float)(nr - 1), dxi, fb);
      const bool outside = (fmaxf(xa, xb) <= lo) || (fminf(xa, xb) >= hi);
      if (__all_sync(0xffffffffu, outside)) continue;  // the band misses these lines
      float sum = 0.0f;
      if (!outside) {
        // byte offset of sample J of this stage, minus the floor's exponent bits
        const unsigned cb =
            (unsigned)(st_off + J * LS_SQ * 4) - 0x4B400000u * (unsigned)(LS_SQ * 4);
        sum = (nr == RB) ? band_sum<RB, RB>(sb, cb, RB, fb, dxi)
                         : band_sum<RB, 0>(sb, cb, nr, fb, dxi);
      }
      const int kl = tk.y + lane;
      if (DIFF) {
        float nb = __shfl_down_sync(0xffffffffu, sum, 1);
        if (lane < 31 && kl <= a.n_s - 2) ep[tk.x * a.NSp + kl] += nb - sum;
      } else {
        if (kl <= a.n_s - 1) ep[tk.x * a.NSp + kl] += sum;
      }
    }
    __syncthreads();
  }

  // line sums (RAW) or differences R_{k+1}-R_k (DIFF), times the Joseph scale
  for (int i = threadIdx.x; i < G.count * a.NSp; i += LS_THREADS) ep[i] *= lmu[i / a.NSp].jscale;
  __syncthreads();

  const float D = fv.D, D2 = D * D;
  const int total = G.count * a.NSp;
  auto s_half = [&](int k) { return s_half_of(k, a.n_s, a.ds); };
  auto Kw = [&](int m, float sh) { return redundancy_k(a.mu[m], fv, sh); };

  if (MODE == M_RAW || MODE == M_GRANGEAT) {
    for (int idx = threadIdx.x; idx < total; idx += LS_THREADS) {
      int ml = idx / a.NSp, k = idx % a.NSp;
      if (k >= a.n_s) continue;
      int m = a.mu_order[G.first + ml];
      float val;
      if (MODE == M_RAW) {
        val = ep[idx];
      } else {
        float sh = s_half(k);
        val = (k <= a.n_s - 2) ? ep[idx] * (fmaf(sh, sh, D2) / D2) / a.ds : 0.0f;
      }
      a.out[(((size_t)b * a.V + v) * a.n_mu + m) * a.n_s + k] = val;
    }
    return;
  }
  if (MODE == M_DIFFSTORE) {
    for (int idx = threadIdx.x; idx < total; idx += LS_THREADS) {
      int ml = idx / a.NSp, k = idx % a.NSp;
      int m = a.mu_order[G.first + ml];
      a.sinoA[((size_t)slot * a.n_mu + m) * a.NSp + k] = (k <= a.n_s - 2) ? ep[idx] : 0.0f;
    }
    return;
  }
  if (MODE == M_FILTER) {
    // Q = W K w_sino (R_{k+1}-R_k)/ds on s_{k+1/2}
    bool bad_w = false;
    for (int idx = threadIdx.x; idx < total; idx += LS_THREADS) {
      int ml = idx / a.NSp, k = idx % a.NSp;
      int m = a.mu_order[G.first + ml];
      float q = 0.0f;
      if (k <= a.n_s - 2) {
        float sh = s_half(k);
        float w = a.Wred ? a.Wred[((size_t)v * a.n_mu + m) * a.n_s + k] : 0.5f;
        bad_w |= !isfinite(w);
        q = w * Kw(m, sh) * (fmaf(sh, sh, D2) / D2) * ep[idx] / a.ds;
        // Grangeat's S (Eq. 7), kept for a reverse mode that reuses it
        if (a.Sout)
          a.Sout[(((size_t)b * a.V + v) * a.n_mu + m) * a.n_s + k] =
              ep[idx] * (fmaf(sh, sh, D2) / D2) / a.ds;
      } else if (a.Sout && k < a.n_s) {
        a.Sout[(((size_t)b * a.V + v) * a.n_mu + m) * a.n_s + k] = 0.0f;
      }
      ep[idx] = q;
    }
    if (bad_w) atomicOr(a.err, DC_FLAG_NONFINITE_W);
    __syncthreads();
    // P = D_b Q, times the A2d^T scale (pi/n_mu)(ds/p^2) and the Joseph scale
    for (int idx = threadIdx.x; idx < total; idx += LS_THREADS) {
      int ml = idx / a.NSp, k = idx % a.NSp;
      int m = a.mu_order[G.first + ml];
      float val = 0.0f;
      if (k < a.n_s) {
        float qm = (k > 0) ? ep[idx - 1] : 0.0f;
        val = (ep[idx] - qm) / a.ds * a.cT * lmu[ml].jscale;
      }
      a.out[((size_t)slot * a.n_mu + m) * a.NSp + k] = val;
    }
    return;
  }
  if (MODE == M_ADJ) {
    // sinoA holds jscale*(R_G[k+1]-R_G[k]) of w_d*dL/dg^F; this launch's
    // line differences are those of w_cos*g (Grangeat's S, recomputed).
    bool bad_w = false;
    for (int idx = threadIdx.x; idx < total; idx += LS_THREADS) {
      int ml = idx / a.NSp, k = idx % a.NSp;
      int m = a.mu_order[G.first + ml];
      size_t o = ((size_t)slot * a.n_mu + m) * a.NSp + k;
      float y = 0.0f, tW = 0.0f;
      if (k <= a.n_s - 2) {
        float sh = s_half(k);
        float wsino = fmaf(sh, sh, D2) / D2;
        float S = wsino * ep[idx] / a.ds;
        float Qg = -a.cT * a.sinoA[o] / a.ds;  // D_b^T of dL/dP
        float Kv = Kw(m, sh);
        float w = a.Wred ? a.Wred[((size_t)v * a.n_mu + m) * a.n_s + k] : 0.5f;
        bad_w |= !isfinite(w);
        tW = Kv * S * Qg;                       // dL/dW contribution
        y = wsino * w * Kv * Qg;                // dL/dS times w_sino
      }
      a.sinoA[o] = tW;
      ep[idx] = y;
    }
    if (bad_w) atomicOr(a.err, DC_FLAG_NONFINITE_W);
    __syncthreads();
    // dL/dR = D_f^T y; times the Joseph scale for the transpose gather
    for (int idx = threadIdx.x; idx < total; idx += LS_THREADS) {
      int ml = idx / a.NSp, k = idx % a.NSp;
      int m = a.mu_order[G.first + ml];
      float val = 0.0f;
      if (k < a.n_s) {
        float ym = (k > 0) ? ep[idx - 1] : 0.0f;
        float y0 = (k <= a.n_s - 2) ? ep[idx] : 0.0f;
        val = (ym - y0) / a.ds * lmu[ml].jscale;
      }
      a.sinoB[((size_t)slot * a.n_mu + m) * a.NSp + k] = val;
    }
  }
}

template <int MODE, int RB>
__global__ void __launch_bounds__(LS_THREADS, 1) k_linesum(LineArgs a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ LineMu lmu[dc::DC_LS_MAX_MG];
  __shared__ short2 ttab[dc::DC_LS_MAX_TASKS];
  linesum_body<MODE, RB, LS_THREADS>(a, blockIdx.x, blockIdx.y, blockIdx.y, smem, lmu, ttab);
}

// ----------------------------------------------------- 2-D backprojection
constexpr int BP2_THREADS = 256;
constexpr int BP2_NQ = 2;   // x positions per thread (lane, lane+32)
constexpr int BP2_RY = 16;  // rows per warp
constexpr int BP2_TX = 32 * BP2_NQ;
constexpr int BP2_TY = 8 * BP2_RY;
constexpr int BP2_MC = 12;  // angles per stage (2 stages: 4 CTAs per SM at 512 s-bins)

enum { OUT_F32 = 0, OUT_BF16 = 1, OUT_F32_ABSMAX = 2, OUT_F32_SLOT = 3 };

struct BP2Args {
  const float *sino;  // [n][n_mu][NSp], pre-scaled by the Joseph and mu scales
  int H, W, n_mu, n_s, NSp;
  int V, B, v0, n_img;  // B = batch items in this chunk
  int b0;
  float pitch, ds;
  const dc::FView *fv;
  const dc::MuRec *mu;
  const dc::VMu *vmu;  // [V][n_mu]
  int weight;          // WT_NONE / WT_COS / WT_D
  int out_kind;        // OUT_*
  void *out;           // user [B][V][H][W] (f32 or bf16) or scratch [n][H][Wp] f32
                       // (OUT_F32_ABSMAX, OUT_F32_SLOT)
  int Wp;
  unsigned *absmax;    // [n] (OUT_F32_ABSMAX)
  unsigned *err;
};

// per-angle constants of one tile: the s-bin position of pixel (j0 + jl,
// r0 + rl) is I00 + F00 + jl*Bc + rl*Bs (I00 integer, F00 in [0, 1))
struct BPMu {
  float F00, Bc, Bs, winv;  // winv: slope of the Joseph hat in s-bins
  float w1c, lo, hi;        // 1 - winv; positions relative to I00 clamp to [lo, hi]
  unsigned cbase;           // byte offset of s-bin I00 in its stage, minus the floor's exponent bits
  int fast;                 // positions stay inside (lo, hi) over the tile: no clamp
  int row0;                 // float offset of s-bin I00 in its stage
  int pad1, pad2;
};

// Barrier of one group of BP2_THREADS threads (named barrier `id`; id 0 with
// a CTA of exactly BP2_THREADS threads is __syncthreads), and its OR-reduction.
__device__ __forceinline__ void group_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(BP2_THREADS) : "memory");
}
__device__ __forceinline__ bool group_sync_or(int id, bool pred) {
  unsigned r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((unsigned)pred), "r"(id), "n"(BP2_THREADS)
      : "memory");
  return r != 0;
}

// One BP2_TX x (8 RY) pixel tile (tile_x, tile_y) of image n (view
// a.v0 + n / a.B, item a.b0 + n % a.B) by a group of BP2_THREADS threads (gt:
// thread within the group; barrier `bar_id`).  The sinograms come from
// work-area slot `slot` of a.sino; OUT_F32_ABSMAX writes slot `slot` of the
// scratch and a.absmax[slot].  `smem` holds the group's two stages, `bars`
// its two mbarriers (initialised by the caller), `bmu` its per-angle
// constants; `it` counts the angle chunks the group has staged so far (the
// stage and the barrier phase of the next chunk follow from it).  Returns
// false if a bounded wait gave up.  OUT_F32_SLOT writes slot `slot` of the
// scratch without the absmax.
//
// MULTI: ds < pitch, where the transposed Joseph hat of an angle (half-width
// 1/winv s-bins, at most 3 for ds >= pitch/3) covers up to six taps; those
// are summed with explicit bounds instead of the two-tap fast paths.
template <bool MULTI, int RY>
__device__ __forceinline__ bool bp2d_tile(const BP2Args &a, int n, int slot, int tile_x,
                                          int tile_y, int gt, int bar_id, float *smem,
                                          uint64_t *bars, BPMu (*bmu)[BP2_MC], unsigned &it) {
  const int v = a.v0 + n / a.B, b = a.b0 + n % a.B;
  const dc::FView fv = a.fv[v];
  const int warp = gt >> 5, lane = gt & 31;
  constexpr int TY = 8 * RY;  // tile rows: RY per warp
  const int j0 = tile_x * BP2_TX, r0 = tile_y * TY;
  const int rstride = a.NSp + PADL + PADR;
  const int stage_sz = BP2_MC * rstride;
  const float *src = a.sino + (size_t)slot * a.n_mu * a.NSp;
  const int nchunk = (a.n_mu + BP2_MC - 1) / BP2_MC;
  const char *sb = reinterpret_cast<const char *>(smem);
  const unsigned it0 = it;

  // zero pads left and right of every stage row (the copies fill the middle)
  for (int i = gt; i < 2 * BP2_MC; i += BP2_THREADS) {
    float *row = smem + (size_t)i * rstride;
    for (int t = 0; t < PADL; ++t) row[t] = 0.0f;
    for (int t = PADL + a.NSp; t < rstride; ++t) row[t] = 0.0f;
  }
  group_sync(bar_id);
  auto issue = [&](int c) {
    const unsigned st = (it0 + c) & 1;
    int m0 = c * BP2_MC, nm = min(BP2_MC, a.n_mu - m0);
    uint64_t *bar = &bars[st];
    dc::fence_proxy_async();
    dc::mbar_arrive_expect_tx(bar, (unsigned)(nm * a.NSp * 4));
    for (int q = 0; q < nm; ++q)
      dc::bulk_g2s(smem + st * stage_sz + (size_t)q * rstride + PADL, src + (size_t)(m0 + q) * a.NSp,
                   (unsigned)(a.NSp * 4), bar);
  };
  // per-angle constants of this tile, from exact float splits of the origin
  auto angle_consts = [&](int c) {
    int mi = gt;
    int m = c * BP2_MC + mi;
    if (mi < BP2_MC && m < a.n_mu) {
      const dc::MuRec R = a.mu[m];
      const dc::VMu Q = a.vmu[(size_t)v * a.n_mu + m];
      float fj0 = (float)j0, fr0 = (float)r0;
      float t = fj0 * R.bc_hi + fr0 * R.bs_hi;  // exact
      float ti = floorf(t);
      float F = Q.xof + (t - ti) + fmaf(fj0, R.bc_lo, fr0 * R.bs_lo);
      float Fi = floorf(F);
      const float I00 = Q.xoi + ti + Fi;
      BPMu M;
      M.F00 = F - Fi;
      M.Bc = R.bc_hi + R.bc_lo;
      M.Bs = R.bs_hi + R.bs_lo;
      M.winv = R.winv;
      M.w1c = 1.0f - R.winv;
      M.lo = -1.0f - I00;
      M.hi = (float)a.n_s - I00;
      M.cbase = (unsigned)((mi * rstride + PADL + (int)I00) * 4) - 4u * 0x4B400000u;
      float ex = (float)(BP2_TX - 1) * M.Bc, ey = (float)(TY - 1) * M.Bs;
      float xmin = M.F00 + fminf(ex, 0.0f) + fminf(ey, 0.0f);
      float xmax = M.F00 + fmaxf(ex, 0.0f) + fmaxf(ey, 0.0f);
      M.fast = (xmin >= M.lo + 0.01f && xmax <= M.hi - 0.01f) ? 1 : 0;
      M.row0 = mi * rstride + PADL + (int)I00;
      M.pad1 = M.pad2 = 0;
      bmu[(it0 + c) & 1][mi] = M;
    }
  };
  if (gt == 0) {
    issue(0);
    if (nchunk > 1) issue(1);
  }
  angle_consts(0);

  // a thread's two pixels of a row (columns lane and lane + 32) are held as
  // the two halves of a float2 and stepped with the packed FP32x2 operations
  // of sm_100+ (one issue slot for both); every component is rounded as the
  // scalar operation would round it
  static_assert(BP2_NQ == 2, "two pixels per thread and row, packed");
  float2 acc[RY];
#pragma unroll
  for (int ry = 0; ry < RY; ++ry) acc[ry] = make_float2(0.0f, 0.0f);
  const float rl0 = (float)(warp * RY);
  float jlf[BP2_NQ], rlf[RY];  // pixel offsets inside the tile, as floats
#pragma unroll
  for (int q = 0; q < BP2_NQ; ++q) jlf[q] = (float)(lane + 32 * q);
#pragma unroll
  for (int ry = 0; ry < RY; ++ry) rlf[ry] = rl0 + (float)ry;
  const float2 jl2 = make_float2(jlf[0], jlf[1]);
  const float2 mM2 = make_float2(-12582912.0f, -12582912.0f);  // -1.5 * 2^23
  const float2 M2 = make_float2(12582912.0f, 12582912.0f);
  const float2 m12 = make_float2(-1.0f, -1.0f);

  bool ok = true;
  for (int c = 0; c < nchunk; ++c) {
    const unsigned st = (it0 + c) & 1;
    if (c + 1 < nchunk) angle_consts(c + 1);
    if (!dc::mbar_wait_bounded(&bars[st], ((it0 + c) >> 1) & 1, a.err)) ok = false;
    if (group_sync_or(bar_id, !ok)) {
      ok = false;
      break;
    }
    const unsigned st_off = st * (unsigned)(stage_sz * 4);  // bytes
    int nm = min(BP2_MC, a.n_mu - c * BP2_MC);
#pragma unroll 2
    for (int mi = 0; mi < nm; ++mi) {
      const BPMu M = bmu[st][mi];
      const unsigned cb = M.cbase + st_off;
      if (MULTI) {
        // taps k = floor(x) - 2 .. floor(x) + 3 (relative to I00) inside the
        // s range [lo + 1, hi - 1]; weight max(0, 1 - winv |x - k|)
        const float *row = smem + st * stage_sz + M.row0;
        const int klo = (int)M.lo + 1, khi = (int)M.hi - 1;
#pragma unroll
        for (int ry = 0; ry < RY; ++ry) {
          float rt = fmaf(rlf[ry], M.Bs, M.F00);
#pragma unroll
          for (int q = 0; q < BP2_NQ; ++q) {
            float f;
            const int k0 = dc::floor_frac(fmaf(jlf[q], M.Bc, rt), f);
            float sum = 0.0f;
#pragma unroll
            for (int t = -2; t <= 3; ++t) {
              const int kk = k0 + t;
              const float w = fmaxf(0.0f, fmaf(-fabsf(f - (float)t), M.winv, 1.0f));
              if (kk >= klo && kk <= khi) sum = fmaf(w, row[kk], sum);
            }
            if (q == 0) acc[ry].x += sum;
            else acc[ry].y += sum;
          }
        }
      } else {
        // two-tap paths (ds >= pitch, so winv >= 1): the hat weights
        // 1 - f winv and 1 - (1 - f) winv never exceed 1, so clamping them
        // below at 0 is a saturation to [0, 1].  The s-bin position of a
        // pixel is (jl Bc + F00) + rl Bs: the first part once per angle, one
        // packed FMA per row.
        const float2 base = __ffma2_rn(jl2, make_float2(M.Bc, M.Bc), make_float2(M.F00, M.F00));
        const float2 Bs2 = make_float2(M.Bs, M.Bs);
        auto pair_row = [&](int ry, bool clamp) {
          float2 x = __ffma2_rn(make_float2(rlf[ry], rlf[ry]), Bs2, base);
          if (clamp)
            x = make_float2(fminf(fmaxf(x.x, M.lo), M.hi), fminf(fmaxf(x.y, M.lo), M.hi));
          // exact floor (rounded-down bits) and fraction, as in band_sum
          const float2 t = __fadd2_rd(x, M2);
          const float2 f = __ffma2_rn(__fadd2_rn(t, mM2), m12, x);
          const unsigned o0 = __float_as_uint(t.x) * 4u + cb, o1 = __float_as_uint(t.y) * 4u + cb;
          const float2 p0 = make_float2(*reinterpret_cast<const float *>(sb + o0),
                                        *reinterpret_cast<const float *>(sb + o1));
          const float2 p1 = make_float2(*reinterpret_cast<const float *>(sb + o0 + 4),
                                        *reinterpret_cast<const float *>(sb + o1 + 4));
          const float2 w0 = make_float2(__saturatef(fmaf(-f.x, M.winv, 1.0f)),
                                        __saturatef(fmaf(-f.y, M.winv, 1.0f)));
          const float2 w1 = make_float2(__saturatef(fmaf(f.x, M.winv, M.w1c)),
                                        __saturatef(fmaf(f.y, M.winv, M.w1c)));
          acc[ry] = __ffma2_rn(w0, p0, __ffma2_rn(w1, p1, acc[ry]));
        };
        if (M.fast) {
#pragma unroll
          for (int ry = 0; ry < RY; ++ry) pair_row(ry, false);
        } else {
#pragma unroll
          for (int ry = 0; ry < RY; ++ry) pair_row(ry, true);
        }
      }
    }
    group_sync(bar_id);
    if (gt == 0 && c + 2 < nchunk) issue(c + 2);
  }
  it = it0 + (unsigned)nchunk;
  if (!ok) {
    for (int s2 = 0; s2 < 2; ++s2) dc::mbar_wait_bounded(&bars[s2], 0, nullptr);
    return false;
  }

  float lmax = 0.0f;
#pragma unroll
  for (int ry = 0; ry < RY; ++ry) {
    int r = r0 + warp * RY + ry;
#pragma unroll
    for (int q = 0; q < BP2_NQ; ++q) {
      int j = j0 + lane + 32 * q;
      if (r >= a.H || j >= a.W) continue;
      float val = (q == 0) ? acc[ry].x : acc[ry].y;
      if (a.weight != WT_NONE) {
        float x = (j - fv.cu) * a.pitch, y = (r - fv.cv) * a.pitch;
        float l2 = fmaf(x, x, fmaf(y, y, fv.D * fv.D));
        val *= (a.weight == WT_D) ? l2 : fv.D * rsqrtf(l2);
      }
      if (a.out_kind == OUT_F32_ABSMAX || a.out_kind == OUT_F32_SLOT) {
        ((float *)a.out)[((size_t)slot * a.H + r) * a.Wp + j] = val;
        lmax = fmaxf(lmax, fabsf(val));
      } else {
        size_t o = (((size_t)b * a.V + v) * a.H + r) * a.W + j;
        if (a.out_kind == OUT_BF16)
          ((__nv_bfloat16 *)a.out)[o] = __float2bfloat16_rn(val);
        else
          ((float *)a.out)[o] = val;
      }
    }
  }
  if (a.out_kind == OUT_F32_ABSMAX) {
    for (int o = 16; o > 0; o >>= 1) lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    if (lane == 0) atomicMax(&a.absmax[slot], __float_as_uint(lmax));
  }
  return true;
}

#include "dc_filter_quad.cuh"

template <bool MULTI>
__global__ void __launch_bounds__(BP2_THREADS) k_bp2d(BP2Args a) {
  extern __shared__ __align__(16) float smem[];
  __shared__ uint64_t bars[2];
  __shared__ BPMu bmu[2][BP2_MC];
  if (threadIdx.x == 0) {
    dc::mbar_init(&bars[0], 1);
    dc::mbar_init(&bars[1], 1);
    dc::fence_barrier_init();
  }
  __syncthreads();
  unsigned it = 0;
  bp2d_tile<MULTI, BP2_RY>(a, blockIdx.z, blockIdx.z, blockIdx.x, blockIdx.y, threadIdx.x, 0, smem,
                           bars, bmu, it);
}

// FP16 storage with a per-view power-of-two scale chosen from the absmax so
// that the largest value maps into [2^14, 2^15): g^F = half * scale.
__global__ void k_to_f16(const float *__restrict__ src, const unsigned *__restrict__ absmax,
                         int H, int W, int Wp, int V, int B, int v0, int b0,
                         __half *__restrict__ dst, float *__restrict__ scale) {
  int n = blockIdx.y;
  int v = v0 + n / B, b = b0 + n % B;
  float am = __uint_as_float(absmax[n]);
  float sc = 1.0f;
  if (am > 0.0f) {
    int e;
    frexpf(am, &e);          // am = m * 2^e, m in [0.5, 1)
    sc = ldexpf(1.0f, e - 15);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) scale[(size_t)b * V + v] = sc;
  float inv = 1.0f / sc;     // exact: power of two
  size_t np = (size_t)H * W;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < np;
       i += (size_t)gridDim.x * blockDim.x) {
    int r = (int)(i / W), j = (int)(i % W);
    float val = src[((size_t)n * H + r) * Wp + j] * inv;
    dst[((size_t)b * V + v) * np + i] = __float2half_rn(val);
  }
}

// FP32 pair storage (DC_F32X2): pixel (r, c) of g^F becomes the pair
// (g[r][c], g[r][c+1] - g[r][c]), with g[r][W] = 0 (the detector's zero
// extension), the tap pair of the backprojection's row interpolation.  A
// thread converts two neighbouring pixels: three loads of the L2-resident
// scratch row, one 16-byte store (W even) or two 8-byte stores.
__global__ void k_to_pairs(const float *__restrict__ src, int H, int W, int Wp, int V, int B,
                           int v0, int b0, float2 *__restrict__ dst) {
  const int n = blockIdx.y;
  const int v = v0 + n / B, b = b0 + n % B;
  const int half = (W + 1) >> 1;  // pixel pairs per row
  const size_t np = (size_t)H * W;
  float2 *out = dst + ((size_t)b * V + v) * np;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < (size_t)H * half;
       i += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(i / half), j = 2 * (int)(i - (size_t)r * half);
    const float *row = src + ((size_t)n * H + r) * Wp;
    const float g0 = row[j];
    const float g1 = (j + 1 < W) ? row[j + 1] : 0.0f;
    const float g2 = (j + 2 < W) ? row[j + 2] : 0.0f;
    float2 *o = out + (size_t)r * W + j;
    if ((W & 1) == 0) {
      *reinterpret_cast<float4 *>(o) = make_float4(g0, g1 - g0, g1, g2 - g1);
    } else {
      o[0] = make_float2(g0, g1 - g0);
      if (j + 1 < W) o[1] = make_float2(g1, g2 - g1);
    }
  }
}

// sum over the batch of the per-image dL/dW contributions (fixed order);
// QUAD: the images are interleaved by four
template <bool QUAD>
__global__ void k_reduce_gradW(const float *__restrict__ sinoA, int n_mu, int n_s, int NSp,
                               int B, int v0, int nv, int accumulate,
                               float *__restrict__ gradW) {
  size_t total = (size_t)nv * n_mu * n_s;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    int k = (int)(i % n_s);
    size_t t = i / n_s;
    int m = (int)(t % n_mu);
    int vl = (int)(t / n_mu);
    float s = 0.0f;
    for (int b = 0; b < B; ++b) {
      const size_t n = (size_t)vl * B + b;
      s += QUAD ? sinoA[(((n >> 2) * n_mu + m) * NSp + k) * 4 + (n & 3)]
                : sinoA[(n * n_mu + m) * NSp + k];
    }
    size_t o = ((size_t)(v0 + vl) * n_mu + m) * n_s + k;
    gradW[o] = accumulate ? gradW[o] + s : s;
  }
}

// copy a user sinogram [B][V][n_mu][n_s] into the padded work layout, times
// the Joseph scale of each angle (for the transpose gather)
__global__ void k_sino_in(const float *__restrict__ R, const dc::MuRec *__restrict__ mu,
                          int n_mu, int n_s, int NSp, int V, int B, int v0, int b0,
                          float *__restrict__ dst) {
  int n = blockIdx.y;
  int v = v0 + n / B, b = b0 + n % B;
  size_t total = (size_t)n_mu * NSp;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    int m = (int)(i / NSp), k = (int)(i % NSp);
    float val = 0.0f;
    if (k < n_s) val = R[(((size_t)b * V + v) * n_mu + m) * n_s + k] * mu[m].jscale;
    dst[(size_t)n * total + i] = val;
  }
}

int round4(int x) { return (x + 3) & ~3; }

// The last step of the filter's reverse mode with Grangeat's S read from
// memory (kept by the forward pass) instead of recomputed by a line-sum
// pass: the same arithmetic as the M_ADJ epilogue of k_linesum.  A CTA
// takes AS_ROWS angles of one image; sinoA holds jscale (R_G[k+1] - R_G[k])
// of w_d dL/dg^F on entry and dL/dW contributions on exit, sinoB receives
// D_f^T of dL/dS (times the Joseph scale) for the 2-D backprojection.
constexpr int AS_ROWS = 4;

__global__ void __launch_bounds__(256) k_adj_from_s(LineArgs a, const float *__restrict__ S) {
  extern __shared__ float ys[];  // [AS_ROWS][NSp]
  const int n = blockIdx.y;
  const int v = a.v0 + n / a.B, b = a.b0 + n % a.B;
  const dc::FView fv = a.fv[v];
  const float D = fv.D, D2 = D * D;
  const int m0 = blockIdx.x * AS_ROWS;
  const int total = min(AS_ROWS, a.n_mu - m0) * a.NSp;
  bool bad_w = false;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int m = m0 + idx / a.NSp, k = idx % a.NSp;
    const size_t o = ((size_t)n * a.n_mu + m) * a.NSp + k;
    float y = 0.0f, tW = 0.0f;
    if (k <= a.n_s - 2) {
      const float sh = s_half_of(k, a.n_s, a.ds);
      const float wsino = fmaf(sh, sh, D2) / D2;
      const float Sv = S[(((size_t)b * a.V + v) * a.n_mu + m) * a.n_s + k];
      const float Qg = -a.cT * a.sinoA[o] / a.ds;  // D_b^T of dL/dP
      const float Kv = redundancy_k(a.mu[m], fv, sh);
      const float w = a.Wred ? a.Wred[((size_t)v * a.n_mu + m) * a.n_s + k] : 0.5f;
      bad_w |= !isfinite(w);
      tW = Kv * Sv * Qg;
      y = wsino * w * Kv * Qg;
    }
    a.sinoA[o] = tW;
    ys[idx] = y;
  }
  if (bad_w) atomicOr(a.err, DC_FLAG_NONFINITE_W);
  __syncthreads();
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int m = m0 + idx / a.NSp, k = idx % a.NSp;
    float val = 0.0f;
    if (k < a.n_s) {
      const float ym = (k > 0) ? ys[idx - 1] : 0.0f;
      const float y0 = (k <= a.n_s - 2) ? ys[idx] : 0.0f;
      val = (ym - y0) / a.ds * a.mu[m].jscale;
    }
    a.sinoB[((size_t)n * a.n_mu + m) * a.NSp + k] = val;
  }
}

size_t linesum_smem_for(int H, int W, int mg, int NSp, int rb) {
  return (size_t)(2 * (std::max(H, W) + 2 * (rb + 1)) * (rb + 1) + mg * NSp) * sizeof(float);
}

// tallest band whose two stages fit the shared-memory budget (0: none)
int linesum_band_rows(int H, int W, int mg, int NSp, size_t budget = LS_SMEM_BUDGET) {
  for (int rb = 32; rb >= 8; rb /= 2)
    if (linesum_smem_for(H, W, mg, NSp, rb) <= budget) return rb;
  return 0;
}

size_t linesum_smem(const dc_geometry *g) {
  return linesum_smem_for(g->d.det_rows, g->d.det_cols, g->mg, g->NSp, g->ls_rb);
}

template <int MODE, int RB>
int launch_linesum_rb(dim3 grid, LineArgs &a, size_t sm, cudaStream_t st) {
  static bool attr_done = false;  // per template instance
  if (!attr_done) {
    DC_CUDA(cudaFuncSetAttribute(k_linesum<MODE, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 LS_SMEM_BUDGET));
    attr_done = true;
  }
  k_linesum<MODE, RB><<<grid, LS_THREADS, sm, st>>>(a);
  DC_CHECK_LAUNCH("k_linesum");
  return DC_OK;
}

size_t bp2d_smem(const dc_geometry *g) {
  return (size_t)(2 * BP2_MC * (g->NSp + PADL + PADR)) * sizeof(float);
}

template <int MODE>
int launch_linesum4(const dc_geometry *g, LineArgs &a, cudaStream_t st) {
  const L4Shape sh = l4_shape(a.H, a.W);
  a.mg = g->q_mg;
  a.groups = g->q_groups;
  DC_CUDA(cudaFuncSetAttribute(k_linesum4<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               L4_SMEM_BUDGET));
  dim3 grid(g->q_n_groups, (a.n_img + 3) / 4);
  k_linesum4<MODE><<<grid, L4_THREADS, l4_smem(sh, a.mg, a.NSp), st>>>(a, sh, g->q_tm_cols,
                                                                       g->q_tm_rows);
  DC_CHECK_LAUNCH("k_linesum4");
  return DC_OK;
}

// line sums of the images that launch_prep staged with the same `quad`
template <int MODE>
int launch_linesum(const dc_geometry *g, LineArgs &a, bool quad, cudaStream_t st) {
  if (quad) {
    dc::ProfScope ps(dc::KID_LINESUM, st);
    return launch_linesum4<MODE>(g, a, st);
  }
  size_t sm = linesum_smem(g);
  dim3 grid(g->n_groups, a.n_img);
  dc::ProfScope ps(dc::KID_LINESUM, st);
  switch (g->ls_rb) {
    case 32: return launch_linesum_rb<MODE, 32>(grid, a, sm, st);
    case 16: return launch_linesum_rb<MODE, 16>(grid, a, sm, st);
    default: return launch_linesum_rb<MODE, 8>(grid, a, sm, st);
  }
}

bool multi_tap(const dc_geometry *g) { return g->d.ds < g->d.pitch * (1.0 - 1e-12); }

template <int NT, int RY>
int launch_bp2d4_t(const dc_geometry *g, BP2Args &a, const B4Shape &sh, const CUtensorMap &tm,
                   cudaStream_t st) {
  const size_t sm = b4_smem(sh);
  // the limit belongs to the kernel, not to the launch: one value for all
  // geometries, so that no thread lowers it under another's launch
  DC_CUDA(cudaFuncSetAttribute(k_bp2d4<NT, RY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               B4_SMEM_MAX));
  const int tx = 32 * sh.nwx, ty = RY * (8 / sh.nwx);
  dim3 grid((a.W + tx - 1) / tx, (a.H + ty - 1) / ty, (a.n_img + 3) / 4);
  k_bp2d4<NT, RY><<<grid, B4_THREADS, sm, st>>>(a, sh, tm);
  DC_CHECK_LAUNCH("k_bp2d4");
  return DC_OK;
}

template <int NT>
int launch_bp2d4(const dc_geometry *g, BP2Args &a, cudaStream_t st) {
  const B4Shape sh = b4_arrange(g->q_nwx, g->d.pitch, g->d.ds, g->q_ry);
  const CUtensorMap &tm = (a.sino == g->w_sinoB) ? g->q_tm_sinoB : g->q_tm_sinoA;
  return g->q_ry == 2 ? launch_bp2d4_t<NT, 2>(g, a, sh, tm, st)
                      : launch_bp2d4_t<NT, 8>(g, a, sh, tm, st);
}

// 2-D backprojection of the sinograms that the same `quad` laid out
int launch_bp2d(const dc_geometry *g, BP2Args &a, bool quad, cudaStream_t st) {
  if (quad) {
    dc::ProfScope ps(dc::KID_BP2D, st);
    switch (b4_taps(g->d.pitch, g->d.ds)) {
      case 2: return launch_bp2d4<2>(g, a, st);
      case 4: return launch_bp2d4<4>(g, a, st);
      default: return launch_bp2d4<6>(g, a, st);
    }
  }
  size_t sm = bp2d_smem(g);
  static bool attr_done = false;
  if (!attr_done) {
    DC_CUDA(cudaFuncSetAttribute(k_bp2d<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 200 * 1024));
    DC_CUDA(cudaFuncSetAttribute(k_bp2d<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 200 * 1024));
    attr_done = true;
  }
  dim3 grid((a.W + BP2_TX - 1) / BP2_TX, (a.H + BP2_TY - 1) / BP2_TY, a.n_img);
  dc::ProfScope ps(dc::KID_BP2D, st);
  if (multi_tap(g))
    k_bp2d<true><<<grid, BP2_THREADS, sm, st>>>(a);
  else
    k_bp2d<false><<<grid, BP2_THREADS, sm, st>>>(a);
  DC_CHECK_LAUNCH("k_bp2d");
  return DC_OK;
}

int launch_prep(const dc_geometry *g, const float *src, int weight, int v0, int n_img, int B,
                int b0, bool quad, cudaStream_t st) {
  const dc_geometry_desc &d = g->d;
  PrepArgs p;
  p.src = src;
  p.img = g->w_img;
  p.fv = g->fv;
  p.H = d.det_rows;
  p.W = d.det_cols;
  p.Wp = g->Wp;
  p.V = d.n_views;
  p.B = B;
  p.v0 = v0;
  p.b0 = b0;
  p.Bt = 0;
  p.n_img = n_img;
  p.pitch = (float)d.pitch;
  p.weight = weight;
  dc::ProfScope ps(dc::KID_PREP, st);
  if (quad) {
    dim3 grid((d.det_cols + 31) / 32, (d.det_rows + 31) / 32, (n_img + 3) / 4);
    k_prep4<<<grid, dim3(32, 8), 0, st>>>(p, (float4 *)g->w_img, (float4 *)g->w_imgT);
    DC_CHECK_LAUNCH("k_prep4");
    return DC_OK;
  }
  dim3 grid((g->Wp + 31) / 32, (d.det_rows + 31) / 32, n_img);
  k_prep<<<grid, dim3(32, 8), 0, st>>>(p);
  DC_CHECK_LAUNCH("k_prep");
  return DC_OK;
}

LineArgs line_args(const dc_geometry *g, int B, int v0, int b0, int n_img) {
  const dc_geometry_desc &d = g->d;
  LineArgs a;
  memset(&a, 0, sizeof(a));
  a.img = g->w_img;
  a.H = d.det_rows;
  a.W = d.det_cols;
  a.Wp = g->Wp;
  a.n_mu = d.n_mu;
  a.n_s = d.n_s;
  a.NSp = g->NSp;
  a.V = d.n_views;
  a.B = B;
  a.v0 = v0;
  a.b0 = b0;
  a.n_img = n_img;
  a.pitch = (float)d.pitch;
  a.ds = (float)d.ds;
  a.cT = (float)((M_PI / d.n_mu) * d.ds / (d.pitch * d.pitch));
  a.mu = g->mu;
  a.vmu = g->vmu;
  a.mu_order = g->mu_order;
  a.groups = g->groups;
  a.fv = g->fv;
  a.err = g->w_flags;
  a.mg = g->mg;
  return a;
}

BP2Args bp2_args(const dc_geometry *g, int B, int v0, int b0, int n_img, const float *sino) {
  const dc_geometry_desc &d = g->d;
  BP2Args a;
  memset(&a, 0, sizeof(a));
  a.sino = sino;
  a.H = d.det_rows;
  a.W = d.det_cols;
  a.n_mu = d.n_mu;
  a.n_s = d.n_s;
  a.NSp = g->NSp;
  a.V = d.n_views;
  a.B = B;
  a.v0 = v0;
  a.b0 = b0;
  a.n_img = n_img;
  a.pitch = (float)d.pitch;
  a.ds = (float)d.ds;
  a.fv = g->fv;
  a.mu = g->mu;
  a.vmu = g->vmu;
  a.Wp = g->Wp;
  a.absmax = g->w_absmax;
  a.err = g->w_flags;
  return a;
}

int check_common(const dc_geometry *g, int B, const char *who) {
  if (!g) return dc::fail(DC_ERR_ARG, std::string(who) + ": NULL geometry");
  if (B < 1) return dc::fail(DC_ERR_ARG, std::string(who) + ": batch must be >= 1");
  int dev = -1;
  cudaGetDevice(&dev);
  if (dev != g->device)
    return dc::fail(DC_ERR_ARG, std::string(who) + ": geometry belongs to another device");
  return DC_OK;
}

// A chunk holds bc batch items of cv views (bc * cv <= chunk_images images).
struct Chunking {
  int bc, cv;
};
Chunking chunking(const dc_geometry *g, int B, int view_limit = 0) {
  Chunking c;
  c.bc = std::min(B, g->chunk_images);
  c.cv = std::max(1, g->chunk_images / c.bc);
  if (view_limit > 0) c.cv = std::min(c.cv, view_limit);
  return c;
}

// Chunks planned for one image (view_chunk or chunk_images of 1) keep the
// per-image kernels.  The rule looks at the plan of the whole call, not at a
// chunk, so that every image of a call takes the same path; a group that is not
// full costs what a full one does, which is still less than one image alone
// (filter of one image: 64 x 64, 180 angles 160 us per image, 57 as a group;
// 384 x 512, 720 angles 689 and 419).
bool use_quad(const dc_geometry *g, int bc, int cv) { return g->quad && bc * cv >= 2; }

// BF16 storage keeps the per-image kernels, so that a stored g^F and what is
// reconstructed from it stay the bits they were.  The two paths' FP32 results
// differ by their rounding (5e-6 relative), which turns 0.1 % of the BF16
// roundings the other way, each by 2^-8 of its value: reconstructions 2.2e-5
// apart (relative L2; 1.5e-3 at most), equally far from FP64.  FP16's roundings
// are eight times finer (5e-6, 6e-5).
bool quad_storage(int dtype) { return dtype != DC_BF16; }

// ------------------------------------------------ batched persistent filter
// One kernel filters every view of a batch of problems (orbits with uneven
// view counts, detectors and angle grids): persistent CTAs of BF_THREADS
// threads, one per SM, take (problem, view) items from a device counter.  An
// item is a whole image: its weighted copy (w_cos, rows padded) goes to the
// CTA's own image scratch, the line sums of every angle group fill the CTA's
// sinogram scratch (the M_FILTER epilogue: D_f, w_sino, W K, D_b), and the
// 2-D backprojection of that sinogram (w_d epilogue) is computed by the
// CTA's two halves, each a group of BP2_THREADS threads with its own stages,
// mbarriers and named barrier, taking alternate pixel tiles.  FP16 storage
// keeps the FP32 result in the image scratch, then converts it with the
// image's power-of-two scale.
constexpr int BF_THREADS = 512;
static_assert(BF_THREADS == 2 * BP2_THREADS, "two 2-D backprojection groups per CTA");
// rows per warp of the 2-D backprojection tiles here: with one CTA per SM a
// warp keeps 16 pixels in flight (64 x 64 tiles) to hide latency with half
// the warps of the standalone kernel's four CTAs per SM
constexpr int BF_RY = 16;
constexpr int DC_BF_MAX = 32;

struct FilterProblem {
  LineArgs la;          // the geometry's tables; img, out and Wred are set per CTA / run
  BP2Args ba;           // out = the problem's g^F; sino, absmax and out (FP16) per CTA
  long long first;      // first item (view 0) of this problem
  int rb;               // line-sum band rows (32, 16, 8)
  int n_groups;         // angle groups of the line sums
  int multi;            // ds < pitch: the bounds-checked multi-tap 2-D backprojection
  int tiles_x, tiles_y;
  int dtype;            // DC_F32 / DC_BF16 / DC_F16
  float *scale;         // [V] FP16 scales
};

struct FilterRun {
  const float *g[DC_BF_MAX];   // [V][H][W] projections of each table entry
  const float *W[DC_BF_MAX];   // [V][n_mu][n_s] weights or NULL (= 1/2)
};

template <int RB>
__device__ __forceinline__ void linesum_all_groups(const LineArgs &la, int v, int n_groups,
                                                   float *smem, LineMu *lmu, short2 *ttab) {
  for (int gi = 0; gi < n_groups; ++gi) {
    linesum_body<M_FILTER, RB, BF_THREADS>(la, gi, v, 0, smem, lmu, ttab);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(BF_THREADS, 1)
    k_filter_batched(const FilterProblem *__restrict__ probs, int nprob, long long total,
                     unsigned long long *counter, FilterRun run, float *img_scratch,
                     size_t img_cap, float *sino_scratch, size_t sino_cap,
                     unsigned *absmax_scratch, int bp2_floats) {
  extern __shared__ __align__(16) float smem[];
  __shared__ LineMu lmu[dc::DC_LS_MAX_MG];
  __shared__ short2 ttab[dc::DC_LS_MAX_TASKS];
  __shared__ uint64_t bars[2][2];
  __shared__ BPMu bmu[2][2][BP2_MC];
  __shared__ long long item;
  __shared__ int failed;
  const int tid = threadIdx.x, grp = tid / BP2_THREADS, gt = tid % BP2_THREADS;
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      dc::mbar_init(&bars[q][0], 1);
      dc::mbar_init(&bars[q][1], 1);
    }
    dc::fence_barrier_init();
    failed = 0;
  }
  float *img = img_scratch + (size_t)blockIdx.x * img_cap;
  float *sino = sino_scratch + (size_t)blockIdx.x * sino_cap;
  unsigned *amax = absmax_scratch + blockIdx.x;
  unsigned it = 0;  // angle chunks staged by this thread's group
  for (;;) {
    __syncthreads();
    if (tid == 0) item = (long long)atomicAdd(counter, 1ull);
    __syncthreads();
    const long long w = item;
    if (w >= total || failed) break;
    int p = 0;
    while (p + 1 < nprob && probs[p + 1].first <= w) ++p;
    const FilterProblem &P = probs[p];
    const int v = (int)(w - P.first);
    LineArgs la = P.la;
    la.img = img;
    la.out = sino;
    la.Wred = run.W[p];
    BP2Args ba = P.ba;
    ba.sino = sino;
    ba.absmax = amax;
    if (P.dtype == DC_F16) ba.out = img;

    // w_cos g of view v into the image scratch, rows padded to Wp with zeros
    {
      const dc::FView f = la.fv[v];
      const float *src = run.g[p] + (size_t)v * la.H * la.W;
      for (int r = tid / 32; r < la.H; r += BF_THREADS / 32)
        for (int j = tid % 32; j < la.Wp; j += 32) {
          float val = 0.0f;
          if (j < la.W) {
            const float x = (j - f.cu) * la.pitch, y = (r - f.cv) * la.pitch;
            val = src[(size_t)r * la.W + j] * (f.D * rsqrtf(fmaf(x, x, fmaf(y, y, f.D * f.D))));
          }
          img[(size_t)r * la.Wp + j] = val;
        }
    }
    if (tid == 0) *amax = 0u;
    __syncthreads();
    switch (P.rb) {
      case 32: linesum_all_groups<32>(la, v, P.n_groups, smem, lmu, ttab); break;
      case 16: linesum_all_groups<16>(la, v, P.n_groups, smem, lmu, ttab); break;
      default: linesum_all_groups<8>(la, v, P.n_groups, smem, lmu, ttab); break;
    }
    // the sinogram was written by ordinary stores and is read back by bulk
    // (async-proxy) copies
    asm volatile("fence.proxy.async.global;" ::: "memory");
    __syncthreads();
    const int ntiles = P.tiles_x * P.tiles_y;
    float *gsm = smem + (size_t)grp * bp2_floats;
    bool ok = true;
    for (int t = grp; t < ntiles && ok; t += 2) {
      ok = P.multi ? bp2d_tile<true, BF_RY>(ba, v, 0, t % P.tiles_x, t / P.tiles_x, gt, 1 + grp,
                                            gsm, bars[grp], bmu[grp], it)
                   : bp2d_tile<false, BF_RY>(ba, v, 0, t % P.tiles_x, t / P.tiles_x, gt, 1 + grp,
                                             gsm, bars[grp], bmu[grp], it);
    }
    if (!ok) failed = 1;
    __syncthreads();
    if (failed) break;
    if (P.dtype == DC_F16) {
      // power-of-two scale mapping the view's absmax into [2^14, 2^15)
      const float am = __uint_as_float(*(volatile unsigned *)amax);
      float sc = 1.0f;
      if (am > 0.0f) {
        int e;
        frexpf(am, &e);
        sc = ldexpf(1.0f, e - 15);
      }
      if (tid == 0) P.scale[v] = sc;
      const float inv = 1.0f / sc;
      __half *dst = (__half *)P.ba.out + (size_t)v * la.H * la.W;
      for (int r = tid / 32; r < la.H; r += BF_THREADS / 32)
        for (int j = tid % 32; j < la.W; j += 32)
          dst[(size_t)r * la.W + j] = __float2half_rn(img[(size_t)r * la.Wp + j] * inv);
    }
  }
  // nothing is left in flight: every staged chunk was waited for
}

}  // namespace

namespace dc {

constexpr long L2_MB = 112, QUAD_MB = 384;

// Images that the work area holds, in `mb` MB of it: the per-image kernels
// want a chunk that stays in the 126 MB L2 (112 MB); the four-image kernels take
// few CTAs per image, so larger chunks keep the last wave of a launch small
// (their L2 working set is the few images in flight): 384 MB, also for few views
// (held to the views, batches of several items take up to 14 % longer: 30 views
// of 300 x 400, 3 items, 2.29 against 2.61 ms).  The autotuner may use fewer
// images per chunk.
static int chunk_capacity(const dc_geometry *g, bool quad, long mb) {
  const dc_geometry_desc &d = g->d;
  const size_t img = (size_t)d.det_rows * round4(d.det_cols), sino = (size_t)d.n_mu * round4(d.n_s);
  const size_t per_img = ((quad ? 2 : 1) * img + 2 * sino) * sizeof(float);
  const char *env = getenv("DC_CHUNK_IMAGES");
  auto clamp = [](long n) { return std::min(std::max(n, 4L), 256L); };
  auto quads = [](long n) { return (n + 3) & ~3L; };
  if (env) return (int)(quad ? quads(clamp(atoi(env))) : clamp(atoi(env)));
  const long most = clamp((mb << 20) / (long)per_img);
  return (int)(quad ? most & ~3L : most);
}

// The four-image line sums share every sample position, so all views need
// the same principal point.  Matrices of one scanner give it up to the
// rounding of their recovery (~1e-10 pixels); 1e-8 pixels is below a
// hundredth of the FP32 positions' own rounding (~1e-6), and a detector
// calibrated view by view differs by far more and keeps the per-image
// kernel, as do rows too long for two stages.  The angles per group are the
// number with the least time for a chunk: waves of CTAs (one per SM) times a
// CTA's rounds of its warps over its tasks plus its set-up and epilogue, 8 us
// against 0.69 us per band and round (64 views of 64 x 64, 180 x 64 lines: 48
// us in two waves of up to 16 angles, 38 us in one of 23).
int quad_plan(dc_geometry *g) {
  const dc_geometry_desc &d = g->d;
  g->quad = 0;
  if (d.det_rows < L4_RB || d.det_cols < L4_RB) return DC_OK;
  for (int i = 1; i < d.n_views; ++i)
    for (int c = 13; c <= 14; ++c)
      if (!(std::fabs(g->host_geo[(size_t)DC_VIEW_GEO_N * i + c] - g->host_geo[c]) < 1e-8))
        return DC_OK;
  const int nch = (d.n_s + 31) / 32, NSp = round4(d.n_s);
  const L4Shape sh = l4_shape(d.det_rows, d.det_cols);
  const int nb[2] = {(d.n_mu + 1) / 2, d.n_mu / 2};  // angles per branch, within one
  const int quads = (std::min(d.n_views, chunk_capacity(g, true, QUAD_MB)) + 3) / 4;
  const double over = 23.2 * L4_RB / (d.det_rows + d.det_cols);
  double best = 0.0;
  for (int mg = 1; mg <= L4_MAX_MG && mg * nch <= L4_TASKS; ++mg) {
    if (l4_smem(sh, mg, NSp) > L4_SMEM_BUDGET) break;
    int groups = 0, most = 0;
    for (int br = 0; br < 2; ++br) {
      const int ng = (nb[br] + mg - 1) / mg;
      groups += ng;
      if (ng) most = std::max(most, (nb[br] + ng - 1) / ng);
    }
    const int rounds = (most * nch + L4_WARPS - 1) / L4_WARPS;
    const double cost = ((groups * quads + g->sms - 1) / g->sms) * (rounds + over);
    if (!g->quad || cost < best) {
      best = cost;
      g->q_mg = mg;
      g->quad = 1;
    }
  }
  return DC_OK;
}

int alloc_workspace(dc_geometry *g) {
  const dc_geometry_desc &d = g->d;
  g->Wp = round4(d.det_cols);
  g->NSp = round4(d.n_s);
  g->img_stride = (size_t)d.det_rows * g->Wp;
  g->sino_stride = (size_t)d.n_mu * g->NSp;
  g->l2_images = chunk_capacity(g, false, L2_MB);
  bp_plan(g);
  g->ls_rb = linesum_band_rows(d.det_rows, d.det_cols, g->mg, g->NSp);
  if (g->ls_rb == 0 || bp2d_smem(g) > 200 * 1024)
    return fail(DC_ERR_UNSUPPORTED, "detector or sinogram rows too long for shared memory");
  // one block (four allocations of this size cost 0.1 ms more), its parts on 1
  // KB.  Where the four-image kernels' does not fit, a smaller one, and the
  // per-image kernels' at the last.
  auto floats = [](size_t n) { return (n + 255) & ~(size_t)255; };
  const struct {
    bool quad;
    long mb;
  } tries[3] = {{true, QUAD_MB}, {true, L2_MB}, {false, L2_MB}};
  int ci = 0;
  cudaError_t e = cudaErrorMemoryAllocation;
  for (int t = g->quad ? 0 : 2; t < 3 && e == cudaErrorMemoryAllocation; ++t) {
    g->quad = tries[t].quad;
    ci = chunk_capacity(g, g->quad, tries[t].mb);
    const size_t n_img = floats(g->img_stride * ci), n_sino = floats(g->sino_stride * ci);
    const size_t n_imgT = g->quad ? floats((size_t)d.det_rows * d.det_cols * ci) : 0;
    e = dmalloc((void **)&g->w_img, sizeof(float) * (n_img + n_imgT + 2 * n_sino));
    if (e != cudaSuccess) {
      cudaGetLastError();  // not the next launch's error
      continue;
    }
    g->w_imgT = g->quad ? g->w_img + n_img : nullptr;
    g->w_sinoA = g->w_img + n_img + n_imgT;
    g->w_sinoB = g->w_sinoA + n_sino;
  }
  if (e != cudaSuccess) return cuda_fail(e, "dc_setup_geometry: work area");
  g->chunk_images = ci;
  g->chunk_capacity = ci;
  if (g->quad) {
    const size_t H = d.det_rows, W = d.det_cols, ng = ci / 4;
    const L4Shape sh = l4_shape(d.det_rows, d.det_cols);
    if (!encode_map_f32(&g->q_tm_cols, g->w_imgT, 4 * H, W, ng, 4 * L4_RB, sh.boxh[0]) ||
        !encode_map_f32(&g->q_tm_rows, g->w_img, 4 * W, H, ng, 4 * L4_RB, sh.boxh[1]))
      g->quad = 0;
  }
  if (g->quad) {
    const size_t ng = ci / 4, n0 = 4 * (size_t)g->NSp, n1 = d.n_mu;
    // of the usual work area: results do not depend on the memory that was free
    const int chunk = chunk_capacity(g, true, QUAD_MB);
    g->q_ry = b4_rows(d.det_rows, d.det_cols, d.pitch, d.ds, d.n_views, chunk, g->sms);
    const B4Shape b4 = b4_shape(d.det_rows, d.det_cols, d.pitch, d.ds, g->q_ry, d.n_views, chunk,
                                g->sms);
    g->q_nwx = b4.nwx;
    const int lwb = b4.lwb;
    if (!encode_map_f32(&g->q_tm_sinoA, g->w_sinoA, n0, n1, ng, 4 * lwb, 1) ||
        !encode_map_f32(&g->q_tm_sinoB, g->w_sinoB, n0, n1, ng, 4 * lwb, 1))
      g->quad = 0;
  }
  DC_CUDA(dmalloc((void **)&g->w_absmax, sizeof(unsigned) * ci));
  DC_CUDA(dmalloc((void **)&g->w_flags, sizeof(unsigned) * 4));
  DC_CUDA(cudaMemset(g->w_flags, 0, sizeof(unsigned) * 4));
  return DC_OK;
}

int filter_check(const dc_geometry *g, int B, const float *gin, const void *gF, int dtype,
                 const float *gF_scale, const char *who) {
  int rc = check_common(g, B, who);
  if (rc) return rc;
  if (!gin || !gF) return fail(DC_ERR_ARG, std::string(who) + ": NULL g or gF");
  if (dtype != DC_F32 && dtype != DC_BF16 && dtype != DC_F16 && dtype != DC_F32X2)
    return fail(DC_ERR_ARG, std::string(who) + ": unknown dtype");
  if (dtype == DC_F16 && !gF_scale)
    return fail(DC_ERR_ARG, std::string(who) + ": DC_F16 needs gF_scale");
  if (dtype == DC_F32X2 && ((uintptr_t)gF & 15) != 0)
    return fail(DC_ERR_ARG, std::string(who) + ": DC_F32X2 g^F must be 16-byte aligned");
  const dc_geometry_desc &d = g->d;
  if (3.0 * d.ds < d.pitch * (1.0 - 1e-12))
    return fail(DC_ERR_UNSUPPORTED, std::string(who) + ": ds < pitch/3 is not supported");
  return DC_OK;
}

void filter_chunk_plan(const dc_geometry *g, int B, int dtype, int *bc, int *cv) {
  // the per-image kernels take chunks that stay in L2
  Chunking ck = chunking(g, B);
  if (g->quad && !quad_storage(dtype)) {
    ck.bc = std::min(ck.bc, g->l2_images);
    ck.cv = std::max(1, std::min(ck.cv, g->l2_images / ck.bc));
  }
  *bc = ck.bc;
  *cv = ck.cv;
}

// the filter of images (view v0 + n / bc, item b0 + n % bc), n < nv * bc
int filter_chunk(const dc_geometry *g, const float *gin, const float *W, void *gF, int dtype,
                 float *gF_scale, int b0, int bc, int v0, int nv, cudaStream_t st, float *S) {
  const dc_geometry_desc &d = g->d;
  const int n_img = nv * bc;
  int rc;
  const bool quad = use_quad(g, g->chunk_images, 1) && quad_storage(dtype);
  if ((rc = launch_prep(g, gin, WT_COS, v0, n_img, bc, b0, quad, st))) return rc;
  LineArgs la = line_args(g, bc, v0, b0, n_img);
  la.Wred = W;
  la.out = g->w_sinoA;
  la.Sout = S;
  if ((rc = launch_linesum<M_FILTER>(g, la, quad, st))) return rc;
  BP2Args ba = bp2_args(g, bc, v0, b0, n_img, g->w_sinoA);
  ba.weight = WT_D;
  if (dtype == DC_F16) {
    DC_CUDA(cudaMemsetAsync(g->w_absmax, 0, sizeof(unsigned) * n_img, st));
    ba.out_kind = OUT_F32_ABSMAX;
    ba.out = g->w_img;
    if ((rc = launch_bp2d(g, ba, quad, st))) return rc;
    dim3 grid(64, n_img);
    ProfScope ps(KID_TO_F16, st);
    k_to_f16<<<grid, 256, 0, st>>>(g->w_img, g->w_absmax, d.det_rows, d.det_cols, g->Wp,
                                   d.n_views, bc, v0, b0, (__half *)gF, gF_scale);
    DC_CHECK_LAUNCH("k_to_f16");
  } else if (dtype == DC_F32X2) {
    // g^F of the chunk into the work area (L2-resident), then the pairs
    ba.out_kind = OUT_F32_SLOT;
    ba.out = g->w_img;
    if ((rc = launch_bp2d(g, ba, quad, st))) return rc;
    const int pairs_per_img = d.det_rows * ((d.det_cols + 1) / 2);
    dim3 grid((unsigned)std::min(64, (pairs_per_img + 255) / 256), n_img);
    ProfScope ps(KID_TO_PAIRS, st);
    k_to_pairs<<<grid, 256, 0, st>>>(g->w_img, d.det_rows, d.det_cols, g->Wp, d.n_views, bc, v0,
                                     b0, (float2 *)gF);
    DC_CHECK_LAUNCH("k_to_pairs");
  } else {
    ba.out_kind = (dtype == DC_BF16) ? OUT_BF16 : OUT_F32;
    ba.out = gF;
    if ((rc = launch_bp2d(g, ba, quad, st))) return rc;
  }
  return DC_OK;
}

// The plan of the batched persistent filter: the problem table (in the
// order the items are handed out: largest per-image work first), the per-CTA
// scratch and the launch shape.
struct BatchFilterPlan {
  int n;
  int grid;
  long long total;
  size_t smem, img_cap, sino_cap;
  int bp2_floats;
  int order[DC_BF_MAX];  // table position -> problem index
  FilterProblem *d_probs;
  unsigned long long *d_counter;
  float *img_scratch, *sino_scratch;
  unsigned *amax;
};

void batch_filter_destroy(BatchFilterPlan *p) {
  if (!p) return;
  cudaFree(p->d_probs);
  cudaFree(p->d_counter);
  cudaFree(p->img_scratch);
  cudaFree(p->sino_scratch);
  cudaFree(p->amax);
  delete p;
}

int batch_filter_create(int n, dc_geometry *const *geoms, int dtype, void *const *gF,
                        float *const *scale, BatchFilterPlan **out) {
  *out = nullptr;
  if (n < 1 || n > DC_BF_MAX) return fail(DC_ERR_ARG, "batched filter: 1 <= n <= 32");
  if (dtype == DC_F32X2)  // the pairs come from a pass over the finished image
    return fail(DC_ERR_UNSUPPORTED, "batched filter: DC_F32X2 uses the chunked filter");
  int dev = 0;
  DC_CUDA(cudaGetDevice(&dev));
  cudaFuncAttributes fa;
  DC_CUDA(cudaFuncGetAttributes(&fa, k_filter_batched));
  int optin = 0;
  DC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t budget = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
  BatchFilterPlan *p = new BatchFilterPlan();
  memset((void *)p, 0, sizeof(BatchFilterPlan));
  p->n = n;
  // largest per-image work first (line-sum steps plus 2-D backprojection pairs)
  auto work = [&](int i) {
    const dc_geometry_desc &d = geoms[i]->d;
    return (double)d.n_mu * d.n_s * std::max(d.det_rows, d.det_cols) +
           (double)d.det_rows * d.det_cols * d.n_mu;
  };
  for (int i = 0; i < n; ++i) p->order[i] = i;
  std::stable_sort(p->order, p->order + n, [&](int x, int y) { return work(x) > work(y); });
  std::vector<FilterProblem> probs(n);
  long long first = 0;
  for (int t = 0; t < n; ++t) {
    const dc_geometry *g = geoms[p->order[t]];
    const dc_geometry_desc &d = g->d;
    FilterProblem &P = probs[t];
    memset((void *)&P, 0, sizeof(P));
    P.la = line_args(g, 1, 0, 0, 1);
    P.ba = bp2_args(g, 1, 0, 0, 1, nullptr);
    P.ba.weight = WT_D;
    P.ba.out_kind = (dtype == DC_BF16) ? OUT_BF16 : (dtype == DC_F16 ? OUT_F32_ABSMAX : OUT_F32);
    P.ba.out = gF[p->order[t]];
    P.rb = linesum_band_rows(d.det_rows, d.det_cols, g->mg, g->NSp, budget);
    P.n_groups = g->n_groups;
    P.multi = multi_tap(g) ? 1 : 0;
    P.tiles_x = (d.det_cols + BP2_TX - 1) / BP2_TX;
    P.tiles_y = (d.det_rows + 8 * BF_RY - 1) / (8 * BF_RY);
    P.dtype = dtype;
    P.scale = (dtype == DC_F16) ? scale[p->order[t]] : nullptr;
    P.first = first;
    first += d.n_views;
    if (P.rb == 0) {
      batch_filter_destroy(p);
      return fail(DC_ERR_UNSUPPORTED, "batched filter: detector rows too long for its shared memory");
    }
    p->img_cap = std::max(p->img_cap, (size_t)d.det_rows * g->Wp);
    p->sino_cap = std::max(p->sino_cap, (size_t)d.n_mu * g->NSp);
    p->bp2_floats = std::max(p->bp2_floats, 2 * BP2_MC * (g->NSp + PADL + PADR));
    p->smem = std::max(p->smem, linesum_smem_for(d.det_rows, d.det_cols, g->mg, g->NSp, P.rb));
  }
  p->total = first;
  p->smem = std::max(p->smem, (size_t)2 * p->bp2_floats * sizeof(float));
  if (p->smem > budget) {
    batch_filter_destroy(p);
    return fail(DC_ERR_UNSUPPORTED, "batched filter: sinogram rows too long for its shared memory");
  }
  // the limit belongs to the kernel: one value for all plans, so that none
  // lowers it under another's launch
  cudaError_t e = cudaFuncSetAttribute(k_filter_batched, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)budget);
  int per_sm = 0, sms = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_batched, BF_THREADS, p->smem);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) {
    batch_filter_destroy(p);
    return cuda_fail(e, "batched filter: launch shape");
  }
  if (per_sm < 1) {
    batch_filter_destroy(p);
    return fail(DC_ERR_UNSUPPORTED, "batched filter: no resident CTA fits");
  }
  p->grid = std::max(1, sms) * per_sm;
  e = dmalloc((void **)&p->d_probs, sizeof(FilterProblem) * n);
  if (e == cudaSuccess) e = dmalloc((void **)&p->d_counter, sizeof(unsigned long long));
  if (e == cudaSuccess) e = dmalloc((void **)&p->img_scratch, sizeof(float) * p->img_cap * p->grid);
  if (e == cudaSuccess) e = dmalloc((void **)&p->sino_scratch, sizeof(float) * p->sino_cap * p->grid);
  if (e == cudaSuccess) e = dmalloc((void **)&p->amax, sizeof(unsigned) * p->grid);
  if (e == cudaSuccess)
    e = cudaMemcpy(p->d_probs, probs.data(), sizeof(FilterProblem) * n, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    batch_filter_destroy(p);
    return cuda_fail(e, "batched filter: allocation");
  }
  *out = p;
  return DC_OK;
}

int batch_filter_run(BatchFilterPlan *p, const float *const *g, const float *const *W,
                     cudaStream_t st) {
  FilterRun run;
  memset(&run, 0, sizeof(run));
  for (int t = 0; t < p->n; ++t) {
    run.g[t] = g[p->order[t]];
    run.W[t] = W ? W[p->order[t]] : nullptr;
  }
  DC_CUDA(cudaMemsetAsync(p->d_counter, 0, sizeof(unsigned long long), st));
  ProfScope ps(KID_FILTER_BATCHED, st);
  k_filter_batched<<<p->grid, BF_THREADS, p->smem, st>>>(
      p->d_probs, p->n, p->total, p->d_counter, run, p->img_scratch, p->img_cap, p->sino_scratch,
      p->sino_cap, p->amax, p->bp2_floats);
  DC_CHECK_LAUNCH("k_filter_batched");
  return DC_OK;
}

}  // namespace dc

extern "C" {

// Every entry point walks the (batch item, view) images chunk by chunk:
// the outer loop takes bc batch items starting at b0, the inner loop cv views
// starting at v0; image n of a chunk is (view v0 + n / bc, item b0 + n % bc).

static int filter_all(const dc_geometry *g, int B, const float *gin, const float *W, void *gF,
                      int dtype, float *gF_scale, float *S, void *stream, const char *who) {
  int rc = dc::filter_check(g, B, gin, gF, dtype, gF_scale, who);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  int bcm, cvm;
  dc::filter_chunk_plan(g, B, dtype, &bcm, &cvm);
  for (int b0 = 0; b0 < B; b0 += bcm) {
    int bc = std::min(bcm, B - b0);
    for (int v0 = 0; v0 < g->d.n_views; v0 += cvm) {
      int nv = std::min(cvm, g->d.n_views - v0);
      if ((rc = dc::filter_chunk(g, gin, W, gF, dtype, gF_scale, b0, bc, v0, nv, st, S)))
        return rc;
    }
  }
  return DC_OK;
}

int dc_filter(const dc_geometry *g, int B, const float *gin, const float *W, void *gF,
              int dtype, float *gF_scale, void *stream) {
  return filter_all(g, B, gin, W, gF, dtype, gF_scale, nullptr, stream, "dc_filter");
}

int dc_filter_with_s(const dc_geometry *g, int B, const float *gin, const float *W, void *gF,
                     int dtype, float *gF_scale, float *S, void *stream) {
  if (!S) return dc::fail(DC_ERR_ARG, "dc_filter_with_s: NULL S");
  return filter_all(g, B, gin, W, gF, dtype, gF_scale, S, stream, "dc_filter_with_s");
}

int dc_filter_adjoint(const dc_geometry *g, int B, const float *grad_gF, const float *gin,
                      const float *W, float *grad_g, float *grad_W, int view_chunk,
                      void *stream) {
  int rc = check_common(g, B, "dc_filter_adjoint");
  if (rc) return rc;
  if (!grad_gF || !gin) return dc::fail(DC_ERR_ARG, "dc_filter_adjoint: NULL grad_gF or g");
  if (view_chunk < 0) return dc::fail(DC_ERR_ARG, "dc_filter_adjoint: negative view_chunk");
  const dc_geometry_desc &d = g->d;
  if (3.0 * d.ds < d.pitch * (1.0 - 1e-12))
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_filter_adjoint: ds < pitch/3 is not supported");
  if (!grad_g && !grad_W) return DC_OK;
  cudaStream_t st = (cudaStream_t)stream;
  Chunking ck = chunking(g, B, view_chunk);
  const bool quad = use_quad(g, ck.bc, ck.cv);
  for (int b0 = 0; b0 < B; b0 += ck.bc) {
    int bc = std::min(ck.bc, B - b0);
    for (int v0 = 0; v0 < d.n_views; v0 += ck.cv) {
      int nv = std::min(ck.cv, d.n_views - v0);
      int n_img = nv * bc;
      // dL/dP up to D_b^T: line differences of w_d * dL/dg^F
      if ((rc = launch_prep(g, grad_gF, WT_D, v0, n_img, bc, b0, quad, st))) return rc;
      LineArgs la = line_args(g, bc, v0, b0, n_img);
      la.Wred = W;
      la.sinoA = g->w_sinoA;
      la.sinoB = g->w_sinoB;
      if ((rc = launch_linesum<M_DIFFSTORE>(g, la, quad, st))) return rc;
      // recompute S from w_cos * g and finish the chain
      if ((rc = launch_prep(g, gin, WT_COS, v0, n_img, bc, b0, quad, st))) return rc;
      if ((rc = launch_linesum<M_ADJ>(g, la, quad, st))) return rc;
      if (grad_W) {
        size_t total = (size_t)nv * d.n_mu * d.n_s;
        int nb = (int)std::min<size_t>((total + 255) / 256, 4096);
        dc::ProfScope ps(dc::KID_REDUCE_W, st);
        auto reduce = quad ? k_reduce_gradW<true> : k_reduce_gradW<false>;
        reduce<<<nb, 256, 0, st>>>(g->w_sinoA, d.n_mu, d.n_s, g->NSp, bc, v0, nv, b0 > 0, grad_W);
        DC_CHECK_LAUNCH("k_reduce_gradW");
      }
      if (grad_g) {
        BP2Args ba = bp2_args(g, bc, v0, b0, n_img, g->w_sinoB);
        ba.weight = WT_COS;
        ba.out_kind = OUT_F32;
        ba.out = grad_g;
        if ((rc = launch_bp2d(g, ba, quad, st))) return rc;
      }
    }
  }
  return DC_OK;
}

int dc_filter_adjoint_from_s(const dc_geometry *g, int B, const float *grad_gF,
                             const float *S, const float *W, float *grad_g, float *grad_W,
                             int view_chunk, void *stream) {
  int rc = check_common(g, B, "dc_filter_adjoint_from_s");
  if (rc) return rc;
  if (!grad_gF || !S)
    return dc::fail(DC_ERR_ARG, "dc_filter_adjoint_from_s: NULL grad_gF or S");
  if (view_chunk < 0) return dc::fail(DC_ERR_ARG, "dc_filter_adjoint_from_s: negative view_chunk");
  const dc_geometry_desc &d = g->d;
  if (3.0 * d.ds < d.pitch * (1.0 - 1e-12))
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_filter_adjoint_from_s: ds < pitch/3 is not supported");
  if (!grad_g && !grad_W) return DC_OK;
  cudaStream_t st = (cudaStream_t)stream;
  Chunking ck = chunking(g, B, view_chunk);
  const bool quad = use_quad(g, ck.bc, ck.cv);
  for (int b0 = 0; b0 < B; b0 += ck.bc) {
    int bc = std::min(ck.bc, B - b0);
    for (int v0 = 0; v0 < d.n_views; v0 += ck.cv) {
      int nv = std::min(ck.cv, d.n_views - v0);
      int n_img = nv * bc;
      // dL/dP up to D_b^T: line differences of w_d * dL/dg^F
      if ((rc = launch_prep(g, grad_gF, WT_D, v0, n_img, bc, b0, quad, st))) return rc;
      LineArgs la = line_args(g, bc, v0, b0, n_img);
      la.Wred = W;
      la.sinoA = g->w_sinoA;
      la.sinoB = g->w_sinoB;
      if ((rc = launch_linesum<M_DIFFSTORE>(g, la, quad, st))) return rc;
      {  // finish the chain with the stored S
        dc::ProfScope ps(dc::KID_ADJ_S, st);
        if (quad) {
          dim3 grid((d.n_mu + AS4_ROWS - 1) / AS4_ROWS, (n_img + 3) / 4);
          DC_CUDA(cudaFuncSetAttribute(k_adj_from_s4, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       AS4_ROWS * 2048 * 16));
          k_adj_from_s4<<<grid, 256, sizeof(float4) * AS4_ROWS * g->NSp, st>>>(la, S);
        } else {
          dim3 grid((d.n_mu + AS_ROWS - 1) / AS_ROWS, n_img);
          k_adj_from_s<<<grid, 256, sizeof(float) * AS_ROWS * g->NSp, st>>>(la, S);
        }
        DC_CHECK_LAUNCH("k_adj_from_s");
      }
      if (grad_W) {
        size_t total = (size_t)nv * d.n_mu * d.n_s;
        int nb = (int)std::min<size_t>((total + 255) / 256, 4096);
        dc::ProfScope ps(dc::KID_REDUCE_W, st);
        auto reduce = quad ? k_reduce_gradW<true> : k_reduce_gradW<false>;
        reduce<<<nb, 256, 0, st>>>(g->w_sinoA, d.n_mu, d.n_s, g->NSp, bc, v0, nv, b0 > 0, grad_W);
        DC_CHECK_LAUNCH("k_reduce_gradW");
      }
      if (grad_g) {
        BP2Args ba = bp2_args(g, bc, v0, b0, n_img, g->w_sinoB);
        ba.weight = WT_COS;
        ba.out_kind = OUT_F32;
        ba.out = grad_g;
        if ((rc = launch_bp2d(g, ba, quad, st))) return rc;
      }
    }
  }
  return DC_OK;
}

int dc_grangeat(const dc_geometry *g, int B, const float *gin, float *S, void *stream) {
  int rc = check_common(g, B, "dc_grangeat");
  if (rc) return rc;
  if (!gin || !S) return dc::fail(DC_ERR_ARG, "dc_grangeat: NULL argument");
  const dc_geometry_desc &d = g->d;
  cudaStream_t st = (cudaStream_t)stream;
  Chunking ck = chunking(g, B);
  const bool quad = use_quad(g, ck.bc, ck.cv);
  for (int b0 = 0; b0 < B; b0 += ck.bc) {
    int bc = std::min(ck.bc, B - b0);
    for (int v0 = 0; v0 < d.n_views; v0 += ck.cv) {
      int n_img = std::min(ck.cv, d.n_views - v0) * bc;
      if ((rc = launch_prep(g, gin, WT_COS, v0, n_img, bc, b0, quad, st))) return rc;
      LineArgs la = line_args(g, bc, v0, b0, n_img);
      la.out = S;
      if ((rc = launch_linesum<M_GRANGEAT>(g, la, quad, st))) return rc;
    }
  }
  return DC_OK;
}

int dc_radon2d(const dc_geometry *g, int B, const float *img, float *R, void *stream) {
  int rc = check_common(g, B, "dc_radon2d");
  if (rc) return rc;
  if (!img || !R) return dc::fail(DC_ERR_ARG, "dc_radon2d: NULL argument");
  const dc_geometry_desc &d = g->d;
  cudaStream_t st = (cudaStream_t)stream;
  Chunking ck = chunking(g, B);
  const bool quad = use_quad(g, ck.bc, ck.cv);
  for (int b0 = 0; b0 < B; b0 += ck.bc) {
    int bc = std::min(ck.bc, B - b0);
    for (int v0 = 0; v0 < d.n_views; v0 += ck.cv) {
      int n_img = std::min(ck.cv, d.n_views - v0) * bc;
      if ((rc = launch_prep(g, img, WT_NONE, v0, n_img, bc, b0, quad, st))) return rc;
      LineArgs la = line_args(g, bc, v0, b0, n_img);
      la.out = R;
      if ((rc = launch_linesum<M_RAW>(g, la, quad, st))) return rc;
    }
  }
  return DC_OK;
}

int dc_radon2d_adjoint(const dc_geometry *g, int B, const float *R, float *img, void *stream) {
  int rc = check_common(g, B, "dc_radon2d_adjoint");
  if (rc) return rc;
  if (!img || !R) return dc::fail(DC_ERR_ARG, "dc_radon2d_adjoint: NULL argument");
  const dc_geometry_desc &d = g->d;
  if (3.0 * d.ds < d.pitch * (1.0 - 1e-12))
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_radon2d_adjoint: ds < pitch/3 is not supported");
  cudaStream_t st = (cudaStream_t)stream;
  Chunking ck = chunking(g, B);
  const bool quad = use_quad(g, ck.bc, ck.cv);
  for (int b0 = 0; b0 < B; b0 += ck.bc) {
    int bc = std::min(ck.bc, B - b0);
    for (int v0 = 0; v0 < d.n_views; v0 += ck.cv) {
      int n_img = std::min(ck.cv, d.n_views - v0) * bc;
      {
        dc::ProfScope ps(dc::KID_SINO_IN, st);
        if (quad)
          k_sino_in4<<<dim3(64, (n_img + 3) / 4), 256, 0, st>>>(
              R, g->mu, d.n_mu, d.n_s, g->NSp, d.n_views, bc, v0, b0, n_img, (float4 *)g->w_sinoA);
        else
          k_sino_in<<<dim3(64, n_img), 256, 0, st>>>(R, g->mu, d.n_mu, d.n_s, g->NSp, d.n_views,
                                                     bc, v0, b0, g->w_sinoA);
        DC_CHECK_LAUNCH("k_sino_in");
      }
      BP2Args ba = bp2_args(g, bc, v0, b0, n_img, g->w_sinoA);
      ba.weight = WT_NONE;
      ba.out_kind = OUT_F32;
      ba.out = img;
      if ((rc = launch_bp2d(g, ba, quad, st))) return rc;
    }
  }
  return DC_OK;
}

// The s-derivatives of Eqs. 7 and 11 alone, on [rows][n_s] sinograms:
// kind 0 D_f (forward difference onto s_{k+1/2}; entry n_s-1 is 0), 1 its
// transpose, 2 D_b (backward difference, zero below k = 0), 3 its transpose;
// all divided by ds.  One thread per entry, rows read from global memory.
__global__ void k_deriv(const float *__restrict__ in, float *__restrict__ out, long long rows,
                        int n_s, float ds, int kind) {
  const long long total = rows * n_s;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(i % n_s);
    const float *x = in + (i - k);
    float v;
    if (kind == 0) {
      v = (k < n_s - 1) ? (x[k + 1] - x[k]) / ds : 0.0f;
    } else if (kind == 1) {
      const float a = (k >= 1) ? x[k - 1] : 0.0f, b = (k < n_s - 1) ? x[k] : 0.0f;
      v = (a - b) / ds;
    } else if (kind == 2) {
      v = (x[k] - (k > 0 ? x[k - 1] : 0.0f)) / ds;
    } else {
      v = (x[k] - (k + 1 < n_s ? x[k + 1] : 0.0f)) / ds;
    }
    out[i] = v;
  }
}

int dc_deriv(const dc_geometry *g, int B, const float *in, float *out, int kind, void *stream) {
  int rc = check_common(g, B, "dc_deriv");
  if (rc) return rc;
  if (!in || !out || in == out) return dc::fail(DC_ERR_ARG, "dc_deriv: NULL or aliased arrays");
  if (kind < 0 || kind > 3) return dc::fail(DC_ERR_ARG, "dc_deriv: kind must be 0..3");
  const dc_geometry_desc &d = g->d;
  const long long rows = (long long)B * d.n_views * d.n_mu;
  const long long total = rows * d.n_s;
  int sms = 0;
  DC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device));
  const int blocks = (int)std::min<long long>((total + 255) / 256, (long long)std::max(sms, 1) * 16);
  k_deriv<<<blocks, 256, 0, (cudaStream_t)stream>>>(in, out, rows, d.n_s, (float)d.ds, kind);
  DC_CHECK_LAUNCH("k_deriv");
  return DC_OK;
}

// Test hook of the timeout path: one thread waits, with the library's bound
// (~2^31 cycles), on an mbarrier that nothing completes, gives up and raises
// the handle's timeout flag, as a staged kernel does when a copy never lands.
__global__ void k_wait_probe(unsigned *err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    dc::mbar_init(&bar, 1);
    dc::fence_barrier_init();
    dc::mbar_wait_bounded(&bar, 0, err);
  }
}

int dc_debug_wait_timeout(const dc_geometry *g, void *stream) {
  if (!g) return dc::fail(DC_ERR_ARG, "dc_debug_wait_timeout: NULL geometry");
  k_wait_probe<<<1, 32, 0, (cudaStream_t)stream>>>(g->w_flags);
  DC_CHECK_LAUNCH("k_wait_probe");
  return DC_OK;
}

int dc_sync_status(const dc_geometry *g, void *stream) {
  if (!g) return dc::fail(DC_ERR_ARG, "dc_sync_status: NULL geometry");
  DC_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
  unsigned flags = 0;
  DC_CUDA(cudaMemcpy(&flags, g->w_flags, sizeof(unsigned), cudaMemcpyDeviceToHost));
  if (flags) {
    DC_CUDA(cudaMemset(g->w_flags, 0, sizeof(unsigned)));
    if (flags & DC_FLAG_TIMEOUT) return dc::fail(DC_ERR_TIMEOUT, "a bounded device wait gave up");
    return dc::fail(DC_ERR_NONFINITE,
                    "a redundancy weight W read by the filter or its adjoint was NaN or infinite");
  }
  return DC_OK;
}

}  // extern "C"

// ------------------------------------------------------------------------
// Allocation-free Joseph line sums.
//
// Callers that cannot allocate device memory (a real-time reconstruction
// loop on a scanner whose memory budget is fixed before the scan and must
// never wait on CUDA's allocator, or a host that embeds this library
// inside another runtime's memory pool and cannot create a geometry handle)
// use dc_radon2d_noalloc.  Its work area is the fixed array below, compiled
// into the library: every GPU that loads the library holds it until exit.
namespace {

constexpr size_t NA_BYTES = 32u << 20;         // 32 MiB per device
constexpr size_t NA_TABLE_BYTES = 256u << 10;  // angle tables and error word
constexpr int NA_MAX_MU = 2048;
constexpr int NA_MAX_DEV = 64;

static_assert((sizeof(dc::MuRec) + sizeof(dc::VMu) + sizeof(int) + sizeof(dc::MuGroup)) *
                      NA_MAX_MU + 1024 <=
                  NA_TABLE_BYTES,
              "angle tables overflow their region");

static __device__ __align__(256) unsigned char g_na_scratch[NA_BYTES];

// set-up: the device address of g_na_scratch, once per device and context
// (a cudaDeviceReset gives the device a new primary context in which the
// array has a new address, so the cache is keyed on the current context)
void *g_na_ptr[NA_MAX_DEV];
void *g_na_ctx[NA_MAX_DEV];
std::mutex g_na_mu;

typedef CUresult (*CtxGetCurrentFn)(CUcontext *);
CtxGetCurrentFn ctx_get_current_fn() {
  static CtxGetCurrentFn fn = nullptr;
  static bool looked = false;
  if (!looked) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (CtxGetCurrentFn)p;
    looked = true;
  }
  return fn;
}

// Angle tables for one call, written into the fixed area: one thread per
// angle for the per-angle records, thread 0 for the ordering and grouping
// (the same as a geometry handle's tables).
__global__ void k_na_tables(int n_mu, int n_s, double pitch, double ds, double cu, double cv,
                            int mg, dc::MuRec *mu, dc::VMu *vmu, int *order,
                            dc::MuGroup *groups, dc::FView *fv, unsigned *err) {
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < n_mu) {
    mu[m] = dc::make_mu_rec(m, n_mu, pitch, ds);
    vmu[m] = dc::make_vmu(m, n_mu, n_s, pitch, ds, cu, cv);
  }
  if (m != 0) return;
  *err = 0u;
  dc::FView f;
  f.D = 1.0f;
  f.cu = (float)cu;
  f.cv = (float)cv;
  f.ax = f.ay = f.az = f.pad0 = f.pad1 = 0.0f;
  *fv = f;
  int nord = 0, ng = 0;
  for (int br = 0; br < 2; ++br) {
    int cnt = 0;
    for (int q = 0; q < n_mu; ++q) {
      bool rows = dc::joseph_rows(q, n_mu);
      if ((br == 0) != rows) continue;
      if (cnt % mg == 0) {
        groups[ng].first = nord;
        groups[ng].count = 0;
        groups[ng].branch = br;
        groups[ng].pad = 0;
        ++ng;
      }
      groups[ng - 1].count += 1;
      order[nord++] = q;
      ++cnt;
    }
  }
}

}  // namespace

extern "C" int dc_radon2d_noalloc(int n_img, int H, int W, int n_mu, int n_s, double pitch,
                                  double ds, double cu, double cv, const float *img, float *R,
                                  void *stream) {
  if (n_img < 1 || H < 2 || W < 2 || n_mu < 1 || n_s < 2)
    return dc::fail(DC_ERR_ARG, "dc_radon2d_noalloc: sizes must be positive (H, W, n_s >= 2)");
  if (!img || !R) return dc::fail(DC_ERR_ARG, "dc_radon2d_noalloc: NULL img or R");
  if (!(pitch > 0) || !(ds > 0) || !std::isfinite(cu) || !std::isfinite(cv))
    return dc::fail(DC_ERR_ARG, "dc_radon2d_noalloc: bad pitch, ds or principal point");
  if (n_mu > NA_MAX_MU)
    return dc::fail(DC_ERR_ARG, "dc_radon2d_noalloc: n_mu above the fixed maximum of " +
                                    std::to_string(NA_MAX_MU));
  const int Wp = round4(W), NSp = round4(n_s);
  const size_t per_img = (size_t)H * Wp * sizeof(float);
  const size_t cap = NA_BYTES - NA_TABLE_BYTES;
  if (per_img > cap)
    return dc::fail(DC_ERR_ARG, "dc_radon2d_noalloc: one " + std::to_string(H) + "x" +
                                    std::to_string(W) + " image needs " +
                                    std::to_string(per_img) + " bytes of work area; the fixed "
                                    "maximum is " + std::to_string(cap) + " bytes");
  const int mg = dc::linesum_group_size(n_s);
  const int rb = linesum_band_rows(H, W, mg, NSp);
  if (rb == 0)
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_radon2d_noalloc: rows too long for shared memory");
  const size_t smem = linesum_smem_for(H, W, mg, NSp, rb);

  int dev = 0;
  DC_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= NA_MAX_DEV)
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_radon2d_noalloc: device index out of range");
  unsigned char *base = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_na_mu);
    CUcontext ctx = nullptr;
    CtxGetCurrentFn cur = ctx_get_current_fn();
    if (cur && cur(&ctx) != CUDA_SUCCESS) ctx = nullptr;
    if (!g_na_ptr[dev] || (ctx && ctx != (CUcontext)g_na_ctx[dev])) {
      void *p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_na_scratch);
      if (e != cudaSuccess) return dc::cuda_fail(e, "cudaGetSymbolAddress(g_na_scratch)");
      g_na_ptr[dev] = p;
      g_na_ctx[dev] = (void *)ctx;
    }
    base = (unsigned char *)g_na_ptr[dev];
  }
  // fixed-area layout: tables first, then the image copies
  dc::MuRec *mu = (dc::MuRec *)base;
  dc::VMu *vmu = (dc::VMu *)(base + sizeof(dc::MuRec) * NA_MAX_MU);
  int *order = (int *)(base + (sizeof(dc::MuRec) + sizeof(dc::VMu)) * NA_MAX_MU);
  dc::MuGroup *groups =
      (dc::MuGroup *)(base + (sizeof(dc::MuRec) + sizeof(dc::VMu) + sizeof(int)) * NA_MAX_MU);
  unsigned char *tail =
      base + (sizeof(dc::MuRec) + sizeof(dc::VMu) + sizeof(int) + sizeof(dc::MuGroup)) * NA_MAX_MU;
  dc::FView *fv = (dc::FView *)tail;
  unsigned *err = (unsigned *)(tail + 256);
  float *work = (float *)(base + NA_TABLE_BYTES);

  cudaStream_t st = (cudaStream_t)stream;
  k_na_tables<<<(n_mu + 127) / 128, 128, 0, st>>>(n_mu, n_s, pitch, ds, cu, cv, mg, mu, vmu,
                                                  order, groups, fv, err);
  DC_CHECK_LAUNCH("k_na_tables");
  // the group count is a host-side launch parameter: recompute it here
  int nb0 = 0, nb1 = 0;
  for (int m = 0; m < n_mu; ++m) (dc::joseph_rows(m, n_mu) ? nb0 : nb1) += 1;
  const int n_groups_h = (nb0 + mg - 1) / mg + (nb1 + mg - 1) / mg;

  const int per_chunk = (int)std::min<size_t>(cap / per_img, 65535);
  float *img_w = work;
  for (int n0 = 0; n0 < n_img; n0 += per_chunk) {
    int nc = std::min(per_chunk, n_img - n0);
    PrepArgs p;
    p.src = img + (size_t)n0 * H * W;
    p.img = img_w;
    p.fv = fv;
    p.H = H;
    p.W = W;
    p.Wp = Wp;
    p.V = 1;    // image n is batch item n of a one-view problem, so it
    p.B = nc;   // reads offset n*H*W and table record 0
    p.v0 = 0;
    p.b0 = 0;
    p.Bt = 0;
    p.n_img = nc;
    p.pitch = (float)pitch;
    p.weight = WT_NONE;
    dim3 gp((Wp + 31) / 32, (H + 31) / 32, nc);
    {
      dc::ProfScope ps(dc::KID_PREP, st);
      k_prep<<<gp, dim3(32, 8), 0, st>>>(p);
      DC_CHECK_LAUNCH("k_prep");
    }
    LineArgs a;
    memset(&a, 0, sizeof(a));
    a.img = img_w;
    a.H = H;
    a.W = W;
    a.Wp = Wp;
    a.n_mu = n_mu;
    a.n_s = n_s;
    a.NSp = NSp;
    a.V = 1;    // output image n lands at ((b*1 + 0)*n_mu + m)*n_s with b = n
    a.B = nc;
    a.v0 = 0;
    a.b0 = 0;
    a.n_img = nc;
    a.pitch = (float)pitch;
    a.ds = (float)ds;
    a.mu = mu;
    a.vmu = vmu;
    a.mu_order = order;
    a.groups = groups;
    a.fv = fv;
    a.out = R + (size_t)n0 * n_mu * n_s;
    a.err = err;
    a.mg = mg;
    dim3 grid(n_groups_h, nc);
    {
      dc::ProfScope ps(dc::KID_LINESUM, st);
      int rc = rb == 32 ? launch_linesum_rb<M_RAW, 32>(grid, a, smem, st)
               : rb == 16 ? launch_linesum_rb<M_RAW, 16>(grid, a, smem, st)
                          : launch_linesum_rb<M_RAW, 8>(grid, a, smem, st);
      if (rc != DC_OK) return rc;
    }
  }
  return DC_OK;
}
