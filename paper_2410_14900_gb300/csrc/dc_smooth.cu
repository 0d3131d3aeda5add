// dc_smooth.cu -- the Gaussian filter layer on the learned redundancy weight
// (Ye et al., DRACO, Sec. 3.1: sigma 20, kernel size 121), and its transpose
// for the reverse mode.
//
// Per view the weight map W[mu][k] is filtered along mu and along s over the
// valid half-grid entries k < n_s - 1 (entry n_s - 1 is unused by the filter
// chain and passes through).  Taps exp(-t^2 / (2 sigma^2)), |t| <= radius,
// normalised to unit sum; each line is extended by mirroring about its end
// samples (index -1 reads 1, index n reads n - 2, repeated for short lines).
// The two axis filters act on different axes and commute.
//
// One kernel (k_smooth_tile) serves both axes and both directions.  A CTA
// stages 128 + 2 radius mirror-extended samples of 64 neighbouring lines as
// [sample][line]; a lane takes a pair of lines and a warp 16 consecutive
// outputs, held in registers with a sliding window of 16 samples, so that a
// tap costs 16 packed FMAs, one 8-byte load and half a 16-byte load of taps.
// Bound by the FMA pipe: the two directions on 360 x 360 x 256 with 121 taps
// are 1.6e10 FMAs, 0.40 ms at the FP32 peak; 4.60 ms with k_smooth_lines (a
// shared-memory load per FMA, taps normalised by one thread), 1.93 with loads
// through registers, 1.10 with two CTAs per SM, 0.99 as it is.
//
// The transpose needs no code of its own: the taps are even, so with D = 2 at
// a line's two end samples and 1 elsewhere (the mirrored line meets an end
// sample once per period and every other sample twice) the filter A satisfies
// A^T = D^-1 A D, exactly, also for lines shorter than the radius.
//
// Radii whose halo does not fit (above 320), and few short lines (few_samples),
// take k_smooth_lines: `cw`
// neighbouring lines of one view whole in shared memory (cw = 16 columns for
// the mu axis, whose elements are n_s apart; one contiguous row for the s
// axis).  The forward pass gathers from a mirror-extended copy of the line;
// the transpose computes the zero-padded correlation c(p) for every extended
// position p and folds it back onto the sample p mirrors to.
#include <algorithm>
#include <cmath>
#include <string>

#include "dc_async.cuh"
#include "dc_common.cuh"

namespace {

constexpr int SM_THREADS = 256;
constexpr size_t SM_SMEM_BUDGET = 200 * 1024;

struct SmoothLines {
  const float *in;
  float *out;
  int n;            // samples per line
  int lines;        // lines per view
  size_t vstride;   // floats between views
  int es;           // floats between samples of a line
  int ls;           // floats between neighbouring lines
  int lcw;          // log2 of the lines per CTA
  int R;            // radius
  float sigma;
  int adjoint;
};

__device__ __forceinline__ int mirror_of(int p, int n) {
  if (n == 1) return 0;
  const int T = 2 * (n - 1);
  p %= T;
  if (p < 0) p += T;
  return p < n ? p : T - p;
}

// taps exp(-t^2 / 2 sigma^2) over their sum, each to one thread.  Every warp sums
// them, a 32nd per lane: one running sum of 121 taps is 4e-7 off, this 1.5e-7.
template <typename Put>
__device__ __forceinline__ void normalised_taps(int R, float sigma, int threads, Put put) {
  const int ntap = 2 * R + 1;
  auto tap = [&](int t) {
    const float d = (float)(t - R);
    return expf(-0.5f * d * d / (sigma * sigma));
  };
  float s = 0.0f;
  for (int t = threadIdx.x & 31; t < ntap; t += 32) s += tap(t);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const float inv = 1.0f / s;
  for (int t = threadIdx.x; t < ntap; t += threads) put(t, tap(t) * inv);
}

// `through` (mu axis): the array whose entry `lines` of every row passes into a.out
__global__ void __launch_bounds__(SM_THREADS)
    k_smooth_lines(SmoothLines a, const float *__restrict__ through) {
  extern __shared__ float sm[];
  const int R = a.R, n = a.n, cw = 1 << a.lcw, cm = cw - 1;
  const int ntap = 2 * R + 1;
  float *w = sm;                              // taps
  float *xe = sm + ((ntap + 3) & ~3);         // staged lines
  const int v = blockIdx.y, l0 = blockIdx.x * cw;
  const float *src = a.in + (size_t)v * a.vstride + (size_t)l0 * a.ls;
  float *dst = a.out + (size_t)v * a.vstride + (size_t)l0 * a.ls;
  const int tid = threadIdx.x;

  if (through && blockIdx.x == 0)
    for (int j = tid; j < n; j += SM_THREADS) {
      const size_t o = (size_t)v * a.vstride + (size_t)j * a.es + (size_t)a.lines * a.ls;
      a.out[o] = through[o];
    }
  normalised_taps(R, a.sigma, SM_THREADS, [&](int t, float v) { w[t] = v; });

  if (!a.adjoint) {
    // xe[(p + R) * cw + c] = line c at mirror(p), p in [-R, n - 1 + R]
    const int ne = n + 2 * R;
    for (int idx = tid; idx < ne * cw; idx += SM_THREADS) {
      const int pp = idx >> a.lcw, c = idx & cm;
      float val = 0.0f;
      if (l0 + c < a.lines) val = src[(size_t)mirror_of(pp - R, n) * a.es + (size_t)c * a.ls];
      xe[idx] = val;
    }
    __syncthreads();
    for (int idx = tid; idx < n * cw; idx += SM_THREADS) {
      const int i = idx >> a.lcw, c = idx & cm;
      if (l0 + c >= a.lines) continue;
      const float *x = xe + (size_t)i * cw + c;
      float acc = 0.0f;
      for (int t = 0; t < ntap; ++t) acc = fmaf(w[t], x[t * cw], acc);
      dst[(size_t)i * a.es + (size_t)c * a.ls] = acc;
    }
    return;
  }

  // transpose: y zero-padded by 2R on each side, then c(p) = sum_t w_t
  // y(p - t) for p in [-R, n - 1 + R], folded onto mirror(p)
  const int ny = n + 4 * R, nc = n + 2 * R;
  float *ye = xe;
  float *ce = xe + (size_t)ny * cw;
  for (int idx = tid; idx < ny * cw; idx += SM_THREADS) {
    const int q = (idx >> a.lcw) - 2 * R, c = idx & cm;
    float val = 0.0f;
    if (q >= 0 && q < n && l0 + c < a.lines) val = src[(size_t)q * a.es + (size_t)c * a.ls];
    ye[idx] = val;
  }
  __syncthreads();
  for (int idx = tid; idx < nc * cw; idx += SM_THREADS) {
    const int pp = idx >> a.lcw, c = idx & cm;  // p = pp - R: y(p - t) sits at ye[pp + 2R - t']
    const float *y = ye + (size_t)(pp + 2 * R) * cw + c;
    float acc = 0.0f;
    for (int t = 0; t < ntap; ++t) acc = fmaf(w[t], y[-(t * cw)], acc);
    ce[idx] = acc;
  }
  __syncthreads();
  for (int idx = tid; idx < n * cw; idx += SM_THREADS) {
    const int j = idx >> a.lcw, c = idx & cm;
    if (l0 + c >= a.lines) continue;
    float acc = 0.0f;
    if (n == 1) {
      for (int pp = 0; pp < nc; ++pp) acc += ce[(size_t)pp * cw + c];
    } else {
      // extended positions p in [-R, n - 1 + R] with mirror(p) = j:
      // p = j or p = -j modulo T = 2(n - 1) (one class at both ends)
      const int T = 2 * (n - 1);
      const int ncls = (j == 0 || j == n - 1) ? 1 : 2;
      for (int cl = 0; cl < ncls; ++cl) {
        const int p0 = cl ? -j : j;
        const int off = p0 + R;  // first p >= -R congruent to p0
        const int k = off >= 0 ? off / T : -((-off + T - 1) / T);
        for (int p = p0 - k * T; p <= n - 1 + R; p += T) acc += ce[(size_t)(p + R) * cw + c];
      }
    }
    dst[(size_t)j * a.es + (size_t)c * a.ls] = acc;
  }
}

constexpr int ST_OUT = 16;                // outputs per thread along the line
constexpr int ST_SEG = 128;               // outputs per CTA along the line
constexpr int ST_LINES = 64;              // lines per CTA, two per lane
constexpr int ST_LS = ST_LINES + 2;       // row stride: transposed stores meet two per bank
constexpr int ST_THREADS = 32 * (ST_SEG / ST_OUT);
constexpr int ST_MAX_R = 320;

size_t tile_smem(int R) {
  return sizeof(float) * ((size_t)(ST_SEG + 2 * R) * ST_LS + 2 * ((2 * R + 1 + 1) & ~1));
}

// a.in filtered into a.out; lanes run over the axis that is contiguous in
// memory when they load and store.  `through` (mu axis): the array whose
// entry `lines` of every row passes into a.out.
__global__ void __launch_bounds__(ST_THREADS, 3)
    k_smooth_tile(SmoothLines a, const float *__restrict__ through) {
  extern __shared__ __align__(16) float sm[];
  const int R = a.R, n = a.n, ntap = 2 * R + 1;
  const int rows = ST_SEG + 2 * R;                 // staged samples
  float *x = sm;                                   // [rows][ST_LS]
  float2 *w2 = reinterpret_cast<float2 *>(sm + (size_t)rows * ST_LS);  // taps, twice each
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i0 = blockIdx.x * ST_SEG, l0 = blockIdx.y * ST_LINES;
  const size_t vo = (size_t)blockIdx.z * a.vstride;
  const float *src = a.in + vo;
  float *dst = a.out + vo;
  const float end = a.adjoint && n > 1 ? 2.0f : 1.0f;  // D

  // every staged element is copied by cp.async, all in flight at once (loads
  // through registers waited for memory three quarters of the time)
  const int used = min(rows, n - i0 + 2 * R);  // samples that some output reads
  auto mirrored = [&](int pp) {
    int q = abs(i0 + pp - R);
    if (q >= n) q = 2 * (n - 1) - q;
    return (q < 0 || q >= n) ? mirror_of(i0 + pp - R, n) : q;
  };
  if (a.es == 1) {
    for (int pp = lane; pp < used; pp += 32) {
      const float *s0 = src + mirrored(pp) + (size_t)l0 * a.ls;
      float *d0 = x + (size_t)pp * ST_LS;
#pragma unroll
      for (int c = 0; c < ST_LINES / (ST_THREADS / 32); ++c) {
        const int cc = warp + c * (ST_THREADS / 32);
        if (l0 + cc < a.lines) dc::cp_async4(d0 + cc, s0 + (size_t)cc * a.ls);
      }
    }
  } else {
    for (int pp = warp; pp < used; pp += ST_THREADS / 32) {
      const float *s0 = src + (size_t)mirrored(pp) * a.es + l0;
      float *d0 = x + (size_t)pp * ST_LS;
      if (l0 + lane < a.lines) dc::cp_async4(d0 + lane, s0 + lane);
      if (l0 + lane + 32 < a.lines) dc::cp_async4(d0 + lane + 32, s0 + lane + 32);
    }
  }
  dc::cp_async_commit();
  normalised_taps(R, a.sigma, ST_THREADS, [&](int t, float v) { w2[t] = make_float2(v, v); });
  dc::cp_async_wait<0>();
  __syncthreads();
  if (end != 1.0f) {  // D: twice the end samples, wherever they are staged
    for (int pp = warp; pp < used; pp += ST_THREADS / 32) {
      const int q = mirrored(pp);
      if (q == 0 || q == n - 1) {
        x[(size_t)pp * ST_LS + lane] *= end;
        x[(size_t)pp * ST_LS + lane + 32] *= end;
      }
    }
    __syncthreads();
  }

  // outputs i0 + ST_OUT warp + i of lines l0 + 2 lane, + 1
  float2 acc[ST_OUT], win[ST_OUT];
  const float *xp = x + (size_t)(warp * ST_OUT) * ST_LS + 2 * lane;
#pragma unroll
  for (int i = 0; i < ST_OUT; ++i) {
    acc[i] = make_float2(0.0f, 0.0f);
    win[i] = *reinterpret_cast<const float2 *>(xp + i * ST_LS);
  }
  xp += ST_OUT * ST_LS;
  const bool some = i0 + warp * ST_OUT < n;
  int t = 0;
  for (; some && t + ST_OUT <= ntap; t += ST_OUT) {
#pragma unroll
    for (int u = 0; u < ST_OUT; ++u) {
      const float2 w = w2[t + u];
#pragma unroll
      for (int i = 0; i < ST_OUT; ++i) acc[i] = __ffma2_rn(w, win[(i + u) % ST_OUT], acc[i]);
      // the window's next sample (rows + ST_OUT in all: one past the last tap's)
      if (t + u + 1 < ntap) win[u] = *reinterpret_cast<const float2 *>(xp);
      xp += ST_LS;
    }
  }
  if (some) {
#pragma unroll
    for (int u = 0; u < ST_OUT; ++u) {
      if (t + u < ntap) {
        const float2 w = w2[t + u];
#pragma unroll
        for (int i = 0; i < ST_OUT; ++i) acc[i] = __ffma2_rn(w, win[(i + u) % ST_OUT], acc[i]);
        if (t + u + 1 < ntap) win[u] = *reinterpret_cast<const float2 *>(xp);
        xp += ST_LS;
      }
    }
  }
  __syncthreads();
  // back through shared memory, so that the stores are contiguous
#pragma unroll
  for (int i = 0; i < ST_OUT; ++i)
    *reinterpret_cast<float2 *>(x + (size_t)(warp * ST_OUT + i) * ST_LS + 2 * lane) = acc[i];
  __syncthreads();
  const float iend = 1.0f / end;
  auto store = [&](int i, int c) {
    const int j = i0 + i, l = l0 + c;
    if (j >= n) return;
    const size_t o = (size_t)j * a.es + (size_t)l * a.ls;
    const float v = x[(size_t)i * ST_LS + c];
    if (l < a.lines) dst[o] = (j == 0 || j == n - 1) ? v * iend : v;
    else if (through && l == a.lines) dst[o] = through[vo + o];
  };
  if (a.es == 1) {
    for (int c = warp; c < ST_LINES; c += ST_THREADS / 32)
      for (int i = lane; i < ST_SEG; i += 32) store(i, c);
  } else {
    for (int e = tid; e < ST_SEG * ST_LINES; e += ST_THREADS) store(e / ST_LINES, e % ST_LINES);
  }
}

int launch_tile(const SmoothLines &a, int views, const float *through, cudaStream_t st) {
  const size_t smem = tile_smem(a.R);
  DC_CUDA(cudaFuncSetAttribute(k_smooth_tile, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)tile_smem(ST_MAX_R)));
  const int lines = a.lines + (through ? 1 : 0);
  dc::ProfScope ps(dc::KID_SMOOTH, st);
  // at most 65535 views per launch (the grid's z limit)
  for (int v0 = 0; v0 < views; v0 += 65535) {
    SmoothLines b = a;
    b.in = a.in + (size_t)v0 * a.vstride;
    b.out = a.out + (size_t)v0 * a.vstride;
    dim3 grid((unsigned)((a.n + ST_SEG - 1) / ST_SEG), (unsigned)((lines + ST_LINES - 1) / ST_LINES),
              (unsigned)std::min(65535, views - v0));
    k_smooth_tile<<<grid, ST_THREADS, smem, st>>>(
        b, through ? through + (size_t)v0 * a.vstride : nullptr);
    DC_CHECK_LAUNCH("k_smooth_tile");
  }
  return DC_OK;
}

size_t smem_floats(int n, int R, int lcw, int adjoint) {
  return (size_t)((2 * R + 1 + 3) & ~3) +
         ((size_t)1 << lcw) * (size_t)(adjoint ? (2 * n + 6 * R) : (n + 2 * R));
}

int launch_lines(const SmoothLines &a, int views, const float *through, cudaStream_t st) {
  const int cw = 1 << a.lcw;
  const size_t smem = smem_floats(a.n, a.R, a.lcw, a.adjoint) * sizeof(float);
  static bool attr_done = false;
  if (!attr_done) {
    DC_CUDA(cudaFuncSetAttribute(k_smooth_lines, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)SM_SMEM_BUDGET));
    attr_done = true;
  }
  dim3 grid((unsigned)((a.lines + cw - 1) / cw), (unsigned)views);
  dc::ProfScope ps(dc::KID_SMOOTH, st);
  k_smooth_lines<<<grid, SM_THREADS, smem, st>>>(a, through);
  DC_CHECK_LAUNCH("k_smooth_lines");
  return DC_OK;
}

// Few short lines leave the tiles' CTAs with nothing to overlap: what counts is
// the time of one CTA, and that of k_smooth_lines, a few lines at a time, is
// shorter.  16 views of 90 x 64, radius 3: 11.1 us with it, 14.4 with tiles
// (radius 60: 23.1 and 22.6; about 1 us less since no copy follows it); 48 views 16.3 and 14.5; one view of 360 x 256 20.1
// and 17.1, six of 250 x 80 with radius 15 21.3 and 19.6.  Its transpose folds the halo back and so takes small radii only
// (4 views of 90 x 64: radius 15 13.4 and 17.6, radius 60 32.5 and 25.2).
bool few_samples(int V, int n_mu, int n_s, int radius, int adjoint) {
  const double n = (double)V * n_mu * n_s;
  return V <= 65535 && n <= 1 << 17 && std::max(n_mu, n_s) <= 224 &&
         (adjoint ? radius <= 16 : n * (2 * radius + 1) <= 1 << 23);
}

// lines per CTA along mu: the widest power of two (<= 16) whose staging fits
int mu_log_width(int n_mu, int R, int adjoint) {
  for (int l = 4; l >= 0; --l)
    if (smem_floats(n_mu, R, l, adjoint) * sizeof(float) <= SM_SMEM_BUDGET) return l;
  return -1;
}

}  // namespace

extern "C" int dc_gauss_smooth(int V, int n_mu, int n_s, float sigma, int radius, int adjoint,
                               const float *in, float *out, float *work, void *stream) {
  if (V < 1 || n_mu < 1 || n_s < 2)
    return dc::fail(DC_ERR_ARG, "dc_gauss_smooth: sizes must be positive (n_s >= 2)");
  if (!in || !out || !work) return dc::fail(DC_ERR_ARG, "dc_gauss_smooth: NULL array");
  if (in == out || in == work || out == work)
    return dc::fail(DC_ERR_ARG, "dc_gauss_smooth: in, out and work must not alias");
  if (!(sigma > 0.0f) || !std::isfinite(sigma) || radius < 0 || radius > 1024)
    return dc::fail(DC_ERR_ARG, "dc_gauss_smooth: sigma > 0 and 0 <= radius <= 1024");
  const int ns1 = n_s - 1;
  const int ad = adjoint ? 1 : 0;
  const int lmu = mu_log_width(n_mu, radius, ad);
  if (lmu < 0 || smem_floats(ns1, radius, 0, ad) * sizeof(float) > SM_SMEM_BUDGET)
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_gauss_smooth: lines too long for shared memory");
  cudaStream_t st = (cudaStream_t)stream;

  SmoothLines s_axis;  // rows: n_mu lines of ns1 contiguous samples
  s_axis.n = ns1;
  s_axis.lines = n_mu;
  s_axis.vstride = (size_t)n_mu * n_s;
  s_axis.es = 1;
  s_axis.ls = n_s;
  s_axis.lcw = 0;
  s_axis.R = radius;
  s_axis.sigma = sigma;
  s_axis.adjoint = ad;
  SmoothLines mu_axis = s_axis;  // columns: ns1 lines of n_mu samples, n_s apart
  mu_axis.n = n_mu;
  mu_axis.lines = ns1;
  mu_axis.es = n_s;
  mu_axis.ls = 1;
  mu_axis.lcw = lmu;

  // in -> work along s, work -> out along mu (the axis filters commute, and
  // so do their transposes); the unused entry n_s - 1 is copied through
  s_axis.in = in;
  s_axis.out = work;
  int rc;
  if (radius <= ST_MAX_R && !few_samples(V, n_mu, n_s, radius, ad)) {
    if ((rc = launch_tile(s_axis, V, nullptr, st))) return rc;
    mu_axis.in = work;
    mu_axis.out = out;
    return launch_tile(mu_axis, V, in, st);
  }
  if ((rc = launch_lines(s_axis, V, nullptr, st))) return rc;
  mu_axis.in = work;
  mu_axis.out = out;
  return launch_lines(mu_axis, V, in, st);
}
