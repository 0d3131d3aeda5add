// dc_crofton.cu -- smooth Crofton weights of Eq. 9 (Ye et al., DRACO, Sec.
// 2.3), the analytic redundancy weight for an arbitrary discrete orbit:
//
//   M(theta, lambda_i) = |a'(lambda_i).theta|^m c(lambda_i)
//                        / sum_alpha |a'(lambda_alpha).theta|^m c(lambda_alpha)
//
// for every view i and plane (mu, s_{k+1/2}) through the source a_i.  The
// intersections lambda_alpha of the plane with the orbit are view i itself
// and every sign change of f_j = (a_j - a_i).theta between consecutive views
// of a segment (wrapping for a closed segment; pairs containing i are
// skipped), where the tangent and the taper c are interpolated linearly.
// With m >= 1 the weight is continuous across tangencies, so FP32 suffices.
#include <cstring>
#include <string>

#include "dc_common.cuh"

namespace {

constexpr int CR_THREADS = 256;

struct CroftonArgs {
  const dc::MuRec *mu;      // cos, sin per angle
  const dc::FView *fv;      // D per view
  const double *geo;        // FP64 records (frame, tangent)
  int V, n_mu, n_s, m, taper;
  float ds;
  int n_seg;
  int seg_start[DC_MAX_SEGMENTS];
  int seg_closed[DC_MAX_SEGMENTS];
  float *W;
};

__device__ float taper_of(int j, const CroftonArgs &a) {
  if (a.taper <= 0) return 1.0f;
  for (int q = 0; q < a.n_seg; ++q) {
    int lo = a.seg_start[q], hi = (q + 1 < a.n_seg) ? a.seg_start[q + 1] : a.V;
    if (j < lo || j >= hi) continue;
    if (a.seg_closed[q]) return 1.0f;
    int d = min(j - lo, hi - 1 - j);
    if (d >= a.taper) return 1.0f;
    float x = sinpif(0.5f * ((float)d + 0.5f) / (float)a.taper);
    return x * x;
  }
  return 1.0f;
}

__device__ __forceinline__ float powi(float x, int m) {
  float r = 1.0f;
  for (int e = 0; e < m; ++e) r *= x;
  return r;
}

// A CTA takes up to CR_MU angles of one view; the orbit relative to a_i lives in
// shared memory, once for all of them.  A warp takes 32 neighbouring s-bins of
// one angle (lane = plane).
//
// Testing every pair of views for every plane is what the time would go to
// (1.2e10 pairs for 360 views and 360 x 256 planes: 9.0 ms), and a plane meets
// the orbit a few times only.  f_j is, up to a positive factor, linear in s,
// so a view whose f keeps one sign at both ends of the warp's s-range keeps it
// for all 32 planes: lanes test 32 views at once at the two ends, and only the
// pairs whose two views are not both positive or both negative are looked at
// plane by plane, in the same order and with the same arithmetic (1.66 ms).
// A view within the rounding of f of zero at an end counts as neither.
constexpr int CR_MU = 16;  // at most: fewer where the grid would not fill the GPU

__global__ void __launch_bounds__(CR_THREADS) k_crofton(CroftonArgs a, int n_ang) {
  extern __shared__ float4 orb[];  // [V] (a_j - a_i, c_j), then [V] (v_j, 0)
  const int i = blockIdx.y;
  const double *gi = a.geo + (size_t)DC_VIEW_GEO_N * i;
  float4 *vt = orb + a.V;
  for (int j = threadIdx.x; j < a.V; j += CR_THREADS) {
    const double *gj = a.geo + (size_t)DC_VIEW_GEO_N * j;
    orb[j] = make_float4((float)(gj[0] - gi[0]), (float)(gj[1] - gi[1]), (float)(gj[2] - gi[2]),
                         taper_of(j, a));
    vt[j] = make_float4((float)gj[15], (float)gj[16], (float)gj[17], 0.0f);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const float D = a.fv[i].D;
  float lx[3], ly[3], lz[3];
  for (int c = 0; c < 3; ++c) {
    lx[c] = (float)gi[3 + c];
    ly[c] = (float)gi[6 + c];
    lz[c] = (float)gi[9 + c];
  }
  const float4 vi = vt[i];
  const float ci = orb[i].w;
  const int nch = (a.n_s + 31) >> 5, m0 = blockIdx.x * n_ang;
  const int items = min(n_ang, a.n_mu - m0) * nch;
  for (int w = threadIdx.x >> 5; w < items; w += CR_THREADS / 32) {
    const int m = m0 + w / nch, k0 = (w % nch) * 32, k = k0 + lane;
    const dc::MuRec mr = a.mu[m];
    auto s_half = [&](int q) { return ((float)q - 0.5f * (float)(a.n_s - 1) + 0.5f) * a.ds; };
    const float sh = s_half(k);
    const float nrm = rsqrtf(fmaf(sh, sh, D * D));
    float th[3];
    for (int c = 0; c < 3; ++c) th[c] = (D * mr.c * lx[c] + D * mr.s * ly[c] + sh * lz[c]) * nrm;
    const float own = powi(fabsf(vi.x * th[0] + vi.y * th[1] + vi.z * th[2]), a.m) * ci;
    // the plane normals (not normalised) at the two ends of the warp's range
    const float se0 = s_half(k0), se1 = s_half(k0 + 31);
    float u0[3], u1[3];
    for (int c = 0; c < 3; ++c) {
      const float b = D * mr.c * lx[c] + D * mr.s * ly[c];
      u0[c] = fmaf(se0, lz[c], b);
      u1[c] = fmaf(se1, lz[c], b);
    }
    // bound on the rounding of f (a few 1e-7 |a_j - a_i|, here times |u|)
    const float tol = 4e-6f * (D + fmaxf(fabsf(se0), fabsf(se1)));
    float sum = own;
    for (int q = 0; q < a.n_seg; ++q) {
      const int lo = a.seg_start[q], hi = (q + 1 < a.n_seg) ? a.seg_start[q + 1] : a.V;
      const int npair = a.seg_closed[q] ? hi - lo : hi - lo - 1;
      // 31 pairs (e, e + 1) at a time; lane 31 holds the last pair's second view
      for (int e0 = 0; e0 < npair; e0 += 31) {
        const int e = e0 + lane;
        const float4 o = orb[lo + (e < hi - lo ? e : (e - (hi - lo)) % (hi - lo))];
        const float f0 = fmaf(o.x, u0[0], fmaf(o.y, u0[1], o.z * u0[2]));
        const float f1 = fmaf(o.x, u1[0], fmaf(o.y, u1[1], o.z * u1[2]));
        const float t = tol * (fabsf(o.x) + fabsf(o.y) + fabsf(o.z));
        const unsigned P = __ballot_sync(0xffffffffu, fminf(f0, f1) > t);
        const unsigned N = __ballot_sync(0xffffffffu, fmaxf(f0, f1) < -t);
        const int cnt = min(31, npair - e0);
        unsigned todo = ~((P & (P >> 1)) | (N & (N >> 1))) & ((1u << cnt) - 1u);
        while (todo) {
          const int b = __ffs(todo) - 1;
          todo &= todo - 1;
          const int j0 = lo + e0 + b, j1 = (j0 + 1 < hi) ? j0 + 1 : lo;
          if (j0 == i || j1 == i) continue;
          const float4 o0 = orb[j0], o1 = orb[j1];
          const float g0 = o0.x * th[0] + o0.y * th[1] + o0.z * th[2];
          const float g1 = o1.x * th[0] + o1.y * th[1] + o1.z * th[2];
          if ((g0 < 0.0f) != (g1 < 0.0f)) {
            const float tt = g0 / (g0 - g1);
            const float4 v0 = vt[j0], v1 = vt[j1];
            const float vx = fmaf(tt, v1.x - v0.x, v0.x), vy = fmaf(tt, v1.y - v0.y, v0.y),
                        vz = fmaf(tt, v1.z - v0.z, v0.z);
            const float ca = fmaf(tt, o1.w - o0.w, o0.w);
            sum += powi(fabsf(vx * th[0] + vy * th[1] + vz * th[2]), a.m) * ca;
          }
        }
      }
    }
    if (k < a.n_s)
      a.W[((size_t)i * a.n_mu + m) * a.n_s + k] =
          (k == a.n_s - 1 || !(own > 0.0f)) ? 0.0f : own / sum;
  }
}

}  // namespace

extern "C" int dc_crofton_weights(const dc_geometry *g, int n_seg, const int *seg_start,
                                  const int *seg_closed, int m, int taper, float *W,
                                  void *stream) {
  if (!g || !W) return dc::fail(DC_ERR_ARG, "dc_crofton_weights: NULL argument");
  const dc_geometry_desc &d = g->d;
  CroftonArgs a;
  memset(&a, 0, sizeof(a));
  if (n_seg == 0) {
    a.n_seg = 1;
    a.seg_start[0] = 0;
    a.seg_closed[0] = d.closed_orbit ? 1 : 0;
  } else {
    if (n_seg < 0 || n_seg > DC_MAX_SEGMENTS || !seg_start || !seg_closed)
      return dc::fail(DC_ERR_ARG, "dc_crofton_weights: 1 <= n_seg <= " +
                                      std::to_string(DC_MAX_SEGMENTS) + " with both arrays");
    if (seg_start[0] != 0) return dc::fail(DC_ERR_ARG, "dc_crofton_weights: first segment must start at view 0");
    for (int q = 0; q < n_seg; ++q) {
      int hi = (q + 1 < n_seg) ? seg_start[q + 1] : d.n_views;
      if (seg_start[q] >= hi)
        return dc::fail(DC_ERR_ARG, "dc_crofton_weights: segment starts must increase below V");
      a.seg_start[q] = seg_start[q];
      a.seg_closed[q] = seg_closed[q] ? 1 : 0;
    }
    a.n_seg = n_seg;
  }
  if (m < 0 || m > 8) return dc::fail(DC_ERR_ARG, "dc_crofton_weights: 0 <= m <= 8");
  if (taper < 0) return dc::fail(DC_ERR_ARG, "dc_crofton_weights: taper must be >= 0");
  size_t smem = sizeof(float4) * 2 * (size_t)d.n_views;
  if (smem > 200 * 1024)
    return dc::fail(DC_ERR_UNSUPPORTED, "dc_crofton_weights: too many views for shared memory");
  a.mu = g->mu;
  a.fv = g->fv;
  a.geo = g->geo64;
  a.V = d.n_views;
  a.n_mu = d.n_mu;
  a.n_s = d.n_s;
  a.m = m;
  a.taper = taper;
  a.ds = (float)d.ds;
  a.W = W;
  cudaStream_t st = (cudaStream_t)stream;
  DC_CUDA(cudaFuncSetAttribute(k_crofton, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               200 * 1024));
  // the grid's y limit is 65535; shared memory allows 6400 views
  // few views: fewer angles per CTA until two CTAs per SM have some (16 views,
  // 90 x 64 planes: 8.6 us with 16 angles, 6.5 with 2; 6 views, 720 x 512: 43 and
  // 34)
  int n_ang = CR_MU;
  while (n_ang > 1 && (long)((d.n_mu + n_ang - 1) / n_ang) * d.n_views < 2 * g->sms) n_ang /= 2;
  dim3 grid((d.n_mu + n_ang - 1) / n_ang, d.n_views);
  k_crofton<<<grid, CR_THREADS, smem, st>>>(a, n_ang);
  DC_CHECK_LAUNCH("k_crofton");
  return DC_OK;
}
