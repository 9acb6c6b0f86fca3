// Batched chi2 of multiple-image constraints (Sec. 2.2, Eq. 6, Fig. 3).
//
// Static cache: when a constraint set is bound to a model, the FP64
// deflection and Hessian of every potential except the two varying ones are
// summed at each constraint position once (one CTA per image, deterministic
// tree reduction).  A parameter set then costs two FP64 potential
// evaluations per image instead of N.
//
// Source-plane kernel: persistent CTAs loop over parameter sets; per set the
// CTA rebuilds the two varying potentials, back-traces every image
// (beta = theta - r alpha, Sec. 2.1 Eq. 1), forms each source's barycentre
// and reduces the chi2 with warp shuffles in a fixed order.
//
// No-cache form: the static sum is recomputed for every parameter set (a
// batch of sets at a time, into scratch memory, in double-float) before the
// same source-plane kernel runs; this is the per-set cost when any potential
// may vary, as in the paper's fit, where every potential is evaluated for
// every model.
//
// The two varying potentials are evaluated in double-float (FP32 pipe,
// ~1e-13 relative; lens_chi2_df.cuh), two images side by side per thread, FP64
// only where that fails; the static cache itself is FP64.
#include <algorithm>

#include "lens_chi2_df.cuh"

namespace lens {
namespace {

constexpr int CACHE_THREADS = 128;
constexpr int NOCACHE_BATCH = 512;  // parameter sets per batch of the no-cache form

// grid (nimg, copies): copy c of the sums goes to stat + c * nimg * 5
__global__ void __launch_bounds__(CACHE_THREADS) k_static_cache(const double *__restrict__ all64, int n, int v0,
                                                                int v1, const double *__restrict__ x,
                                                                const double *__restrict__ y, double *stat) {
  __shared__ double s_red[(CACHE_THREADS / 32) * 5];
  const int img = blockIdx.x;
  stat += (size_t)blockIdx.y * gridDim.x * 5;
  const double X = x[img], Y = y[img];
  double v[5] = {0, 0, 0, 0, 0};
  for (int h = threadIdx.x; h < n; h += CACHE_THREADS) {
    if (h == v0 || h == v1) continue;
    double ax, ay, k, g1, g2;
    eval64<true>(all64 + (size_t)h * REC64, X, Y, ax, ay, k, g1, g2);
    v[0] += ax;
    v[1] += ay;
    v[2] += k;
    v[3] += g1;
    v[4] += g2;
  }
  block_sum<5, CACHE_THREADS>(v, s_red);
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; ++k) stat[(size_t)img * 5 + k] = v[k];
}

struct Chi2SrcArgs {
  const double *stat, *x, *y, *isig2, *ratio, *params;
  long long stat_stride;  // doubles between the static sums of consecutive sets (0: one shared cache)
  int pstride;            // doubles per parameter set (14; 16 with the members' scaling factors)
  const int32_t *img_off, *src_of;
  int nsrc, nimg, P, variant;
  int type0, type1;
  double *chi2;
  int keep_xy;  // the images' positions as float pairs fit in shared memory
};

// Parameter sets whose varying potentials' records two warps build at a
// time (one thread per record: the FP64 record arithmetic runs 32 lanes wide
// instead of on two threads per set).
constexpr int SRC_BATCH = 16;
constexpr int SRC_INV = 16;  // image counts whose reciprocals are kept

// The FP64 record (kind 0; returns whether the parameters are inside the
// domain) or the double-float record (kind 1) of varying potential v of a
// parameter set, out of line.
__device__ __noinline__ bool var_rec_cold(const double *q, int type0, int type1, int v, int kind, double *s_rec,
                                          float2 *s_rdf) {
  if (kind == 0) return load_var_rec64(q, type0, type1, v, s_rec);
  const double *w = q + 7 * v;
  make_recdf(v == 0 ? type0 : type1, w[0], w[1], w[3], w[2], w[4], w[5], w[6], s_rdf + v * RECDF);
  record_consts<true>(s_rdf + v * RECDF);
  return true;
}

__device__ __forceinline__ Df<float> d_from_double(double d) {
  const df v = df_from_double(d);
  return {v.hi, v.lo};
}
// A finite float as a double by integer operations (conversions run on the
// FP64 pipe, at 1/64 of the FP32 rate); subnormals become zero.
__device__ __forceinline__ double f_to_double(float f) {
  const int i = __float_as_int(f);
  const bool zero = (i & 0x7f800000) == 0;
  return __hiloint2double(zero ? 0 : (i & 0x80000000) | (((i >> 3) & 0x0fffffff) + (896 << 20)), zero ? 0 : i << 29);
}
__device__ __forceinline__ double d_to_double(float hi, float lo) {
  if (!(fabsf(hi) < INFINITY)) return (double)hi;  // (rare: keeps NaN and infinity)
  return f_to_double(hi) + f_to_double(lo);
}

// r alpha and r H of image j from its sums acc (static cache + varying
// potentials): beta into s_beta and, if HESS, r hxx, r hyy, r hxy into s_m.
template <bool HESS>
__device__ __forceinline__ void store_image(const Chi2SrcArgs &a, int j, double X, double Y, const double *acc,
                                            double *s_beta, double *s_m) {
  const double r = a.ratio[a.src_of[j]];
  s_beta[2 * j] = X - r * acc[0];
  s_beta[2 * j + 1] = Y - r * acc[1];
  if (HESS) {
    s_m[3 * j] = r * (acc[2] + acc[3]);
    s_m[3 * j + 1] = r * (acc[2] - acc[3]);
    s_m[3 * j + 2] = r * acc[4];
  }
}

// Back-trace of every image, two images per thread side by side (j and j +
// ceil(nimg / 2)), which with the called division and polynomial and fewer
// FP64 operations (positions as pairs, integer conversions) takes 0.284
// instead of 0.341 ms per 4096 sets x 372 images: both varying potentials in double-float, summed in
// double-float and added to the static cache with one conversion each; FP64
// for a potential whose double-float evaluation fails.
template <int THREADS, bool HESS>
__device__ __forceinline__ void backtrace_pairs(const Chi2SrcArgs &a, const double *stat, const double *s_rec,
                                                const float2 *s_rdf, const float4 *s_xy, double *s_beta, double *s_m) {
  const int half = (a.nimg + 1) / 2;
  for (int j0 = threadIdx.x; j0 < half; j0 += THREADS) {
    const int j1 = j0 + half < a.nimg ? j0 + half : j0;  // (alone: a copy of itself, not stored)
    Df<float2> X, Y, sum[5];
    double acc[2][5];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int j = k ? j1 : j0;
      float4 xy;
      if (a.keep_xy) {
        xy = s_xy[j];
      } else {
        const Df<float> x = d_from_double(a.x[j]), y = d_from_double(a.y[j]);
        xy = make_float4(x.hi, x.lo, y.hi, y.lo);
      }
      part2(X.hi, k) = xy.x;
      part2(X.lo, k) = xy.y;
      part2(Y.hi, k) = xy.z;
      part2(Y.lo, k) = xy.w;
#pragma unroll
      for (int q = 0; q < (HESS ? 5 : 2); ++q) acc[k][q] = 0.0;
    }
    bool cold = false;
#pragma unroll 1
    for (int v = 0; v < 2; ++v) {  // one copy of the (large) evaluator in the code
      Df<float2> t[5];
      const unsigned ok = any_fixed<HESS, true>(s_rdf + v * RECDF, X, Y, t[0], t[1], t + 2);
      if (ok != f_all<float2>) {
        const Df<float2> zero = d_dup<float2>(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < (HESS ? 5 : 2); ++q) t[q] = d_sel(ok, t[q], zero);
        cold = true;
#pragma unroll
        for (int k = 0; k < 2; ++k)
          if (!(ok >> k & 1u)) {
            double e[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
            const int j = k ? j1 : j0;
            eval64_cold<HESS>(s_rec + v * REC64, a.x[j], a.y[j], e);
#pragma unroll
            for (int q = 0; q < (HESS ? 5 : 2); ++q) acc[k][q] = v == 0 || acc[k][q] == 0.0 ? e[q] : acc[k][q] + e[q];
          }
      }
#pragma unroll
      for (int q = 0; q < (HESS ? 5 : 2); ++q) sum[q] = v == 0 ? t[q] : d_add(sum[q], t[q]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int j = k ? j1 : j0;
      if (k && j1 == j0) break;
      const double *st = stat + (size_t)j * 5;
      double o[5];
#pragma unroll
      for (int q = 0; q < (HESS ? 5 : 2); ++q)
        o[q] = (cold ? st[q] + acc[k][q] : st[q]) + d_to_double(part2(sum[q].hi, k), part2(sum[q].lo, k));
      store_image<HESS>(a, j, a.x[j], a.y[j], o, s_beta, s_m);
    }
  }
}

// The same with a thread per (image, potential), for calls of so few sets
// that a CTA has an SM to itself: half the chain per thread.
template <int THREADS, bool HESS>
__device__ __forceinline__ void backtrace_split(const Chi2SrcArgs &a, const double *stat, const double *s_rec,
                                                const float2 *s_rdf, double *s_beta, double *s_m) {
  const int v = threadIdx.x & 1, lane0 = threadIdx.x & ~31;
  for (int t0 = 0; 2 * a.nimg > t0 + lane0; t0 += THREADS) {  // whole warps
    const int j = min((t0 + (int)threadIdx.x) >> 1, a.nimg - 1);
    const double X = a.x[j], Y = a.y[j];
    Df<float> t[5];
    double e[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const unsigned ok = any_fixed<HESS, true>(s_rdf + v * RECDF, d_from_double(X), d_from_double(Y), t[0], t[1], t + 2);
    if (!ok) {
      eval64_cold<HESS>(s_rec + v * REC64, X, Y, e);
#pragma unroll
      for (int q = 0; q < (HESS ? 5 : 2); ++q) t[q] = {0.f, 0.f};
    }
    const bool cold = __any_sync(0xffffffffu, !ok);
    const double *st = stat + (size_t)j * 5;
    double o[5];
#pragma unroll
    for (int q = 0; q < (HESS ? 5 : 2); ++q) {  // the odd thread's result joins the even one's
      const Df<float> u = {__shfl_xor_sync(0xffffffffu, t[q].hi, 1), __shfl_xor_sync(0xffffffffu, t[q].lo, 1)};
      double s = st[q];
      if (cold) s = (s + e[q]) + __shfl_xor_sync(0xffffffffu, e[q], 1);
      const Df<float> w = d_add(t[q], u);
      o[q] = s + d_to_double(w.hi, w.lo);
    }
    if (v == 0 && (t0 + (int)threadIdx.x) >> 1 < a.nimg) store_image<HESS>(a, j, X, Y, o, s_beta, s_m);
  }
}

// HESS: the variants that need the Hessian (the plain residuals take fewer
// registers without it).  SPLIT: a thread per (image, varying potential),
// else two images per thread.
template <int THREADS, bool HESS, bool SPLIT>
__global__ void __launch_bounds__(THREADS) k_chi2_source(const Chi2SrcArgs a) {
  static_assert(THREADS >= 4 * SRC_BATCH, "one thread per record of a batch");
  extern __shared__ double sm[];
  double *s_beta = sm;                   // [nimg][2]
  double *s_m = s_beta + 2 * a.nimg;     // [nimg][3]: r hxx, r hyy, r hxy
  double *s_bary = s_m + 3 * a.nimg;     // [nsrc][2]
  double *s_red = s_bary + 2 * a.nsrc;   // [THREADS/32]
  // the images' positions as float pairs (two images per thread: read once per set)
  float4 *s_xy = reinterpret_cast<float4 *>(sm + ((5 * a.nimg + 2 * a.nsrc + THREADS / 32 + 1) & ~1));
  if (!SPLIT && a.keep_xy)
    for (int j = threadIdx.x; j < a.nimg; j += THREADS) {
      const Df<float> x = d_from_double(a.x[j]), y = d_from_double(a.y[j]);
      s_xy[j] = make_float4(x.hi, x.lo, y.hi, y.lo);
    }
  __shared__ double s_rec[SRC_BATCH][2 * REC64];   // FP64 records of the batch's varying potentials
  __shared__ float2 s_rdf[SRC_BATCH][2 * RECDF];   // the same in double-float
  __shared__ int s_ok[SRC_BATCH][2];
  __shared__ double s_inv[SRC_INV];                // 1 / (a source's images)
  if (const int k = (int)threadIdx.x - (THREADS - SRC_INV); k >= 0) s_inv[k] = k > 0 ? 1.0 / k : 0.0;  // (a warp that builds no records, where there is one)
  // this CTA's sets are p = blockIdx.x + j gridDim.x, taken SRC_BATCH at a time
  for (long long p0 = blockIdx.x; p0 < a.P; p0 += (long long)gridDim.x * SRC_BATCH) {
    __syncthreads();  // the previous batch's records are no longer read
    if (threadIdx.x < 4 * SRC_BATCH) {  // one warp builds the FP64 records, the next the double-float ones
      const int kind = threadIdx.x / (2 * SRC_BATCH), k = threadIdx.x % (2 * SRC_BATCH) >> 1, v = threadIdx.x & 1;
      const long long p = p0 + (long long)k * gridDim.x;
      if (p < a.P) {
        const bool ok = var_rec_cold(a.params + p * a.pstride, a.type0, a.type1, v, kind, s_rec[k], s_rdf[k]);
        if (kind == 0) s_ok[k][v] = ok;
      }
    }
    __syncthreads();
    for (int k = 0; k < SRC_BATCH; ++k) {
      const long long p = p0 + (long long)k * gridDim.x;
      if (p >= a.P) break;  // uniform over the CTA
      if (!(s_ok[k][0] && s_ok[k][1])) {
        if (threadIdx.x == 0) a.chi2[p] = __longlong_as_double(0x7ff8000000000000ll);
        continue;
      }
      const double *stat = a.stat + p * a.stat_stride;
      if (SPLIT)
        backtrace_split<THREADS, HESS>(a, stat, s_rec[k], s_rdf[k], s_beta, s_m);
      else
        backtrace_pairs<THREADS, HESS>(a, stat, s_rec[k], s_rdf[k], s_xy, s_beta, s_m);
      __syncthreads();
      for (int i = threadIdx.x; i < a.nsrc; i += THREADS) {  // each source's barycentre (Fig. 3)
        const int b = a.img_off[i], e = a.img_off[i + 1];
        double sx = 0, sy = 0;
        for (int j = b; j < e; ++j) {
          sx += s_beta[2 * j];
          sy += s_beta[2 * j + 1];
        }
        const double im = e - b < SRC_INV ? s_inv[e - b] : 1.0 / (e - b);
        s_bary[2 * i] = sx * im;
        s_bary[2 * i + 1] = sy * im;
      }
      __syncthreads();
      double acc[1] = {0.0};
      for (int j = threadIdx.x; j < a.nimg; j += THREADS) {
        const int i = a.src_of[j];
        const double dbx = s_bary[2 * i] - s_beta[2 * j], dby = s_bary[2 * i + 1] - s_beta[2 * j + 1];
        const double is2 = a.isig2[j];
        if (!HESS) {
          acc[0] += (dbx * dbx + dby * dby) * is2;
        } else {
          // A^-1 = I - r H (Sec. 2.1 Eq. 4)
          const double a11 = 1.0 - s_m[3 * j], a22 = 1.0 - s_m[3 * j + 1], a12 = -s_m[3 * j + 2];
          const double det = a11 * a22 - a12 * a12;
          const double id = det != 0.0 ? rcp64(det) : 1.0 / det;
          if (a.variant == LENS_CHI2_SRC_MU) {
            acc[0] += (dbx * dbx + dby * dby) * fabs(id) * is2;
          } else {
            const double rx = (a22 * dbx - a12 * dby) * id, ry = (a11 * dby - a12 * dbx) * id;
            acc[0] += (rx * rx + ry * ry) * is2;
          }
        }
      }
      block_sum<1, THREADS>(acc, s_red);
      if (threadIdx.x == 0) a.chi2[p] = acc[0];
    }
  }
}

}  // namespace

// Synchronous on the context's upload stream (no other stream waits).
int build_static_cache(lens_ctx *ctx, const Model *m, CSet *c) {
  cudaStream_t st = upload_stream(ctx);
  if (!st) return fail(LENS_ECUDA, "upload stream creation failed");
  k_static_cache<<<c->nimg, CACHE_THREADS, 0, st>>>(m->all64, m->n, c->var[0], c->var[1], c->x, c->y, c->stat);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(LENS_ECUDA, "static cache: %s", cudaGetErrorString(e));
  return LENS_OK;
}

template <int T, bool SPLIT = false>
static int launch_src_cfg(lens_ctx *ctx, const CSet *c, const double *d_params, int32_t P, int32_t variant,
                          double *d_chi2, cudaStream_t st, int blocks_per_sm, const double *stat = nullptr,
                          long long stat_stride = 0, int pstride = 14) {
  const size_t words = 5 * (size_t)c->nimg + 2 * (size_t)c->nsrc + T / 32;
  if (sizeof(double) * words > 200 * 1024) return fail(LENS_EINVAL, "constraint set too large for one CTA (%d images)", c->nimg);
  // the pair form also keeps the positions there when they fit
  const size_t with_xy = sizeof(double) * ((words + 1) & ~(size_t)1) + sizeof(float4) * (size_t)c->nimg;
  const bool keep_xy = !SPLIT && with_xy <= 100 * 1024;
  const size_t smem = keep_xy ? with_xy : sizeof(double) * words;
  auto kern = variant == LENS_CHI2_SRC_PLAIN ? k_chi2_source<T, false, SPLIT> : k_chi2_source<T, true, SPLIT>;
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  int per_sm = 0, nsm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T, smem);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device);
  per_sm = std::max(1, per_sm);
  if (blocks_per_sm > 0) per_sm = std::min(per_sm, blocks_per_sm);
  const int blocks = std::max(1, std::min(P, per_sm * nsm));
  Chi2SrcArgs a;
  a.stat = stat ? stat : c->stat;
  a.stat_stride = stat_stride;
  a.x = c->x;
  a.y = c->y;
  a.isig2 = c->isig2;
  a.ratio = c->ratio;
  a.params = d_params;
  a.pstride = pstride;
  a.img_off = c->img_off;
  a.src_of = c->src_of;
  a.nsrc = c->nsrc;
  a.nimg = c->nimg;
  a.P = P;
  a.variant = variant;
  a.type0 = c->var_type[0];
  a.type1 = c->var_type[1];
  a.chi2 = d_chi2;
  a.keep_xy = keep_xy;
  kern<<<blocks, T, smem, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(LENS_ECUDA, "chi2 source launch: %s", cudaGetErrorString(e));
  return LENS_OK;
}

// Launch shapes the autotuner sets against the untuned rule
// (launch_src_default): threads per CTA x CTAs per SM (0 = as many as fit).
static const int SRC_CFG[][2] = {{64, 0}, {64, 4}, {64, 2}, {128, 0}, {128, 2}, {128, 1}, {256, 0}, {256, 1}};
constexpr int N_SRC_CFG = sizeof(SRC_CFG) / sizeof(SRC_CFG[0]);

static int launch_src(lens_ctx *ctx, const CSet *c, const double *d_params, int32_t P, int32_t variant, double *d_chi2,
                      cudaStream_t st, int threads, int cap, const double *stat = nullptr, long long stat_stride = 0,
                      int pstride = 14) {
  switch (threads) {
    case 64: return launch_src_cfg<64>(ctx, c, d_params, P, variant, d_chi2, st, cap, stat, stat_stride, pstride);
    case 96: return launch_src_cfg<96>(ctx, c, d_params, P, variant, d_chi2, st, cap, stat, stat_stride, pstride);
    case 192: return launch_src_cfg<192>(ctx, c, d_params, P, variant, d_chi2, st, cap, stat, stat_stride, pstride);
    case 256: return launch_src_cfg<256>(ctx, c, d_params, P, variant, d_chi2, st, cap, stat, stat_stride, pstride);
    default: return launch_src_cfg<128>(ctx, c, d_params, P, variant, d_chi2, st, cap, stat, stat_stride, pstride);
  }
}

// The launch shape without a tuned one, from a sweep of 100 to 4096 sets x 18
// to 340 images (us; each pair of numbers with and without the Hessian):
//   - up to 64 images: a thread per (image, potential), 128 threads (4096 sets
//     x 44 images 76.5 / 57.0; image pairs leave half the warps idle: 101 / 76);
//   - a set per SM, or up to 160 images and 1000 sets: the same with 512 or 256
//     threads (100 x 340: 31.0 / 24.9 against 39 / 31; 700 x 93: 37 / 29
//     against 41 / 33);
//   - else image pairs: in one round while every CTA is resident (700 x 340: 192
//     threads 70 / 50, 64 82 / 64), then the threads that leave the fewest idle
//     in the last round, small CTAs when they are many (4096 x 340: 64 threads
//     282 / 223, 96 297 / 199, 192 297 / 217).
static int launch_src_default(lens_ctx *ctx, const CSet *c, const double *d_params, int32_t P, int32_t variant,
                              double *d_chi2, cudaStream_t st, const double *stat = nullptr, long long stat_stride = 0,
                              int pstride = 14) {
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device);
  const bool few = P <= nsm, some = P <= 8 * nsm;
  if (c->nimg <= 64)
    return launch_src_cfg<128, true>(ctx, c, d_params, P, variant, d_chi2, st, 0, stat, stat_stride, pstride);
  if (few && c->nimg > 128)
    return launch_src_cfg<512, true>(ctx, c, d_params, P, variant, d_chi2, st, 0, stat, stat_stride, pstride);
  if (few || (some && c->nimg <= 160))
    return launch_src_cfg<256, true>(ctx, c, d_params, P, variant, d_chi2, st, 0, stat, stat_stride, pstride);
  const int pairs = (c->nimg + 1) / 2;
  int best = 96;
  if (some) {
    best = pairs <= 128 ? 128 : 192;
  } else {
    int least = INT32_MAX;
    const bool many = P > 20 * nsm && variant != LENS_CHI2_SRC_PLAIN;
    for (int t : {many ? 64 : 96, many ? 96 : 64, 128, 192}) {
      const int slots = (pairs + t - 1) / t * t;
      if (slots < least) {
        least = slots;
        best = t;
      }
    }
  }
  return launch_src(ctx, c, d_params, P, variant, d_chi2, st, best, 0, stat, stat_stride, pstride);
}

int launch_chi2_source(lens_ctx *ctx, const Model *m, const CSet *c, const double *d_params, int32_t P,
                       int32_t variant, double *d_chi2, cudaStream_t st) {
  (void)m;
  if (c->tuned_cfg >= 0 && c->tuned_cfg < N_SRC_CFG)
    return launch_src(ctx, c, d_params, P, variant, d_chi2, st, SRC_CFG[c->tuned_cfg][0], SRC_CFG[c->tuned_cfg][1]);
  return launch_src_default(ctx, c, d_params, P, variant, d_chi2, st);
}

// Static sums of the no-cache form, grid (nimg, sets): every static potential
// at the image in double-float (FP64 where that fails), per-thread sums in
// double-float, deterministic CTA reduction in FP64; copy c goes to
// stat + c * nimg * 5.
__global__ void __launch_bounds__(CACHE_THREADS) k_static_df(const float2 *__restrict__ recdf,
                                                             const double *__restrict__ all64, int n, int v0, int v1,
                                                             const double *__restrict__ x,
                                                             const double *__restrict__ y, double *stat) {
  __shared__ double s_red[(CACHE_THREADS / 32) * 5];
  const int img = blockIdx.x;
  stat += (size_t)blockIdx.y * gridDim.x * 5;
  const double X = x[img], Y = y[img];
  const df Xd = df_kept(X), Yd = df_kept(Y);
  double v[5] = {0, 0, 0, 0, 0};
  // per-thread sums in double-float, converted once (FP64 only for the
  // potentials whose double-float evaluation fails)
  df sum[5] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  for (int h = threadIdx.x; h < n; h += CACHE_THREADS) {
    if (h == v0 || h == v1) continue;
    const float2 *r = recdf + h;
    df ax, ay, hh[3];
    bool ok = true;
    if (r[F_U2 * n].x < 0.f)
      circ_df<true>(r, n, Xd, Yd, ax, ay, hh);
    else
      ok = dpie_df<true, true>(r, n, Xd, Yd, ax, ay, hh);
    if (ok) {
      sum[0] = df_add(sum[0], ax);
      sum[1] = df_add(sum[1], ay);
      sum[2] = df_add(sum[2], hh[0]);
      sum[3] = df_add(sum[3], hh[1]);
      sum[4] = df_add(sum[4], hh[2]);
    } else {
      double e[5] = {0, 0, 0, 0, 0};
      eval64<true>(all64 + (size_t)h * REC64, X, Y, e[0], e[1], e[2], e[3], e[4]);
#pragma unroll
      for (int k = 0; k < 5; ++k) v[k] += e[k];
    }
  }
#pragma unroll
  for (int k = 0; k < 5; ++k) v[k] += df_to_double(sum[k]);
  block_sum<5, CACHE_THREADS>(v, s_red);
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; ++k) stat[(size_t)img * 5 + k] = v[k];
}

size_t chi2_nocache_scratch_bytes(const CSet *c) { return (size_t)NOCACHE_BATCH * c->nimg * 5 * sizeof(double); }

int launch_chi2_source_nocache(lens_ctx *ctx, const Model *m, const CSet *c, const double *d_params, int32_t P,
                               int32_t variant, double *d_chi2, cudaStream_t st) {
  CallScratch scratch(ctx, st);  // the static sums of a batch, on this call's stream
  int rc0 = scratch.alloc(chi2_nocache_scratch_bytes(c));
  if (rc0) return rc0;
  double *stat = (double *)scratch.p;
  for (int32_t p0 = 0; p0 < P; p0 += NOCACHE_BATCH) {
    const int B = std::min(NOCACHE_BATCH, P - p0);
    k_static_df<<<dim3(c->nimg, B), CACHE_THREADS, 0, st>>>(m->recdf, m->all64, m->n, c->var[0], c->var[1], c->x,
                                                             c->y, stat);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(LENS_ECUDA, "static sums launch: %s", cudaGetErrorString(e));
    const int rc = launch_src_default(ctx, c, d_params + (size_t)p0 * 14, B, variant, d_chi2 + p0, st, stat,
                                       (long long)c->nimg * 5);
    if (rc) return rc;
  }
  return LENS_OK;
}

// Static sums with the members' scaling relations applied, grid (nimg, sets):
// every static potential's b0 times f_b = params[14] and every static dPIE's
// r_cut times f_t = params[15] (b0_i = b0* s_i, r_cut,i = r_cut* s_i: varying
// b0* and r_cut*).  The sum is linear in b0, so f_b scales the result; the
// r_cut-dependent fields of each double-float record are rebuilt from
// st' = f_t st in double-float (q^2 st', q^2 st'^2, (1+q^2) st'^2, u^2 st'^2,
// st' + sc, q^2 (st' +- sc), q^2 (st'^2 - sc^2)).  FP64 (a record rescaled the
// same way) where the double-float evaluation fails.  Outside the domain
// (f_b <= 0, f_t r_cut,i <= r_core,i) the set's sums are NaN.
// A CTA takes two images side by side (grid (pairs, sets)): a potential's
// record is rescaled once for both.  Bound: instruction fetch and the FMA pipe
// (60 % busy); 512 sets x 372 images x 998 potentials 15.3 -> 11.0 ms (compiled
// for 4 or 5 CTAs per SM instead of 3: 11.2, 11.5).
__global__ void __launch_bounds__(CACHE_THREADS) k_static_scaled(const float2 *__restrict__ recdf,
                                                                 const double *__restrict__ all64, int n, int v0,
                                                                 int v1, const double *__restrict__ x,
                                                                 const double *__restrict__ y, int nimg,
                                                                 const double *__restrict__ params, double *stat) {
  __shared__ double s_red[(CACHE_THREADS / 32) * 16];
  const int img[2] = {(int)blockIdx.x, min((int)(blockIdx.x + gridDim.x), nimg - 1)};
  stat += (size_t)blockIdx.y * nimg * 5;
  const double fb = params[(size_t)blockIdx.y * 16 + 14], ft = params[(size_t)blockIdx.y * 16 + 15];
  Df<float2> X, Y, sum[5];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const df xd = df_kept(x[img[k]]), yd = df_kept(y[img[k]]);
    part2(X.hi, k) = xd.hi;
    part2(X.lo, k) = xd.lo;
    part2(Y.hi, k) = yd.hi;
    part2(Y.lo, k) = yd.lo;
  }
#pragma unroll
  for (int q = 0; q < 5; ++q) sum[q] = d_dup<float2>(0.f, 0.f);
  const df fd = df_kept(ft), f2 = df_mul(fd, fd);
  double v[16] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  bool bad = !(fb > 0.0 && ft > 0.0 && isfinite(fb) && isfinite(ft));
  for (int h = threadIdx.x; h < n && !bad; h += CACHE_THREADS) {
    if (h == v0 || h == v1) continue;
    float2 r[RECDF];
#pragma unroll
    for (int k = 0; k < RECDF; ++k) r[k] = recdf[h + (size_t)k * n];
    if (!(r[F_U2].x < 0.f)) {
      auto D = [&](int k) { return df{r[k].x, r[k].y}; };
      auto put = [&](int k, df d) { r[k] = make_float2(d.hi, d.lo); };
      const df st = df_mul(D(F_ST), fd), sc = D(F_SC), q2st = df_mul(D(F_Q2ST), fd);
      const df ss = df_add_ss(st, sc), q2ds = df_sub(q2st, D(F_Q2SC));
      if (!(st.hi > sc.hi)) bad = true;  // r_cut' <= r_core
      put(F_ST, st);
      put(F_Q2ST, q2st);
      put(F_SS, ss);
      put(F_Q2SS, df_add_ss(q2st, D(F_Q2SC)));
      put(F_Q2DS, q2ds);
      put(F_KT, df_mul(D(F_KT), f2));
      put(F_DT0, df_mul(D(F_DT0), f2));
      put(F_U2ST2, df_mul(D(F_U2ST2), f2));
      put(F_KTC, df_mul(q2ds, ss));
      record_consts<false>(r);
    }
    Df<float2> t[5];
    const unsigned ok = any_fixed<true, false>(r, X, Y, t[0], t[1], t + 2);
    if (ok != f_all<float2>) {
      const Df<float2> zero = d_dup<float2>(0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 5; ++q) t[q] = d_sel(ok, t[q], zero);
      double g[REC64];
      for (int k = 0; k < REC64; ++k) g[k] = all64[(size_t)h * REC64 + k];
      g[D_ST] *= ft;
      g[D_DS] = g[D_ST] - g[D_SC];
      g[D_SS] = g[D_ST] + g[D_SC];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (!(ok >> k & 1u)) {
          double e[5] = {0, 0, 0, 0, 0};
          eval64_cold<true>(g, x[img[k]], y[img[k]], e);
#pragma unroll
          for (int q = 0; q < 5; ++q) v[5 * k + q] += e[q];
        }
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) sum[q] = d_add(sum[q], t[q]);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int q = 0; q < 5; ++q)
      v[5 * k + q] = fb * (v[5 * k + q] + d_to_double(part2(sum[q].hi, k), part2(sum[q].lo, k)));
  const int any_bad = __syncthreads_or(bad);
  // the CTA's sums: a warp's lanes halve the values they carry at every step
  // of the butterfly (16 additions a lane instead of 50; block_sum's tree, so
  // its bits), lane 2 m then holds value m
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16, w = 8; o >= 2; o >>= 1, w >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (k < w) {
        const double mine = up ? v[k + w] : v[k], other = up ? v[k] : v[k + w];
        v[k] = mine + __shfl_xor_sync(0xffffffffu, other, o);
      }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
  // the value this lane holds: bit 3 from lane bit 4, ... bit 0 from lane bit 1
  const int m = lane >> 1;
  if ((lane & 1) == 0) s_red[warp * 16 + m] = v[0];
  __syncthreads();
  if (threadIdx.x < 10 && (threadIdx.x < 5 || blockIdx.x + gridDim.x < nimg)) {
    double t = 0.0;
    for (int w = 0; w < CACHE_THREADS / 32; ++w) t += s_red[w * 16 + threadIdx.x];
    stat[(size_t)img[threadIdx.x / 5] * 5 + threadIdx.x % 5] = any_bad ? __longlong_as_double(0x7ff8000000000000ll) : t;
  }
}

// Static sums of each set from the scaling cache, grid (sets of the batch):
// the barycentric Chebyshev interpolant in f_t of the cached sums (second
// kind points xs with weights (-1)^k, halved at both ends: Berrut and
// Trefethen, "Barycentric Lagrange interpolation", SIAM Review 2004), times
// f_b; NaN for f_t outside the cached interval or f_b not positive.
constexpr int MAX_SCALE_NODES = 128;
__global__ void __launch_bounds__(CACHE_THREADS) k_scaled_interp(const double *__restrict__ cache,
                                                                 const double *__restrict__ xs, int nodes,
                                                                 double ft_min, double ft_max, int nimg,
                                                                 const double *__restrict__ params, double *stat) {
  __shared__ double s_w[MAX_SCALE_NODES];
  __shared__ int s_hit;
  const double fb = params[(size_t)blockIdx.x * 16 + 14], ft = params[(size_t)blockIdx.x * 16 + 15];
  stat += (size_t)blockIdx.x * nimg * 5;
  const bool ok = fb > 0.0 && isfinite(fb) && ft >= ft_min && ft <= ft_max;
  if (threadIdx.x == 0) s_hit = -1;
  __syncthreads();
  for (int k = threadIdx.x; k < nodes; k += CACHE_THREADS) {
    const double xk = xs[k];
    const double wk = ((k & 1) ? -1.0 : 1.0) * ((k == 0 || k == nodes - 1) ? 0.5 : 1.0);
    if (ft == xk) s_hit = k;
    s_w[k] = wk / (ft - xk);
  }
  __syncthreads();
  const int hit = s_hit;
  double den = 0.0;
  if (hit < 0)
    for (int k = 0; k < nodes; ++k) den += s_w[k];
  const double iden = hit < 0 ? 1.0 / den : 0.0;
  for (int j = threadIdx.x; j < nimg; j += CACHE_THREADS) {
    double v[5];
    if (hit >= 0) {
#pragma unroll
      for (int q = 0; q < 5; ++q) v[q] = cache[((size_t)hit * nimg + j) * 5 + q];
    } else {
      double num[5] = {0, 0, 0, 0, 0};
      for (int k = 0; k < nodes; ++k) {
        const double w = s_w[k];
#pragma unroll
        for (int q = 0; q < 5; ++q) num[q] = fma(w, cache[((size_t)k * nimg + j) * 5 + q], num[q]);
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) v[q] = num[q] * iden;
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) stat[(size_t)j * 5 + q] = ok ? fb * v[q] : __longlong_as_double(0x7ff8000000000000ll);
  }
}

// Synchronous on the context's upload stream.
int build_scaling_cache(lens_ctx *ctx, const Model *m, CSet *c, const double *d_nodes16, int32_t nodes) {
  cudaStream_t st = upload_stream(ctx);
  if (!st) return fail(LENS_ECUDA, "upload stream creation failed");
  k_static_scaled<<<dim3((c->nimg + 1) / 2, nodes), CACHE_THREADS, 0, st>>>(m->recdf, m->all64, m->n, c->var[0], c->var[1],
                                                                  c->x, c->y, c->nimg, d_nodes16, c->scale_cache);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail(LENS_ECUDA, "scaling cache: %s", cudaGetErrorString(e));
  return LENS_OK;
}

int launch_chi2_source_scaled(lens_ctx *ctx, const Model *m, const CSet *c, const double *d_params, int32_t P,
                              int32_t variant, double *d_chi2, cudaStream_t st) {
  CallScratch scratch(ctx, st);  // the static sums of a batch, on this call's stream
  int rc0 = scratch.alloc(chi2_nocache_scratch_bytes(c));
  if (rc0) return rc0;
  double *stat = (double *)scratch.p;
  for (int32_t p0 = 0; p0 < P; p0 += NOCACHE_BATCH) {
    const int B = std::min(NOCACHE_BATCH, P - p0);
    if (c->scale_cache)
      k_scaled_interp<<<B, CACHE_THREADS, 0, st>>>(c->scale_cache, c->scale_x, c->scale_nodes, c->ft_min,
                                                    c->ft_max, c->nimg, d_params + (size_t)p0 * 16, stat);
    else
      k_static_scaled<<<dim3((c->nimg + 1) / 2, B), CACHE_THREADS, 0, st>>>(m->recdf, m->all64, m->n, c->var[0], c->var[1],
                                                                   c->x, c->y, c->nimg, d_params + (size_t)p0 * 16, stat);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(LENS_ECUDA, "scaled static sums launch: %s", cudaGetErrorString(e));
    const int rc = launch_src_default(ctx, c, d_params + (size_t)p0 * 16, B, variant, d_chi2 + p0, st, stat,
                                       (long long)c->nimg * 5, 16);
    if (rc) return rc;
  }
  return LENS_OK;
}

// Time the untuned rule (k = -1) and every launch shape on this constraint set
// and P (each once to warm up, then best of 3) and keep the fastest shape, or
// the rule where no shape beats it by 2 % (it has shapes of its own: pinned to
// image pairs, 4096 sets x 42 images took 98 instead of 77 us).  Synchronous
// on st.
int autotune_chi2_source(lens_ctx *ctx, CSet *c, const double *d_params, int32_t P, double *d_chi2, cudaStream_t st,
                         int32_t *chosen, float *best_ms) {
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return fail(LENS_ECUDA, "event creation failed");
  int best = 0;  // fastest of the listed shapes
  float best_t = 1e30f, rule_t = 1e30f;
  int rc = LENS_OK;
  for (int k = -1; k < N_SRC_CFG && rc == LENS_OK; ++k) {
    auto launch = [&]() {
      return k < 0 ? launch_src_default(ctx, c, d_params, P, 0, d_chi2, st)
                   : launch_src(ctx, c, d_params, P, 0, d_chi2, st, SRC_CFG[k][0], SRC_CFG[k][1]);
    };
    rc = launch();
    for (int r = 0; r < 3 && rc == LENS_OK; ++r) {
      cudaEventRecord(e0, st);
      rc = launch();
      cudaEventRecord(e1, st);
      if (cudaEventSynchronize(e1) != cudaSuccess) rc = fail(LENS_ECUDA, "autotune timing failed");
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (rc == LENS_OK && k < 0) rule_t = std::min(rule_t, ms);
      if (rc == LENS_OK && k >= 0 && ms < best_t) {
        best_t = ms;
        best = k;
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  const bool rule = !(best_t < 0.98f * rule_t);
  c->tuned_cfg = rule ? -1 : best;
  if (chosen) *chosen = SRC_CFG[best][0] * 100 + SRC_CFG[best][1];
  if (best_ms) *best_ms = rule ? rule_t : best_t;
  return LENS_OK;
}

}  // namespace lens
