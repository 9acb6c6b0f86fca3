// LENS_MIXED maps with the far potentials interpolated (Sec. 4.1, Eq. 10;
// Sec. 2.4, Eqs. 7-9).
//
// What bounds a map when every node evaluates every potential is the FP32
// pipe (k_map_mixed in lens_maps.cu: 65 operations per pair, 4.2e9 pairs for
// 2048^2 nodes x 1000 potentials), but most potentials are far from any one
// tile of the map and smooth over it.  A potential's deflection, Hessian and
// lensing potential are analytic in the node's position out to the complex
// displacement at which psi^2 = q^2 (s^2 + x^2) + y^2 vanishes, whose length
// is at least the real psi there (|t|^2 = psi^2 / (q^2 cos^2 + sin^2) along
// any direction), so on a tile of half-diagonal R polynomial interpolation
// at P x P Chebyshev nodes converges like rho^-P with rho growing with
// psi / R (Trefethen, "Approximation Theory and Approximation Practice",
// ch. 8).  Measured over random dPIE terms at the worst place psi = K R of
// the tile's centre: P = 10, K = 3 gives 1.2e-8 of the term's own deflection,
// P = 12, K = 2.5 gives 4e-9 -- below the 1e-7 an FP32 term carries -- and
// the error falls as psi^-P beyond.
//
// Two levels.  k_far_coarse: per coarse tile (ct x ct nodes, ct = 64..512),
// the potentials with psi >= KC R are summed at 12 x 12 nodes; the others'
// bits are set in the tile's mask.  k_far_map: per 32 x 32 or 64 x 64 tile, the
// potentials left by the coarse tile (all of them without a coarse level)
// with psi >= KF R are summed at 10 x 10 nodes, the coarse tile's
// interpolant is added there, and every map node then takes the near
// potentials one by one plus the interpolant.  Cluster-scale potentials go
// through the same levels in double-float, with wider margins.
//
// Precision.  A potential's terms at the nodes are the FP32 terms the direct
// kernel would sum, with the same compensated accumulation; the node sums
// are kept in double-float, a plane (slopes of 8 significant bits, so that
// its products with node offsets are exact) is taken out of them, and only
// the remainder is interpolated in FP32.  The map node's value is the plane
// plus the remainder plus the near sum in double-float, scaled by D_ls/D_s
// and rounded once.  The magnitude sum that decides the double-float repair
// is interpolated as well (a few percent off where a far term changes sign).
// It stands for the FP32 terms' rounding, not for that of the remainders,
// which the cluster-scale potentials' deflections feed as well: where those
// cancel, that rounding shows (2e-7 to 7e-7 arcsec between two b0 = 30"
// clusters, 7 times the 1e-6 |alpha| bound).  Per tile it is at most 14.4
// 2^-24 = 8.6e-7 of the largest remainder of the coarse plus that of the fine
// interpolation (restated on the CPU: 1 to 3 random cluster-scale terms beyond
// the margins, 16000 tiles of every size, every map node; rms 3 2^-24).  It is
// independent of the FP32 terms' rounding, so a node is listed where |alpha| is
// below the root of (ratio x magnitude sum)^2 + (those two remainders)^2 -- also
// in a model without FP32 potentials and with the FP32 terms' repair off.  (The
// plain sum lists a sixth more nodes of 8192^2 x 2000: 8.8 instead of 7.8 ms.)
// A potential map is stored in double and its cluster-scale terms are FP64, so
// its remainders (tens of arcsec^2) are interpolated as pairs, weights and all
// (in FP32 they left 1.5e-5 arcsec^2 where the members leave none; now 3e-9.
// 1537 x 1021 x 500 potentials 263 -> 269 us).
#include <algorithm>
#include <cmath>

#include "lens_device.cuh"

namespace lens {
namespace {

constexpr int FP = FAR_P;  // interpolation nodes per axis of a fine tile
constexpr int CP = 12;   // a coarse tile's
// Coarse kernel: its few CTAs (256 for 2048^2 x 1000) are one wave bound by the
// latency of each thread's chain of potentials, so 5 threads share a node pair's
// potentials (256 threads are 3, of which 40 threads idle; 448 are 6 and spill).
// Whole map with 256 / 288 / 384 / 448 threads: Hessian 2048^2 x 1000 719 / 714 /
// 710 / 721 us, deflection 5000^2 x 217 439 / 435 / 425 / 425, potential 1537 x
// 1021 x 500 258 / 254 / 247 / 247.
constexpr int CO_THREADS = 384;
constexpr int FF_CH = 64;            // potentials per staged chunk
// the coarse kernel's: with 64 / 128 / 256 the Hessian map above took 714 / 702 /
// 712 us on another GPU (fewer waits for records against shared memory for L1)
constexpr int CO_CH = 128;
constexpr int REC_STRIDE4 = REC32 / 4 + 1;  // float4 slots per staged record (the pad spreads the records a warp reads)
constexpr int FF_SUB = 16;           // partial sums folded every FF_SUB potentials
constexpr double DET_TERM_ERR = 2e-7, DET_REPAIR_ABS = 1e-5;  // as in lens_maps.cu
constexpr int CT_MAX = 512;

enum FarMode : int { FAR_GRAD = 0, FAR_HESS = 1, FAR_POT = 2 };
// interpolated values: deflection (2), kappa, gamma1, gamma2 (HESS) or the
// potential alone, then the magnitude sum (not POT)
__host__ __device__ constexpr int nval(int mode) { return mode == FAR_HESS ? 5 : mode == FAR_GRAD ? 2 : 1; }
__host__ __device__ constexpr int ncmp(int mode) { return nval(mode) + (mode == FAR_POT ? 0 : 1); }
__host__ __device__ constexpr int ncmp2(int mode) { return (ncmp(mode) + 1) / 2; }
// floats per remainder: a pair for the potential (hi values, then lo)
__host__ __device__ constexpr int nrem(int mode) { return mode == FAR_POT ? 2 : 1; }

// CTAs per SM of the fine kernel with 128, 256 or 512 threads (launch_far_map)
__host__ __device__ constexpr int fi_blocks(int mode, int th) { return th == 512 ? 1 : th == 256 ? 2 : mode == FAR_GRAD ? 5 : 4; }

// Chebyshev nodes of a fine tile of FT x FT map nodes (FT = 32 or 64), in
// units of 1/64 grid step about its centre, and of the coarse tile in units
// of its half-width / 512.
template <int FT>
struct XiTab {
  static constexpr int v[FP] = {980, 884, 701, 450, 155, -155, -450, -701, -884, -980};
};
template <>
struct XiTab<64> {
  static constexpr int v[FP] = {1991, 1796, 1426, 915, 315, -315, -915, -1426, -1796, -1991};
};
constexpr int ZC512[CP] = {508, 473, 406, 312, 196, 67, -67, -196, -312, -406, -473, -508};
__device__ const float D_ZC[CP] = {508 / 512.f, 473 / 512.f, 406 / 512.f, 312 / 512.f, 196 / 512.f, 67 / 512.f,
                                   -67 / 512.f, -196 / 512.f, -312 / 512.f, -406 / 512.f, -473 / 512.f, -508 / 512.f};

// A fine tile's nodes in steps and the Lagrange weights at its map nodes,
// formed in FP64 at compile time.
template <int FT>
struct FineTab {
  float w[FT][FP];    // at map node m - (FT - 1) / 2 steps
  float wlo[FT][FP];  // w + wlo: in double-float (repair)
  float xi[FP];
};
template <int FT>
constexpr FineTab<FT> fine_tab() {
  FineTab<FT> t{};
  for (int i = 0; i < FP; ++i) t.xi[i] = (float)(XiTab<FT>::v[i] / 64.0);
  for (int m = 0; m < FT; ++m)
    for (int i = 0; i < FP; ++i) {
      double v = 1.0;
      for (int k = 0; k < FP; ++k)
        if (k != i) v *= ((m - 0.5 * (FT - 1)) * 64.0 - XiTab<FT>::v[k]) / (double)(XiTab<FT>::v[i] - XiTab<FT>::v[k]);
      t.w[m][i] = (float)v;
      t.wlo[m][i] = (float)(v - (double)t.w[m][i]);
    }
  return t;
}
__device__ const FineTab<32> D_FINE32 = fine_tab<32>();
__device__ const FineTab<64> D_FINE64 = fine_tab<64>();
// the coarse basis at the fine tile's nodes: fine tile c of SUBT along an
// axis, node i, coarse node k
template <int SUBT>
struct CoarseTab {
  float w[SUBT][FP][CP], wlo[SUBT][FP][CP];  // (wlo: the potential's)
};
template <int FT, int SUBT>
constexpr CoarseTab<SUBT> coarse_tab() {
  CoarseTab<SUBT> t{};
  const double half = 0.5 * FT * SUBT;  // half-width in steps
  for (int c = 0; c < SUBT; ++c)
    for (int i = 0; i < FP; ++i)
      for (int k = 0; k < CP; ++k) {
        const double x = (FT * (c + 0.5) - half + XiTab<FT>::v[i] / 64.0) / half * 512.0;
        double v = 1.0;
        for (int l = 0; l < CP; ++l)
          if (l != k) v *= (x - ZC512[l]) / (double)(ZC512[k] - ZC512[l]);
        t.w[c][i][k] = (float)v;
        t.wlo[c][i][k] = (float)(v - (double)t.w[c][i][k]);
      }
  return t;
}
__device__ const CoarseTab<2> D_CO32_2 = coarse_tab<32, 2>(), D_CO64_2 = coarse_tab<64, 2>();
__device__ const CoarseTab<4> D_CO32_4 = coarse_tab<32, 4>(), D_CO64_4 = coarse_tab<64, 4>();
__device__ const CoarseTab<8> D_CO32_8 = coarse_tab<32, 8>(), D_CO64_8 = coarse_tab<64, 8>();
__device__ const CoarseTab<16> D_CO32_16 = coarse_tab<32, 16>();
template <int FT>
__device__ __forceinline__ const FineTab<FT> &fine_table();
template <>
__device__ __forceinline__ const FineTab<32> &fine_table<32>() { return D_FINE32; }
template <>
__device__ __forceinline__ const FineTab<64> &fine_table<64>() { return D_FINE64; }
// CoarseTab::w of the table with `sub` fine tiles per axis (wlo follows it)
template <int FT>
__device__ __forceinline__ const float *coarse_weights(int sub) {
  if (FT == 32)
    return sub == 2 ? &D_CO32_2.w[0][0][0] : sub == 4 ? &D_CO32_4.w[0][0][0] : sub == 8 ? &D_CO32_8.w[0][0][0]
                                                                                       : &D_CO32_16.w[0][0][0];
  return sub == 2 ? &D_CO64_2.w[0][0][0] : sub == 4 ? &D_CO64_4.w[0][0][0] : &D_CO64_8.w[0][0][0];
}

struct FarArgs {
  const float *rec32;
  const float4 *cen32;
  int n_light;
  const double *heavy;
  const float2 *heavydf;
  int n_heavy;
  int nwl, nw;       // mask words of the FP32 potentials / of all (the cluster-scale ones start at word nwl)
  double xmin, ymin, dx, dy;
  int nx, ny;        // ny: rows of this launch
  int row0;
  double dls;
  float dls_h, dls_l;  // as a float pair
  float thr_c, thr_ch, thr_f, thr_fh;  // squared psi beyond which a potential is far: coarse / fine, FP32 / cluster-scale
  // coarse level: tile (0, 0) covers the grid's first nodes
  int ct, nct;       // nodes a side (0: no coarse level), tiles per row
  float *cval;       // per coarse tile: remainders [nrem][ncmp][CP * CP], planes [nval][4], s_kb [KB]
  unsigned *cmask;   // per coarse tile: nw words, bit set = left to the fine level
  float *out;
  double *out64;
  long long plane;
  int tau;
  double bx, by;
  float repair_f;    // 2 * ratio, 0: only the remainders' part of the repair
  int *rep_count, *rep_list;  // NULL: no repair
  DenseRepair dense;
  int dense_min;     // listed nodes from which a tile is dense
};

constexpr int KB = 6;  // a tile's s_kb (repair_bound)
__host__ __device__ constexpr int coarse_floats(int mode) { return nrem(mode) * ncmp(mode) * CP * CP + nval(mode) * 4 + KB; }

// Is the potential far from a tile centred at (dx, dy) from it?
__device__ __forceinline__ bool far32(const float4 *r4, float dX, float dY, float thr) {
  const float4 A = r4[0];
  const int kind = __float_as_int(r4[7].x);
  if (kind == K32_SIS || kind == K32_POINT) return fmaf(dX, dX, dY * dY) >= thr;
  const float x = fmaf(A.x, dX, A.y * dY), y = fmaf(A.x, dY, -A.y * dX);
  return fmaf(A.z, x * x, fmaf(y, y, r4[1].x)) >= thr;
}
__device__ __forceinline__ bool far_df(const float2 *r, float dX, float dY, float thr) {
  if (r[F_U2].x < 0.f) return fmaf(dX, dX, dY * dY) >= thr;
  const float c = r[F_C].x, s = r[F_S].x, x = fmaf(c, dX, s * dY), y = fmaf(c, dY, -s * dX);
  return fmaf(r[F_Q2].x, x * x, fmaf(y, y, r[F_KC].x)) >= thr;
}

// One cluster-scale potential in double-float at (X, Y), added to sum
// (out of line: it is large and taken rarely).
template <int MODE>
__device__ __noinline__ void add_heavy(const float2 *rdf, const double *r64, df X, df Y, df *sum) {
  const double Xd = df_to_double(X), Yd = df_to_double(Y);
  if constexpr (MODE == FAR_POT)
    sum[0] = df_add(sum[0], df_from_double(pot64(r64, Xd, Yd)));
  else
    add_potential_dfs<MODE == FAR_HESS>(rdf, 1, r64, Xd, Yd, X, Y, sum);
}

// The FP32 potentials h0, h0 + step, ... < cnt of a staged chunk at one
// point pair of the tile: offsets (ox) shared, (oy) per point, from the
// tile's centre as hi/lo pairs.
template <int MODE>
struct Sums {
  Acc2<MODE == FAR_HESS, 1> tot, cmp, part;
  int seen;
  __device__ __forceinline__ void zero() {
    tot.zero();
    cmp.zero();
    part.zero();
    seen = 0;
  }
  __device__ __forceinline__ void fold() {
    if constexpr (MODE == FAR_POT)
      fold2_pot(tot, cmp, part);
    else
      fold2(tot, cmp, part);
    seen = 0;
  }
  __device__ __forceinline__ void sweep(const float4 *s_rec, const float4 *s_off, int h0, int cnt, int step, float2 ox,
                                        float2 oyh, float2 oyl) {
    constexpr bool HESS = MODE == FAR_HESS, POT = MODE == FAR_POT;
    for (int h = h0; h < cnt; h += step) {
      const float4 *r4 = s_rec + h * REC_STRIDE4;
      const float4 o = s_off[h];
      const float dX = (o.x + ox.x) + (o.y + ox.y);
      const float2 dY[1] = {add2(add2(dup2(o.z), oyh), add2(dup2(o.w), oyl))};
      const int kind = __float_as_int(r4[7].x);
      if (kind == K32_DPIE)
        dpie32x2<HESS, 1, false, !POT, false, POT>(r4, dX, dY, part);
      else if (kind == K32_DPIE_SERIES)
        dpie32x2<HESS, 1, true, !POT, false, POT>(r4, dX, dY, part);
      else if (kind == K32_SIS)
        circ32x2<HESS, 1, false, !POT, POT>(r4, dX, dY, part);
      else
        circ32x2<HESS, 1, true, !POT, POT>(r4, dX, dY, part);
      if (++seen == FF_SUB) fold();
    }
  }
  // value c of point h as a double-float number
  __device__ __forceinline__ df value(int c, int h) const {
    const float2 *t, *m;
    if constexpr (MODE == FAR_POT) {
      t = tot.k;
      m = cmp.k;
    } else {
      t = c == 0 ? tot.ax : c == 1 ? tot.ay : c == 2 ? tot.k : c == 3 ? tot.g1 : tot.g2;
      m = c == 0 ? cmp.ax : c == 1 ? cmp.ay : c == 2 ? cmp.k : c == 3 ? cmp.g1 : cmp.g2;
    }
    return df{part2(t[0], h), -part2(m[0], h)};
  }
  __device__ __forceinline__ float mag(int h) const { return part2(tot.mag[0], h); }
};

// Potential idx of the list (FP32) into staging slot h: its record, and the
// tile centre's offset from its centre as hi/lo pairs.
template <int TH>
__device__ __forceinline__ void stage_chunk(const FarArgs &a, const unsigned short *list, int cnt, df Tx, df Ty,
                                            float4 *s_rec, float4 *s_off) {
  const float4 *g_rec = reinterpret_cast<const float4 *>(a.rec32);
  for (int q = threadIdx.x; q < cnt * (REC32 / 4); q += TH)
    s_rec[(q >> 3) * REC_STRIDE4 + (q & 7)] = __ldg(g_rec + (size_t)list[q >> 3] * (REC32 / 4) + (q & 7));
  if (threadIdx.x < cnt) {
    const float4 c = __ldg(a.cen32 + list[threadIdx.x]);
    const df ox = df_sub(Tx, df{c.x, c.z}), oy = df_sub(Ty, df{c.y, c.w});
    s_off[threadIdx.x] = make_float4(ox.hi, ox.lo, oy.hi, oy.lo);
  }
}

// Classify the potentials whose bit is set in `in` (NULL: all) as far from
// the tile or near, and list the far ones then the near ones, each in index
// order.  s_far / s_near: nw words each.  cnt: far FP32, far cluster-scale,
// near FP32, near cluster-scale.  Ends synchronised.
template <int TH>
__device__ __forceinline__ void classify(const FarArgs &a, const unsigned *in, df Tx, df Ty, float thr, float thr_h,
                                         unsigned *s_far, unsigned *s_near, unsigned short *s_list, int *s_cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float4 *g_rec = reinterpret_cast<const float4 *>(a.rec32);
  for (int w = warp; w < a.nw; w += (TH / 32)) {
    const bool hv = w >= a.nwl;
    const int i = (hv ? w - a.nwl : w) * 32 + lane;
    bool mine = i < (hv ? a.n_heavy : a.n_light);
    if (in) mine = mine && (in[w] >> lane & 1u);
    bool far = false;
    if (mine) {
      if (hv) {
        const float2 *r = a.heavydf + (size_t)i * RECDF;
        far = far_df(r, df_sub(Tx, df{r[F_X0].x, r[F_X0].y}).hi, df_sub(Ty, df{r[F_Y0].x, r[F_Y0].y}).hi, thr_h);
      } else {
        const float4 c = __ldg(a.cen32 + i);
        far = far32(g_rec + (size_t)i * (REC32 / 4), df_sub(Tx, df{c.x, c.z}).hi, df_sub(Ty, df{c.y, c.w}).hi, thr);
      }
    }
    const unsigned f = __ballot_sync(0xffffffffu, mine && far), n = __ballot_sync(0xffffffffu, mine && !far);
    if (lane == 0) {
      s_far[w] = f;
      s_near[w] = n;
    }
  }
  __syncthreads();
  // positions: warp 0 scans the words' populations, the far words first
  int *pos = reinterpret_cast<int *>(s_near + a.nw);  // [2 nw]
  if (warp == 0) {
    int base = 0;
    for (int w0 = 0; w0 < 2 * a.nw; w0 += 32) {
      const int w = w0 + lane;
      const int c = w < 2 * a.nw ? __popc(w < a.nw ? s_far[w] : s_near[w - a.nw]) : 0;
      int s = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += t;
      }
      if (w < 2 * a.nw) pos[w] = base + s - c;
      base += __shfl_sync(0xffffffffu, s, 31);
    }
    __syncwarp();
    if (lane == 0) {
      const int fl = a.nwl < a.nw ? pos[a.nwl] : pos[a.nw], fa = pos[a.nw];
      const int nl = a.nwl < a.nw ? pos[a.nw + a.nwl] : base;
      s_cnt[0] = fl;
      s_cnt[1] = fa - fl;
      s_cnt[2] = nl - fa;
      s_cnt[3] = base - nl;
    }
  }
  __syncthreads();
  for (int w = warp; w < 2 * a.nw; w += (TH / 32)) {
    const int wi = w < a.nw ? w : w - a.nw;
    const unsigned m = w < a.nw ? s_far[wi] : s_near[wi];
    const int i = (wi >= a.nwl ? wi - a.nwl : wi) * 32 + lane;
    if (m >> lane & 1u) s_list[pos[w] + __popc(m & ((1u << lane) - 1u))] = (unsigned short)i;
  }
  __syncthreads();
}

// det's error, 2 |1 - kappa| d kappa + 2 |gamma| d gamma, in units of 2
// DET_TERM_ERR: above DET_LIST a node's planes are all recomputed.  A
// remainder's rounding (below 5 DET_TERM_ERR of it) adds to the FP32 terms' as
// the root of both squares, like the deflection's.
constexpr float REM_TERM = 5.f, DET_LIST = (float)(DET_REPAIR_ABS / (2.0 * DET_TERM_ERR));

// Slope with 8 significant bits: its products with node offsets (up to 15
// bits) are exact in FP32.
__device__ __forceinline__ float slope8(float v) { return __int_as_float(__float_as_int(v) & 0xffff0000); }

// P x P node sums of the far potentials of one tile: s_val[c][node] in
// double-float (node = y index * P + x index).  Ends synchronised.
// kb: the FP32 potentials' largest |kappa|, |gamma1|, |gamma2| at the nodes
// (HESS), added to what is there.
template <int MODE, int P, int TH, int CH>
__device__ __forceinline__ void node_sums(const FarArgs &a, const unsigned short *list, int n_far, int n_far_h,
                                          df Tx, df Ty, const float2 *s_nx, const float2 *s_ny, float4 *s_rec,
                                          float4 *s_off, float2 *s_part, float2 *s_val, float *s_kb) {
  constexpr int NODES = P * P, PAIRS = NODES / 2, SPLITS = TH / PAIRS, NC = ncmp(MODE), NV = nval(MODE);
  const int tid = threadIdx.x, split = tid / PAIRS, pr = tid % PAIRS, ix = pr % P, jy = 2 * (pr / P);
  const bool active = split < SPLITS;
  Sums<MODE> S;
  S.zero();
  const float2 ox = s_nx[ix], y0 = s_ny[jy], y1 = s_ny[jy + 1];
  static_assert(CH <= TH, "stage_chunk: one offset per thread");
  for (int c0 = 0; c0 < n_far; c0 += CH) {
    const int cnt = min(CH, n_far - c0);
    if (c0) __syncthreads();  // the previous chunk has been used
    stage_chunk<TH>(a, list + c0, cnt, Tx, Ty, s_rec, s_off);
    __syncthreads();
    if (active)
      S.sweep(s_rec, s_off, split, cnt, SPLITS, ox, make_float2(y0.x, y1.x), make_float2(y0.y, y1.y));
  }
  S.fold();
  if (active) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float2 *o = s_part + ((size_t)split * NODES + (jy + h) * P + ix) * NC;
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        const df v = S.value(c, h);
        o[c] = make_float2(v.hi, v.lo);
      }
      if (MODE != FAR_POT) o[NV] = make_float2(S.mag(h), 0.f);
    }
  }
  __syncthreads();
  for (int q = tid; q < NODES * NC; q += TH) {
    df v = {s_part[q].x, s_part[q].y};
    for (int s = 1; s < SPLITS; ++s) {
      const float2 t = s_part[(size_t)s * NODES * NC + q];
      v = df_add(v, df{t.x, t.y});
    }
    const int node = q / NC, c = q % NC;
    s_val[c * NODES + node] = make_float2(v.hi, v.lo);
    if (MODE == FAR_HESS && c >= 2 && c < 5)
      atomicMax(reinterpret_cast<int *>(s_kb) + c - 2, __float_as_int(fabsf(v.hi)));
  }
  __syncthreads();
  if (n_far_h > 0) {
    for (int node = tid; node < NODES; node += TH) {
      const float2 nx = s_nx[node % P], ny = s_ny[node / P];
      const df X = df_add(Tx, df{nx.x, nx.y}), Y = df_add(Ty, df{ny.x, ny.y});
      df sum[5] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
      for (int k = 0; k < n_far_h; ++k) {
        const int h = list[n_far + k];
        add_heavy<MODE>(a.heavydf + (size_t)h * RECDF, a.heavy + (size_t)h * REC64, X, Y, sum);
      }
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        float2 &o = s_val[c * NODES + node];
        const df v = df_add(df{o.x, o.y}, sum[c]);
        o = make_float2(v.hi, v.lo);
      }
    }
    __syncthreads();
  }
}

// acc + (w + wlo) (f + flo), pairs
__device__ __forceinline__ df fma_pair(float w, float wlo, float f, float flo, df acc) {
  const float p = __fmul_rn(w, f);
  const float e = fmaf(wlo, f, fmaf(w, flo, fmaf(w, f, -p)));
  const df s = two_sum(acc.hi, p);
  return {s.hi, acc.lo + (s.lo + e)};
}

// Plane of value c: the middle node's value and slopes (per grid step)
// between the outermost nodes of the middle row and column.
template <int P>
__device__ __forceinline__ float4 plane_of(const float2 *v, float span) {
  const int m = P / 2;
  return make_float4(v[m * P + m].x, slope8((v[m * P].x - v[m * P + P - 1].x) / span),
                     slope8((v[m].x - v[(P - 1) * P + m].x) / span), 0.f);
}

// Entry `lane` of a tile's s_kb, for the repair (one warp): the far FP32
// potentials' largest |kappa|, |gamma1|, |gamma2| (kb), then the largest
// remainders of the deflection, of kappa and of gamma; the remainder of value c
// at a node is f[(c NODES + node) stride].
template <int MODE, int NODES>
__device__ __forceinline__ float repair_bound(const float *kb, const float *f, int stride, int lane) {
  float rm[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int c = 0; c < nval(MODE); ++c) {
    for (int node = lane; node < NODES; node += 32) rm[c] = fmaxf(rm[c], fabsf(f[(c * NODES + node) * stride]));
    rm[c] = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(rm[c])));
  }
  if (lane < 3) return kb[lane];
  return lane == 3 ? fmaxf(rm[0], rm[1]) : lane == 4 ? rm[2] : sqrtf(fmaf(rm[3], rm[3], rm[4] * rm[4]));
}

template <int MODE>
__global__ void __launch_bounds__(CO_THREADS, 2) k_far_coarse(const FarArgs a) {
  constexpr int NODES = CP * CP, NC = ncmp(MODE), NV = nval(MODE), NR = nrem(MODE) * NC, SPLITS = CO_THREADS / (NODES / 2);
  extern __shared__ __align__(16) unsigned char s_dyn[];
  float4 *s_rec = reinterpret_cast<float4 *>(s_dyn);
  float4 *s_off = s_rec + CO_CH * REC_STRIDE4;
  float2 *s_part = reinterpret_cast<float2 *>(s_off + CO_CH);
  float2 *s_val = s_part + SPLITS * NODES * NC;
  unsigned *s_far = reinterpret_cast<unsigned *>(s_val + NODES * NC);
  unsigned *s_near = s_far + a.nw;
  unsigned short *s_list = reinterpret_cast<unsigned short *>(s_near + 3 * a.nw);
  __shared__ float2 s_nx[CP], s_ny[CP];
  __shared__ float s_kb[KB];
  __shared__ float4 s_plane[NV];
  __shared__ int s_cnt[4];
  const int tid = threadIdx.x, tile = blockIdx.y * a.nct + blockIdx.x;
  const double half = 0.5 * a.ct;
  // centre of the tile: half a step past its middle node pair's first
  const df Tx = df_from_double(a.xmin + (blockIdx.x * (double)a.ct + half - 0.5) * a.dx);
  const df Ty = df_from_double(a.ymin + (blockIdx.y * (double)a.ct + half - 0.5) * a.dy);
  if (tid < CP) {
    // the coarse basis is laid out about the centre of the tile's fine
    // tiles, each 32 steps wide about its own centre: the same point
    const df ox = df_from_double(D_ZC[tid] * half * a.dx), oy = df_from_double(D_ZC[tid] * half * a.dy);
    s_nx[tid] = make_float2(ox.hi, ox.lo);
    s_ny[tid] = make_float2(oy.hi, oy.lo);
  }
  if (tid < KB) s_kb[tid] = 0.f;
  classify<CO_THREADS>(a, nullptr, Tx, Ty, a.thr_c, a.thr_ch, s_far, s_near, s_list, s_cnt);
  for (int w = tid; w < a.nw; w += CO_THREADS) a.cmask[(size_t)tile * a.nw + w] = s_near[w];
  node_sums<MODE, CP, CO_THREADS, CO_CH>(a, s_list, s_cnt[0], s_cnt[1], Tx, Ty, s_nx, s_ny, s_rec, s_off, s_part, s_val, s_kb);
  if (tid < NV) s_plane[tid] = plane_of<CP>(s_val + tid * NODES, (D_ZC[0] - D_ZC[CP - 1]) * (float)half);
  __syncthreads();
  float *o = a.cval + (size_t)tile * coarse_floats(MODE);
  for (int q = tid; q < NODES * NC; q += CO_THREADS) {
    const int c = q / NODES, node = q % NODES;
    const float2 v = s_val[q];
    float r = v.x;
    if (c < NV) {
      const float4 p = s_plane[c];
      const float zx = D_ZC[node % CP] * (float)half, zy = D_ZC[node / CP] * (float)half;
      df d = df_sub(df{v.x, v.y}, df{p.x, 0.f});
      d = df_sub(d, df{p.y * zx, 0.f});
      d = df_sub(d, df{p.z * zy, 0.f});
      r = d.hi + d.lo;
      s_val[q].x = r;
      if (MODE == FAR_POT) o[NC * NODES + q] = (d.hi - r) + d.lo;
    }
    o[q] = r;
  }
  if (tid < NV * 4) o[NR * NODES + tid] = reinterpret_cast<const float *>(s_plane)[tid];
  if (MODE == FAR_POT) return;
  __syncthreads();
  if (tid < 32) {
    const float b = repair_bound<MODE, NODES>(s_kb, reinterpret_cast<const float *>(s_val), 2, tid);
    if (tid < KB) o[NR * NODES + NV * 4 + tid] = b;
  }
}

// 1 / (hi + lo), one Newton step on the MUFU reciprocal
__device__ __forceinline__ float rcp_dff(float hi, float lo) {
  const float r = rcp_a(hi);
  const float e = fmaf(-lo, r, fmaf(-hi, r, 1.f));
  return fabsf(e) < 1e-3f ? fmaf(r, e, r) : 1.f / hi;
}

template <int MODE, int FT, int FI_THREADS>
__global__ void __launch_bounds__(FI_THREADS, fi_blocks(MODE, FI_THREADS)) k_far_map(const FarArgs a) {
  constexpr bool HESS = MODE == FAR_HESS, POT = MODE == FAR_POT;
  constexpr int NODES = FP * FP, NC = ncmp(MODE), NV = nval(MODE), NC2 = ncmp2(MODE), SPLITS = FI_THREADS / (NODES / 2);
  constexpr int NR = nrem(MODE) * NC, CV_PLANE = NR * CP * CP;  // floats of a coarse tile's values before its planes
  extern __shared__ __align__(16) unsigned char s_dyn[];
  float4 *s_rec = reinterpret_cast<float4 *>(s_dyn);                      // [FF_CH][REC_STRIDE4]
  float4 *s_off = s_rec + FF_CH * REC_STRIDE4;                            // [FF_CH]
  float4 *s_c = s_off + FF_CH;                                            // [FT / 2][FP][NC2]: row-pair coefficients
  float2 *s_part = reinterpret_cast<float2 *>(s_c + (FT / 2) * FP * NC2);  // [SPLITS][NODES][NC]
  float2 *s_val = s_part + SPLITS * NODES * NC;                           // [NC][NODES]
  unsigned *s_far = reinterpret_cast<unsigned *>(s_val + NODES * NC);
  unsigned *s_near = s_far + a.nw;
  unsigned short *s_list = reinterpret_cast<unsigned short *>(s_near + 3 * a.nw);
  float *s_tmp = reinterpret_cast<float *>(s_part);  // coarse level: [NR][CP * CP] values, [NR][FP][CP] (after node_sums)
  float *s_rem = s_tmp;                              // then the remainders [NR][NODES]
  __shared__ float2 s_nx[FP], s_ny[FP];
  __shared__ float2 s_cx[FT], s_ry[FT];  // offsets of the tile's columns and rows from its centre, hi/lo
  __shared__ float s_L[FT][FP + 1], s_xi[FP];  // (odd stride: lanes read a column each)
  __shared__ float s_Ll[POT ? FT : 1][FP + 1];
  __shared__ float4 s_T;                 // the centre, hi/lo
  __shared__ unsigned s_m[FT * FT / 32], s_mh[HESS ? FT * FT / 32 : 1];  // nodes to recompute: deflection alone / all planes
  __shared__ double s_tau[POT ? 2 : 1][POT ? FT : 1];  // half the squared offsets from beta
  __shared__ float s_kb[KB];  // for the repair: repair_bound (here and of the coarse tile), [3] squared
  __shared__ float4 s_plane[NV];
  __shared__ int s_cnt[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = blockIdx.x * FT, j0 = a.row0 + blockIdx.y * FT;  // grid column and row of the tile's first node
  // the few FP64 operations once per tile
  constexpr double HALF = 0.5 * (FT - 1);
  for (int q = tid; q < 2 + 2 * FP + 2 * FT; q += FI_THREADS) {
    if (q < 2) {
      const df t = df_from_double(q == 0 ? a.xmin + (i0 + HALF) * a.dx : a.ymin + (j0 + HALF) * a.dy);
      reinterpret_cast<float2 *>(&s_T)[q] = make_float2(t.hi, t.lo);
    } else if (q < 2 + 2 * FP) {
      const int k = (q - 2) % FP;
      const df o = df_from_double(fine_table<FT>().xi[k] * (q < 2 + FP ? a.dx : a.dy));
      (q < 2 + FP ? s_nx : s_ny)[k] = make_float2(o.hi, o.lo);
      s_xi[k] = fine_table<FT>().xi[k];
    } else {
      const int e = q - 2 - 2 * FP, k = e % FT;
      const df o = df_from_double((k - HALF) * (e < FT ? a.dx : a.dy));
      (e < FT ? s_cx : s_ry)[k] = make_float2(o.hi, o.lo);
      if (POT && a.tau) {
        const double d = e < FT ? a.xmin + (i0 + k) * a.dx - a.bx : a.ymin + (j0 + k) * a.dy - a.by;
        s_tau[POT && e >= FT][POT ? k : 0] = 0.5 * d * d;
      }
    }
  }
  if (tid < KB) s_kb[tid] = 0.f;
  for (int q = tid; q < FT * FP; q += FI_THREADS) {
    s_L[q / FP][q % FP] = (&fine_table<FT>().w[0][0])[q];
    if (POT) s_Ll[POT ? q / FP : 0][q % FP] = (&fine_table<FT>().wlo[0][0])[q];
  }
  __syncthreads();
  const df Tx = {s_T.x, s_T.y}, Ty = {s_T.z, s_T.w};
  const int ctile = a.ct ? (j0 / a.ct) * a.nct + i0 / a.ct : 0;
  classify<FI_THREADS>(a, a.ct ? a.cmask + (size_t)ctile * a.nw : nullptr, Tx, Ty, a.thr_f, a.thr_fh, s_far, s_near, s_list, s_cnt);
  const int n_far = s_cnt[0], n_far_h = s_cnt[1], n_near = s_cnt[2], n_near_h = s_cnt[3];
  node_sums<MODE, FP, FI_THREADS, FF_CH>(a, s_list, n_far, n_far_h, Tx, Ty, s_nx, s_ny, s_rec, s_off, s_part, s_val, s_kb);
  if (a.ct) {
    // the coarse tile's interpolant at this tile's nodes: rows of the tensor
    // product, then columns; its plane (exact products) in double-float
    const float *cv = a.cval + (size_t)ctile * coarse_floats(MODE);
    const int sub = a.ct / FT, cx = (i0 % a.ct) / FT, cy = (j0 % a.ct) / FT;
    const float *W = coarse_weights<FT>(sub);
    const float *Wx = W + cx * FP * CP, *Wy = W + cy * FP * CP;
    const int wlo = sub * FP * CP;  // from a weight to its low part
    float *s_t1 = s_tmp + NR * CP * CP;
    for (int q = tid; q < NR * CP * CP; q += FI_THREADS) s_tmp[q] = cv[q];
    __syncthreads();
    for (int q = tid; q < NC * CP * FP; q += FI_THREADS) {  // (c, coarse row, fine column)
      const int i = q % FP, cr = q / FP;
      const float *f = s_tmp + cr * CP;
      if constexpr (POT) {
        df v = {0.f, 0.f};
#pragma unroll
        for (int k = 0; k < CP; ++k) v = fma_pair(Wx[i * CP + k], Wx[wlo + i * CP + k], f[k], f[NC * CP * CP + k], v);
        v = fast_two_sum(v.hi, v.lo);
        s_t1[q] = v.hi;
        s_t1[NC * CP * FP + q] = v.lo;
      } else {
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < CP; ++k) v = fmaf(Wx[i * CP + k], f[k], v);
        s_t1[q] = v;
      }
    }
    __syncthreads();
    const float bx0 = FT * (cx + 0.5f) - 0.5f * a.ct, by0 = FT * (cy + 0.5f) - 0.5f * a.ct;
    for (int q = tid; q < NC * NODES; q += FI_THREADS) {
      const int c = q / NODES, node = q % NODES, i = node % FP, j = node / FP;
      df v = {0.f, 0.f};
#pragma unroll
      for (int k = 0; k < CP; ++k) {
        const float *f = s_t1 + (c * CP + k) * FP + i;
        if constexpr (POT)
          v = fma_pair(Wy[j * CP + k], Wy[wlo + j * CP + k], f[0], f[NC * CP * FP], v);
        else
          v.hi = fmaf(Wy[j * CP + k], f[0], v.hi);
      }
      df d = {s_val[q].x, s_val[q].y};
      d = df_add(d, v);
      if (c < NV) {
        const float *p = cv + CV_PLANE + c * 4;
        d = df_add(d, df{p[0], 0.f});
        d = df_add(d, df{p[1] * (bx0 + s_xi[i]), 0.f});
        d = df_add(d, df{p[2] * (by0 + s_xi[j]), 0.f});
      }
      s_val[q] = make_float2(d.hi, d.lo);
    }
    __syncthreads();
  }
  if (tid < NV) s_plane[tid] = plane_of<FP>(s_val + tid * NODES, s_xi[0] - s_xi[FP - 1]);
  __syncthreads();
  for (int q = tid; q < NC * NODES; q += FI_THREADS) {
    const int c = q / NODES, node = q % NODES;
    const float2 v = s_val[q];
    float r = v.x;
    if (c < NV) {
      const float4 p = s_plane[c];
      df d = df_sub(df{v.x, v.y}, df{p.x, 0.f});
      d = df_sub(d, df{p.y * s_xi[node % FP], 0.f});
      d = df_sub(d, df{p.z * s_xi[node / FP], 0.f});
      r = d.hi + d.lo;
      if (POT) s_rem[NC * NODES + q] = (d.hi - r) + d.lo;
    }
    s_rem[q] = r;
  }
  __syncthreads();
  if (!POT && warp == 0) {
    float b = repair_bound<MODE, NODES>(s_kb, s_rem, 1, lane);
    if (lane < KB) {
      if (a.ct) b += a.cval[(size_t)ctile * coarse_floats(MODE) + CV_PLANE + NV * 4 + lane];
      s_kb[lane] = lane == 3 ? b * b : b;
    }
  }
  // coefficients of every row pair: the remainders interpolated in y at the
  // tile's rows, one float4 = two values at two rows
  for (int q = tid; q < (FT / 2) * FP * NC2 * 2; q += FI_THREADS) {
    const int c = q % (2 * NC2), i = q / (2 * NC2) % FP, rp = q / (2 * NC2 * FP);
    float u = 0.f, v = 0.f;
    if constexpr (POT) {  // c = 1: the low parts
      df x = {0.f, 0.f}, y = {0.f, 0.f};
#pragma unroll
      for (int j = 0; j < FP; ++j) {
        const float f = s_rem[j * FP + i], g = s_rem[NODES + j * FP + i];
        x = fma_pair(s_L[2 * rp][j], s_Ll[POT ? 2 * rp : 0][j], f, g, x);
        y = fma_pair(s_L[2 * rp + 1][j], s_Ll[POT ? 2 * rp + 1 : 0][j], f, g, y);
      }
      x = fast_two_sum(x.hi, x.lo);
      y = fast_two_sum(y.hi, y.lo);
      u = c ? x.lo : x.hi;
      v = c ? y.lo : y.hi;
    } else if (c < NC) {
#pragma unroll
      for (int j = 0; j < FP; ++j) {
        const float f = s_rem[c * NODES + j * FP + i];
        u = fmaf(s_L[2 * rp][j], f, u);
        v = fmaf(s_L[2 * rp + 1][j], f, v);
      }
    }
    reinterpret_cast<float2 *>(s_c)[q] = make_float2(u, v);
  }
  // the near potentials and the interpolant at the map nodes: lane = column,
  // a warp takes row pairs warp, warp + (FI_THREADS / 32)
  bool staged = false;
#pragma unroll 1
  for (int task = warp; task < (FT / 2) * (FT / 32); task += (FI_THREADS / 32)) {
    const int rp = task % (FT / 2), m = task / (FT / 2) * 32 + lane, i = i0 + m;
    const float mx = m - (float)HALF;
    const float2 ox = s_cx[m], r0 = s_ry[2 * rp], r1 = s_ry[2 * rp + 1];
    const float2 oyh = make_float2(r0.x, r1.x), oyl = make_float2(r0.y, r1.y);
    Sums<MODE> S;
    S.zero();
    for (int c0 = 0; c0 < n_near || (c0 == 0 && !staged); c0 += FF_CH) {
      const int cnt = min(FF_CH, n_near - c0);
      if (n_near > FF_CH || !staged) {
        __syncthreads();
        stage_chunk<FI_THREADS>(a, s_list + n_far + n_far_h + c0, cnt, Tx, Ty, s_rec, s_off);
        __syncthreads();
        staged = true;
      }
      S.sweep(s_rec, s_off, 0, cnt, 1, ox, oyh, oyl);
    }
    S.fold();
    float2 v[2 * NC2];
#pragma unroll
    for (int c = 0; c < 2 * NC2; ++c) v[c] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < FP; ++k) {
      const float2 L = dup2(s_L[m][k]);
#pragma unroll
      for (int c = 0; c < NC2; ++c) {
        const float4 t = s_c[(rp * FP + k) * NC2 + c];
        if constexpr (POT) {  // v[0], v[1]: hi and lo sums of pairs
          const float2 f = make_float2(t.x, t.y), p = mul2(L, f);
          const float2 e = fma2(dup2(s_Ll[POT ? m : 0][k]), f, fma2(L, make_float2(t.z, t.w), fma2(L, f, neg2(p))));
          const df2 r = two_sum2(v[0], p);
          v[0] = r.hi;
          v[1] = add2(v[1], add2(r.lo, e));
          continue;
        }
        v[2 * c] = fma2(L, make_float2(t.x, t.y), v[2 * c]);
        v[2 * c + 1] = fma2(L, make_float2(t.z, t.w), v[2 * c + 1]);
      }
    }
    // plane + near + remainder, per value and point pair, in double-float
    const float2 my = make_float2(2 * rp - (float)HALF, 2 * rp + 1 - (float)HALF);
    float2 vh[NV], vl[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      const float4 p = s_plane[c];
      const df x = two_sum(p.x, p.y * mx);
      const df2 y = two_sum2(dup2(x.hi), mul2(dup2(p.z), my));
      const df n0 = S.value(c, 0), n1 = S.value(c, 1);
      const df2 z = two_sum2(y.hi, make_float2(n0.hi, n1.hi));
      float2 lo = add2(add2(y.lo, dup2(x.lo)), add2(z.lo, make_float2(n0.lo, n1.lo)));
      df2 w = {z.hi, v[c]};
      if constexpr (POT) {
        w = two_sum2(z.hi, v[0]);
        w.lo = add2(w.lo, v[1]);
      }
      const df2 r = two_sum2(w.hi, add2(lo, w.lo));
      vh[c] = r.hi;
      vl[c] = r.lo;
    }
    if (n_near_h > 0) {
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const df X = df_add(Tx, df{ox.x, ox.y}), Y = df_add(Ty, df{h ? oyh.y : oyh.x, h ? oyl.y : oyl.x});
        df sum[5] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        for (int k = 0; k < n_near_h; ++k) {
          const int hh = s_list[n_far + n_far_h + n_near + k];
          add_heavy<MODE>(a.heavydf + (size_t)hh * RECDF, a.heavy + (size_t)hh * REC64, X, Y, sum);
        }
#pragma unroll
        for (int c = 0; c < NV; ++c) {
          const df t = df_add(df{h ? vh[c].y : vh[c].x, h ? vl[c].y : vl[c].x}, sum[c]);
          if (h) {
            vh[c].y = t.hi;
            vl[c].y = t.lo;
          } else {
            vh[c].x = t.hi;
            vl[c].x = t.lo;
          }
        }
      }
    }
    const int jl = blockIdx.y * FT + 2 * rp;  // row of the launch
    if constexpr (POT) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = jl + h;
        if (i < a.nx && j < a.ny) {
          const long long o = (long long)j * a.nx + i;
          const double phi = a.dls * ((double)part2(vh[0], h) + (double)part2(vl[0], h));
          a.out64[o] = phi;
          if (a.tau) a.out64[a.plane + o] = s_tau[0][m] + s_tau[1][2 * rp + h] - phi;
        }
      }
    } else {
      const float dh = a.dls_h, dl = a.dls_l;
      // which nodes the double-float repair recomputes (see k_map_mixed);
      // the far potentials' kappa and gamma enter by their bounds on the tile
      if (a.rep_count) {
        bool rep[2], rep_h[2] = {false, false};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool in = i < a.nx && jl + h < a.ny;
          const float mg = a.repair_f * (part2(v[NV], h) + S.mag(h)), fx = part2(vh[0], h), fy = part2(vh[1], h);
          rep[h] = in && fmaf(fx, fx, fy * fy) < fmaf(mg, mg, s_kb[3]);
          if (HESS) {
            const float kl = dh * (fabsf(S.value(2, h).hi) + s_kb[0]);
            const float g1l = dh * (fabsf(S.value(3, h).hi) + s_kb[1]), g2l = dh * (fabsf(S.value(4, h).hi) + s_kb[2]);
            const float kap = dh * part2(vh[NV > 2 ? 2 : 0], h), g1 = dh * part2(vh[NV > 3 ? 3 : 0], h),
                        g2 = dh * part2(vh[NV > 4 ? 4 : 0], h);
            const float gm = sqrtf(fmaf(g1, g1, g2 * g2)), gl = sqrtf(fmaf(g1l, g1l, g2l * g2l));
            const float om = fabsf(1.f - kap), e1 = a.repair_f > 0.f ? fmaf(om, kl, gm * (kl + gl)) : 0.f;
            const float e2 = REM_TERM * dh * fmaf(om, s_kb[4], gm * s_kb[5]);
            rep_h[h] = in && fmaf(e1, e1, e2 * e2) > DET_LIST * DET_LIST;
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const unsigned mh = __ballot_sync(0xffffffffu, rep_h[h]), m1 = __ballot_sync(0xffffffffu, rep[h] && !rep_h[h]);
          if (lane == 0) {
            s_m[(2 * rp + h) * (FT / 32) + m / 32] = m1;
            if (HESS) s_mh[(2 * rp + h) * (FT / 32) + m / 32] = mh;
          }
        }
      }
      // scaled by D_ls/D_s in double-float, rounded once
#pragma unroll
      for (int c = 0; c < NV; ++c) {
        const float2 p = mul2(vh[c], dup2(dh));
        const float2 e = fma2(vl[c], dup2(dh), fma2(vh[c], dup2(dl), fma2(vh[c], dup2(dh), neg2(p))));
        vh[c] = add2(p, e);
        vl[c] = sub2(e, sub2(vh[c], p));
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = jl + h;
        if (i >= a.nx || j >= a.ny) continue;
        float *o = a.out + (long long)j * a.nx + i;
        o[0] = part2(vh[0], h);
        o[a.plane] = part2(vh[1], h);
        if constexpr (HESS) {
          const float kh = part2(vh[2], h), kl = part2(vl[2], h), g1 = part2(vh[3], h), g1l = part2(vl[3], h),
                      g2 = part2(vh[4], h), g2l = part2(vl[4], h);
          // det = (1 - kappa)^2 - gamma1^2 - gamma2^2 with the products' errors
          df om = two_sum(1.f, -kh);
          om = fast_two_sum(om.hi, om.lo - kl);
          const float p0 = __fmul_rn(om.hi, om.hi), p1 = __fmul_rn(g1, g1), p2 = __fmul_rn(g2, g2);
          const float e0 = fmaf(2.f * om.hi, om.lo, fmaf(om.hi, om.hi, -p0));
          const float e1 = fmaf(2.f * g1, g1l, fmaf(g1, g1, -p1)), e2 = fmaf(2.f * g2, g2l, fmaf(g2, g2, -p2));
          const df d0 = two_sum(p0, -p1), d1 = two_sum(d0.hi, -p2);
          const df det = fast_two_sum(d1.hi, (d0.lo + d1.lo) + (e0 - (e1 + e2)));
          o[2 * a.plane] = kh;
          o[3 * a.plane] = g1;
          o[4 * a.plane] = g2;
          o[5 * a.plane] = rcp_dff(det.hi, det.lo);
        }
      }
    }
  }
  if (POT || !a.rep_count) return;
  // the nodes to recompute: a tile with many of them goes to the dense tiles
  // (all planes' nodes with it where they are many), the others' to the list
  constexpr int NW = FT * FT / 32;
  __shared__ int s_pos[2 * NW], s_to[3];  // list positions; listed nodes, dense slot (or -1), its all-planes flag
  __syncthreads();
  if (warp == 0) {
    int n1 = 0, nh = 0;
    for (int w = lane; w < NW; w += 32) {
      n1 += __popc(s_m[w]);
      if (HESS) nh += __popc(s_mh[w]);
    }
    n1 = __reduce_add_sync(0xffffffffu, n1);
    nh = __reduce_add_sync(0xffffffffu, nh);
    int slot = -1;
    const bool full = HESS && nh >= a.dense_min;
    if (lane == 0 && a.dense.cap && (full || n1 >= a.dense_min)) {
      slot = atomicAdd(a.dense.count, 1);
      if (slot >= a.dense.cap) slot = -1;
    }
    slot = __shfl_sync(0xffffffffu, slot, 0);
    const bool list_h = slot < 0 || !full;
    const int nl = (list_h ? nh : 0) + (slot < 0 ? n1 : 0);
    int base = 0;
    if (lane == 0 && nl) base = atomicAdd(a.rep_count, nl);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int w0 = 0; w0 < 2 * NW && nl; w0 += 32) {  // all-plane words, then the others
      const int w = w0 + lane;
      const int c = __popc(w < NW ? (HESS && list_h ? s_mh[HESS ? w : 0] : 0u) : slot < 0 ? s_m[w - NW] : 0u);
      int sum = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += t;
      }
      s_pos[w] = base + sum - c;
      base += __shfl_sync(0xffffffffu, sum, 31);
    }
    if (lane == 0) {
      s_to[0] = nl;
      s_to[1] = slot;
      s_to[2] = full;
      if (slot >= 0) a.dense.tile[slot] = (blockIdx.y * gridDim.x + blockIdx.x) | (full ? (int)0x80000000u : 0);
    }
  }
  __syncthreads();
  const int nl = s_to[0], slot = s_to[1];
  const bool full = s_to[2] != 0, list_h = slot < 0 || !full;
  if (slot >= 0)
    for (int w = tid; w < NW; w += FI_THREADS) {
      unsigned *m = a.dense.mask + (size_t)slot * (HESS ? 2 : 1) * NW + w;
      m[0] = s_m[w];
      if (HESS) m[NW] = full ? s_mh[HESS ? w : 0] : 0u;
    }
  if (nl)
    for (int w = warp; w < 2 * NW; w += (FI_THREADS / 32)) {
      const int wi = w % NW;
      const unsigned mask = w < NW ? (HESS && list_h ? s_mh[HESS ? wi : 0] : 0u) : slot < 0 ? s_m[wi] : 0u;
      const int j = blockIdx.y * FT + wi / (FT / 32), i = i0 + wi % (FT / 32) * 32 + lane;
      if (mask >> lane & 1u)
        a.rep_list[s_pos[w] + __popc(mask & ((1u << lane) - 1u))] = (j * a.nx + i) | (w < NW ? (int)0x80000000u : 0);
    }
}

// The listed nodes of the densely listed tiles: a CTA takes some of a tile's
// nodes, FR_LANES lanes each (launch_far_repair); the near potentials (those
// the interpolation nodes left out) in double-float, dealt to the lanes, their
// records staged, then the far ones' values interpolated in double-float
// (weights and values as pairs: the FP32 weights' 6e-8 of a far sum of tens of
// arcsec would show where the deflection is near zero).  8192^2 x 2000: the
// repair spends its time on 100 instead of up to 4096 evaluations of every
// potential per tile.  Bound: latency on small maps, else issue (74 %).
constexpr int FR_THREADS = 128;
struct FarRepairArgs {
  const float2 *recdf;
  const double *all64;
  int n;
  double xmin, ymin, dx, dy;
  int nx, row0;
  double dls;
  float *out;
  long long plane;
  DenseRepair dense;
};

template <int FT, bool HESS, int FR_LANES>
__global__ void __launch_bounds__(FR_THREADS) k_far_repair(const FarRepairArgs a) {
  constexpr int FR_NODES = FR_THREADS / FR_LANES;
  constexpr int NW = FT * FT / 32, PARTS = FT * FT / FR_NODES, NODES = FP * FP, NV = HESS ? 5 : 2, NM = HESS ? 2 : 1;
  __shared__ unsigned s_w[NW], s_wh[HESS ? NW : 1];
  __shared__ int s_pos[NW + 1], s_near[FR_THREADS], s_nn[FR_THREADS / 32];
  __shared__ float2 s_val[NV][NODES];
  __shared__ float2 s_rdf[RECDF][FR_THREADS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nh = min(*a.dense.count, a.dense.cap);
  for (long long item = blockIdx.x; item < (long long)nh * PARTS; item += gridDim.x) {
    // part by part: the tiles' last parts, often empty, come last (tile by tile
    // a CTA's items all had the same part number: 5000^2 x 1500 9.93 ms, so 9.39)
    const int slot = (int)(item % nh), part = (int)(item / nh);
    __syncthreads();  // the previous item's shared data has been used
    const int entry = a.dense.tile[slot], tile = entry & 0x7fffffff;
    const bool full = HESS && entry < 0;  // the tile's Hessian values are there too
    for (int w = tid; w < NW; w += FR_THREADS) {
      const unsigned *m = a.dense.mask + (size_t)slot * NM * NW + w;
      const unsigned mh = HESS ? m[HESS ? NW : 0] : 0u;
      s_w[w] = m[0] | mh;
      if (HESS) s_wh[HESS ? w : 0] = mh;
    }
    for (int q = tid; q < (full ? NV : 2) * NODES; q += FR_THREADS) (&s_val[0][0])[q] = a.dense.val[(size_t)slot * NV * NODES + q];
    __syncthreads();
    if (warp == 0) {
      int base = 0;
      for (int w0 = 0; w0 < NW; w0 += 32) {
        const int c = __popc(s_w[w0 + lane]);
        int sum = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, sum, o);
          if (lane >= o) sum += t;
        }
        s_pos[w0 + lane] = base + sum - c;
        base += __shfl_sync(0xffffffffu, sum, 31);
      }
      if (lane == 0) s_pos[NW] = base;
    }
    __syncthreads();
    const int listed = s_pos[NW];
    if (part * FR_NODES >= listed) continue;  // uniform over the CTA
    // this lane group's node
    const int want = part * FR_NODES + tid / FR_LANES, sub = tid % FR_LANES;
    const int rank = min(want, listed - 1);
    const bool mine = want < listed && sub == 0;
    int lo = 0, hi = NW;  // s_pos[lo] <= rank < s_pos[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) / 2;
      if (s_pos[mid] <= rank)
        lo = mid;
      else
        hi = mid;
    }
    unsigned bits = s_w[lo];
    for (int k = rank - s_pos[lo]; k > 0; --k) bits &= bits - 1u;
    const int jr = lo / (FT / 32), ic = lo % (FT / 32) * 32 + __ffs(bits) - 1;
    const bool all = HESS && mine && (s_wh[HESS ? lo : 0] >> (__ffs(bits) - 1) & 1u);  // every plane of this node
    const int i0 = tile % a.dense.tpr * FT, j0 = tile / a.dense.tpr * FT;
    const df Cx = tile_centre(a.xmin, (double)i0, FT, a.dx), Cy = tile_centre(a.ymin, (double)(a.row0 + j0), FT, a.dy);
    const double X = a.xmin + (i0 + ic) * a.dx, Y = a.ymin + (a.row0 + j0 + jr) * a.dy;
    const df Xd = df_kept(X), Yd = df_kept(Y);
    df sum[5] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    for (int h0 = 0; h0 < a.n; h0 += FR_THREADS) {
      const int h = h0 + tid;
      const bool near = h < a.n && !repair_far(a.recdf + h, a.n, Cx, Cy, a.dense.thr, a.dense.thr_h);
      const unsigned b = __ballot_sync(0xffffffffu, near);
      __syncthreads();  // the previous chunk's records have been used
      if (lane == 0) s_nn[warp] = __popc(b);
      __syncthreads();
      int base = 0, nn = 0;
      for (int w = 0; w < FR_THREADS / 32; ++w) {
        if (w < warp) base += s_nn[w];
        nn += s_nn[w];
      }
      if (near) s_near[base + __popc(b & ((1u << lane) - 1u))] = h;
      __syncthreads();
      for (int q = tid; q < RECDF * nn; q += FR_THREADS) s_rdf[q / nn][q % nn] = a.recdf[(size_t)(q / nn) * a.n + s_near[q % nn]];
      __syncthreads();
      for (int k = sub; k < nn; k += FR_LANES)
        if (HESS && full)
          add_potential_dfs<true>(&s_rdf[0][k], FR_THREADS, a.all64 + (size_t)s_near[k] * REC64, X, Y, Xd, Yd, sum);
        else
          add_potential_dfs<false>(&s_rdf[0][k], FR_THREADS, a.all64 + (size_t)s_near[k] * REC64, X, Y, Xd, Yd, sum);
    }
    // the lanes' sums (every lane gets the same bits)
#pragma unroll
    for (int c = 0; c < NV; ++c)
#pragma unroll
      for (int o = 1; o < FR_LANES; o <<= 1)
        sum[c] = df_add(sum[c], df{__shfl_xor_sync(0xffffffffu, sum[c].hi, o), __shfl_xor_sync(0xffffffffu, sum[c].lo, o)});
    // the far potentials: rows of the tensor product (spread over the lanes),
    // then the column
    const FineTab<FT> &t = fine_table<FT>();
    double val[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      if (c >= 2 && !full) break;
      df v = {0.f, 0.f};
#pragma unroll 1
      for (int j = sub; j < FP; j += FR_LANES) {
        df r = {0.f, 0.f};
#pragma unroll
        for (int i = 0; i < FP; ++i) {
          const float2 f = s_val[c][j * FP + i];
          r = df_add(r, df_mul(df{t.w[ic][i], t.wlo[ic][i]}, df{f.x, f.y}));
        }
        v = df_add(v, df_mul(df{t.w[jr][j], t.wlo[jr][j]}, r));
      }
#pragma unroll
      for (int o = 1; o < FR_LANES; o <<= 1)
        v = df_add(v, df{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
      val[c] = a.dls * df_to_double(df_add(v, sum[c]));
    }
    float *o = a.out + (long long)(j0 + jr) * a.nx + i0 + ic;
    if (mine) {
      o[0] = (float)val[0];
      o[a.plane] = (float)val[1];
    }
    if constexpr (HESS) {
      if (all) {
        const double kap = val[2], g1 = val[3], g2 = val[4];
        const double det = (1.0 - kap) * (1.0 - kap) - g1 * g1 - g2 * g2;
        o[2 * a.plane] = (float)kap;
        o[3 * a.plane] = (float)g1;
        o[4 * a.plane] = (float)g2;
        o[5 * a.plane] = (float)(1.0 / det);
      }
    }
  }
}

// ft = 0: the coarse kernel
size_t far_smem(int mode, int ft, int nw, int n, int threads = 256) {
  const bool coarse = ft == 0;
  const int nodes = coarse ? CP * CP : FP * FP, splits = threads / (nodes / 2), nc = ncmp(mode);
  size_t b = sizeof(float4) * (size_t)(coarse ? CO_CH : FF_CH) * (REC_STRIDE4 + 1);
  if (!coarse) b += sizeof(float4) * (ft / 2) * FP * ncmp2(mode);
  // the partial sums' space also holds the coarse tile's values (fine kernel)
  const size_t part = std::max(sizeof(float2) * splits * nodes * nc, coarse ? 0 : sizeof(float) * nrem(mode) * nc * (CP * CP + CP * FP));
  b += (part + 15) / 16 * 16 + sizeof(float2) * nodes * nc;
  b += sizeof(unsigned) * 4 * (size_t)nw + sizeof(unsigned short) * (size_t)n;
  return (b + 15) / 16 * 16;
}

// Margins: squared psi (K R)^2 of the tile's half-diagonal R beyond which a
// potential is far.  The FP32 potentials' interpolation error stays below
// 1.2e-8 of the term; the cluster-scale ones', whose deflection is ten times
// the rest, below 1e-9.
constexpr double KF = 3.0, KF_H = 3.5, KC = 2.5, KC_H = 3.0;
// fixed work in evaluations of one FP32 potential: per fine tile, per map node
constexpr double TILE_COST = 4000.0, NODE_COST = 3.0;
// densely listed tiles of the repair: from this many nodes, on maps of at
// least this many nodes and potentials (below, the extra launch costs more
// than the repair) and at most this many tiles (2.1 KB each, 5 KB with the Hessian)
constexpr int DENSE_MIN = 150, DENSE_NODES = 1 << 19, DENSE_N = 64;
constexpr long long DENSE_TILES = 65536;
// margins of the repair: interpolation error below 4e-11 of a potential's own
// deflection at the edge of its far region (4e-14 for the strong ones)
constexpr double KR = 5.0, KR_H = 8.0;
// Potential maps are stored in double, so the FP32 terms' rounding shows in
// them.  Both forms are as far from 64 bits, but they round differently: they
// differ by 0.5e-10 to 7.3e-10 of the map where Model::pot_light is below this
// (50 models of 60 to 2000 potentials; 8.3e-10 to 6.4e-9 from 0.003 on).  Which
// form a grid takes depends on its size and on the memory at hand, and a map is
// not to move with that by more than 1e-9 of itself: beyond, every size takes
// the direct kernel (2048^2 x 1000, 0.00303: 8 ms; interpolated 0.52).
constexpr double POT_LIGHT = 0.0025;
constexpr int FAR_MAX_N = 16384;  // potentials (two bytes each of shared memory)

// Fraction of the map's nodes within psi < r of a potential of axis ratio q
// and core s: the area of the ellipse q^2 (s^2 + x^2) + y^2 < r^2.
double near_frac(double r, double q, double s, double area) {
  const double r2 = r * r - q * q * s * s;
  return r2 <= 0.0 ? 0.0 : std::min(1.0, M_PI * r2 / (q * area));
}

// The lists' and masks' words, and what a launch of this size needs.
int far_words(const Model *m) { return (m->n_light + 31) / 32 + (m->n_heavy + 31) / 32; }

}  // namespace

// Expected cost per map node of the direct kernel and of the interpolated
// one with each coarse level, in evaluations of one FP32 potential (HV of
// them for a cluster-scale potential in double-float), idle SMs of small
// grids included (152 SMs: 4 CTAs of the direct kernel, 1 of the coarse or 2 of
// the fine one each).
FarPlan plan_far(const lens_ctx *ctx, const Model *m, const lens_grid *g, int mode) {
  FarPlan p;
  if (m->n > FAR_MAX_N || m->n < 1) return p;
  if (mode == FAR_POT && m->pot_light > POT_LIGHT) return p;
  const double dx = (g->xmax - g->xmin) / (g->nx - 1), dy = (g->ymax - g->ymin) / (g->ny - 1);
  const double area = (g->xmax - g->xmin) * (g->ymax - g->ymin), nodes = (double)g->nx * g->ny;
  const double HV = mode == FAR_HESS ? 20.0 : 10.0, step = std::max(dx, dy);
  auto light = [&](double r) { return m->n_light * near_frac(r, 1.0 / m->invq_light, 0.0, area); };
  auto heavy = [&](double r) {
    double s = 0.0;
    for (const auto &h : m->heavy_shape) s += near_frac(r, h.first, h.second, area);
    return s;
  };
  double best = 0.85 * (m->n_light + HV * m->n_heavy + 2.0) * std::max(1.0, 608.0 * 256.0 / nodes);
  for (int ft = 32; ft <= 64; ft *= 2) {
    const double tiles = std::ceil(g->nx / (double)ft) * std::ceil(g->ny / (double)ft);
    const double Rf = std::sqrt(2.0) * 0.5 * (ft - 1) * step;
    const double near = light(KF * Rf) + HV * heavy(KF_H * Rf);
    for (int ct = 0; ct <= CT_MAX; ct = ct ? 2 * ct : 2 * ft) {
      if (ct && ct >= 2 * std::max(g->nx, g->ny)) break;
      double mid = m->n_light, mid_h = m->n_heavy, coarse = 0.0;
      if (ct) {
        const double Rc = std::sqrt(2.0) * 0.5 * ct * step;
        const double ctiles = std::ceil(g->nx / (double)ct) * std::ceil(g->ny / (double)ct);
        coarse = (m->n_light + 2.0 * HV * m->n_heavy) * 170.0 * ctiles / nodes * std::max(1.0, 152.0 / ctiles);
        mid = light(KC * Rc);
        mid_h = heavy(KC_H * Rc);
      }
      const double fine = (TILE_COST + (mid + 2.5 * HV * mid_h) * (FP * FP)) / (double)(ft * ft);
      const double c = coarse + (NODE_COST + fine + near) * tiles * ft * ft / nodes * std::max(1.0, 304.0 / tiles);
      if (c < best) {
        best = c;
        p.use = true;
        p.ft = ft;
        p.ct = ct;
        p.cost = c;
      }
    }
  }
  if (p.use && p.ct) {
    p.nct = (g->nx + p.ct - 1) / p.ct;
    p.ncr = (g->ny + p.ct - 1) / p.ct;
    const size_t t = (size_t)p.nct * p.ncr;
    p.val_bytes = (t * coarse_floats(mode) * sizeof(float) + 255) & ~(size_t)255;
    p.bytes = (p.val_bytes + t * far_words(m) * sizeof(unsigned) + 255) & ~(size_t)255;
  }
  if (p.use && mode != FAR_POT && ctx->repair_ratio > 0.0 && nodes >= DENSE_NODES && m->n >= DENSE_N && m->n_light > 0) {
    const long long tiles = (long long)((g->nx + p.ft - 1) / p.ft) * ((g->ny + p.ft - 1) / p.ft);
    p.rep_cap = tiles <= DENSE_TILES ? (int)tiles : 0;
    const size_t h = mode == FAR_HESS;
    p.rep_bytes = ((size_t)p.rep_cap * (sizeof(float2) * (h ? 5 : 2) * FP * FP + sizeof(int) + (h ? 2 : 1) * (size_t)p.ft * p.ft / 8) + 255) & ~(size_t)255;
    p.bytes += p.rep_bytes;
  }
  return p;
}

DenseRepair dense_repair(const lens_grid *g, const FarPlan &p, bool hess, void *mem, int *count) {
  DenseRepair d;
  if (!mem || !p.rep_cap) return d;
  d.count = count;
  d.cap = p.rep_cap;
  d.ft = p.ft;
  d.tpr = (g->nx + p.ft - 1) / p.ft;
  d.nv = hess ? 5 : 2;
  d.val = (float2 *)mem;
  d.tile = (int *)(d.val + (size_t)p.rep_cap * d.nv * FP * FP);
  d.mask = (unsigned *)(d.tile + p.rep_cap);
  const double dx = (g->xmax - g->xmin) / (g->nx - 1), dy = (g->ymax - g->ymin) / (g->ny - 1);
  const double R = std::sqrt(2.0) * 0.5 * (p.ft - 1) * std::max(dx, dy);
  d.thr = (float)(KR * R * KR * R);
  d.thr_h = (float)(KR_H * R * KR_H * R);
  for (int k = 0; k < FP; ++k) d.xi[k] = (float)((p.ft == 32 ? XiTab<32>::v[k] : XiTab<64>::v[k]) / 64.0);
  return d;
}

int launch_far_repair(const Model *m, const lens_grid *g, const DenseRepair &dense, double dls, void *out, int row0,
                      int rows, int device, cudaStream_t st) {
  FarRepairArgs a;
  a.recdf = m->recdf;
  a.all64 = m->all64;
  a.n = m->n;
  a.xmin = g->xmin;
  a.ymin = g->ymin;
  a.dx = (g->xmax - g->xmin) / (g->nx - 1);
  a.dy = (g->ymax - g->ymin) / (g->ny - 1);
  a.nx = g->nx;
  a.row0 = row0;
  a.dls = dls;
  a.out = (float *)out;
  a.plane = (long long)g->nx * rows;
  a.dense = dense;
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
  const bool hess = dense.nv == 5;
  // Lanes per node: the near potentials of one node are a long chain, and a map
  // of few nodes has few listed ones to fill the chip with; more lanes repeat
  // the search for the near potentials more often.  Whole Hessian map with 1 /
  // 2 / 4 lanes: 768^2 x 1000 705 / 595 / 556 us, 1024^2 x 300 298 / 278 / 266,
  // 1536^2 x 500 439 / 423 / 422, 2048^2 x 1000 795 / 780 / 800; 64 x 64 tiles,
  // 8192^2 x 2000 7.83 / 8.13 ms.  By the whole map, so that bands keep its bits.
  const bool few = (long long)g->nx * g->ny < 1 << 21;
  auto kern = dense.ft == 64 ? (hess ? k_far_repair<64, true, 1> : k_far_repair<64, false, 1>)
              : few          ? (hess ? k_far_repair<32, true, 4> : k_far_repair<32, false, 4>)
                             : (hess ? k_far_repair<32, true, 2> : k_far_repair<32, false, 2>);
  kern<<<4 * nsm, FR_THREADS, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(LENS_ECUDA, "dense map repair launch: %s", cudaGetErrorString(e));
  return LENS_OK;
}

static FarArgs far_args(const Model *m, const lens_grid *g, const FarPlan &p, int mode, void *mem) {
  FarArgs a;
  a.rec32 = m->rec32;
  a.cen32 = (const float4 *)m->cen32;
  a.n_light = m->n_light;
  a.heavy = m->heavy;
  a.heavydf = m->heavydf;
  a.n_heavy = m->n_heavy;
  a.nwl = (m->n_light + 31) / 32;
  a.nw = far_words(m);
  a.xmin = g->xmin;
  a.ymin = g->ymin;
  a.dx = (g->xmax - g->xmin) / (g->nx - 1);
  a.dy = (g->ymax - g->ymin) / (g->ny - 1);
  a.nx = g->nx;
  a.ny = g->ny;
  a.row0 = 0;
  a.dls = 1.0;
  a.dls_h = 1.f;
  a.dls_l = 0.f;
  const double step = std::sqrt(2.0) * std::max(a.dx, a.dy), rf = 0.5 * (p.ft - 1) * step, rc = 0.5 * p.ct * step;
  auto sq = [](double v) { return (float)(v * v); };
  a.thr_c = sq(KC * rc);
  a.thr_ch = sq(KC_H * rc);
  a.thr_f = sq(KF * rf);
  a.thr_fh = sq(KF_H * rf);
  a.ct = p.ct;
  a.nct = p.nct;
  a.cval = (float *)mem;
  a.cmask = (unsigned *)((char *)mem + p.val_bytes);
  a.out = nullptr;
  a.out64 = nullptr;
  a.plane = 0;
  a.tau = 0;
  a.bx = a.by = 0.0;
  a.repair_f = 0.f;
  a.rep_count = a.rep_list = nullptr;
  a.dense_min = DENSE_MIN;
  return a;
}

// A kernel's shared memory limit: what the largest model takes, whatever this
// call's takes.  It belongs to the kernel on the device, not to the context, and
// another context's thread may be between setting it and launching.
template <typename K>
static int far_limit(K kern, int mode, int ft, int threads) {
  const size_t most = far_smem(mode, ft, FAR_MAX_N / 32 + 1, FAR_MAX_N, threads);
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  return e == cudaSuccess ? LENS_OK : fail(LENS_ECUDA, "interpolated map's shared memory: %s", cudaGetErrorString(e));
}

template <int MODE>
static int coarse_launch(const FarArgs &a, const FarPlan &p, int n, cudaStream_t st) {
  const size_t smem = far_smem(MODE, 0, a.nw, n, CO_THREADS);
  const int rc = far_limit(k_far_coarse<MODE>, MODE, 0, CO_THREADS);
  if (rc) return rc;
  k_far_coarse<MODE><<<dim3(p.nct, p.ncr), CO_THREADS, smem, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(LENS_ECUDA, "coarse map level launch: %s", cudaGetErrorString(e));
  return LENS_OK;
}

template <int MODE, int FT, int TH>
static int fine_launch(const FarArgs &a, int n, cudaStream_t st) {
  const size_t smem = far_smem(MODE, FT, a.nw, n, TH);
  const int rc = far_limit(k_far_map<MODE, FT, TH>, MODE, FT, TH);
  if (rc) return rc;
  k_far_map<MODE, FT, TH><<<dim3((a.nx + FT - 1) / FT, (a.ny + FT - 1) / FT), TH, smem, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(LENS_ECUDA, "interpolated map launch: %s", cudaGetErrorString(e));
  return LENS_OK;
}

// 128 threads where there are many tiles (small CTAs overlap each other's
// phases), 256 where the longest tile shows.  Both, whole map (256 / 128):
// Hessian x 1000, 256 tiles 422 / 627 us, 1024 tiles 654 / 700, 2304 tiles 651
// / 667, 4096 tiles 824 / 798; deflection x 200, 2304 tiles 197 / 181, 2304 of
// 64 x 64 299 / 323, 4096 tiles 250 / 210, 6241 (5000^2 x 217) 524 / 451.
// The potential's FP64 terms want the 256 (0.266 against 0.279 ms).
// 512 threads (one CTA per SM) where not every SM has two tiles: a tile is a
// chain of phases, and twice the threads shorten it.  256 / 512 threads, us:
// Hessian x 1000, 100 tiles 480 / 355, 196 tiles 395 / 299, 256 tiles 396 / 331;
// x 300, 175 / 135, 147 / 115, 145 / 129; deflection x 300, 256 tiles 122 / 104;
// potential x 1000, 256 tiles 389 / 294.  With 10 potentials there is little to
// share: Hessian, 196 tiles 40.2 / 36.5, 256 tiles 40.3 / 42.9 (60 potentials
// 60.5 / 59.7), hence the lower line there.
// Counted over the whole map, also where a band of it is launched: the split of
// the node sums, and with it the last bits, is then the same.
constexpr int FI_TILES = 3072, FI_FEW = 304, FI_FEW_SMALL = 200, FI_SMALL = 32;
template <int MODE, int FT>
static int fine_threads(const FarArgs &a, const lens_grid *g, int n, cudaStream_t st) {
  const long long tiles = (long long)((g->nx + FT - 1) / FT) * ((g->ny + FT - 1) / FT);
  if constexpr (MODE != FAR_POT)
    if (tiles >= FI_TILES) return fine_launch<MODE, FT, 128>(a, n, st);
  if constexpr (FT == 32)
    if (tiles <= (MODE != FAR_POT && n < FI_SMALL ? FI_FEW_SMALL : FI_FEW)) return fine_launch<MODE, FT, 512>(a, n, st);
  return fine_launch<MODE, FT, 256>(a, n, st);
}

int launch_far_coarse(const Model *m, const lens_grid *g, const FarPlan &p, int mode, void *mem, cudaStream_t st) {
  if (!p.ct) return LENS_OK;
  const FarArgs a = far_args(m, g, p, mode, mem);
  return mode == FAR_HESS   ? coarse_launch<FAR_HESS>(a, p, m->n, st)
         : mode == FAR_GRAD ? coarse_launch<FAR_GRAD>(a, p, m->n, st)
                            : coarse_launch<FAR_POT>(a, p, m->n, st);
}

int launch_far_map(const Model *m, const lens_grid *g, const FarPlan &p, int mode, void *mem, double dls, void *out,
                   int row0, int rows, double repair, int *rep_count, int *rep_list, const DenseRepair &dense,
                   const double *beta, cudaStream_t st) {
  FarArgs a = far_args(m, g, p, mode, mem);
  a.ny = rows;
  a.row0 = row0;
  a.dls = dls;
  a.dls_h = (float)dls;
  a.dls_l = (float)(dls - (double)a.dls_h);
  a.plane = (long long)g->nx * rows;
  a.repair_f = (float)(2.0 * repair);
  a.rep_count = rep_count;
  a.rep_list = rep_list;
  a.dense = dense;
  if (mode == FAR_POT) {
    a.out64 = (double *)out;
    a.tau = beta != nullptr;
    a.bx = beta ? beta[0] : 0.0;
    a.by = beta ? beta[1] : 0.0;
    return p.ft == 32 ? fine_threads<FAR_POT, 32>(a, g, m->n, st) : fine_threads<FAR_POT, 64>(a, g, m->n, st);
  }
  a.out = (float *)out;
  if (mode == FAR_HESS) return p.ft == 32 ? fine_threads<FAR_HESS, 32>(a, g, m->n, st) : fine_threads<FAR_HESS, 64>(a, g, m->n, st);
  return p.ft == 32 ? fine_threads<FAR_GRAD, 32>(a, g, m->n, st) : fine_threads<FAR_GRAD, 64>(a, g, m->n, st);
}

}  // namespace lens
