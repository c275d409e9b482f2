// Catalogue scalars (alpha, I22, I33, N0, S3) and deterministic CIC/TSC interlaced painting.
//
// Painting (Sec. 3.1 mass assignment; interlacing as cited there):
//   1. k_brick_count  grid coordinate s = (x - origin) * (n/box) in float64, base cell floor(s)
//                     (wrapped), brick of BS^3 cells; per-brick counts and in-brick ranks.
//   2. k_scan         exclusive scan of the brick counts.
//   3. k_scatter      particles regrouped by brick as records {x, y, z, weight coefficient}.
//   4. k_paint_brick  one CTA per brick accumulates every tap of its particles into a
//                     (BS+4)^3 shared-memory tile (the brick plus the cells its particles can
//                     reach) in 64-bit fixed point (words of 32 bits), so the sum is independent of
//                     thread order;
//                     the tile is written out once.
//   5. k_fold         each mesh cell sums, in a fixed order, the (up to 8) tiles that cover it.
// The mesh is therefore bitwise reproducible run to run without any floating-point atomics.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "npc_internal.cuh"

namespace {

constexpr int RED_THREADS = 256;
constexpr int RED_CHUNK = 4096;   // objects per block, until the blocks number four per SM
constexpr int NSUM = 6;  // sum w, w^2, w^3, nbar w^2, nbar^2 w^3, max |w|

template <typename T>
__device__ __forceinline__ void cat_partial(const T* __restrict__ w, const T* __restrict__ nbar, int64_t n,
                                            int nblk, int blk, double* __restrict__ part) {
  __shared__ double sh[NSUM][RED_THREADS];
  const int64_t chunk = (n + nblk - 1) / nblk;
  const int64_t beg = (int64_t)blk * chunk;
  const int64_t end = min(n, beg + chunk);
  double a[NSUM] = {0, 0, 0, 0, 0, 0};
  if constexpr (sizeof(T) == 4) {
    // float inputs: products and per-thread sums in float-float arithmetic (error-free products by
    // FMA, two-sum accumulation, about 48 significant bits) instead of the slow FP64 pipe; the
    // per-thread results are exact in double and enter the same fixed-order tree
    float hs[NSUM - 1] = {0, 0, 0, 0, 0}, ls[NSUM - 1] = {0, 0, 0, 0, 0};
    float wmax = 0.0f;
    // explicit _rn operations: the compiler must not fuse a product into the sums below
    auto acc = [&](int k, float vh, float vl) {
      const float s = __fadd_rn(hs[k], vh);
      const float bb = __fsub_rn(s, hs[k]);
      const float e = __fadd_rn(__fadd_rn(__fsub_rn(hs[k], __fsub_rn(s, bb)), __fsub_rn(vh, bb)), __fadd_rn(ls[k], vl));
      hs[k] = __fadd_rn(s, e);
      ls[k] = __fsub_rn(e, __fsub_rn(hs[k], s));
    };
    auto add = [&](float wi, float nb) {
      const float p2 = __fmul_rn(wi, wi), e2 = fmaf(wi, wi, -p2);             // w^2
      const float p3 = __fmul_rn(p2, wi), e3 = fmaf(p2, wi, -p3) + e2 * wi;   // w^3
      const float p4 = __fmul_rn(nb, p2), e4 = fmaf(nb, p2, -p4) + nb * e2;   // nbar w^2
      const float pt = __fmul_rn(nb, p3), et = fmaf(nb, p3, -pt) + nb * e3;   // nbar w^3
      const float p5 = __fmul_rn(nb, pt), e5 = fmaf(nb, pt, -p5) + nb * et;   // nbar^2 w^3
      acc(0, wi, 0.0f);
      acc(1, p2, e2);
      acc(2, p3, e3);
      acc(3, p4, e4);
      acc(4, p5, e5);
      wmax = fmaxf(wmax, fabsf(wi));
    };
    // four objects' loads in flight per thread
    int64_t i = beg + threadIdx.x;
    for (; i + 3 * RED_THREADS < end; i += 4 * RED_THREADS) {
      float wv[4], nv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        wv[k] = w ? (float)w[i + k * RED_THREADS] : 1.0f;
        nv[k] = nbar ? (float)nbar[i + k * RED_THREADS] : 0.0f;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) add(wv[k], nv[k]);
    }
    for (; i < end; i += RED_THREADS) add(w ? (float)w[i] : 1.0f, nbar ? (float)nbar[i] : 0.0f);
#pragma unroll
    for (int k = 0; k < NSUM - 1; ++k) a[k] = (double)hs[k] + (double)ls[k];
    a[NSUM - 1] = (double)wmax;
  } else {
    for (int64_t i = beg + threadIdx.x; i < end; i += blockDim.x) {
      const double wi = w ? (double)w[i] : 1.0;
      const double nb = nbar ? (double)nbar[i] : 0.0;
      const double w2 = wi * wi;
      a[0] += wi;
      a[1] += w2;
      a[2] += w2 * wi;
      a[3] += nb * w2;
      a[4] += nb * nb * w2 * wi;
      a[5] = fmax(a[5], fabs(wi));
    }
  }
#pragma unroll
  for (int k = 0; k < NSUM; ++k) sh[k][threadIdx.x] = a[k];
  __syncthreads();
  // warp k reduces sum k over the block in a fixed tree: float64 adds are scarce on this part (16 cycles
  // per warp instruction), so they are spread over the warps, with one barrier
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  if (k >= NSUM) return;
  auto comb = [&](double x, double y) { return k == NSUM - 1 ? fmax(x, y) : x + y; };
  double v[RED_THREADS / 32];
#pragma unroll
  for (int j = 0; j < RED_THREADS / 32; ++j) v[j] = sh[k][lane + 32 * j];
#pragma unroll
  for (int off = RED_THREADS / 64; off > 0; off >>= 1)
#pragma unroll
    for (int j = 0; j < off; ++j) v[j] = comb(v[j], v[j + off]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v[0] = comb(v[0], __shfl_down_sync(0xffffffffu, v[0], off));
  if (lane == 0) part[blk * NSUM + k] = v[0];
}

// grid (blocks, 1 or 2): per-block partial sums of the data (y = 0) and of the randoms (y = 1)
template <typename T, typename U>
__global__ void __launch_bounds__(RED_THREADS)
k_cat_partials(const T* __restrict__ wd, const T* __restrict__ nd, int64_t n_d, const U* __restrict__ wr,
               const U* __restrict__ nr, int64_t n_r, double* __restrict__ pd, double* __restrict__ pr) {
  if (blockIdx.y == 0) cat_partial<T>(wd, nd, n_d, gridDim.x, blockIdx.x, pd);
  else cat_partial<U>(wr, nr, n_r, gridDim.x, blockIdx.x, pr);
}

// Warp w sums sum w % NSUM of catalogue w / NSUM: lane l takes the partials of blocks l, l+32, ... in
// order, then a fixed shuffle tree; the order depends only on nblk (bitwise reproducible).  One warp for
// all twelve took 25 us over 1024 blocks.
__global__ void __launch_bounds__(2 * NSUM * 32)
k_cat_final(const double* __restrict__ pd, const double* __restrict__ pr, int nblk, int have_randoms, double box,
            double* __restrict__ sc) {
  __shared__ double s_sum[2 * NSUM];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, k = warp % NSUM;
  double v = 0.0;
  if (warp < NSUM || have_randoms) {
    const double* __restrict__ p = warp < NSUM ? pd : pr;
    for (int b = lane; b < nblk; b += 32) v = k == NSUM - 1 ? fmax(v, p[b * NSUM + k]) : v + p[b * NSUM + k];
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double o = __shfl_down_sync(0xffffffffu, v, off);
    v = k == NSUM - 1 ? fmax(v, o) : v + o;
  }
  if (lane == 0) s_sum[warp] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double *g = s_sum, *r = s_sum + NSUM;
  for (int k = 0; k < SC_COUNT; ++k) sc[k] = 0.0;
  if (have_randoms) {
    const double alpha = g[0] / r[0];
    const double i22 = alpha * r[3];
    sc[SC_ALPHA] = alpha;
    sc[SC_I22] = i22;
    sc[SC_I33] = alpha * r[4];
    sc[SC_N0] = (g[1] + alpha * alpha * r[1]) / i22;
    sc[SC_S3] = g[2] - alpha * alpha * alpha * r[2];
    sc[SC_SUMWG] = g[0];
    sc[SC_SUMWR] = r[0];
    sc[SC_SUMW2] = g[1] + alpha * alpha * r[1];
    sc[SC_MAXW_F] = fmax(g[5], fabs(alpha) * r[5]);
    sc[SC_MAXW_N] = fmax(g[5] * g[5], alpha * alpha * r[5] * r[5]);
  } else {
    const double vol = box * box * box;
    const double ws = g[0];
    const double i22 = ws * ws / vol;
    sc[SC_ALPHA] = 0.0;
    sc[SC_I22] = i22;
    sc[SC_I33] = ws * ws * ws / (vol * vol);
    sc[SC_N0] = g[1] / i22;
    sc[SC_S3] = g[2];
    sc[SC_SUMWG] = ws;
    sc[SC_SUMWR] = 0.0;
    sc[SC_SUMW2] = g[1];
    sc[SC_MAXW_F] = g[5];
    sc[SC_MAXW_N] = g[5] * g[5];
  }
}

// ---------------------------------------------------------------------------------------------
// Painting
// ---------------------------------------------------------------------------------------------
struct PaintGeo {
  int n, bs, nb, ts;     // mesh cells, brick size, bricks per side, tile side (bs + 4)
  int bshift;            // log2(bs)
  double o[3];           // origin
  double inv_h;          // n / box
  float o_hi[3], o_lo[3];      // origin and n / box as float pairs (hi + lo) for the scatter's
  float ih_hi, ih_lo;          // float fast path
};

// i modulo n; the integer division only outside the box
__device__ __forceinline__ int wrapi(long long i, int n) {
  if (i >= 0 && i < n) return (int)i;
  const long long r = i % n;
  return (int)(r < 0 ? r + n : r);
}

// One or two catalogues of the same type sorted together: object i is the first's for i < n0, else the
// second's (randoms).
template <typename P> struct CatPair {
  const P* pos[2];
  const P* w[2];
  int64_t n0, n;
};

// Brick of an object, -1 when its position is not finite (or absurdly far).
template <typename P>
__device__ __forceinline__ int brick_of(const P* __restrict__ pos, int64_t i, const PaintGeo& g) {
  int bidx[3];
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // floor(s) decided in float when s is farther from an integer than a bound on the float
    // rounding error (three roundings of relative size 2^-24 on |x| n/box, |origin| n/box and
    // |s|, with a factor 8 of margin), otherwise in float64 exactly as everywhere else
    const P pa = pos[3 * i + a];
    if (sizeof(P) == 4) {
      const float ih = (float)g.inv_h;
      const float sf = ((float)pa - (float)g.o[a]) * ih;
      const float ff = floorf(sf);
      const float fr = sf - ff;
      const float tol = 1.0e-6f * ((fabsf((float)pa) + fabsf((float)g.o[a])) * ih + fabsf(sf)) + 1.0e-6f;
      if (fabsf(sf) < 1.0e6f && fr > tol && fr < 1.0f - tol) {
        bidx[a] = wrapi((int)ff, g.n) >> g.bshift;
        continue;
      }
    }
    const double s = ((double)pa - g.o[a]) * g.inv_h;
    if (!(fabs(s) < 1e15)) {
      ok = false;
      bidx[a] = 0;
      continue;
    }
    bidx[a] = wrapi((long long)floor(s), g.n) >> g.bshift;
  }
  return ok ? (bidx[2] * g.nb + bidx[1]) * g.nb + bidx[0] : -1;
}

// Brick and in-brick rank of every object, and the objects per brick.  Up to COUNT_SHARED_MAX bricks the
// CTA counts its COUNT_CHUNK objects in shared memory and takes one range per brick from the global
// counter: a global counter then sees one add per CTA instead of one per object (the adds that return
// a rank serialise per 32-byte sector at about 10 ns each: 189 us for 1.4 M objects in 512 bricks, 10 ms
// of a batch's 34 ms; for the same reason every counter has a sector of its own).  Above it the counters
// are too many for that to help (less than one object per CTA and brick) and each object adds to its own.
constexpr int COUNT_THREADS = 512, COUNT_ITEMS = 8;
constexpr int COUNT_SHARED_MAX = 8192;
constexpr int COUNT_STRIDE = 8;   // ints between the counters of consecutive bricks
template <typename P, bool SHARED>
__global__ void __launch_bounds__(COUNT_THREADS)
k_brick_count(const CatPair<P> c, PaintGeo g, int nbricks, int* __restrict__ count, int* __restrict__ brick,
              int* __restrict__ rank) {
  extern __shared__ int s_hist[];
  const int64_t beg = blockIdx.x * (int64_t)(COUNT_THREADS * COUNT_ITEMS);
  if constexpr (SHARED) {
    for (int b = threadIdx.x; b < nbricks; b += COUNT_THREADS) s_hist[b] = 0;
    __syncthreads();
  }
  int br[COUNT_ITEMS], rk[COUNT_ITEMS];
#pragma unroll
  for (int k = 0; k < COUNT_ITEMS; ++k) {
    const int64_t i = beg + k * COUNT_THREADS + threadIdx.x;
    br[k] = -1;
    rk[k] = 0;
    if (i >= c.n) continue;
    br[k] = i < c.n0 ? brick_of<P>(c.pos[0], i, g) : brick_of<P>(c.pos[1], i - c.n0, g);
    if (br[k] >= 0) rk[k] = atomicAdd(SHARED ? s_hist + br[k] : count + (size_t)br[k] * COUNT_STRIDE, 1);
  }
  if constexpr (SHARED) {
    __syncthreads();
    for (int b = threadIdx.x; b < nbricks; b += COUNT_THREADS) {
      const int m = s_hist[b];
      if (m > 0) s_hist[b] = atomicAdd(count + (size_t)b * COUNT_STRIDE, m);
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < COUNT_ITEMS; ++k) {
    const int64_t i = beg + k * COUNT_THREADS + threadIdx.x;
    if (i >= c.n) continue;
    brick[i] = br[k];
    rank[i] = br[k] < 0 ? 0 : (SHARED ? s_hist[br[k]] + rk[k] : rk[k]);
  }
}

// Exclusive scan of the m brick counts into start[0..m), the total into start[m]: one CTA per SCAN_CHUNK entries writes its chunk's scan
// and total; with more than one chunk k_scan_add adds the totals of the chunks before (one CTA over
// everything took 428 us for the 262,144 bricks of a 1024^3 mesh).
constexpr int SCAN_THREADS = 1024, SCAN_PER = 8, SCAN_CHUNK = SCAN_THREADS * SCAN_PER;
__global__ void __launch_bounds__(SCAN_THREADS) k_scan(const int* __restrict__ count, int m, int* __restrict__ start,
                                                       int* __restrict__ total) {
  __shared__ int s_warp[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int beg = blockIdx.x * SCAN_CHUNK + threadIdx.x * SCAN_PER;
  int v[SCAN_PER], sum = 0;
#pragma unroll
  for (int k = 0; k < SCAN_PER; ++k) {
    v[k] = beg + k < m ? count[(size_t)(beg + k) * COUNT_STRIDE] : 0;
    sum += v[k];
  }
  int inc = sum;   // inclusive over the warp's threads
  for (int off = 1; off < 32; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += o;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int w = s_warp[lane];
    for (int off = 1; off < 32; off <<= 1) {
      const int o = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += o;
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  int run = inc - sum + (warp > 0 ? s_warp[warp - 1] : 0);
#pragma unroll
  for (int k = 0; k < SCAN_PER; ++k) {
    if (beg + k <= m) start[beg + k] = run;
    run += v[k];
  }
  if (threadIdx.x == SCAN_THREADS - 1) total[blockIdx.x] = run;
}
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_add(const int* __restrict__ total, int m,
                                                           int* __restrict__ start) {
  __shared__ int s_before;
  if (threadIdx.x < 32) {
    int v = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += 32) v += total[b];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (threadIdx.x == 0) s_before = v;
  }
  __syncthreads();
  for (int k = 0; k < SCAN_PER; ++k) {
    const int i = blockIdx.x * SCAN_CHUNK + k * SCAN_THREADS + threadIdx.x;
    if (i <= m) start[i] += s_before;
  }
}

template <typename R> struct RecOf;
template <> struct RecOf<float> { using type = float4; };
template <> struct RecOf<double> { using type = double4_32a; };

// Per particle, per axis: the float64 decisions of the oracle are taken here once and stored as
//   meta bits 8a..8a+4: base cell floor(s) relative to its brick (< 16)
//   meta bits 8a+5   : phase-a tap centre minus base (TSC floor(s+1/2) - floor(s); CIC 0)
//   meta bits 8a+6..7: phase-b tap centre minus base (TSC floor((s+1/2)+1/2) - floor(s);
//                      CIC floor(s+1/2) - floor(s))
// and the record keeps frac = s - floor(s) (exact in float64, rounded once to R) and the weight.
template <int ASSIGN>
__device__ __forceinline__ uint32_t axis_meta(double s, int n, int bs, double* frac) {
  const double f = floor(s);
  const long long fb = (long long)f;
  const double sb = s + 0.5;
  long long ia, ib;
  if (ASSIGN == 2) {
    ia = fb;
    ib = (long long)floor(sb);
  } else {
    ia = (long long)floor(s + 0.5);
    ib = (long long)floor(sb + 0.5);
  }
  *frac = s - f;
  const uint32_t local = (uint32_t)(wrapi(fb, n) & (bs - 1));
  return local | ((uint32_t)(ia - fb) << 5) | ((uint32_t)(ib - fb) << 6);
}

// The same decisions and fraction from a float position in float arithmetic: s = (x - origin) n/box
// as a float pair (exact difference by two-sum, exact product error by fma; about 2^-46 relative),
// its floor and the fraction s - floor(s) to float precision.  For TSC floor(s + 1/2) - floor(s) is
// [frac >= 1/2] and floor(s + 1) - floor(s) = 1; for CIC the phase-a offset is 0 and the phase-b one
// [frac >= 1/2], exactly as the float64 expressions give them.  Returns false (the caller takes the
// float64 path) when |s| >= 2^22 or the fraction lies within 1e-6 of 0, 1/2 or 1, where the float64
// rounding of s could decide differently.
template <int ASSIGN>
__device__ __forceinline__ bool axis_meta_fast(float x, float o_hi, float o_lo, float ih_hi, float ih_lo, int n, int bs,
                                               float* frac, uint32_t* meta) {
  const float d1 = __fsub_rn(x, o_hi);
  const float bv = __fsub_rn(d1, x);
  const float d2 = __fsub_rn(__fadd_rn(__fsub_rn(x, __fsub_rn(d1, bv)), __fsub_rn(-o_hi, bv)), o_lo);
  // the rounded product is never fused into a later add: s2 carries its exact error
  const float s1 = __fmul_rn(d1, ih_hi);
  float s2 = fmaf(d1, ih_hi, -s1);
  s2 = fmaf(d1, ih_lo, s2);
  s2 = fmaf(d2, ih_hi, s2);
  if (!(fabsf(s1) < 4194304.0f)) return false;
  float f = floorf(s1);
  float fr = __fadd_rn(__fsub_rn(s1, f), s2);
  if (fr < 0.0f) {
    f -= 1.0f;
    fr += 1.0f;
  } else if (fr >= 1.0f) {
    f += 1.0f;
    fr -= 1.0f;
  }
  const float tol = 1.0e-6f;
  if (fr < tol || fr > 1.0f - tol || fabsf(fr - 0.5f) < tol) return false;
  const int fb = (int)f;
  const uint32_t half = fr >= 0.5f ? 1u : 0u;
  const uint32_t local = (uint32_t)(wrapi(fb, n) & (bs - 1));
  const uint32_t da = ASSIGN == 2 ? 0u : half, db = ASSIGN == 2 ? half : 1u;
  *meta = local | (da << 5) | (db << 6);
  *frac = fr;
  return true;
}

// coefficient * w^power per object: 1 for the first catalogue, -alpha (power 1) or alpha^2 for the randoms
template <int ASSIGN, typename P, typename R>
__global__ void k_scatter(const CatPair<P> c, int power, bool randoms_first, const double* __restrict__ sc, PaintGeo g,
                          const int* __restrict__ brick, const int* __restrict__ rank, const int* __restrict__ start,
                          typename RecOf<R>::type* __restrict__ rec, uint32_t* __restrict__ meta) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < c.n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int b = brick[t];
    if (b < 0) continue;
    const int dst = start[b] + rank[t];
    const bool second = t >= c.n0;
    const P* __restrict__ pos = second ? c.pos[1] : c.pos[0];
    const P* __restrict__ w = second ? c.w[1] : c.w[0];
    const int64_t i = second ? t - c.n0 : t;
    double coef = 1.0;
    if (second || randoms_first) coef = power == 2 ? sc[SC_ALPHA] * sc[SC_ALPHA] : -sc[SC_ALPHA];
    const float coef_f = (float)coef;
    if constexpr (sizeof(R) == 4 && sizeof(P) == 4) {
      // float records from float positions: the float pair path, float64 only near a decision
      uint32_t u[3];
      float wcf;
      {
        const float wf = w ? (float)w[i] : 1.0f;
        wcf = coef_f * (power == 2 ? wf * wf : wf);
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float x = (float)pos[3 * i + a];
        float frf;
        uint32_t ma;
        if (!axis_meta_fast<ASSIGN>(x, g.o_hi[a], g.o_lo[a], g.ih_hi, g.ih_lo, g.n, g.bs, &frf, &ma)) {
          double frd;
          ma = axis_meta<ASSIGN>(((double)x - g.o[a]) * g.inv_h, g.n, g.bs, &frd);
          frf = (float)frd;
        }
        const uint32_t q = __float2uint_rz(frf * 16777216.0f);
        u[a] = (q > 0xffffffu ? 0xffffffu : q) | ((ma & 255u) << 24);
      }
      typename RecOf<R>::type r;
      r.x = __uint_as_float(u[0]);
      r.y = __uint_as_float(u[1]);
      r.z = __uint_as_float(u[2]);
      r.w = wcf;
      rec[dst] = r;
      continue;
    }
    const double wi = w ? (double)w[i] : 1.0;
    const double wc = coef * (power == 2 ? wi * wi : wi);
    double fr[3];
    uint32_t m = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double s = ((double)pos[3 * i + a] - g.o[a]) * g.inv_h;
      m |= axis_meta<ASSIGN>(s, g.n, g.bs, &fr[a]) << (8 * a);
    }
    typename RecOf<R>::type r;
    if constexpr (sizeof(R) == 4) {
      // one 16-byte record: per axis the fraction in 24-bit fixed point (truncated, |error| < 2^-24
      // of a cell) with that axis's 8 decision bits on top, and the float weight
      uint32_t u[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const uint32_t q = __float2uint_rz((float)fr[a] * 16777216.0f);
        u[a] = (q > 0xffffffu ? 0xffffffu : q) | (((m >> (8 * a)) & 255u) << 24);
      }
      r.x = __uint_as_float(u[0]);
      r.y = __uint_as_float(u[1]);
      r.z = __uint_as_float(u[2]);
      r.w = (float)wc;
    } else {
      r.x = (R)fr[0];
      r.y = (R)fr[1];
      r.z = (R)fr[2];
      r.w = (R)wc;
      meta[dst] = m;
    }
    rec[dst] = r;
  }
}

// Per-axis taps of one phase: up to 3 (TSC) or 2 (CIC) cells with weights, from the stored fraction
// and decision bits.  Returns the first tap's tile index; the others follow it.  The rounding of the
// middle float weight 3/4 - d^2 is spelled out (FUSED: the square is not rounded by itself), so that
// the mesh does not depend on which products the compiler fuses.
__device__ __forceinline__ float middle_weight(float d, bool fused) {
  return fused ? fmaf(-d, d, 0.75f) : __fsub_rn(0.75f, __fmul_rn(d, d));
}
__device__ __forceinline__ double middle_weight(double d, bool) { return 0.75 - d * d; }

template <int ASSIGN, typename T, bool FUSED = true>
__device__ __forceinline__ int axis_taps(T frac, uint32_t m8, int phase, T* wt) {
  const int local = (int)(m8 & 31u);
  const int off = phase ? (int)((m8 >> 6) & 3u) : (int)((m8 >> 5) & 1u);
  // d = s - centre (phase a) or (s + 1/2) - centre (phase b)
  const T d = frac + (phase ? T(0.5) : T(0)) - T(off);
  const int rel = local + off + 1;   // tile index of the centre (tile starts one cell below the brick)
  if (ASSIGN == 2) {
    wt[0] = T(1) - d;
    wt[1] = d;
    return rel;
  }
  const T a = T(0.5) - d, b = T(0.5) + d;
  wt[0] = T(0.5) * a * a;
  wt[1] = middle_weight(d, FUSED);
  wt[2] = T(0.5) * b * b;
  return rel - 1;
}

// Pairs of floats in one 64-bit register: the packed add, multiply and fused multiply-add of this
// architecture round each half as the scalar instruction does and issue once for both.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Two float tap values as integer parts: |v| < 2^43 (the tile kernel's scale guarantees it),
// rn(v) = 2^22 h + l with |h|, |l| <= 2^21, without a conversion instruction: h = rn(v / 2^22) and the
// exact remainder v - 2^22 h are rounded to integers by adding 1.5 * 2^23 (the float add rounds to
// nearest even, and the integer sits in the low mantissa bits); since 2^22 h is an even integer,
// 2^22 h + rn(remainder) = rn(v).
__device__ __forceinline__ void fixed_parts2(f32x2 v, int (&h)[2], int (&l)[2]) {
  const f32x2 magic = pack2(12582912.0f, 12582912.0f);                                       // 1.5 * 2^23
  const f32x2 th = fma2(v, pack2(2.384185791015625e-07f, 2.384185791015625e-07f), magic);   // rn(v 2^-22) + magic
  const f32x2 hf = add2(th, pack2(-12582912.0f, -12582912.0f));                              // exact
  const f32x2 tl = add2(fma2(hf, pack2(-4194304.0f, -4194304.0f), v), magic);                // (v - 2^22 h) + magic
  float a, b;
  unpack2(th, a, b);
  h[0] = __float_as_int(a) - 0x4B400000;
  h[1] = __float_as_int(b) - 0x4B400000;
  unpack2(tl, a, b);
  l[0] = __float_as_int(a) - 0x4B400000;
  l[1] = __float_as_int(b) - 0x4B400000;
}

// 64-bit fixed point back to T times 2^-e; the float path uses two 32-bit conversions.
__device__ __forceinline__ float from_fixed(long long q, float inv) {
  const int hi = (int)(q >> 32);
  const unsigned lo = (unsigned)(q & 0xffffffffull);
  return fmaf((float)hi, 4294967296.0f, (float)lo) * inv;
}
__device__ __forceinline__ double from_fixed(long long q, double inv) { return (double)q * inv; }

// The tile sums are 64-bit integers, but shared memory has no native 64-bit atomic add (it runs as a
// compare-and-swap loop: 21 cycles per warp instruction measured here), so every sum is kept as two
// 32-bit words with native adds:
//   float, at most NARROW_MAX objects in the brick: sums of the h and of the l parts, two adds without
//     a return value; no word can overflow (1023 * 2^21 < 2^31).  10 cycles at 671 objects.
//   float, more objects: the adds return the old word, so that an overflow of l is carried into h
//     (2^32 = 1024 * 2^22) and one of h into the cell's signed byte of a third array (the whole sum is
//     at most 127/128 of 2^61, so h overflows at most 127 times either way).  9 cycles at 20,000
//     objects, where the tile's clearing and writing no longer count.
//   double: low and high halves of the 64-bit integer, the high add taking the carry of the low one.
constexpr int NARROW_MAX = 1023;
__device__ __forceinline__ bool add_overflows(int old, int q) {
  const int now = (int)((unsigned)old + (unsigned)q);
  return ((old ^ now) & (q ^ now)) < 0;
}
template <bool WIDE>
__device__ __forceinline__ void tile_add(int* lo, int* hi, unsigned* top, int idx, int h, int l) {
  if constexpr (!WIDE) {
    atomicAdd(lo + idx, l);
    atomicAdd(hi + idx, h);
  } else {
    if (add_overflows(atomicAdd(lo + idx, l), l)) h += l < 0 ? -1024 : 1024;
    if (add_overflows(atomicAdd(hi + idx, h), h)) atomicAdd(top + (idx >> 2), (h < 0 ? 0xffffffffu : 1u) << (8 * (idx & 3)));
  }
}
__device__ __forceinline__ void tile_add(int* lo, int* hi, int idx, double v) {
  const long long q = __double2ll_rn(v);
  const unsigned ql = (unsigned)q;
  const unsigned old = atomicAdd(reinterpret_cast<unsigned*>(lo) + idx, ql);
  const int h = (int)(q >> 32) + (old + ql < old ? 1 : 0);
  if (h != 0) atomicAdd(hi + idx, h);
}

// Sum of cell idx from its words.  The bytes of `top` hold signed digits that borrowed from their
// upper neighbours: digit d is the sign-extended low byte once the digits below it are taken out.
template <typename T>
__device__ __forceinline__ long long tile_sum(int lo, int hi, unsigned topw, int digit) {
  if constexpr (sizeof(T) == 8) return ((long long)hi << 32) | (unsigned)lo;
  int d = 0;
  if (topw != 0u) {
    for (int k = 0; k <= digit; ++k) {
      d = (int)(signed char)(topw & 0xffu);
      topw = (topw - (unsigned)d) >> 8;
    }
  }
  return (((long long)d << 32) + hi) * 4194304LL + lo;
}

// Every tap of the brick's objects into the tile words.
template <int ASSIGN, typename T, int BS, bool WIDE>
__device__ __forceinline__ void tile_taps(const typename RecOf<T>::type* __restrict__ rec,
                                          const uint32_t* __restrict__ meta, int cnt, int ph, T scale, int* lo, int* hi,
                                          unsigned* top) {
  constexpr int TS = BS + 4;
  constexpr int NT = ASSIGN == 2 ? 2 : 3;
  // NT adjacent lanes share one object, lane xt taking its x tap: the atomics of one instruction
  // then hit runs of NT neighbouring cells instead of 32 scattered ones (fewer bank wavefronts; nine
  // lanes per object, x and y, measured 1.6 times slower: three times the record decoding per tap)
  constexpr int OPW = 32 / NT;   // objects per warp and pass
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int xt = lane % NT, slot = lane / NT;
  for (int k0 = warp * OPW; k0 < cnt; k0 += nwarp * OPW) {
    const int k = k0 + slot;
    if (slot >= OPW || k >= cnt) continue;
    const typename RecOf<T>::type r = rec[k];
    T wx[NT], wy[NT], wz[NT];
    int ix, iy, iz;
    if constexpr (sizeof(T) == 4) {
      const uint32_t ux = __float_as_uint(r.x), uy = __float_as_uint(r.y), uz = __float_as_uint(r.z);
      const float sc24 = 5.9604644775390625e-8f;   // 2^-24
      ix = axis_taps<ASSIGN, T>((float)(ux & 0xffffffu) * sc24, ux >> 24, ph, wx);
      iy = axis_taps<ASSIGN, T>((float)(uy & 0xffffffu) * sc24, uy >> 24, ph, wy);
      iz = axis_taps<ASSIGN, T, false>((float)(uz & 0xffffffu) * sc24, uz >> 24, ph, wz);
    } else {
      const uint32_t m = meta[k];
      ix = axis_taps<ASSIGN, T>(r.x, m & 255u, ph, wx);
      iy = axis_taps<ASSIGN, T>(r.y, (m >> 8) & 255u, ph, wy);
      iz = axis_taps<ASSIGN, T, false>(r.z, (m >> 16) & 255u, ph, wz);
    }
    // the taps of a brick's object lie inside its tile by construction; the test only protects shared memory
    if (max(max(ix, iy), iz) > TS - NT) continue;
    T wxs = wx[0];
#pragma unroll
    for (int a = 1; a < NT; ++a)
      if (xt == a) wxs = wx[a];
    const T wgt = r.w * scale * wxs;
    const int base = (iz * TS + iy) * TS + ix + xt;
    // tap values (w 2^e W_x) W_z W_y, formed once per tap in a fixed order
    if constexpr (sizeof(T) == 4) {
      int h[2], l[2];
      float wc[NT];
#pragma unroll
      for (int c = 0; c < NT; ++c) {
        wc[c] = wgt * wz[c];
        fixed_parts2(mul2(pack2(wc[c], wc[c]), pack2(wy[0], wy[1])), h, l);
        tile_add<WIDE>(lo, hi, top, base + c * TS * TS, h[0], l[0]);
        tile_add<WIDE>(lo, hi, top, base + (c * TS + 1) * TS, h[1], l[1]);
      }
      if constexpr (NT == 3) {
        fixed_parts2(mul2(pack2(wc[0], wc[1]), pack2(wy[2], wy[2])), h, l);
        tile_add<WIDE>(lo, hi, top, base + 2 * TS, h[0], l[0]);
        tile_add<WIDE>(lo, hi, top, base + (TS + 2) * TS, h[1], l[1]);
        fixed_parts2(mul2(pack2(wc[2], 0.0f), pack2(wy[2], 0.0f)), h, l);
        tile_add<WIDE>(lo, hi, top, base + (2 * TS + 2) * TS, h[0], l[0]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < NT; ++c) {
#pragma unroll
        for (int bb = 0; bb < NT; ++bb) tile_add(lo, hi, base + (c * TS + bb) * TS, wgt * wz[c] * wy[bb]);
      }
    }
  }
}

template <typename T, int BS> constexpr size_t tile_smem() {
  return (sizeof(T) == 4 ? 9 : 8) * (size_t)(BS + 4) * (BS + 4) * (BS + 4);
}

// One CTA per (brick, phase): fixed-point accumulation of all taps in a (BS+4)^3 tile.  Bound by the
// shared-memory atomics and the instructions that form a tap's integer parts (27 taps per object and
// phase for TSC, 8 for CIC); 72 KB of tile words, three CTAs of 512 threads per SM.
template <int ASSIGN, typename T, int BS>
__global__ void __launch_bounds__(512, sizeof(T) == 4 ? 3 : 2)
k_paint_brick(const typename RecOf<T>::type* __restrict__ rec, const uint32_t* __restrict__ meta,
              const int* __restrict__ start, int nphase, const double* __restrict__ sc, int maxw_slot,
              T* __restrict__ tiles) {
  constexpr int TS = BS + 4, TS3 = TS * TS * TS;
  static_assert(TS3 % 16 == 0, "the tile words are cleared and read in 16-byte steps");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* lo = reinterpret_cast<int*>(smem_raw);
  int* hi = lo + TS3;
  unsigned* top = reinterpret_cast<unsigned*>(hi + TS3);   // one signed byte per cell (float tiles)
  __shared__ int s_exp;
  const int b = blockIdx.x / nphase, ph = blockIdx.x % nphase;
  const int beg = start[b], cnt = start[b + 1] - beg;
  for (int i = threadIdx.x; i < (int)(tile_smem<T, BS>() / 16); i += blockDim.x)
    reinterpret_cast<int4*>(smem_raw)[i] = make_int4(0, 0, 0, 0);
  if (threadIdx.x == 0) {
    // fixed-point scale 2^e with cnt * max|w| * 2^e < 2^61 (no overflow of the tile sums)
    const double bound = (double)cnt * sc[maxw_slot];
    int ex = 0;
    double mant = 0.0;
    if (bound > 0) mant = frexp(bound, &ex);
    int e = 61 - ex;
    if constexpr (sizeof(T) == 4) {
      // float: at most 127/128 of 2^61 (the words' range) and every tap |w W| 2^e < 2^43 (that of fixed_parts)
      int exw = 0;
      if (sc[maxw_slot] > 0) frexp(sc[maxw_slot], &exw);
      e = max(-126, min(126, min(mant > 127.0 / 128.0 ? e - 1 : e, 43 - exw)));
    }
    s_exp = e;
  }
  __syncthreads();
  const int e = s_exp;
  T scale, inv;   // 2^e and 2^-e
  if constexpr (sizeof(T) == 4) {
    scale = __int_as_float((127 + e) << 23);
    inv = __int_as_float((127 - e) << 23);
  } else {
    scale = ldexp(1.0, e);
    inv = ldexp(1.0, -e);
  }
  const uint32_t* bmeta = sizeof(T) == 8 ? meta + beg : nullptr;
  if (cnt <= NARROW_MAX)
    tile_taps<ASSIGN, T, BS, false>(rec + beg, bmeta, cnt, ph, scale, lo, hi, top);
  else
    tile_taps<ASSIGN, T, BS, true>(rec + beg, bmeta, cnt, ph, scale, lo, hi, top);
  __syncthreads();
  T* out = tiles + ((size_t)b * nphase + ph) * TS3;
  for (int i = threadIdx.x; i < TS3 / 4; i += blockDim.x) {
    const int4 l = reinterpret_cast<const int4*>(lo)[i];
    const int4 h = reinterpret_cast<const int4*>(hi)[i];
    const unsigned t = sizeof(T) == 4 ? top[i] : 0u;
    const T v0 = from_fixed(tile_sum<T>(l.x, h.x, t, 0), inv), v1 = from_fixed(tile_sum<T>(l.y, h.y, t, 1), inv);
    const T v2 = from_fixed(tile_sum<T>(l.z, h.z, t, 2), inv), v3 = from_fixed(tile_sum<T>(l.w, h.w, t, 3), inv);
    if constexpr (sizeof(T) == 4) {
      reinterpret_cast<float4*>(out)[i] = make_float4(v0, v1, v2, v3);
    } else {
      reinterpret_cast<double2*>(out)[2 * i] = make_double2(v0, v1);
      reinterpret_cast<double2*>(out)[2 * i + 1] = make_double2(v2, v3);
    }
  }
}

// Each cell sums the tiles covering it, in a fixed order (brick offset -1, 0, +1 per axis, z
// outermost).  One CTA per (brick, phase); the tile of brick B covers cells [BS B - 1, BS B + BS + 2].
// Thread (x, y) of the CTA owns one column of the brick along z: its x and y options (own tile, the
// lower neighbour's for the first three cells, the upper neighbour's for the last) are fixed per
// thread, only the z options change per cell.
template <typename T, int BS>
__global__ void __launch_bounds__(BS * BS)
k_fold(const T* __restrict__ tiles, PaintGeo g, int nphase, const double* __restrict__ sc, int subtract_mean,
       T* __restrict__ mesh_a, T* __restrict__ mesh_b) {
  constexpr int TS = BS + 4, TS3 = TS * TS * TS;
  const int n = g.n, nb = g.nb;
  const int b = blockIdx.x / nphase, ph = blockIdx.x % nphase;
  const int B[3] = {b % nb, (b / nb) % nb, b / (nb * nb)};
  int nbm[3], nbp[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    nbm[a] = B[a] == 0 ? nb - 1 : B[a] - 1;
    nbp[a] = B[a] == nb - 1 ? 0 : B[a] + 1;
  }
  const T mean = subtract_mean ? (T)(sc[SC_SUMWG] / ((double)n * n * n)) : T(0);
  T* mesh = ph ? mesh_b : mesh_a;
  const int lx = threadIdx.x % BS, ly = threadIdx.x / BS;
  // x and y options: brick coordinate and tile coordinate, lower neighbour first
  int nx = 0, ny = 0, bx[2], tx[2], by[2], ty[2];
  if (lx <= 2) { bx[nx] = nbm[0]; tx[nx] = lx + BS + 1; ++nx; }
  bx[nx] = B[0]; tx[nx] = lx + 1; ++nx;
  if (lx == BS - 1) { bx[nx] = nbp[0]; tx[nx] = 0; ++nx; }
  if (ly <= 2) { by[ny] = nbm[1]; ty[ny] = ly + BS + 1; ++ny; }
  by[ny] = B[1]; ty[ny] = ly + 1; ++ny;
  if (ly == BS - 1) { by[ny] = nbp[1]; ty[ny] = 0; ++ny; }
  // per (iy, ix) option (2 x 2 slots, slot valid when iy < ny and ix < nx): pointer into the tile
  // of the brick in the same z layer; invalid slots hold a valid address and are predicated off
  const size_t zstride = (size_t)nb * nb * nphase * TS3;   // between z layers of bricks
  const T* p_yx[2][2];
  bool ok[2][2];
#pragma unroll
  for (int iy = 0; iy < 2; ++iy)
#pragma unroll
    for (int ix = 0; ix < 2; ++ix) {
      ok[iy][ix] = iy < ny && ix < nx;
      const int yy = ok[iy][ix] ? iy : 0, xx = ok[iy][ix] ? ix : 0;
      const size_t brick = ((size_t)B[2] * nb + by[yy]) * nb + bx[xx];
      p_yx[iy][ix] = tiles + (brick * nphase + ph) * TS3 + ty[yy] * TS + tx[xx];
    }
  const ptrdiff_t dzm = (ptrdiff_t)(nbm[2] - B[2]) * (ptrdiff_t)zstride;   // to the lower z layer
  const ptrdiff_t dzp = (ptrdiff_t)(nbp[2] - B[2]) * (ptrdiff_t)zstride;   // to the upper z layer
  T* col = mesh + ((size_t)(B[2] * BS) * n + (B[1] * BS + ly)) * n + (B[0] * BS + lx);
  // z cells 0..2 also take the lower z layer's tiles, cell BS-1 the upper one's; the loop is unrolled
  // so that the independent loads of several cells are in flight together
#pragma unroll
  for (int lz = 0; lz < BS; ++lz) {
    T v = T(0);
    if (lz <= 2) {
      const ptrdiff_t o = dzm + (ptrdiff_t)(lz + BS + 1) * TS * TS;
#pragma unroll
      for (int iy = 0; iy < 2; ++iy)
#pragma unroll
        for (int ix = 0; ix < 2; ++ix)
          if (ok[iy][ix]) v += p_yx[iy][ix][o];
    }
    {
      const int o = (lz + 1) * TS * TS;
#pragma unroll
      for (int iy = 0; iy < 2; ++iy)
#pragma unroll
        for (int ix = 0; ix < 2; ++ix)
          if (ok[iy][ix]) v += p_yx[iy][ix][o];
    }
    if (lz == BS - 1) {
#pragma unroll
      for (int iy = 0; iy < 2; ++iy)
#pragma unroll
        for (int ix = 0; ix < 2; ++ix)
          if (ok[iy][ix]) v += p_yx[iy][ix][dzp];
    }
    col[(size_t)lz * n * n] = v - mean;
  }
}

// A catalogue and its randoms (r may be null) as one object list; of one type only.
template <typename P>
CatPair<P> cat_pair(const DevCatalog* d, const DevCatalog* r) {
  CatPair<P> c{};
  c.pos[0] = (const P*)d->pos;
  c.w[0] = (const P*)d->w;
  c.n0 = c.n = d->n;
  if (r) {
    c.pos[1] = (const P*)r->pos;
    c.w[1] = (const P*)r->w;
    c.n += r->n;
  }
  return c;
}

template <typename P>
npc_status paint_count(npc_ctx* ctx, const CatPair<P>& c, const PaintGeo& g, int nbricks, int* count, int* brick,
                       int* rank) {
  if (c.n == 0) return NPC_OK;
  const int chunk = COUNT_THREADS * COUNT_ITEMS;
  const unsigned blocks = (unsigned)((c.n + chunk - 1) / chunk);
  if (nbricks <= COUNT_SHARED_MAX)
    k_brick_count<P, true><<<blocks, COUNT_THREADS, sizeof(int) * nbricks, ctx->stream>>>(c, g, nbricks, count, brick,
                                                                                          rank);
  else
    k_brick_count<P, false><<<blocks, COUNT_THREADS, 0, ctx->stream>>>(c, g, nbricks, count, brick, rank);
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

template <int ASSIGN, typename P, typename R>
npc_status paint_scatter(npc_ctx* ctx, const CatPair<P>& c, int power, bool randoms_first, const double* sc,
                         const PaintGeo& g, const int* brick, const int* rank, const int* start, void* rec,
                         uint32_t* meta) {
  if (c.n == 0) return NPC_OK;
  const int blocks = (int)std::min<int64_t>((c.n + 255) / 256, (int64_t)1 << 20);   // one object per thread
  k_scatter<ASSIGN, P, R><<<blocks, 256, 0, ctx->stream>>>(c, power, randoms_first, sc, g, brick, rank, start,
                                                           (typename RecOf<R>::type*)rec, meta);
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

template <typename T>
npc_status launch_fold(npc_ctx* ctx, const void* tiles, const PaintGeo& g, int nphase, const double* sc, int sub,
                       void* mesh_a, void* mesh_b) {
  const int grid = g.nb * g.nb * g.nb * nphase;
  switch (g.bs) {
    case 4: k_fold<T, 4><<<grid, 16, 0, ctx->stream>>>((const T*)tiles, g, nphase, sc, sub, (T*)mesh_a, (T*)mesh_b); break;
    case 8: k_fold<T, 8><<<grid, 64, 0, ctx->stream>>>((const T*)tiles, g, nphase, sc, sub, (T*)mesh_a, (T*)mesh_b); break;
    default: k_fold<T, 16><<<grid, 256, 0, ctx->stream>>>((const T*)tiles, g, nphase, sc, sub, (T*)mesh_a, (T*)mesh_b); break;
  }
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

template <int ASSIGN, typename T, int BS>
npc_status launch_tiles(npc_ctx* ctx, const void* rec, const uint32_t* meta, const int* start, int nbricks,
                        int nphase, const double* sc, int slot, void* tiles) {
  const size_t smem = tile_smem<T, BS>();
  auto kern = k_paint_brick<ASSIGN, T, BS>;
  NPC_TRY(allow_smem(ctx, (const void*)kern, smem));
  kern<<<nbricks * nphase, 512, smem, ctx->stream>>>((const typename RecOf<T>::type*)rec, meta, start, nphase, sc,
                                                     slot, (T*)tiles);
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

template <int ASSIGN, typename T>
npc_status paint_impl(npc_ctx* ctx, const DevCatalog& d, const DevCatalog* r, const npc_mesh_spec& m,
                      int weight_power, const double* sc, void* mesh_a, void* mesh_b, bool sorted) {
  PaintGeo g;
  g.n = m.n;
  g.bs = (m.n >= 48 && m.n % 16 == 0) ? 16 : m.n / 4;   // 16 for every size >= 48; 4, 8 at n = 16, 32
  g.bshift = g.bs == 16 ? 4 : (g.bs == 8 ? 3 : 2);
  g.nb = m.n / g.bs;
  g.ts = g.bs + 4;
  for (int a = 0; a < 3; ++a) g.o[a] = m.origin[a];
  g.inv_h = (double)m.n / m.box;
  for (int a = 0; a < 3; ++a) {
    g.o_hi[a] = (float)g.o[a];
    g.o_lo[a] = (float)(g.o[a] - (double)g.o_hi[a]);
  }
  g.ih_hi = (float)g.inv_h;
  g.ih_lo = (float)(g.inv_h - (double)g.ih_hi);
  const int nphase = m.interlace ? 2 : 1;
  const int nbricks = g.nb * g.nb * g.nb;
  const int64_t ntot = d.n + (r ? r->n : 0);
  // brick starts and ranks are 32-bit offsets into one record array
  if (ntot >= (int64_t)1 << 31)
    return set_err(ctx, NPC_ERR_UNSUPPORTED, "painting takes at most 2^31-1 objects (data + randoms)");
  int *count, *start, *brick, *rank;
  uint32_t* meta;
  void* rec;
  void* tiles;
  const size_t ts3 = (size_t)g.ts * g.ts * g.ts;
  NPC_TRY(ws_get(ctx, "paint.count", sizeof(int) * nbricks * COUNT_STRIDE, (void**)&count));
  NPC_TRY(ws_get(ctx, "paint.start", sizeof(int) * (nbricks + 1), (void**)&start));
  NPC_TRY(ws_get(ctx, "paint.brick", sizeof(int) * std::max<int64_t>(ntot, 1), (void**)&brick));
  NPC_TRY(ws_get(ctx, "paint.rank", sizeof(int) * std::max<int64_t>(ntot, 1), (void**)&rank));
  NPC_TRY(ws_get(ctx, "paint.meta", sizeof(uint32_t) * std::max<int64_t>(ntot, 1), (void**)&meta));
  NPC_TRY(ws_get(ctx, "paint.rec", sizeof(typename RecOf<T>::type) * std::max<int64_t>(ntot, 1), &rec));
  NPC_TRY(ws_get(ctx, "paint.tiles", sizeof(T) * ts3 * nbricks * nphase, &tiles));
  // data and randoms share the brick counters (ranks continue): one launch each for counting and for
  // scattering when both catalogues have one type
  const bool joint = r && r->dtype == d.dtype;
  auto each = [&](auto&& run) -> npc_status {   // run(catalogue pair's parts, offset, randoms first)
    NPC_TRY(run(&d, joint ? r : nullptr, (int64_t)0, false));
    if (r && !joint) NPC_TRY(run(r, (const DevCatalog*)nullptr, d.n, true));
    return NPC_OK;
  };
  if (!sorted) {
    NPC_CUDA(ctx, cudaMemsetAsync(count, 0, sizeof(int) * nbricks * COUNT_STRIDE, ctx->stream));
    NPC_TRY(each([&](const DevCatalog* a, const DevCatalog* b, int64_t off, bool) {
      return a->dtype == 1 ? paint_count<double>(ctx, cat_pair<double>(a, b), g, nbricks, count, brick + off, rank + off)
                           : paint_count<float>(ctx, cat_pair<float>(a, b), g, nbricks, count, brick + off, rank + off);
    }));
    const int chunks = nbricks / SCAN_CHUNK + 1;   // of the nbricks + 1 entries
    int* total;
    NPC_TRY(ws_get(ctx, "paint.total", sizeof(int) * chunks, (void**)&total));
    k_scan<<<chunks, SCAN_THREADS, 0, ctx->stream>>>(count, nbricks, start, total);
    NPC_LAUNCH(ctx);
    if (chunks > 1) {
      k_scan_add<<<chunks, SCAN_THREADS, 0, ctx->stream>>>(total, nbricks, start);
      NPC_LAUNCH(ctx);
    }
  }
  NPC_TRY(stage_mark(ctx, "paint_count"));
  NPC_TRY(each([&](const DevCatalog* a, const DevCatalog* b, int64_t off, bool rf) {
    return a->dtype == 1 ? paint_scatter<ASSIGN, double, T>(ctx, cat_pair<double>(a, b), weight_power, rf, sc, g,
                                                            brick + off, rank + off, start, rec, meta)
                         : paint_scatter<ASSIGN, float, T>(ctx, cat_pair<float>(a, b), weight_power, rf, sc, g,
                                                           brick + off, rank + off, start, rec, meta);
  }));
  NPC_TRY(stage_mark(ctx, "paint_scatter"));
  const int slot = weight_power == 1 ? SC_MAXW_F : SC_MAXW_N;
  switch (g.bs) {
    case 4: NPC_TRY((launch_tiles<ASSIGN, T, 4>(ctx, rec, meta, start, nbricks, nphase, sc, slot, tiles))); break;
    case 8: NPC_TRY((launch_tiles<ASSIGN, T, 8>(ctx, rec, meta, start, nbricks, nphase, sc, slot, tiles))); break;
    default: NPC_TRY((launch_tiles<ASSIGN, T, 16>(ctx, rec, meta, start, nbricks, nphase, sc, slot, tiles)));
  }
  NPC_TRY(stage_mark(ctx, "paint_tiles"));
  const int sub = (m.periodic && weight_power == 1) ? 1 : 0;
  return launch_fold<T>(ctx, tiles, g, nphase, sc, sub, mesh_a, mesh_b);
}

// Partial sums of one or two catalogues (types 0 float, 1 double) in one launch.
void launch_cat_partials(const void* wd, const void* nd, int64_t n_d, int type_d, const void* wr, const void* nr,
                         int64_t n_r, int type_r, int ncat, int nblk, double* pd, double* pr, cudaStream_t st) {
  auto run = [&](auto* t, auto* u) {
    using T = std::remove_pointer_t<decltype(t)>;
    using U = std::remove_pointer_t<decltype(u)>;
    k_cat_partials<T, U><<<dim3(nblk, ncat), RED_THREADS, 0, st>>>((const T*)wd, (const T*)nd, n_d, (const U*)wr,
                                                                   (const U*)nr, n_r, pd, pr);
  };
  float* f = nullptr;
  double* d = nullptr;
  if (type_d == 1) type_r == 1 ? run(d, d) : run(d, f);
  else type_r == 1 ? run(f, d) : run(f, f);
}

// Scalars of a cross spectrum from those of tracers A and B: the normalisation sqrt(I22^A I22^B)
// in the I22 slot, no shot noise, and the tracers' own values for the output (layout in npc.h).
__global__ void k_cross_scalars(const double* __restrict__ sa, const double* __restrict__ sb, double* __restrict__ sx) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int i = 0; i < SC_COUNT; ++i) sx[i] = 0.0;
  sx[SC_ALPHA] = sa[SC_ALPHA];
  sx[SC_I22] = sqrt(sa[SC_I22] * sb[SC_I22]);
  sx[SC_I33] = sb[SC_ALPHA];
  sx[SC_N0] = 0.0;
  sx[SC_S3] = sa[SC_I22];
  sx[SC_SUMWG] = sb[SC_I22];
  sx[SC_SUMWR] = sa[SC_SUMWG];
  sx[SC_SUMW2] = sb[SC_SUMWG];
}

// Scalars of a three-tracer bispectrum: tracer 1's values with I33 replaced by the geometric mean
// (I33^1 I33^2 I33^3)^(1/3) (the normalisation of the cross bispectra, Sec. 6 reading) and S3 = 0
// (no shot noise is subtracted from the raw cross estimates).
__global__ void k_cross3_scalars(const double* __restrict__ s1, const double* __restrict__ s2,
                                 const double* __restrict__ s3, double* __restrict__ sx) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  for (int i = 0; i < SC_COUNT; ++i) sx[i] = s1[i];
  sx[SC_I33] = cbrt(s1[SC_I33] * s2[SC_I33] * s3[SC_I33]);
  sx[SC_S3] = 0.0;
}

}  // namespace

npc_status launch_cross3_scalars(npc_ctx* ctx, const double* s1, const double* s2, const double* s3, double* sx) {
  k_cross3_scalars<<<1, 32, 0, ctx->stream>>>(s1, s2, s3, sx);
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

npc_status launch_cross_scalars(npc_ctx* ctx, const double* sa, const double* sb, double* sx) {
  k_cross_scalars<<<1, 32, 0, ctx->stream>>>(sa, sb, sx);
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

npc_status launch_catalog_scalars(npc_ctx* ctx, const DevCatalog& d, const DevCatalog* r, double box,
                                  double* dev_scalars) {
  const int64_t nmax = std::max<int64_t>(d.n, r ? r->n : 0);
  const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>((nmax + RED_CHUNK - 1) / RED_CHUNK, 4 * ctx->num_sms));
  double* part;
  NPC_TRY(ws_get(ctx, "scalars.part", sizeof(double) * NSUM * 4 * ctx->num_sms * 2, (void**)&part));
  double* part_r = part + (size_t)NSUM * nblk;
  launch_cat_partials(d.w, d.nbar, d.n, d.dtype, r ? r->w : nullptr, r ? r->nbar : nullptr, r ? r->n : 0,
                      r ? r->dtype : d.dtype, r ? 2 : 1, nblk, part, part_r, ctx->stream);
  NPC_LAUNCH(ctx);
  k_cat_final<<<1, 2 * NSUM * 32, 0, ctx->stream>>>(part, part_r, nblk, r ? 1 : 0, box, dev_scalars);
  NPC_LAUNCH(ctx);
  return NPC_OK;
}

npc_status launch_paint(npc_ctx* ctx, const DevCatalog& d, const DevCatalog* r, const npc_mesh_spec& m,
                        int weight_power, int prec, const double* dev_scalars, void* mesh_a, void* mesh_b,
                        bool sorted) {
  const bool any_double = d.dtype == 1 || (r && r->dtype == 1);
  if (prec == NPC_PREC_FP64) {
    if (m.assign == 2) return paint_impl<2, double>(ctx, d, r, m, weight_power, dev_scalars, mesh_a, mesh_b, sorted);
    return paint_impl<3, double>(ctx, d, r, m, weight_power, dev_scalars, mesh_a, mesh_b, sorted);
  }
  // records keep the fraction s - floor(s) (< 1) in float32 in the mixed path
  (void)any_double;
  if (m.assign == 2) return paint_impl<2, float>(ctx, d, r, m, weight_power, dev_scalars, mesh_a, mesh_b, sorted);
  return paint_impl<3, float>(ctx, d, r, m, weight_power, dev_scalars, mesh_a, mesh_b, sorted);
}

// ---------------------------------------------------------------------------------------------
// Allocation-free catalogue scalars.
//
// Some callers cannot call cudaMalloc at all: a host framework that owns every byte of device
// memory through its own pool (a raw allocation would sit outside its accounting), a plugin that
// is only handed device pointers, or a latency-bound loop where the implicit synchronisation of an
// allocation stalls the pipeline.  This entry point serves them: it reuses the reduction kernels
// above, but its scratch (the per-block partial sums and the 16 scalar slots) lives in a
// file-scope device array instead of context workspace, so the call allocates nothing.
// ---------------------------------------------------------------------------------------------
#include <cuda.h>

#include <mutex>

namespace {

constexpr int NOALLOC_CHUNK = 4096;            // objects reduced by one block
constexpr int NOALLOC_MAX_BLOCKS = 8192;       // blocks per catalogue
constexpr int64_t NOALLOC_MAX_OBJECTS = (int64_t)NOALLOC_CHUNK * NOALLOC_MAX_BLOCKS;  // 33,554,432
constexpr size_t NOALLOC_PART = (size_t)NOALLOC_MAX_BLOCKS * NSUM;                     // per catalogue

// 2 catalogues x 8192 blocks x 6 sums + 16 scalar slots, doubles: 786,560 bytes, resident on every
// device that loads this library until the process exits.
static __device__ __align__(256) double g_noalloc_scratch[2 * NOALLOC_PART + SC_COUNT];

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mutex;

// Address of the static array per device, remembered together with the identity of the context it
// was looked up in: a cudaDeviceReset (or another context made current) gives the device a new
// context in which the array may sit elsewhere, so a changed context id triggers a new look-up.
struct NoallocSlot {
  double* ptr = nullptr;
  unsigned long long ctx_id = 0;
  bool ctx_known = false;
};
NoallocSlot g_noalloc_slot[NOALLOC_MAX_DEVICES];

// Identity of the calling thread's current context, through driver entry points the runtime hands
// out (no link-time dependence on the driver library).  False when there is no current context or
// the entry points are unavailable; the caller then looks the address up again on every call.
bool current_context_id(unsigned long long* id) {
  static decltype(&cuCtxGetCurrent) get_current = nullptr;
  static decltype(&cuCtxGetId) get_id = nullptr;
  static bool resolved = false;
  if (!resolved) {
    resolved = true;
    cudaDriverEntryPointQueryResult q1, q2;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", (void**)&get_current, 12000, cudaEnableDefault, &q1) !=
            cudaSuccess || q1 != cudaDriverEntryPointSuccess)
      get_current = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", (void**)&get_id, 12000, cudaEnableDefault, &q2) !=
            cudaSuccess || q2 != cudaDriverEntryPointSuccess)
      get_id = nullptr;
    cudaGetLastError();
  }
  if (!get_current || !get_id) return false;
  CUcontext c = nullptr;
  if (get_current(&c) != CUDA_SUCCESS || !c) return false;
  return get_id(c, id) == CUDA_SUCCESS;
}

npc_status noalloc_err(char* err, size_t errlen, npc_status s, const char* msg) {
  if (err && errlen) {
    std::strncpy(err, msg, errlen - 1);
    err[errlen - 1] = '\0';
  }
  return s;
}

}  // namespace

extern "C" npc_status npc_catalog_scalars_noalloc(const npc_catalog* data, const npc_catalog* randoms, double box,
                                                  double* out_device, void* cuda_stream, char* err, size_t errlen) {
  if (err && errlen) err[0] = '\0';
  if (!data || !out_device) return noalloc_err(err, errlen, NPC_ERR_INVALID_ARG, "data and out_device are required");
  const npc_catalog* cats[2] = {data, randoms};
  for (int c = 0; c < 2; ++c) {
    const npc_catalog* k = cats[c];
    if (!k) continue;
    if (k->n < 0 || (k->n > 0 && !k->pos) || (k->dtype != 0 && k->dtype != 1))
      return noalloc_err(err, errlen, NPC_ERR_INVALID_ARG, "malformed catalogue");
    if (!k->on_device)
      return noalloc_err(err, errlen, NPC_ERR_INVALID_ARG, "catalogue arrays must be device pointers (on_device = 1)");
    if (k->n > NOALLOC_MAX_OBJECTS)
      return noalloc_err(err, errlen, NPC_ERR_INVALID_ARG,
                         "catalogue larger than 33554432 objects, the capacity of the static scratch");
    if (c == 1 && k->n > 0 && !k->nbar) return noalloc_err(err, errlen, NPC_ERR_INVALID_ARG, "randoms need nbar");
  }
  if (!randoms && !(box > 0.0)) return noalloc_err(err, errlen, NPC_ERR_INVALID_ARG, "periodic scalars need box > 0");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
    cudaGetLastError();
    return noalloc_err(err, errlen, NPC_ERR_CUDA, "no usable current CUDA device");
  }
  double* scratch;
  {
    // Set-up per device and context, with that device current: host code cannot take the address
    // of a __device__ array directly, so ask the runtime for it (done on the first call on a
    // device, and again only after that device's context has changed).
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    NoallocSlot& slot = g_noalloc_slot[dev];
    unsigned long long id = 0;
    const bool known = current_context_id(&id);
    if (!slot.ptr || !known || !slot.ctx_known || slot.ctx_id != id) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) {
        cudaGetLastError();
        slot = NoallocSlot{};
        return noalloc_err(err, errlen, NPC_ERR_CUDA, "cudaGetSymbolAddress of the static scratch failed");
      }
      slot.ptr = static_cast<double*>(p);
      // the look-up makes the device's primary context current when none was
      slot.ctx_known = current_context_id(&slot.ctx_id);
    }
    scratch = slot.ptr;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int64_t nmax = std::max<int64_t>(data->n, randoms ? randoms->n : 0);
  const int nblk = (int)std::max<int64_t>(1, (nmax + NOALLOC_CHUNK - 1) / NOALLOC_CHUNK);
  double* part_d = scratch;
  double* part_r = scratch + NOALLOC_PART;
  double* sc = scratch + 2 * NOALLOC_PART;
  // every partial that k_cat_final reads is written by this call's k_cat_partials (blocks past the
  // end of a catalogue write zeros), so nothing needs clearing first
  launch_cat_partials(data->w, data->nbar, data->n, data->dtype, randoms ? randoms->w : nullptr,
                      randoms ? randoms->nbar : nullptr, randoms ? randoms->n : 0,
                      randoms ? randoms->dtype : data->dtype, randoms ? 2 : 1, nblk, part_d, part_r, st);
  k_cat_final<<<1, 2 * NSUM * 32, 0, st>>>(part_d, part_r, nblk, randoms ? 1 : 0, box, sc);
  // peek, not get: an error that the caller's earlier asynchronous work left pending is reported
  // as this call's failure but stays pending for the caller to read
  cudaError_t e = cudaPeekAtLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(out_device, sc, 8 * sizeof(double), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return noalloc_err(err, errlen, NPC_ERR_CUDA, cudaGetErrorString(e));
  return NPC_OK;
}
