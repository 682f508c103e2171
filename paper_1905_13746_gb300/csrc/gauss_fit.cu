// Gaussian fit (real-valued features): per-class means and maximum-likelihood
// variances by two passes over the rows, the mean and then the squared
// deviations about it, with eps = var_smoothing * max_j Var(x_.j) added to
// every variance.
//
// What bounds it.  FP64 runs at about two lanes per clock and SM on this part
// (an FP32 operation at 128), so a warp holds the sums of a run of rows in three
// FP32 numbers, the sum, its error and the error of that, the first two joined
// exactly (Knuth's two-sum, and the FMA product error): the run's sum is then
// exact to about 2^-70 of its largest term and is rounded once, to FP64, for ~8
// (pass 1) and ~22 (pass 2) packed FP32 instructions a value, where FP64 sums of each
// class and of all rows cost eight slots of the FP64 pipe, i.e. 512 of an FP32 one.
// Sums of runs are added in FP64.  (Two numbers a sum, about 48 bits, took the fit of
// 64,000 rows at C = 64, F = 256 110 us instead of 123, 447,355 rows at C = 3, F = 18
// 86 instead of 99, and left the variances 1e-14 off, where FP64 sums are 4e-16 off and
// these 2e-16.  Three numbers a sum in the reductions too, without FP64: 127 and 121.)
// The additions are written as intrinsics: a product that the compiler fused into one
// of them would break the error terms.  A run whose FP32 sum overflows is summed again
// in FP64 by itself (400,000 rows of such values x 32 features: 55 ms while a feature's
// lane walked all rows instead).  The overall variance behind eps comes from the class
// moments (n_c, mu_c, var_c), not from sums of its own.
//
// Pass 2 sums (x - K)^2 with K = fl32(mean) of the class and feature, and
// var = S2 / n_c - (mean - K)^2; x - K is formed exactly as a pair.  Values
// are scaled by the power of two of the class's largest |x| of the feature, so
// that no square overflows, and none that matters underflows: scaled, either
// some value lies at least 1/4 from the mean or all are at least 1/4 in
// magnitude, where differences are multiples of 2^-26.
//
// Split.  A block takes `rows` rows x 32 features (lane = feature: 128-byte
// row segments).  It sorts its rows by class in shared memory (stable, so the
// order of every sum is fixed), deals the sorted rows evenly to its 8 warps,
// and each warp sums runs of one class in registers; a class that several
// warps share is joined in warp order.  So no class count or class size leaves
// warps idle, and a (chunk, class, feature) partial is 12 bytes (an FP64 sum and
// the largest |x|).  Chunks are sized for four blocks per SM; the partials are
// reduced by a block per class and 32 features in a fixed order: the results are
// the same bits on every run, and the same with any scratch (nb_refit and the
// allocation-free re-fit).
// C = 64, F = 256: re-fit on 64,000 rows (65.5 MB), scoring of 200,000 and
// reading the parameters: 4.90 -> 0.84 ms, of which the fit was 3.45 ms of
// device time with FP64 sums in shared memory, 32-row chunks (266 MB of
// partials, mapped anew by every call) and a one-block finish, and is 0.12 ms
// now (passes 37 and 52 us, reductions 8 and 19, finish 10, tensor-core tables
// 16, each launch by itself); C = 2, F = 64, 2,000 rows: the fit 30 us.
#include <math.h>

#include "device.cuh"
#include "internal.cuh"

namespace nbg {

constexpr int kGfWarps = 8;
constexpr int kGfMaxRows = 2048;              // rows per chunk (the sort's shared memory)

struct GfArgs {
  const float* X;
  int64_t ld, n;
  int F, C, rows;
  unsigned nchunk;      // chunks of rows; block: (feature tile) x nchunk + chunk
  const int32_t* y;
  double* part0;        // C x F sums of chunk 0 ...
  double* part;         // ... and of chunks 1, 2, ...
  float* amax0;         // C x F max |x| of chunk 0 (pass 1)
  float* amax;          // ... and of the others
  const double* mean;   // C x F (pass 2)
  const float* scale;   // C x F power-of-two scale (pass 2)
  unsigned long long* nc;
  int* status;
};

// Two rows at a time, one in each half of a packed instruction (the same roundings, half
// the issue slots).
__device__ __forceinline__ uint64_t neg2(uint64_t a) {
  return f32x2_fma(a, f32x2_pack(-1.f, -1.f), f32x2_pack(-0.f, -0.f));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  return f32x2_fma(b, f32x2_pack(-1.f, -1.f), a);
}
// s = a + b rounded, e = what the rounding lost (Knuth)
__device__ __forceinline__ void two_sum2(uint64_t a, uint64_t b, uint64_t& s, uint64_t& e) {
  s = f32x2_add(a, b);
  const uint64_t t = sub2(s, a);
  e = f32x2_add(sub2(a, sub2(s, t)), sub2(b, t));
}

// One run's sums of this lane's feature, of its even and its odd rows.
struct GfAcc {
  uint64_t s = 0, e = 0, l = 0;
  unsigned int m = 0u;   // pass 1: max of |x| as bits (NaN above infinity)
  __device__ __forceinline__ double sum() const;
};

// The FP64 sum of a run, or of several.
struct GfSum {
  double s = 0.0;
  unsigned int m = 0u;
};
__device__ __forceinline__ void gf_join(GfSum& a, const GfSum& b) {
  a.s += b.s;
  a.m = max(a.m, b.m);
}

// Both halves joined (as exactly as a row is), then one rounding to FP64.
__device__ __forceinline__ double GfAcc::sum() const {
  float s0, s1, e0, e1, l0, l1, t[3];
  f32x2_unpack(s, s0, s1);
  f32x2_unpack(e, e0, e1);
  f32x2_unpack(l, l0, l1);
  auto two_sum = [](float a, float b, float& r) {
    const float c = __fadd_rn(a, b), d = __fsub_rn(c, a);
    r = __fadd_rn(__fsub_rn(a, __fsub_rn(c, d)), __fsub_rn(b, d));
    return c;
  };
  s0 = two_sum(s0, s1, t[0]);
  e0 = two_sum(e0, e1, t[1]);
  e0 = two_sum(e0, t[0], t[2]);
  l0 = __fadd_rn(__fadd_rn(l0, l1), __fadd_rn(t[1], t[2]));
  return (double)s0 + ((double)e0 + (double)l0);
}

// Pass 1: x the two rows' values.  Pass 2: x their values, scaled; nK = -K twice.
template <int PASS>
__device__ __forceinline__ void gf_add(GfAcc& a, uint64_t x, uint64_t nK) {
  uint64_t r, t;
  if (PASS == 1) {
    two_sum2(a.s, x, a.s, r);
    two_sum2(a.e, r, a.e, t);
    a.l = f32x2_add(a.l, t);
  } else {
    // d + dl = x - K exactly; its square is p + q + w + u, u of w's product error and dl^2
    uint64_t d, dl, t2, t3, t4;
    two_sum2(x, nK, d, dl);
    const uint64_t p = f32x2_mul(d, d), q = f32x2_fma(d, d, neg2(p));
    const uint64_t d2 = f32x2_add(d, d), w = f32x2_mul(d2, dl);
    const uint64_t u = f32x2_fma(dl, dl, f32x2_fma(d2, dl, neg2(w)));
    two_sum2(a.s, p, a.s, r);
    two_sum2(a.e, r, a.e, t2);
    two_sum2(a.e, q, a.e, t3);
    two_sum2(a.e, w, a.e, t4);
    a.l = f32x2_add(a.l, f32x2_add(f32x2_add(t2, t3), f32x2_add(t4, u)));
  }
}

template <int PASS>
__device__ __forceinline__ void gf_store(const GfArgs& a, unsigned chunk, int c, int j,
                                         const GfSum& v) {
  if (j >= a.F) return;
  const int64_t at = (int64_t)c * a.F + j;
  const int64_t off = chunk == 0 ? at : ((int64_t)(chunk - 1) * a.C) * a.F + at;
  (chunk == 0 ? a.part0 : a.part)[off] = v.s;
  if (PASS == 1) {
    (chunk == 0 ? a.amax0 : a.amax)[off] = __uint_as_float(v.m);
    if (v.m >= 0x7F800000u) atomicOr(a.status, ST_BAD_VALUE);
  }
}

template <int PASS>
__global__ void __launch_bounds__(kGfWarps * 32) k_gauss_pass(const GfArgs a) {
  extern __shared__ __align__(16) unsigned char gf_sm[];
  __shared__ uint16_t s_order[kGfMaxRows];
  __shared__ int s_off[kTcMaxC + 1];
  __shared__ GfSum s_frag[2 * kGfWarps][32];
  __shared__ int s_fc[2 * kGfWarps];
  uint16_t* cnt = reinterpret_cast<uint16_t*>(gf_sm);   // [label group][class]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int C = a.C;
  // one grid dimension: the others end at 65,535, fewer than the tiles of 2.1M features
  const unsigned chunk = blockIdx.x % a.nchunk, ft = blockIdx.x / a.nchunk;
  const int64_t r0 = (int64_t)chunk * a.rows;
  const int nr = (int)min((int64_t)a.rows, a.n - r0);
  const int ng = (nr + 31) / 32;
  const int j = (int)ft * 32 + lane;
  for (int k = threadIdx.x; k < ng * C; k += kGfWarps * 32) cnt[k] = 0;
  if (threadIdx.x < 2 * kGfWarps) s_fc[threadIdx.x] = -1;
  pdl_wait();   // the cleared counters, or the means of pass 1
  __syncthreads();

  // ---- stable counting sort of the chunk's rows by class
  auto label_of = [&](int g) {
    const int r = 32 * g + lane;
    int c = r < nr ? a.y[r0 + r] : -1;
    if (r < nr && (c < 0 || c >= C)) {
      if (PASS == 1 && ft == 0) atomicOr(a.status, ST_BAD_LABEL);
      c = -1;
    }
    return c;
  };
  for (int g = warp; g < ng; g += kGfWarps) {
    const int c = label_of(g);
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    if (c >= 0 && lane == __ffs(peers) - 1) cnt[g * C + c] = (uint16_t)__popc(peers);
  }
  __syncthreads();
  if (threadIdx.x < 64) {   // counts per label group -> exclusive offsets inside the class
    int run = 0;
    if (threadIdx.x < C) {
#pragma unroll 4
      for (int g = 0; g < ng; ++g) {
        const int t = cnt[g * C + threadIdx.x];
        cnt[g * C + threadIdx.x] = (uint16_t)run;
        run += t;
      }
      if (PASS == 1 && ft == 0 && run) atomicAdd(&a.nc[threadIdx.x], (unsigned long long)run);
    }
    // exclusive scan of the class totals over both warps
    int inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= o) inc += v;
    }
    if (threadIdx.x < C) s_off[threadIdx.x + 1] = inc;
    if (threadIdx.x == 0) s_off[0] = 0;
  }
  __syncthreads();
  if (threadIdx.x >= 32 && threadIdx.x < C) s_off[threadIdx.x + 1] += s_off[32];
  __syncthreads();
  for (int g = warp; g < ng; g += kGfWarps) {
    const int c = label_of(g);
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    if (c >= 0)
      s_order[s_off[c] + cnt[g * C + c] + __popc(peers & ((1u << lane) - 1u))] =
          (uint16_t)(32 * g + lane);
  }
  __syncthreads();

  // ---- this warp's share of the sorted rows, run by run
  const int total = s_off[C];
  const int a0 = total * warp / kGfWarps, a1 = total * (warp + 1) / kGfWarps;
  const bool in = j < a.F;
  const float* xb = a.X + r0 * a.ld + (in ? j : 0);
  int c = 0;
  for (int pos = a0; pos < a1;) {
    while (s_off[c + 1] <= pos) ++c;
    const int start = pos, end = min(a1, s_off[c + 1]);
    float K = 0.f, sc = 1.f;
    if (PASS == 2 && in) {
      const int64_t at = (int64_t)c * a.F + j;
      sc = a.scale[at];
      K = (float)a.mean[at] * sc;
    }
    const uint64_t nK = f32x2_pack(-K, -K);
    GfAcc v;
    constexpr int U = 8;   // rows in flight per lane
    auto rows = [&](const float (&x)[U], int n) {   // a row past the run: nothing to add
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        if (u >= n) break;
        if (PASS == 1) {
          v.m = max(v.m, max(__float_as_uint(x[u]) & 0x7FFFFFFFu, __float_as_uint(x[u + 1]) & 0x7FFFFFFFu));
          gf_add<PASS>(v, f32x2_pack(x[u], x[u + 1]), nK);
        } else {
          gf_add<PASS>(v, f32x2_pack(__fmul_rn(x[u], sc), u + 1 < n ? __fmul_rn(x[u + 1], sc) : K), nK);
        }
      }
    };
    for (; pos + U <= end; pos += U) {
      float x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = in ? __ldg(xb + (int64_t)s_order[pos + u] * a.ld) : 0.f;
      rows(x, U);
    }
    if (pos < end) {
      float x[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        x[u] = in && pos + u < end ? __ldg(xb + (int64_t)s_order[pos + u] * a.ld) : 0.f;
      rows(x, end - pos);
      pos = end;
    }
    GfSum sum{v.sum(), v.m};
    if (PASS == 1 && in && !isfinite(sum.s) && v.m < 0x7F800000u) {
      // finite values whose FP32 sum overflowed (above 2^127): the run again in FP64
      sum.s = 0.0;
      for (int k = start; k < end; ++k) sum.s += (double)__ldg(xb + (int64_t)s_order[k] * a.ld);
    }
    if (start == s_off[c] && end == s_off[c + 1]) {
      gf_store<PASS>(a, chunk, c, j, sum);
    } else {   // the class is shared with a neighbouring warp: slot 0 begins, slot 1 ends a share
      const int slot = 2 * warp + (start == a0 ? 0 : 1);
      s_frag[slot][lane] = sum;
      if (lane == 0) s_fc[slot] = c;
    }
  }
  // classes without rows in this chunk
  for (int k = warp; k < C; k += kGfWarps)
    if (s_off[k] == s_off[k + 1]) gf_store<PASS>(a, chunk, k, j, GfSum{});
  __syncthreads();
  if (warp == 0) {   // join the shared classes' pieces in order
    GfSum v;
    int cur = -1;
    for (int k = 0; k < 2 * kGfWarps; ++k) {
      const int fc = s_fc[k];
      if (fc < 0) continue;
      if (fc != cur) {
        if (cur >= 0) gf_store<PASS>(a, chunk, cur, j, v);
        v = s_frag[k][lane];
        cur = fc;
      } else {
        gf_join(v, s_frag[k][lane]);
      }
    }
    if (cur >= 0) gf_store<PASS>(a, chunk, cur, j, v);
  }
}

// ---------------------------------------------------------------------------
// reductions: block (features 32 ft .., class c), 8 warps over the chunks
// ---------------------------------------------------------------------------
struct GfRed {
  GfArgs a;
  double* mu;               // C x F
  double* var;              // C x F
  float* scale;             // C x F
  unsigned int* done_ft;    // per 32-feature tile: blocks that wrote their variances
  unsigned int* done_c;     // per class: finished blocks of the finish kernel
  unsigned long long* vmax; // bits of max_j Var(x_.j)
  TcgHeader* tcg_hdr;       // cleared here when present
};

// the sum of this lane's (class, feature) over all chunks (valid in warp 0)
template <int PASS>
__device__ __forceinline__ GfSum gf_reduce(const GfRed& r, int c, int j) {
  __shared__ GfSum sh[kGfWarps][32];
  const GfArgs& a = r.a;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  GfSum v;
  if (j < a.F) {
    const int64_t at = (int64_t)c * a.F + j, step = (int64_t)a.C * a.F;
#pragma unroll 4
    for (int k = warp; k < (int)a.nchunk; k += kGfWarps) {
      const int64_t off = k == 0 ? at : (int64_t)(k - 1) * step + at;
      v.s += (k == 0 ? a.part0 : a.part)[off];
      if (PASS == 1) v.m = max(v.m, __float_as_uint((k == 0 ? a.amax0 : a.amax)[off]));
    }
  }
  sh[warp][lane] = v;
  __syncthreads();
  if (warp == 0)
    for (int k = 1; k < kGfWarps; ++k) gf_join(v, sh[k][lane]);
  return v;
}

__global__ void __launch_bounds__(kGfWarps * 32) k_gauss_mean(const GfRed r) {
  const GfArgs& a = r.a;
  const int c = blockIdx.y, j = blockIdx.x * 32 + (threadIdx.x & 31);
  pdl_wait();
  if (threadIdx.x == 0) {   // counters of the kernels that follow
    if (c == 0) r.done_ft[blockIdx.x] = 0u;
    if (blockIdx.x == 0) r.done_c[c] = 0u;
    if (blockIdx.x == 0 && c == 0) {
      *r.vmax = 0ull;
      if (r.tcg_hdr) r.tcg_hdr->bad = 0;
    }
  }
  const GfSum v = gf_reduce<1>(r, c, j);
  if (threadIdx.x >= 32 || j >= a.F) return;
  const double nc = (double)a.nc[c];
  const double mean = nc > 0 ? v.s / nc : 0.0;
  const int64_t at = (int64_t)c * a.F + j;
  r.mu[at] = mean;
  // 2^-floor(log2 max |x|), from the exponent field (subnormal maxima: 2^126)
  const int ex = max((int)(v.m >> 23), 1);   // biased exponent
  r.scale[at] = v.m == 0u ? 1.f
                          : (ex >= 254 ? __uint_as_float(0x00400000u)   // 2^-127
                                       : __uint_as_float((unsigned)(254 - ex) << 23));
}

__global__ void __launch_bounds__(kGfWarps * 32) k_gauss_var(const GfRed r) {
  const GfArgs& a = r.a;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.y, j = blockIdx.x * 32 + lane;
  pdl_wait();
  const GfSum v = gf_reduce<2>(r, c, j);
  if (warp == 0 && j < a.F) {
    const int64_t at = (int64_t)c * a.F + j;
    const double nc = (double)a.nc[c], mean = r.mu[at], sc = (double)r.scale[at];
    const double dk = mean - (double)(float)mean;
    double var = nc > 0 ? v.s / (nc * sc * sc) - dk * dk : 0.0;
    if (var < 0.0) var = 0.0;
    __stcg(&r.var[at], var);
  }
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&r.done_ft[blockIdx.x], 1u) == (unsigned)(a.C - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the tile's last block: Var(x_.j) of all rows from the class moments
  __shared__ double sh[kGfWarps][32];
  double t = 0.0;
  if (j < a.F)
    for (int k = warp; k < a.C; k += kGfWarps) t += (double)a.nc[k] * r.mu[(int64_t)k * a.F + j];
  sh[warp][lane] = t;
  __syncthreads();
  double mu_all = 0.0;
  for (int k = 0; k < kGfWarps; ++k) mu_all += sh[k][lane];
  mu_all /= (double)a.n;
  __syncthreads();
  t = 0.0;
  if (j < a.F)
    for (int k = warp; k < a.C; k += kGfWarps) {
      const double d = r.mu[(int64_t)k * a.F + j] - mu_all;
      t += (double)a.nc[k] * (__ldcg(&r.var[(int64_t)k * a.F + j]) + d * d);
    }
  sh[warp][lane] = t;
  __syncthreads();
  if (warp == 0) {
    double m2 = 0.0;
    for (int k = 0; k < kGfWarps; ++k) m2 += sh[k][lane];
    m2 /= (double)a.n;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m2 = fmax(m2, __shfl_xor_sync(0xFFFFFFFFu, m2, o));
    // non-negative doubles order like their bit patterns
    if (lane == 0) atomicMax(r.vmax, (unsigned long long)__double_as_longlong(m2));
  }
}

// ---------------------------------------------------------------------------
// finish: var += eps, log prior, Gaussian constants, FP32 tables.  Block (256
// features, class); classes past C clear the tables' padding.  sum_j log(2 pi
// var_cj) takes one logarithm per warp: the mantissas of 2 pi var are
// multiplied and the exponents added (an FP64 logarithm costs some 60
// multiplications).
// ---------------------------------------------------------------------------
struct GfFin {
  int F, F_pad, C, CP, jt, prior_given;
  int64_t n;
  double var_smoothing;
  const unsigned long long* nc;
  const unsigned long long* vmax;
  const double* mu;
  double* var;
  double* log_pi;
  double* gconst;
  float* g_nms;
  float* g_isd;
  float* g_const;
  double* part;           // per class and tile: sum of logs, sum of m^2 v
  unsigned int* done_c;
  int* status;
};

__global__ void __launch_bounds__(256) k_gauss_finish(const GfFin a) {
  const int c = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = blockIdx.x * 256 + threadIdx.x;
  pdl_wait();
  float nm32 = 0.f, is32 = 0.f;
  double m = 1.0, s4 = 0.0;
  int e = 0;
  if (c < a.C && j < a.F) {
    const double eps = a.var_smoothing * __longlong_as_double((long long)*a.vmax);
    const int64_t at = (int64_t)c * a.F + j;
    const double v = a.var[at] + eps;
    if (!(v > 0.0) || !isfinite(v)) atomicOr(a.status, ST_BAD_TABLE);
    a.var[at] = v;
    is32 = (float)rsqrt(v);
    nm32 = (float)(-a.mu[at] * (double)is32);
    m = frexp(6.283185307179586476925 * v, &e);   // zero, infinities and NaN pass through
    s4 = (double)nm32 * (double)nm32;
  }
  if (j < a.F_pad) {   // feature-major, gauss_cpad(C) classes per feature
    a.g_nms[(int64_t)j * a.CP + c] = nm32;
    a.g_isd[(int64_t)j * a.CP + c] = is32;
  }
  if (c >= a.C) return;
  // 32 mantissas in [1/2, 1): the product stays above 2^-33
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m *= __shfl_xor_sync(0xFFFFFFFFu, m, o);
    e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
    s4 += __shfl_xor_sync(0xFFFFFFFFu, s4, o);
  }
  __shared__ double sl[8], s4s[8];
  if (lane == 0) {
    sl[warp] = log(m) + (double)e * 0.693147180559945309417;
    s4s[warp] = s4;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double t = 0.0, t4 = 0.0;
  for (int w = 0; w < 8; ++w) {
    t += sl[w];
    t4 += s4s[w];
  }
  if (a.jt > 1) {   // the class's last block adds the tiles in order
    __stcg(&a.part[2 * ((int64_t)c * a.jt + blockIdx.x)], t);
    __stcg(&a.part[2 * ((int64_t)c * a.jt + blockIdx.x) + 1], t4);
    __threadfence();
    if (atomicAdd(&a.done_c[c], 1u) != (unsigned)(a.jt - 1)) return;
    __threadfence();
    t = t4 = 0.0;
    for (int k = 0; k < a.jt; ++k) {
      t += __ldcg(&a.part[2 * ((int64_t)c * a.jt + k)]);
      t4 += __ldcg(&a.part[2 * ((int64_t)c * a.jt + k) + 1]);
    }
  }
  a.g_const[a.C + c] = (float)t4;
  if (!a.prior_given) {
    if (a.nc[c] == 0) atomicOr(a.status, ST_BAD_LABEL);
    a.log_pi[c] = a.nc[c] ? log((double)a.nc[c]) - log((double)a.n) : 0.0;
  }
  a.gconst[c] = a.log_pi[c] - 0.5 * t;
  a.g_const[c] = (float)a.gconst[c];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// Rows per chunk: four blocks per SM of this part (152, whatever the device: the
// chunks fix the order of the sums) over chunks x feature tiles, but at least
// eight rows per class (smaller chunks write more partials than they read
// rows), at least 64 rows, 512 past 65,536 rows (the bound on the scratch that
// the allocation-free re-fit's limit relies on), and what the sort can hold.
// It depends on n, F and C alone, so that every caller sums in one order.
static int64_t gf_rows(int64_t n, int F, int C) {
  const int64_t nft = (F + 31) / 32, want = 4 * 152;
  int64_t rows = (n * nft + want - 1) / want;
  rows = (rows + 31) / 32 * 32;
  const int64_t least = n <= 65536 ? 64 : 512;
  if (rows < least) rows = least;
  if (rows < 8 * C) rows = (8 * C + 31) / 32 * 32;
  return rows < kGfMaxRows ? rows : kGfMaxRows;
}

size_t gauss_scratch_bytes(int64_t n, int F, int C) {
  const int64_t rows = gf_rows(n, F, C), nchunk = (n + rows - 1) / rows;
  const size_t cf = (size_t)C * F, jt = (F + 255) / 256;
  return (size_t)(nchunk - 1) * cf * 12 + 16 * (size_t)C * jt +
         sizeof(unsigned int) * ((size_t)(F + 31) / 32 + C) + 64;
}

nb_status launch_fit_gaussian(nb_model* m, const float* X, int64_t n, int64_t ld,
                              const int32_t* y, bool prior_given, void* scratch,
                              cudaStream_t st) {
  const int C = m->C, F = m->F;
  ModelDev& d = m->d;
  // nc and the status word follow one another in the model's allocation
  NB_TRY_CUDA(cudaMemsetAsync(d.nc, 0,
                              (size_t)(reinterpret_cast<char*>(d.status + 1) -
                                       reinterpret_cast<char*>(d.nc)),
                              st),
              "memset");
  const int64_t rows = gf_rows(n, F, C), nchunk = (n + rows - 1) / rows;
  const size_t cf = (size_t)C * F;
  const int nft = (F + 31) / 32, jt = (F + 255) / 256, CP = gauss_cpad(C);
  // scratch: sums and maxima of the chunks after the first, the finish
  // kernel's tile sums, counters.  The first chunk's go to the model's count
  // table (which a Gaussian model does not use) and, before the variances are
  // written there, to its variance table.
  char* s = static_cast<char*>(scratch);
  GfArgs a{};
  a.X = X;
  a.ld = ld;
  a.n = n;
  a.F = F;
  a.C = C;
  a.rows = (int)rows;
  a.nchunk = (unsigned)nchunk;
  a.y = y;
  a.part0 = reinterpret_cast<double*>(d.counts);
  a.amax0 = reinterpret_cast<float*>(d.p1);
  double* part = reinterpret_cast<double*>(s);
  s += 16 * (size_t)C * jt;
  a.part = reinterpret_cast<double*>(s);
  s += (size_t)(nchunk - 1) * cf * 8;
  a.amax = reinterpret_cast<float*>(s);
  s += (size_t)(nchunk - 1) * cf * 4;
  unsigned int* done = reinterpret_cast<unsigned int*>(s);
  // the scales wait in the 1/sd table, which the finish kernel writes
  float* scale = d.g_isd;
  a.mean = d.p0;
  a.scale = scale;
  a.nc = reinterpret_cast<unsigned long long*>(d.nc);
  a.status = d.status;
  GfRed r{a, d.p0, d.p1, scale, done, done + nft, d.fin, d.tcg_kc ? d.tcg_hdr : nullptr};
  const int smem = (int)(sizeof(uint16_t) * ((rows + 31) / 32) * C);
  const dim3 grid((unsigned)(nchunk * nft)), rgrid((unsigned)nft, (unsigned)C);
  const dim3 block(kGfWarps * 32);
  count_launch();
  k_gauss_pass<1><<<grid, block, smem, st>>>(a);
  NB_TRY_CUDA(cudaGetLastError(), "k_gauss_pass<1>");
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_gauss_mean, rgrid, block, 0, st, r), "k_gauss_mean");
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_gauss_pass<2>, grid, block, smem, st, a), "k_gauss_pass<2>");
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_gauss_var, rgrid, block, 0, st, r), "k_gauss_var");
  GfFin f{F, m->F_pad, C, CP, jt, prior_given ? 1 : 0, n, m->var_smoothing, a.nc, d.fin, d.p0,
          d.p1, d.log_pi, d.gconst, d.g_nms, d.g_isd, d.g_const, part, done + nft, d.status};
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_gauss_finish, dim3((unsigned)((m->F_pad + 255) / 256), (unsigned)CP),
                         dim3(256), 0, st, f),
              "k_gauss_finish");
  if (d.tcg_kc) return launch_derive_tcg(m, st);
  return NB_OK;
}

}  // namespace nbg
