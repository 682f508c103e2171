// FP64 recheck of marked rows (the fast scorers mark a row by writing the
// reserved label 255 when their rigorous error bound cannot guarantee the
// FP64 decision, or the log posteriors to 1e-5).
//
// A warp scans 32 labels at a time; for every marked row the whole warp
// recomputes the joint log scores from the stored features and the FP64
// tables exactly as defined (Sec. 4):
//   multinomial  s_c = log pi_c + sum_j x_j log theta_cj
//   Gaussian     s_c = log pi_c - 1/2 sum_j [log(2 pi var_cj) + (x_j - mu_cj)^2 / var_cj]
// then the label (lowest index among the maxima), the top-2 margin and the
// log posteriors, in FP64, rounded to FP32 only for the outputs.
#include <cuda_fp16.h>
#include <math.h>

#include "device.cuh"
#include "internal.cuh"
#include "seg.cuh"

namespace nbg {

// FP64 tables of one model
struct RModel {
  int C;
  const double* p0;       // log theta | mu
  const double* p1;       // var
  const double* log_pi;
  const double* gconst;
};

// one stored matrix and its outputs
struct RView {
  const char* X;
  int64_t ld;   // elements
  int F;
  const int64_t* ovf_ptr;
  const uint16_t* ovf_col;
  const uint16_t* ovf_add;
  const int8_t* row_exp;
  uint8_t* label;
  float* margin;
  float* logpost;
  const int32_t* cols;   // feature j is stored column cols[j] (nullptr: column j)
};

template <int DT>
__device__ __forceinline__ double load_x(const char* rp, int j, double scale) {
  if (DT == NB_F32) return (double)reinterpret_cast<const float*>(rp)[j];
  if (DT == NB_U16) return (double)reinterpret_cast<const uint16_t*>(rp)[j];
  if (DT == NB_U8) return (double)reinterpret_cast<const uint8_t*>(rp)[j];
  if (DT == NB_BF16) {
    const uint32_t b = reinterpret_cast<const uint16_t*>(rp)[j];
    return (double)__uint_as_float(b << 16);
  }
  const uint16_t b = reinterpret_cast<const uint8_t*>(rp)[j];
  return (double)e4m3x2_to_f32(b).x * scale;
}

// Sums of classes c0 .. c0 + nc - 1 (nc <= CB) over the features j = lane,
// lane + 32, ... of one row, in ascending order per lane.  U features are
// loaded at a time, then their CB table entries together: the loads, not the
// FP64 additions, are what a marked row waits for (one feature at a time, 57
// marked rows of 4,096 counts took 130 us).
template <int DT, int KIND, int CB, int U>
__device__ __forceinline__ void recheck_sums(const RView& v, const RModel& md, const char* rp,
                                             double scale, int c0, int nc, double (&acc)[CB]) {
  const int lane = threadIdx.x & 31, F = v.F;
  const double* t0 = md.p0 + (int64_t)c0 * F;   // log theta | mu
  const double* t1 = KIND == NB_GAUSSIAN ? md.p1 + (int64_t)c0 * F : nullptr;
  for (int j0 = lane; j0 < F; j0 += 32 * U) {
    double x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + 32 * u;
      x[u] = j < F ? load_x<DT>(rp, v.cols ? v.cols[j] : j, scale) : 0.0;
    }
    double w[U][CB], z[KIND == NB_GAUSSIAN ? U : 1][KIND == NB_GAUSSIAN ? CB : 1];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = j0 + 32 * u;
      // a zero count adds nothing to a multinomial score (log theta is finite
      // for alpha > 0)
      const bool need = j < F && (KIND == NB_GAUSSIAN || x[u] != 0.0);
#pragma unroll
      for (int k = 0; k < CB; ++k) {
        w[u][k] = need && k < nc ? t0[(int64_t)k * F + j] : 0.0;
        if (KIND == NB_GAUSSIAN) z[u][k] = need && k < nc ? t1[(int64_t)k * F + j] : 1.0;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j0 + 32 * u >= F || (KIND == NB_MULTINOMIAL && x[u] == 0.0)) continue;
#pragma unroll
      for (int k = 0; k < CB; ++k) {
        if (KIND == NB_MULTINOMIAL) {
          acc[k] = fma(x[u], w[u][k], acc[k]);
        } else {
          const double dx = x[u] - w[u][k];
          acc[k] += dx * dx / z[u][k];
        }
      }
    }
  }
}

// The whole warp sums classes c0 .. c0 + nc - 1 (nc <= CB) of row r of v; their
// scores go to s_sh.  The row's value is loaded once for the CB classes; per class
// the lane's sum and the butterfly over the lanes are those of one class at a
// time, so that CB changes no bit.
template <int DT, int KIND, int CB, int U>
__device__ __forceinline__ void recheck_classes(const RView& v, const RModel& md, int64_t r,
                                                int c0, int nc, double* s_sh) {
  const int lane = threadIdx.x & 31;
  constexpr int es = DT == NB_F32 ? 4 : ((DT == NB_U16 || DT == NB_BF16) ? 2 : 1);
  const char* rp = v.X + r * v.ld * es;
  const double scale = (DT == NB_FP8E4M3 && v.row_exp) ? ldexp(1.0, (int)v.row_exp[r]) : 1.0;
  double acc[CB];
#pragma unroll
  for (int k = 0; k < CB; ++k) acc[k] = 0.0;
  recheck_sums<DT, KIND, CB, U>(v, md, rp, scale, c0, nc, acc);
  if (DT == NB_U8 && KIND == NB_MULTINOMIAL && v.ovf_ptr) {
    const double* lt = md.p0 + (int64_t)c0 * v.F;
    for (int64_t e = v.ovf_ptr[r] + lane; e < v.ovf_ptr[r + 1]; e += 32) {
      const int j = v.ovf_col[e];
      if (j >= v.F) continue;
      const double add = (double)v.ovf_add[e];
#pragma unroll
      for (int k = 0; k < CB; ++k)
        if (k < nc) acc[k] = fma(add, lt[(int64_t)k * v.F + j], acc[k]);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
    for (int k = 0; k < CB; ++k) acc[k] += __shfl_xor_sync(0xFFFFFFFFu, acc[k], off);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < CB; ++k) {
      const int c = c0 + k;
      if (k < nc)
        s_sh[c] = KIND == NB_MULTINOMIAL ? md.log_pi[c] + acc[k] : md.gconst[c] - 0.5 * acc[k];
    }
  }
}

// The whole warp writes row r's outputs from its scores.
__device__ __forceinline__ void recheck_finish(const RView& v, const RModel& md, int64_t r,
                                               int want_lp, const double* s_sh) {
  const int lane = threadIdx.x & 31;
  // the lanes share the classes: arg-max (lowest index among the maxima; class
  // 0 when its score is NaN or none is a number), second best, log-sum-exp (an
  // FP64 exponential per class: one lane alone took them one after another)
  double b = -INFINITY;
  int best = 0x7FFFFFFF;
  for (int c = lane; c < md.C; c += 32) {
    const double sc = s_sh[c];
    if (sc > b || (sc == b && c < best)) {
      b = sc;
      best = c;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double ob = __shfl_xor_sync(0xFFFFFFFFu, b, off);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, best, off);
    if (ob > b || (ob == b && oi < best)) {
      b = ob;
      best = oi;
    }
  }
  if (best >= md.C || s_sh[0] != s_sh[0]) best = 0;
  const double sb = s_sh[best];
  double second = -INFINITY, sum = 0.0;
  for (int c = lane; c < md.C; c += 32) {
    if (c != best && s_sh[c] > second) second = s_sh[c];
    if (want_lp) sum += exp(s_sh[c] - sb);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    second = fmax(second, __shfl_xor_sync(0xFFFFFFFFu, second, off));
    sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
  }
  if (lane == 0) {
    v.label[r] = (uint8_t)best;
    v.margin[r] = (float)(sb - second);
  }
  if (want_lp) {
    const double lse = sb + log(sum);
    for (int c = lane; c < md.C; c += 32) v.logpost[r * md.C + c] = (float)(s_sh[c] - lse);
  }
}

// The whole warp recomputes row r of v with model md.
template <int DT, int KIND, int CB, int U>
__device__ __forceinline__ void recheck_row(const RView& v, const RModel& md, int64_t r,
                                            int want_lp, double* s_sh) {
  for (int c0 = 0; c0 < md.C; c0 += CB)
    recheck_classes<DT, KIND, CB, U>(v, md, r, c0, md.C - c0 < CB ? md.C - c0 : CB, s_sh);
  __syncwarp();
  recheck_finish(v, md, r, want_lp, s_sh);
  __syncwarp();
}

struct RArgs {
  RView v;
  RModel md;
  int64_t n;
  int want_lp;
  int counted;   // *n_rechecked already holds the marked rows (skip when 0, do not add)
  int rows;      // rows per warp chunk (a power of two <= 32)
  unsigned long long* n_rechecked;
};

// CB classes and U features in flight: 16 table entries per lane either way.
template <int DT, int KIND, int CB>
__global__ void __launch_bounds__(256) k_recheck(const RArgs a) {
  __shared__ double s_sh[8][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_wait();   // the scorer's labels and mark count
  if (a.counted && *a.n_rechecked == 0ull) return;   // the scorer marked no row
  // a warp takes chunks of a.rows rows (lanes below a.rows read a label) and
  // recomputes the chunk's marked rows one after another; small calls use short
  // chunks, so that densely marked rows spread over many warps
  const int64_t nwarps = (int64_t)gridDim.x * 8;
  unsigned long long cnt = 0;
  for (int64_t base = ((int64_t)blockIdx.x * 8 + warp) * a.rows; base < a.n;
       base += nwarps * a.rows) {
    const int64_t row = base + lane;
    const bool f = lane < a.rows && row < a.n && a.v.label[row] == kLabelRecheck;
    unsigned m = __ballot_sync(0xFFFFFFFFu, f);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      recheck_row<DT, KIND, CB, 16 / CB>(a.v, a.md, base + src, a.want_lp, s_sh[warp]);
      ++cnt;
    }
  }
  if (lane == 0 && cnt && a.n_rechecked && !a.counted) atomicAdd(a.n_rechecked, cnt);
}

using RKernel = void (*)(RArgs);
template <int DT>
static RKernel recheck_kernel(int C) {
  return C == 2 ? (RKernel)k_recheck<DT, NB_MULTINOMIAL, 2> : (RKernel)k_recheck<DT, NB_MULTINOMIAL, 8>;
}
static RKernel recheck_kernel(nb_kind kind, nb_dtype dt, int C) {
  if (kind == NB_GAUSSIAN) return k_recheck<NB_F32, NB_GAUSSIAN, 4>;
  switch (dt) {
    case NB_U8: return recheck_kernel<NB_U8>(C);
    case NB_U16: return recheck_kernel<NB_U16>(C);
    case NB_F32: return recheck_kernel<NB_F32>(C);
    case NB_BF16: return recheck_kernel<NB_BF16>(C);
    default: return recheck_kernel<NB_FP8E4M3>(C);
  }
}

static RView view_of(const void* X, int64_t ld, int F, const nb_aux* aux, const ScoreOut& o) {
  RView v{};
  v.X = static_cast<const char*>(X);
  v.ld = ld;
  v.F = F;
  v.ovf_ptr = aux ? aux->ovf_ptr : nullptr;
  v.ovf_col = aux ? aux->ovf_col : nullptr;
  v.ovf_add = aux ? aux->ovf_add : nullptr;
  v.row_exp = aux ? aux->row_exp : nullptr;
  v.label = o.label;
  v.margin = o.margin;
  v.logpost = o.logpost;
  return v;
}

nb_status launch_recheck(const nb_model* m, const void* X, nb_dtype dt, int64_t n, int64_t ld,
                         const nb_aux* aux, const ScoreOut& o, cudaStream_t st) {
  // NB_RECHECK_OFF still recomputes the rows a scorer could not compute at all
  // (see NB_RECHECK_OFF in the header); in that mode nothing else is marked
  if (n == 0) return NB_OK;
  RArgs a{};
  a.v = view_of(X, ld, m->F, aux, o);
  a.md = RModel{m->C, m->d.p0, m->d.p1, m->d.log_pi, m->d.gconst};
  a.n = n;
  a.want_lp = o.want_lp;
  a.counted = o.counted ? 1 : 0;
  a.n_rechecked = reinterpret_cast<unsigned long long*>(o.n_rechecked);
  // rows per warp chunk: 32, halved while the call has fewer chunks than the
  // grid has warps (down to one row per warp)
  const int64_t cap = (int64_t)num_sms() * 8;   // blocks of 8 warps
  int rows = 32;
  while (rows > 1 && (n + rows - 1) / rows < cap * 8) rows >>= 1;
  a.rows = rows;
  const int64_t blocks = ((n + rows - 1) / rows + 7) / 8;
  count_launch();
  NB_TRY_CUDA(launch_pdl(recheck_kernel(m->kind, dt, m->C), dim3((unsigned)(blocks < cap ? blocks : cap)), dim3(256), 0,
                         st, a),
              "k_recheck launch");
  return NB_OK;
}

// ---------------------------------------------------------------------------
// listed rows (FP8 and BF16 rows of 2^17 and more counts): a block per row, its
// warps two classes each
// ---------------------------------------------------------------------------
// The bits of k_recheck, which gives a marked row to one warp: with few rows that
// warp's loads, one batch of features after another for all classes, are what the
// call waits for (BF16, F = 2,048, C = 16: 64 batches one after another, here 8).
struct RListArgs {
  RView v;
  RModel md;
  const int* list;
  const unsigned long long* count;
  int cap, want_lp;
};

template <int DT>
__global__ void __launch_bounds__(256) k_recheck_list(const RListArgs a) {
  __shared__ double s_sh[kTcMaxC];
  const int warp = threadIdx.x >> 5;
  pdl_wait();   // the scorer's list
  const int n = (int)min(*a.count, (unsigned long long)a.cap);
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const int64_t r = a.list[i];
    for (int c0 = 2 * warp; c0 < a.md.C; c0 += 16)
      recheck_classes<DT, NB_MULTINOMIAL, 2, 8>(a.v, a.md, r, c0, a.md.C - c0 < 2 ? 1 : 2, s_sh);
    __syncthreads();
    if (warp == 0) recheck_finish(a.v, a.md, r, a.want_lp, s_sh);
    __syncthreads();
  }
}

nb_status launch_recheck_list(const nb_model* m, const void* X, nb_dtype dt, int64_t ld,
                              const nb_aux* aux, const ScoreOut& o, const int* list,
                              const unsigned long long* count, int cap, cudaStream_t st) {
  RListArgs a{view_of(X, ld, m->F, aux, o), RModel{m->C, m->d.p0, m->d.p1, m->d.log_pi, m->d.gconst},
              list, count, cap, o.want_lp};
  const int grid = num_sms() * 2;
  count_launch();
  NB_TRY_CUDA(launch_pdl(dt == NB_BF16 ? k_recheck_list<NB_BF16> : k_recheck_list<NB_FP8E4M3>,
                         dim3((unsigned)(cap < grid ? cap : grid)), dim3(256), 0, st, a),
              "k_recheck_list launch");
  return NB_OK;
}

// ---------------------------------------------------------------------------
// segmented recheck: warps take contiguous ranges of 32-row chunks of each
// group list of a batch and walk its groups
// ---------------------------------------------------------------------------
constexpr int kRSegLists = 3;

struct RSegArgs {
  struct List {
    const SegGroup* groups;
    const SegHeader* hdr;
    int model0;            // its models start here in md
    int two;               // two-class models
  } list[kRSegLists];
  RModel md[2 * kSegMaxModels];   // the two-class models and the many-class ones
  int n_lists, F, want_lp;
  const unsigned long long* marks;   // rows that the scorers marked
};

template <int DT>
__global__ void __launch_bounds__(256) k_recheck_seg(const RSegArgs a) {
  __shared__ double s_sh[8][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_wait();   // the scorers' labels and mark count
  if (*a.marks == 0ull) return;
  const long long W = (long long)gridDim.x * 8, w = (long long)blockIdx.x * 8 + warp;
  for (int f = 0; f < a.n_lists; ++f) {
    const RSegArgs::List& L = a.list[f];
    const int n_groups = L.hdr->n_groups;
    const long long chunks = L.hdr->chunks;
    const long long c0 = chunks * w / W, c1 = chunks * (w + 1) / W;
    if (c0 >= c1 || n_groups == 0) continue;
    const SegGroup* gr = L.groups;
    int g = seg_find(n_groups, c0, [gr](int i) { return gr[i].chunk0; });
    for (long long c = c0; c < c1; ++c) {
      while (g + 1 < n_groups && gr[g + 1].chunk0 <= c) ++g;
      const SegGroup& G = gr[g];
      const long long base = (c - G.chunk0) * 32;
      const long long row = base + lane;
      const bool mk = row < G.n && G.label[row] == kLabelRecheck;
      unsigned m = __ballot_sync(0xFFFFFFFFu, mk);
      if (!m) continue;
      RView v;
      v.cols = nullptr;
      v.X = G.X;
      v.F = a.F;
      constexpr int es = DT == NB_F32 ? 4 : ((DT == NB_U16 || DT == NB_BF16) ? 2 : 1);
      v.ld = G.ld_bytes / es;
      v.ovf_ptr = G.ovf_ptr;
      v.ovf_col = G.ovf_col;
      v.ovf_add = G.ovf_add;
      v.row_exp = G.row_exp;
      v.label = G.label;
      v.margin = G.margin;
      v.logpost = G.logpost;
      const RModel& md = a.md[L.model0 + G.model];
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        if (L.two)
          recheck_row<DT, NB_MULTINOMIAL, 2, 8>(v, md, base + src, a.want_lp, s_sh[warp]);
        else
          recheck_row<DT, NB_MULTINOMIAL, 8, 2>(v, md, base + src, a.want_lp, s_sh[warp]);
      }
    }
  }
}

nb_status launch_recheck_seg(const RecheckList* lists, int n_lists, nb_dtype dt, int F, int want_lp,
                             const unsigned long long* marks, cudaStream_t st) {
  RSegArgs a{};
  int at = 0;
  for (int f = 0; f < n_lists && a.n_lists < kRSegLists; ++f) {
    const RecheckList& l = lists[f];
    if (l.n_models < 1) continue;
    // the many-class lists share their models' order but not their number: each
    // list brings its own entries
    if (at + l.n_models > 2 * kSegMaxModels) {
      set_error("recheck: too many models");
      return NB_EINVAL;
    }
    RSegArgs::List& L = a.list[a.n_lists++];
    L = {l.groups, l.hdr, at, l.models[0]->C == 2 ? 1 : 0};
    for (int i = 0; i < l.n_models; ++i) {
      const nb_model* m = l.models[i];
      a.md[at++] = RModel{m->C, m->d.p0, m->d.p1, m->d.log_pi, m->d.gconst};
    }
  }
  if (a.n_lists == 0) return NB_OK;
  a.F = F;
  a.want_lp = want_lp;
  a.marks = marks;
  void (*k)(RSegArgs) = dt == NB_U8     ? k_recheck_seg<NB_U8>
                        : dt == NB_F32  ? k_recheck_seg<NB_F32>
                        : dt == NB_U16  ? k_recheck_seg<NB_U16>
                        : dt == NB_BF16 ? k_recheck_seg<NB_BF16>
                                        : k_recheck_seg<NB_FP8E4M3>;
  count_launch();
  NB_TRY_CUDA(launch_pdl(k, dim3((unsigned)(num_sms() * 4)), dim3(256), 0, st, a),
              "k_recheck_seg launch");
  return NB_OK;
}

}  // namespace nbg

namespace nbg {

// ---------------------------------------------------------------------------
// group-wise recheck: rows in the files' order, each with the model of its
// size group and that model's opcode selection (feature t = column cols[t] of
// the full histogram), the arithmetic of recheck_row unchanged
// ---------------------------------------------------------------------------
struct RGwArgs {
  const unsigned char* X;
  int64_t ld;
  int64_t n;
  const int64_t* sizes;
  int64_t bin_bytes;
  int n_bins, k;
  const int32_t* model_of;   // size group -> model slot
  const int32_t* cols;       // n_models x k
  RModel md[kSegMaxModels];
  uint8_t* label;
  float* margin;
  float* logpost;
  int want_lp;
  int counted;   // *n_rechecked already holds the marked rows (skip when 0, do not add)
  unsigned long long* n_rechecked;
};

__global__ void __launch_bounds__(256) k_recheck_gw(const RGwArgs a) {
  __shared__ double s_sh[8][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pdl_wait();   // the scorer's labels and mark count
  if (a.counted && *a.n_rechecked == 0ull) return;   // the scorer marked no row
  const int64_t nwarps = (int64_t)gridDim.x * 8;
  unsigned long long cnt = 0;
  for (int64_t base = ((int64_t)blockIdx.x * 8 + warp) * 32; base < a.n; base += nwarps * 32) {
    const int64_t row = base + lane;
    const bool f = row < a.n && a.label[row] == kLabelRecheck;
    unsigned m = __ballot_sync(0xFFFFFFFFu, f);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      const int64_t r = base + src;
      long long sz = a.sizes[r];
      sz = sz < 0 ? 0 : sz;
      long long bin = sz / a.bin_bytes;
      if (bin > a.n_bins - 1) bin = a.n_bins - 1;
      const int g = a.model_of[bin];
      RView v;
      v.X = reinterpret_cast<const char*>(a.X);
      v.ld = a.ld;
      v.F = a.k;
      v.ovf_ptr = nullptr;
      v.ovf_col = nullptr;
      v.ovf_add = nullptr;
      v.row_exp = nullptr;
      v.label = a.label;
      v.margin = a.margin;
      v.logpost = a.logpost;
      v.cols = a.cols + (int64_t)g * a.k;
      recheck_row<NB_U8, NB_MULTINOMIAL, 2, 8>(v, a.md[g], r, a.want_lp, s_sh[warp]);
      ++cnt;
    }
  }
  if (lane == 0 && cnt && a.n_rechecked && !a.counted) atomicAdd(a.n_rechecked, cnt);
}

nb_status launch_recheck_gw(const unsigned char* X, int64_t ld, int64_t n, const int64_t* sizes,
                            int64_t bin_bytes, int n_bins, int k, const int32_t* model_of,
                            const int32_t* cols, const nb_model* const* models, int n_models,
                            uint8_t* label, float* margin, float* logpost, int want_lp,
                            int64_t* n_rechecked, bool counted, cudaStream_t st) {
  if (n == 0) return NB_OK;
  RGwArgs a{};
  a.X = X;
  a.ld = ld;
  a.n = n;
  a.sizes = sizes;
  a.bin_bytes = bin_bytes;
  a.n_bins = n_bins;
  a.k = k;
  a.model_of = model_of;
  a.cols = cols;
  for (int i = 0; i < n_models && i < kSegMaxModels; ++i) {
    const nb_model* m = models[i];
    a.md[i] = RModel{m->C, m->d.p0, m->d.p1, m->d.log_pi, m->d.gconst};
  }
  a.label = label;
  a.margin = margin;
  a.logpost = logpost;
  a.want_lp = want_lp;
  a.counted = counted ? 1 : 0;
  a.n_rechecked = reinterpret_cast<unsigned long long*>(n_rechecked);
  const int64_t chunks = (n + 255) / 256;
  const int64_t cap = (int64_t)num_sms() * 8;
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_recheck_gw, dim3((unsigned)(chunks < cap ? chunks : cap)), dim3(256),
                         0, st, a),
              "k_recheck_gw launch");
  return NB_OK;
}

}  // namespace nbg
