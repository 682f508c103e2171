// Internal declarations of the nbgpu library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "nbgpu.h"

namespace nbg {

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
void set_error(const char* fmt, ...);
nb_status cuda_status(cudaError_t e, const char* what);

#define NB_TRY_CUDA(expr, what)                          \
  do {                                                   \
    cudaError_t e__ = (expr);                            \
    if (e__ != cudaSuccess) return ::nbg::cuda_status(e__, what); \
  } while (0)

// device status word bits (model / call error words)
enum : int {
  ST_BAD_LABEL = 1,       // a label outside [0, C)
  ST_BAD_VALUE = 2,       // negative, fractional or non-finite count
  ST_TIMEOUT = 4,         // a bounded wait gave up
  ST_BAD_TABLE = 8,       // non-finite parameter table
  ST_OVF_RANGE = 16,      // overflow column outside [0, F)
  ST_BAD_ROUTE = 32       // routing / gather input: negative size, group, label or column out of range
};

constexpr uint8_t kLabelRecheck = 255;   // internal marker in label[]

// Dynamic shared memory above this size is requested through the kernel's
// max-dynamic-shared-memory attribute; the default limit of 48 KB covers
// dynamic and static shared memory together, and the kernels declare a few
// static barriers.
constexpr int kSmemOptIn = 32 * 1024;

inline int elem_size(nb_dtype d) {
  switch (d) {
    case NB_F32: return 4;
    case NB_U16: return 2;
    case NB_BF16: return 2;
    case NB_U8: return 1;
    case NB_FP8E4M3: return 1;
  }
  return 0;
}

// ---------------------------------------------------------------------------
// two-class scalars produced on the device by the fit (one struct in HBM)
// ---------------------------------------------------------------------------
struct C2Header {
  float b;            // log pi_1 - log pi_0 (FP32)
  float maxabs;       // max_j |Delta_j| of the FP32 table
  float inv_scale;    // 2^-S: fixed-point step of the integer Delta table
  float maxabs_q;     // max_j |Delta_j| bound used with the fixed-point table
  double b64;         // FP64 b
  int32_t S;          // Delta_q = round(Delta * 2^S), |Delta_q| <= 2^22
  int32_t pad;
};

// fixed-point scalars of the many-class tensor-core tables (one struct in HBM)
struct TcHeader {
  float scale;        // 2^-S: step of the fixed-point weights Q = round(w 2^S)
  float tau_unit;     // 2^-(S+1): largest rounding error of one weight
  int32_t S;
  int32_t pad;
};

// tensor-core scorer limits: classes, features
constexpr int kTcMaxC = 64;
// classes of a Gaussian model's FP32 tables per feature: blocks of 4 (C <= 4)
// or 16, the class blocks of the CUDA-core scorer
__host__ __device__ constexpr int gauss_cpad(int C) { return C <= 4 ? 4 : ((C + 15) / 16) * 16; }
constexpr int kTcMaxF = 32768;
constexpr int kTcgMaxF = 8192;   // Gaussian tensor-core tables
constexpr int kTcgFS = 32;       // ... features per stage (a multiple of 8 dividing 32)

// scalars of the Gaussian tensor-core tables (one struct in HBM)
struct TcgHeader {
  int bad;            // a weight outside the FP16 range: the tables are not used
  float wsum;         // sum_j (max_c |B_cj| + max_c |A_cj|), rounded up
};

// Two-class U16 and BF16 rows of up to 16 vectors of 16 bytes take the exact sums of
// k_score2_fix.
inline bool fix_rows(int F) { return F <= 16 * 8; }

// Two-class FP8 rows of fewer than 32 vectors of 16 bytes take five limbs of Delta (see
// k_score2_u8).
inline bool fp8_narrow(int F) { return F <= 31 * 16; }

// ---------------------------------------------------------------------------
// model (library-owned)
// ---------------------------------------------------------------------------
struct ModelDev {
  // all pointers into one device allocation
  uint64_t* counts;    // C x F      (multinomial)
  uint64_t* nc;        // C
  double* p0;          // C x F      log theta (multinomial) | mu (Gaussian)
  double* p1;          // C x F      var (Gaussian)
  double* log_pi;      // C
  double* gconst;      // C          Gaussian: log pi_c - 1/2 sum_j log(2 pi var_cj);
                       //            multinomial: log(N_c + alpha F)
  int* status;         // 1 int: ST_* bits raised while fitting (cleared by each fit)
  int* sstatus;        // 1 int: ST_* bits raised by scoring calls (kept until
                       // nb_model_check reports them)
  unsigned long long* fin;   // 4 words of the two-class fit finish (zero between fits)
  // two-class multinomial tables
  C2Header* c2;        // 1
  float* delta;        // F_pad      FP32 Delta, plain order
  int32_t* delta_q;    // F_pad      fixed-point Delta
  int2* delta_pr;      // F_pad      fixed-point Delta, eight bits finer (step 2^-(S+8)), and in
                       //            FP32 what it leaves of Delta
  int32_t* delta_p;    // 2 F_pad    the same one after the other for short 16-bit rows
                       //            (fix_rows), else nullptr
  uint4* limbs;        // 3 * nvec8  int8 limbs of delta_q, interleaved (u8 path), then
                       //            F_pad packed words (limb l in byte l)
  uint4* limbs5;       // 5 * nvec8  the three limbs and two more (step 2^-(S+15)) for narrow FP8
                       //            rows (fp8_narrow), else nullptr
  float4* il[3];       // interleaved FP32 quads for 4/8/16 elements per vector
  // general-C tables (CUDA-core scorer)
  float* w;            // C x F_pad  centred weights log theta_cj - mean_c log theta_cj
  float* bias;         // C          log pi_c
  float* wmax;         // 1          max |w|
  // many-class tensor-core tables (3 <= C <= kTcMaxC), else nullptr
  uint8_t* tc_w;       // ceil(F/64) stages x 3*Cp x 64 FP16 limbs (MMA operand layout)
  int32_t* tc_q;       // C x F fixed-point weights
  TcHeader* tc_hdr;    // 1
  double* wmean;       // F          mean_c log theta_cj
  char* tc_scratch;    // tc_scratch_bytes(C): heavy rows of one scoring call (ScoreScratch)
  // Gaussian FP32 tables
  float* g_nms;        // -mu / sd: F_pad x gauss_cpad(C), feature-major (past F and C: 0)
  float* g_isd;        // same layout, 1 / sd
  float* g_const;      // 2C         gconst in FP32, then a4_c = sum_j g_nms^2
  // Gaussian tensor-core tables (3 <= C <= kTcMaxC, F <= kTcgMaxF), else nullptr;
  // the FP16 limbs of B and A go to tc_w
  float* tcg_kc;       // C          K_c
  float* tcg_ctr;      // F rounded up to kTcgFS: centres m_j
  float* tcg_bmax;     // ... max_c |B_cj|
  float* tcg_amax;     // ... max_c |A_cj|
  TcgHeader* tcg_hdr;  // 1
};

// The model's scratch for one scoring call at a time: whether a call holds it,
// and the stream and end of the last call that did.
struct ScoreSlot {
  std::mutex mu;
  bool busy = false, used = false;
  unsigned long long stream_id = 0;
  cudaEvent_t end = nullptr;
};

}  // namespace nbg

struct nb_model {
  nb_kind kind;
  int C;
  int F;
  int F_pad;        // F rounded up to a multiple of 32
  int nvec8;        // F_pad / 16 (u8 vectors of 16 bytes)
  double alpha;
  double var_smoothing;
  int device;
  nb_tile_config tile;   // scorer kernel configuration (autotuned or set)
  cudaStream_t stream;   // stream of the fit
  void* mem;
  size_t mem_bytes;
  void* work;            // fit workspace kept between re-fits (see FitScratch), or nullptr
  size_t work_bytes;
  bool refit;            // the model has been fitted: later fits keep their workspace
  mutable nbg::ScoreSlot slot;
  nbg::ModelDev d;
};

namespace nbg {

// launchers implemented in fit.cu / score2.cu / recheck.cu / pack.cu
nb_status launch_fit_multinomial(nb_model* m, const void* X, nb_dtype dt,
                                 int64_t n, int64_t ld, const int32_t* y,
                                 const nb_aux* aux, const double* log_prior_dev,
                                 cudaStream_t st);
// Gaussian fit (gauss_fit.cu): device scratch it needs, and the launches
// (log priors, when given, already stand in the model's log_pi)
size_t gauss_scratch_bytes(int64_t n, int F, int C);
nb_status launch_fit_gaussian(nb_model* m, const float* X, int64_t n, int64_t ld,
                              const int32_t* y, bool prior_given, void* scratch,
                              cudaStream_t st);

// Device scratch of a scoring call: the model's own when no other call can be
// using it on the GPU (the last one was on this stream or has finished), else,
// and on a stream being captured, memory allocated and freed in stream order.
class ScoreScratch {
 public:
  ScoreScratch(const nb_model* m, cudaStream_t st) : m_(m), st_(st) {}
  ~ScoreScratch() { release(); }
  nb_status take(size_t bytes, char* kept, size_t kept_bytes, char** p);
  nb_status release();

 private:
  const nb_model* m_;
  cudaStream_t st_;
  unsigned long long id_ = 0;
  void* own_ = nullptr;
  bool slot_ = false;
};

// Device scratch of a fit: the model's own workspace, kept between re-fits
// (up to kKeepWork bytes; larger ones, the first fit's and those of a stream
// being captured are allocated and freed in stream order).
constexpr size_t kKeepWork = size_t(64) << 20;
class FitScratch {
 public:
  FitScratch(nb_model* m, cudaStream_t st) : m_(m), st_(st) {}
  ~FitScratch() { release(); }
  nb_status take(size_t bytes, void** p);
  nb_status release();

 private:
  nb_model* m_;
  cudaStream_t st_;
  void* own_ = nullptr;
};

struct ScoreOut {
  uint8_t* label;
  float* margin;
  float* logpost;
  int64_t* n_rechecked;
  int want_lp;
  int recheck;
  bool counted = false;   // the scorer counted its marked rows into n_rechecked
};

// 16-byte aligned rows (base and pitch)
inline bool c2_aligned(const void* X, nb_dtype dt, int64_t ld) {
  return (reinterpret_cast<uintptr_t>(X) & 15) == 0 && (ld * elem_size(dt)) % 16 == 0;
}
nb_status launch_score2(const nb_model* m, const void* X, nb_dtype dt,
                        int64_t n, int64_t ld, const nb_aux* aux,
                        const ScoreOut& o, cudaStream_t st);
nb_status launch_fit2_pipe(nb_model* m, const void* X, nb_dtype dt, int64_t n, int64_t ld,
                           const int32_t* y, const nb_aux* aux, cudaStream_t st);
nb_status launch_counts_rows(nb_model* m, const void* X, nb_dtype dt, int64_t n, int64_t ld,
                             const int32_t* y, const nb_aux* aux, cudaStream_t st);
struct S2Args;
nb_status launch_score2_pipe(const S2Args& a, nb_dtype dt, int stages, int rows_per_stage,
                             int rows_per_warp, int stage_entries, cudaStream_t st);
nb_status launch_score_general(const nb_model* m, const void* X, nb_dtype dt,
                               int64_t n, int64_t ld, const nb_aux* aux,
                               const ScoreOut& o, cudaStream_t st);
nb_status launch_recheck(const nb_model* m, const void* X, nb_dtype dt,
                         int64_t n, int64_t ld, const nb_aux* aux,
                         const ScoreOut& o, cudaStream_t st);
// The listed rows (FP8 or BF16, at most cap) in FP64.
nb_status launch_recheck_list(const nb_model* m, const void* X, nb_dtype dt, int64_t ld,
                              const nb_aux* aux, const ScoreOut& o, const int* list,
                              const unsigned long long* count, int cap, cudaStream_t st);

// many-class tensor-core scorer (score_tc.cu)
inline int tc_classes_padded(int C) { return (C + 15) / 16 * 16; }
inline size_t tc_w_bytes(int C, int F) {
  return (size_t)((F + 63) / 64) * 3 * tc_classes_padded(C) * 128;
}
inline bool tc_tables(nb_kind kind, int C, int F) {
  return kind == NB_MULTINOMIAL && C >= 3 && C <= kTcMaxC && F <= kTcMaxF;
}
size_t tc_scratch_bytes(int C);
bool tc_eligible(const nb_model* m, nb_dtype dt, const void* X, int64_t ld);
nb_status launch_derive_tc(nb_model* m, cudaStream_t st);

// many-class Gaussian tensor-core scorer (score_tcg.cu)
inline size_t tcg_w_bytes(int C, int F) {
  return (size_t)((F + kTcgFS - 1) / kTcgFS) * tc_classes_padded(C) * (16 * kTcgFS);
}
inline bool tcg_tables(nb_kind kind, int C, int F) {
  return kind == NB_GAUSSIAN && C >= 3 && C <= kTcMaxC && F <= kTcgMaxF;
}
bool tcg_eligible(const nb_model* m, const void* X, int64_t ld, int recheck);
nb_status launch_derive_tcg(nb_model* m, cudaStream_t st);
nb_status launch_score_tcg(const nb_model* m, const float* X, int64_t n, int64_t ld,
                           const ScoreOut& o, cudaStream_t st);
nb_status launch_score_tc(const nb_model* m, const void* X, nb_dtype dt, int64_t n, int64_t ld,
                          const nb_aux* aux, const ScoreOut& o, cudaStream_t st);

int num_sms();

// Launch k with programmatic stream serialisation (see pdl_wait()).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}
// process-wide count of kernels this library has launched
void count_launch();

// ST_* bits of a status word -> status code and error text (first error wins)
nb_status status_from_word(int w);

// Looks up the allocation-free re-fit's device scratch for the current device
// (noalloc.cu); under lazy module loading this is what commits it.
nb_status noalloc_scratch_prepare();

}  // namespace nbg
