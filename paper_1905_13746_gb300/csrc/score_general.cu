// CUDA-core scorers for any class count (Sec. 4 posterior and decision rule).
//
// Multinomial, C >= 2: s_c = log pi_c + sum_j x_j w_cj with the centred table
// w_cj = log theta_cj - mean_c log theta_cj (the per-feature shift is the same
// for every class, so it cancels in the label, the margin and the log
// posterior, and it keeps |w| small for the error bound).  A block scores 64
// files x 64 classes per pass as a register-tiled FP32 product over 32-feature
// chunks staged in shared memory; the epilogue takes the arg-max (lowest
// index among the maxima), the top-2 margin and the log-sum-exp.
//
// Gaussian: s_c = k_c - 1/2 sum_j (x_j - mu_cj)^2 / var_cj with
// k_c = log pi_c - 1/2 sum_j log(2 pi var_cj) from the FP64 fit.
//
// Both mark rows for the FP64 recheck when a rigorous bound on the FP32
// rounding error cannot guarantee the decision (or the log posteriors).
#include <cuda_fp16.h>
#include <math.h>

#include "device.cuh"
#include "internal.cuh"
#include "seg.cuh"

namespace nbg {

constexpr int GBM = 64;   // rows per tile
constexpr int GBK = 32;   // features per chunk
constexpr int GCB = 64;   // classes per pass

struct GArgs {
  const char* X;
  int64_t ld;        // elements
  int64_t n;
  int F, F_pad, C, dtype, aligned;
  const int64_t* ovf_ptr;
  const uint16_t* ovf_col;
  const uint16_t* ovf_add;
  const int8_t* row_exp;
  const float* w;      // C x F_pad
  const float* bias;   // C
  const float* wmax;
  const double* log_pi;
  uint8_t* label;
  float* margin;
  float* logpost;
  int want_lp, recheck;
  unsigned long long* marks;   // counts the rows marked for the recheck, or nullptr
  int* status;
};

// element j of a row as float (scalar path, any alignment)
__device__ __forceinline__ float gload1(int dt, const char* rp, int j) {
  switch (dt) {
    case NB_F32: return reinterpret_cast<const float*>(rp)[j];
    case NB_U16: return (float)reinterpret_cast<const uint16_t*>(rp)[j];
    case NB_U8: return (float)reinterpret_cast<const uint8_t*>(rp)[j];
    case NB_BF16: return __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(rp)[j] << 16);
    default: return e4m3x2_to_f32((uint16_t)reinterpret_cast<const uint8_t*>(rp)[j]).x;
  }
}

__device__ __forceinline__ void decode16(int dt, const uint4& x, float* v, int& cnt) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
  switch (dt) {
    case NB_F32:
      cnt = 4;
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = __uint_as_float(w[k]);
      break;
    case NB_U16:
      cnt = 8;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[2 * k] = u_field_to_f32(w[k], kSelU16Lo);
        v[2 * k + 1] = u_field_to_f32(w[k], kSelU16Hi);
      }
      break;
    case NB_BF16:
      cnt = 8;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[2 * k] = __uint_as_float(w[k] << 16);
        v[2 * k + 1] = __uint_as_float(w[k] & 0xFFFF0000u);
      }
      break;
    case NB_U8:
      cnt = 16;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int b = 0; b < 4; ++b) v[4 * k + b] = u_field_to_f32(w[k], sel_u8(b));
      break;
    default:
      cnt = 16;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float2 lo = e4m3x2_to_f32((uint16_t)(w[k] & 0xFFFFu));
        const float2 hi = e4m3x2_to_f32((uint16_t)(w[k] >> 16));
        v[4 * k] = lo.x;
        v[4 * k + 1] = lo.y;
        v[4 * k + 2] = hi.x;
        v[4 * k + 3] = hi.y;
      }
  }
}

// One tile of GBM rows starting at r0 (all class blocks, epilogue included).
__device__ __forceinline__ void gen_tile(const GArgs& a, int64_t r0, float* gsm) {
  float* Xs = gsm;                         // [GBK][GBM + 4]
  float* Ws = Xs + GBK * (GBM + 4);        // [GBK][GCB + 4]
  float* Ss = Ws + GBK * (GCB + 4);        // [GBM][C_pad]
  const int C_pad = ((a.C + 3) / 4) * 4;
  float* Ts = Ss + GBM * C_pad;            // [GBM]
  float* Tslot = Ts + GBM;                 // [GBM * 8] per-slot |x| sums
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int es = a.dtype == NB_F32 ? 4 : ((a.dtype == NB_U16 || a.dtype == NB_BF16) ? 2 : 1);
  const int epv = 16 / es;
  const int vpr = GBK / epv;               // vectors per row per chunk (2, 4 or 8)
  const float wmax = *a.wmax;
  float bmax = 0.f;
  for (int c = 0; c < a.C; ++c) bmax = fmaxf(bmax, fabsf(a.bias[c]));
  const int nchunk = (a.F + GBK - 1) / GBK;
  float tpart[2] = {0.f, 0.f};   // |x| sums of the (row, vector) slots this thread loads
  for (int cb = 0; cb < a.C; cb += GCB) {
    float run[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) run[i][j] = 0.f;
    for (int ch = 0; ch < nchunk; ++ch) {
      const int k0 = ch * GBK;
      // X tile -> Xs[k][row] (FP32)
      for (int s = 0, slot = tid; slot < GBM * vpr; ++s, slot += 256) {
        const int row = slot / vpr, vv = slot % vpr;
        const int64_t gr = r0 + row;
        float v[16];
        int cnt = epv;
        const int kb = k0 + vv * epv;
        if (gr < a.n) {
          const char* rp = a.X + gr * a.ld * es;
          if (a.aligned && kb + epv <= a.F) {
            decode16(a.dtype, ld_stream16(rp + (int64_t)kb * es), v, cnt);
          } else {
            for (int e = 0; e < epv; ++e) v[e] = kb + e < a.F ? gload1(a.dtype, rp, kb + e) : 0.f;
          }
          if (a.dtype == NB_FP8E4M3 && a.row_exp) {
            const float sc = exp2f((float)a.row_exp[gr]);
            for (int e = 0; e < epv; ++e) v[e] *= sc;
          }
        } else {
          for (int e = 0; e < epv; ++e) v[e] = 0.f;
        }
        float tsum = 0.f;
        for (int e = 0; e < epv; ++e) {
          Xs[(vv * epv + e) * (GBM + 4) + row] = v[e];
          tsum += fabsf(v[e]);
        }
        if (cb == 0) tpart[s] += tsum;
      }
      // W tile -> Ws[k][c]
      for (int slot = tid; slot < GCB * (GBK / 4); slot += 256) {
        const int c = slot / (GBK / 4), kq = slot % (GBK / 4);
        float4 wv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (cb + c < a.C)
          wv = *reinterpret_cast<const float4*>(a.w + (int64_t)(cb + c) * a.F_pad + k0 + kq * 4);
        Ws[(kq * 4 + 0) * (GCB + 4) + c] = wv.x;
        Ws[(kq * 4 + 1) * (GCB + 4) + c] = wv.y;
        Ws[(kq * 4 + 2) * (GCB + 4) + c] = wv.z;
        Ws[(kq * 4 + 3) * (GCB + 4) + c] = wv.w;
      }
      __syncthreads();
      float acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 8
      for (int k = 0; k < GBK; ++k) {
        const float4 ra = *reinterpret_cast<const float4*>(&Xs[k * (GBM + 4) + ty * 4]);
        const float4 rb = *reinterpret_cast<const float4*>(&Ws[k * (GCB + 4) + tx * 4]);
        const float A[4] = {ra.x, ra.y, ra.z, ra.w};
        const float B[4] = {rb.x, rb.y, rb.z, rb.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(A[i], B[j], acc[i][j]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) run[i][j] += acc[i][j];
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = cb + tx * 4 + j;
        if (c < a.C) Ss[(ty * 4 + i) * C_pad + c] = run[i][j];
      }
  }
  // row |x| totals, summed over the row's slots in a fixed order
  for (int s = 0, slot = tid; slot < GBM * vpr; ++s, slot += 256) Tslot[slot] = tpart[s];
  __syncthreads();
  if (tid < GBM) {
    float t = 0.f;
    for (int vv = 0; vv < vpr; ++vv) t += Tslot[tid * vpr + vv];
    Ts[tid] = t;
  }
  __syncthreads();
  // overflow entries (u8 storage): one thread per (row, class), entries in order
  if (a.dtype == NB_U8 && a.ovf_ptr) {
    for (int q = tid; q < GBM * a.C; q += 256) {
      const int row = q / a.C, c = q % a.C;
      const int64_t gr = r0 + row;
      if (gr >= a.n) continue;
      float s = Ss[row * C_pad + c];
      float t = 0.f;
      for (int64_t k = a.ovf_ptr[gr]; k < a.ovf_ptr[gr + 1]; ++k) {
        const int j = a.ovf_col[k];
        if (j >= a.F) continue;
        const float add = (float)a.ovf_add[k];
        s = fmaf(add, a.w[(int64_t)c * a.F_pad + j], s);
        t += add;
      }
      Ss[row * C_pad + c] = s;
      if (c == 0) Tslot[row] = t;
    }
    __syncthreads();
    if (tid < GBM) Ts[tid] += Tslot[tid];
    __syncthreads();
  }
  // epilogue: a warp per row
  const int warp = tid >> 5, lane = tid & 31;
  for (int row = warp; row < GBM; row += 8) {
    const int64_t gr = r0 + row;
    if (gr >= a.n) continue;
    float best = -INFINITY;
    int bi = 0x7FFFFFFF;
    for (int c = lane; c < a.C; c += 32) {
      const float s = Ss[row * C_pad + c] + a.bias[c];
      if (s > best) { best = s; bi = c; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float ob = __shfl_xor_sync(0xFFFFFFFFu, best, off);
      const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, off);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    float second = -INFINITY, se = 0.f;
    for (int c = lane; c < a.C; c += 32) {
      const float s = Ss[row * C_pad + c] + a.bias[c];
      if (c != bi) second = fmaxf(second, s);
      se += expf(s - best);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      second = fmaxf(second, __shfl_xor_sync(0xFFFFFFFFu, second, off));
      se += __shfl_xor_sync(0xFFFFFFFFu, se, off);
    }
    const float lse = best + logf(se);
    const float margin = best - second;
    const int64_t novf = (a.dtype == NB_U8 && a.ovf_ptr) ? a.ovf_ptr[gr + 1] - a.ovf_ptr[gr] : 0;
    const float k = (float)(GBK + nchunk + 3 + novf);
    const float gam = k * 5.9604645e-8f / (1.f - k * 5.9604645e-8f);
    const float tau = 2.f * (gam * (Ts[row] * wmax + bmax) * 1.01f + 1e-12f * (Ts[row] * wmax + bmax)) + 1e-30f;
    bool flag = false;
    if (a.recheck != NB_RECHECK_OFF) {
      flag = !(margin > tau);
      if (a.recheck == NB_RECHECK_LP && tau > 5e-6f * fmaxf(1.f, margin)) flag = true;
    }
    if (lane == 0) {
      a.label[gr] = flag ? kLabelRecheck : (uint8_t)bi;
      a.margin[gr] = margin;
      if (flag && a.marks) atomicAdd(a.marks, 1ull);
    }
    if (a.want_lp)
      for (int c = lane; c < a.C; c += 32)
        a.logpost[gr * a.C + c] = Ss[row * C_pad + c] + a.bias[c] - lse;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(256) k_score_gen(const GArgs a) {
  extern __shared__ __align__(16) float gsm[];
  const int64_t ntile = (a.n + GBM - 1) / GBM;
  for (int64_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) gen_tile(a, tile * GBM, gsm);
}

// ---------------------------------------------------------------------------
// Gaussian scorer on the CUDA cores (any 2 <= C <= 64, FP32 rows)
// ---------------------------------------------------------------------------
// s_c = k_c - 1/2 sum_j z_cj^2, z = (x_j - mu_cj) / sd_cj (Sec. 4 with Gaussian
// class conditionals; k_c = log pi_c - 1/2 sum_j log(2 pi var_cj)).  The tables hold
// -mu/sd and 1/sd, so that a term costs two fused operations, z = x (1/sd) - mu/sd
// and q + z^2, and a pair of classes shares each instruction (f32x2).
// A group of LPR lanes scores R rows at once: lane li takes features j = li,
// li + LPR, ..., and for each block of CB classes keeps CB x R partial sums
// q = sum z^2.  Slices of FC features go to shared memory with cp.async while the
// slice before is summed: the tables (feature-major, CB consecutive classes per
// feature) once per block of rows, the rows once per class block.  The group's
// partial sums are combined by a reduce-scatter (each exchange halves the values a
// lane holds: CB R (LPR - 1) / LPR shuffles instead of CB R log2 LPR), which leaves
// lane li with the finished sums of classes-and-rows li CB R / LPR ...; their scores
// and bounds go to shared memory, and the LPR lanes then share each row's
// arg-max, sum of exponentials, recheck tests and log-posterior stores.
//
// Against 64 bits the two operations lose little (twice the rounding of 1/sd, one
// product less) and the differences of the epilogue win more: 7.2e-8 -> 6.9e-8 at 64
// classes; over 64 models of six shapes (2 to 40 classes, 16 to 300 features) the log
// posteriors' error is 0.87 to 0.96 of the (x - mu)^2 v form's on average in each
// shape.  Both forms round their tables at random, so single models lie between 0.75
// and 1.40 of it.
// Bound by the FP32 pipe (51 % busy) and the shared-memory reads of the tables (62 %
// of the wavefronts) at four warps a scheduler.  200,000 rows x 256 features x 64
// classes with log posteriors: 636 us with (x - mu)^2 v, one class an instruction and
// loads in place, 441 with two operations a term on pairs, 411 with the slices
// staged ahead, 404 with the classes of a row in registers; 20 classes 371 -> 197,
// 400,000 x 200 x 4: 316 -> 126.  Blocks of 8
// rows x 8 classes halve the table reads and were slower (501): twice the row
// reads.
struct GGArgs {
  const float* X;
  int64_t ld, n;
  int F, F_pad, C;
  const float* nms;   // -mu / sd
  const float* isd;   // 1 / sd
  const float* kc;
  int vec4;           // rows start on 16-byte boundaries
  uint8_t* label;
  float* margin;
  float* logpost;
  int want_lp, recheck;
  unsigned long long* marks;   // counts the rows marked for the recheck, or nullptr
};

constexpr int kGaussWarps = 8;

// lowest index among equal maxima; NaN never wins
__device__ __forceinline__ void gauss_top(float& b, int& i, float ob, int oi) {
  if (ob > b || (ob == b && oi < i)) {
    b = ob;
    i = oi;
  }
}

__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// 16 (4) bytes to shared memory, of which `bytes` are read and the rest are zeros
__device__ __forceinline__ void cp_async16_zfill(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async4_zfill(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// floats per row of the staged scores: 2 past a multiple of 16 puts the rows that
// a warp's lanes write and read at once on different banks
__host__ __device__ constexpr int gauss_cm(int C) { return (C + 15) / 16 * 16 + 2; }
template <int LPR, int R, int CB>
struct GaussLayout {
  static constexpr int RPW = 32 / LPR * R;            // rows per warp
  static constexpr int RPB = kGaussWarps * RPW;       // rows per block tile
  static constexpr int FC = LPR == 8 ? 32 : 64;       // features per staged slice
  // floats per staged feature (-mu/sd of CB classes, then 1/sd): eight lanes' 16-byte
  // reads of consecutive slots touch distinct banks
  static constexpr int SR = 2 * CB + 4;
  // floats of a warp's staged rows: LPR more per group puts the groups' reads on
  // different banks
  static constexpr int XG = R * FC + LPR, XW = 32 / LPR * XG;
  static constexpr int BUF = FC * SR + kGaussWarps * XW;   // one of the two buffers
  static int smem(int C) { return 4 * (2 * BUF + 2 * RPB * gauss_cm(C)); }
};

template <int LPR, int R, int CB>
__global__ void __launch_bounds__(kGaussWarps * 32, CB == 4 ? 4 : 2) k_score_gauss(const GGArgs a) {
  using L = GaussLayout<LPR, R, CB>;
  constexpr int NP = CB * R;      // sums q of a class block
  constexpr int OWN = NP / LPR;   // pairs a lane finishes
  constexpr int FC = L::FC, SR = L::SR, FPL = FC / LPR;   // FPL: features per lane and slice
  static_assert(NP % LPR == 0, "the reduce-scatter ends with whole pairs per lane");
  extern __shared__ __align__(16) float gsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = lane / LPR, li = lane % LPR;
  const int C = a.C, F = a.F, CP = gauss_cpad(C), CM = gauss_cm(C);
  float* s_q = gsm + 2 * L::BUF + (warp * L::RPW + grp * R) * CM;   // [R][CM] of this group
  float* s_t = s_q + kGaussWarps * L::RPW * CM;
  constexpr float u = 5.9604645e-8f;

  // rounding depth of each sum: F / LPR sequential adds, the log2 LPR
  // combining levels, and 8 for the remaining operations
  int lg = 0;
  while ((1 << lg) < LPR) ++lg;
  const int kdepth = (F + LPR - 1) / LPR + lg + 8;
  const float gam = kdepth * u / (1.f - kdepth * u);

  // Slice -> shared memory: the tables of features f0 .. f0 + FC - 1 and classes
  // cb .. cb + CB - 1 (by the block), the same features of the warp's rows from
  // row w0 (rows past the end: the last one)
  auto stage = [&](int buf, int cb, int f0, int64_t w0) {
    float* st = gsm + buf * L::BUF;
    constexpr int Q = CB / 4, TN = FC * Q * 2;
#pragma unroll
    for (int s = 0; s < (TN + kGaussWarps * 32 - 1) / (kGaussWarps * 32); ++s) {
      const int e = threadIdx.x + s * kGaussWarps * 32;
      const int fl = e / (2 * Q), rem = e % (2 * Q), which = rem / Q, q4 = rem % Q;
      const int j = f0 + fl;
      if (TN % (kGaussWarps * 32) == 0 || e < TN)
        cp_async16_zfill(st + fl * SR + which * CB + 4 * q4,
                         (which ? a.isd : a.nms) + (int64_t)(j < a.F_pad ? j : 0) * CP + cb + 4 * q4,
                         j < a.F_pad ? 16 : 0);
    }
    float* sx = st + FC * SR + warp * L::XW;
    if (a.vec4) {
      constexpr int V = FC / 4;   // 16-byte pieces per row, V lanes a row
#pragma unroll
      for (int s = 0; s < L::RPW * V / 32; ++s) {
        const int r = s * (32 / V) + lane / V, v = lane % V;
        const int64_t row = w0 + r < a.n ? w0 + r : a.n - 1;
        const int j = f0 + 4 * v, b = 4 * (F - j);
        cp_async16_zfill(sx + r / R * L::XG + r % R * FC + 4 * v, a.X + row * a.ld + (j < F ? j : 0),
                         b < 0 ? 0 : (b < 16 ? b : 16));
      }
    } else {
#pragma unroll 4
      for (int s = 0; s < L::RPW * FC / 32; ++s) {
        const int r = s / (FC / 32), v = s % (FC / 32) * 32 + lane;
        const int64_t row = w0 + r < a.n ? w0 + r : a.n - 1;
        const int j = f0 + v;
        cp_async4_zfill(sx + r / R * L::XG + r % R * FC + v, a.X + row * a.ld + (j < F ? j : 0),
                        j < F ? 4 : 0);
      }
    }
  };

  const int64_t nbt = (a.n + L::RPB - 1) / L::RPB;
  int buf = 0;
  if ((int64_t)blockIdx.x < nbt) stage(0, 0, 0, (int64_t)blockIdx.x * L::RPB + warp * L::RPW);
  for (int64_t bt = blockIdx.x; bt < nbt; bt += gridDim.x) {   // uniform over the block
    const int64_t w0 = bt * L::RPB + warp * L::RPW, r0 = w0 + grp * R;
    for (int cb = 0; cb < C; cb += CB) {
      // sums of class pairs: pq2[k][i] holds classes cb + 2 k, cb + 2 k + 1 of row
      // r0 + i
      uint64_t pq2[CB / 2][R];
#pragma unroll
      for (int k = 0; k < CB / 2; ++k)
#pragma unroll
        for (int i = 0; i < R; ++i) pq2[k][i] = 0ull;
      for (int f0 = 0; f0 < F; f0 += FC) {
        cp_async_wait_all();
        __syncthreads();   // this slice is there; nobody reads the other buffer any more
        const float* tab = gsm + buf * L::BUF + li * SR;
        const float* xs = gsm + buf * L::BUF + FC * SR + warp * L::XW + grp * L::XG + li;
        buf ^= 1;
        if (f0 + FC < F)
          stage(buf, cb, f0 + FC, w0);
        else if (cb + CB < C)
          stage(buf, cb + CB, 0, w0);
        else if (bt + gridDim.x < nbt)
          stage(buf, 0, 0, w0 + (int64_t)gridDim.x * L::RPB);
#pragma unroll
        for (int jj = 0; jj < FPL; ++jj) {
          if (f0 + LPR * jj >= F) break;   // uniform; the features past F are zeros
          uint64_t xx[R];
#pragma unroll
          for (int i = 0; i < R; ++i) {
            const float xv = xs[i * FC + LPR * jj];
            xx[i] = f32x2_pack(xv, xv);
          }
          const float* tb = tab + jj * LPR * SR;
#pragma unroll
          for (int k4 = 0; k4 < CB / 4; ++k4) {
            const ulonglong2 m2 = *reinterpret_cast<const ulonglong2*>(tb + 4 * k4);
            const ulonglong2 v2 = *reinterpret_cast<const ulonglong2*>(tb + CB + 4 * k4);
#pragma unroll
            for (int i = 0; i < R; ++i) {
              const uint64_t z0 = f32x2_fma(xx[i], v2.x, m2.x), z1 = f32x2_fma(xx[i], v2.y, m2.y);
              pq2[2 * k4][i] = f32x2_fma(z0, z0, pq2[2 * k4][i]);
              pq2[2 * k4 + 1][i] = f32x2_fma(z1, z1, pq2[2 * k4 + 1][i]);
            }
          }
        }
      }
      // sum p = k R + i: class cb + k, row r0 + i
      float pq[NP];
#pragma unroll
      for (int k = 0; k < CB / 2; ++k)
#pragma unroll
        for (int i = 0; i < R; ++i)
          f32x2_unpack(pq2[k][i], pq[2 * k * R + i], pq[(2 * k + 1) * R + i]);
      // reduce-scatter over the group
#pragma unroll
      for (int off = LPR / 2, n = NP; off > 0; off >>= 1, n >>= 1) {
        const bool up = (li & off) != 0;   // this lane keeps the upper half
#pragma unroll
        for (int p = 0; p < n / 2; ++p) {
          const float sq = up ? pq[p] : pq[p + n / 2], kq = up ? pq[p + n / 2] : pq[p];
          pq[p] = kq + __shfl_xor_sync(0xFFFFFFFFu, sq, off);
        }
      }
      // lane li now holds pairs li OWN .. li OWN + OWN - 1
#pragma unroll
      for (int o = 0; o < OWN; ++o) {
        const int p = li * OWN + o, k = p / R, i = p % R, c = cb + k;
        if (c >= C) continue;
        const float qq = pq[o], kc = __ldg(a.kc + c);
        // |s - s_FP64| with u = 2^-24: w = fl(1/sd) is within u relative, m =
        // fl(mu w) within u |m| of mu w, and z = fl(x w - m) rounds once, so z
        // is within u (2 |z| + |m|) of (x - mu) / sd (to first order) and each
        // z^2 within u (4 z^2 + 2 |z| |m|) (1 + 2 u) + 2 u^2 (z^2 + m^2); the
        // FP32 sums add gam q; k_c and the final subtraction add u (|k_c| +
        // |s|).  sum |z| |m| <= sqrt(sum z^2 sum m^2) (Cauchy-Schwarz on the
        // FP32 values; 1e-3 covers the rounding of the two computed sums and
        // of the root, which is within 2^-22); 1% slack covers the FP32
        // evaluation of the bound.
        const float a4 = __ldg(a.kc + C + c);   // sum_j m^2, from the fit
        const float aa = sqrt_approx(qq * a4) * 1.001f;
        const float sc = kc - 0.5f * qq;
        s_q[i * CM + c] = qq;
        s_t[i * CM + c] = (0.5f * (u * (4.f * qq + 2.f * aa) * (1.f + 2.f * u) +
                                   2.f * u * u * (qq + a4) + gam * qq) +
                           u * (fabsf(kc) + fabsf(sc))) * 1.01f +
                          1e-12f * (qq + fabsf(kc)) + 1e-30f;
      }
    }
    __syncwarp();
    // epilogue: the group's lanes share each row's classes, M a lane
    constexpr int M = CB == 4 ? 1 : kTcMaxC / LPR;
    float kv[M], kmax = 0.f;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const int c = li + LPR * m;
      kv[m] = c < C ? __ldg(a.kc + c) : -INFINITY;
      if (c < C) kmax = fmaxf(kmax, fabsf(kv[m]));
    }
#pragma unroll
    for (int off = LPR / 2; off > 0; off >>= 1)
      kmax = fmaxf(kmax, __shfl_xor_sync(0xFFFFFFFFu, kmax, off));
    const unsigned gmask = LPR == 32 ? 0xFFFFFFFFu : ((1u << (LPR & 31)) - 1) << (grp * LPR);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float* qr = s_q + i * CM;
      const float* tr = s_t + i * CM;
      float b1 = -INFINITY, tmax = 0.f;
      int i1 = 0x7FFFFFFF;
      bool nan = false;
      float qv[M], tv[M];   // classes li + LPR m
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (m > 0 && LPR * m >= C) break;   // uniform
        const int c = li + LPR * m;
        qv[m] = c < C ? qr[c] : 0.f;
        tv[m] = c < C ? tr[c] : 0.f;
        const float sv = kv[m] - 0.5f * qv[m];
        nan |= !(sv == sv) || !(tv[m] == tv[m]);
        tmax = fmaxf(tmax, tv[m]);
        gauss_top(b1, i1, sv, c);
      }
#pragma unroll
      for (int off = LPR / 2; off > 0; off >>= 1) {
        const float ob1 = __shfl_xor_sync(0xFFFFFFFFu, b1, off);
        const int oi1 = __shfl_xor_sync(0xFFFFFFFFu, i1, off);
        gauss_top(b1, i1, ob1, oi1);
        tmax = fmaxf(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, off));
      }
      nan = (__ballot_sync(0xFFFFFFFFu, nan) & gmask) != 0;
      const int bi = i1 < C ? i1 : 0;   // every score NaN: class 0, and the row is marked
      const float qb = qr[bi], tb = tr[bi], kb = __ldg(a.kc + bi);
      const float sb = kb - 0.5f * qb;
      // d_c = s_c - s_top from the constants' and the sums' differences: two
      // roundings less than from the scores, at smaller magnitudes
      float dv[M], d2 = -INFINITY, P = 0.f;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (m > 0 && LPR * m >= C) break;
        const int c = li + LPR * m;
        dv[m] = (kv[m] - kb) - 0.5f * (qv[m] - qb);
        if (c < C && c != bi) {
          P += expf(dv[m]);
          d2 = fmaxf(d2, dv[m]);
        }
      }
#pragma unroll
      for (int off = LPR / 2; off > 0; off >>= 1) {
        P += __shfl_xor_sync(0xFFFFFFFFu, P, off);
        d2 = fmaxf(d2, __shfl_xor_sync(0xFFFFFFFFu, d2, off));
      }
      // a runner-up within rounding may come out ahead; no number where s_top is none
      const float margin = (d2 > 0.f ? 0.f : -d2) + (sb - sb);
      // lp_c = d_c - L: formed from the differences, so that no
      // rounding at the scores' magnitude enters (lp_top = -L exactly)
      const float lg1 = log1pf(P);
      bool flag = false;
      if (a.recheck != NB_RECHECK_OFF) {
        flag = nan;   // a NaN score or bound: FP64 decides
        // label: the top class stays ahead of every other class c by more than
        // the two classes' bounds (a far class's large bound does not matter) and
        // what the difference's own roundings add to them: u |k_c - k_top| and u
        // |q_c - q_top| / 2 <= u (|k_c - k_top| + |d_c|), the parts relative to
        // d_c within the factor.
        // lp_c = d_c - L with L = log(1 + sum_{k != top} e^{d_k}); each d_k is
        // off by at most D = t_top + t_max + 4 u max |k|, so L is off by at most
        // D e^{2D} P / (1 + P) (mean value; the softmax weights at the
        // intermediate point are within e^{2D} of the computed ones), and lp_c
        // by that plus t_c + t_top (c != top)
        const bool lp = a.recheck == NB_RECHECK_LP;
        const float D = tb + tmax + 4.f * u * kmax;
        const float eL = lp ? D * expf(2.f * D) * __fdividef(P, 1.f + P) * 1.01f + 1e-30f : 0.f;
#pragma unroll
        for (int m = 0; m < M; ++m) {
          if (m > 0 && LPR * m >= C) break;
          const int c = li + LPR * m;
          if (c >= C) continue;
          const float tt = tb + tv[m] + 2.f * u * fabsf(kv[m] - kb);
          if (c != bi && !(-dv[m] > tt * 1.0001f)) flag = true;
          if (lp && (c == bi ? 0.f : tt) + eL > 5e-6f * fmaxf(1.f, fabsf(dv[m] - lg1))) flag = true;
        }
      }
      const bool fl = (__ballot_sync(0xFFFFFFFFu, flag) & gmask) != 0;
      if (r0 + i < a.n) {
        const int64_t r = r0 + i;
        if (li == 0) {
          a.label[r] = fl ? kLabelRecheck : (uint8_t)bi;
          a.margin[r] = margin;
          if (fl && a.marks) atomicAdd(a.marks, 1ull);
        }
        if (a.want_lp) {
#pragma unroll
          for (int m = 0; m < M; ++m) {
            if (m > 0 && LPR * m >= C) break;
            const int c = li + LPR * m;
            if (c < C) a.logpost[r * C + c] = dv[m] - lg1;
          }
        }
      }
    }
    __syncwarp();
  }
}

template <int LPR, int R, int CB>
static nb_status run_score_gauss(const GGArgs& a, cudaStream_t st) {
  using L = GaussLayout<LPR, R, CB>;
  const int smem = L::smem(a.C);
  NB_TRY_CUDA(cudaFuncSetAttribute(k_score_gauss<LPR, R, CB>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
              "smem attr(k_score_gauss)");
  int occ = 0;
  NB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                  &occ, k_score_gauss<LPR, R, CB>, kGaussWarps * 32, smem),
              "occupancy(k_score_gauss)");
  const int64_t cap = (int64_t)num_sms() * (occ > 0 ? occ : 1);
  int64_t blocks = (a.n + L::RPB - 1) / L::RPB;
  if (blocks > cap) blocks = cap;
  count_launch();
  k_score_gauss<LPR, R, CB><<<(unsigned)blocks, kGaussWarps * 32, smem, st>>>(a);
  NB_TRY_CUDA(cudaGetLastError(), "k_score_gauss launch");
  return NB_OK;
}

// Lanes per row: the features a lane sums in sequence stay at most 32 (the rounding
// depth of the bound; 16 for many classes).  Up to 4 classes take 4-class blocks at four
// blocks per SM (400,000 x 200 x 4: 158 us against 200 at two, before the epilogue kept
// the classes in registers; 126 since).  More take 16-class blocks; between 129 and 512
// features 8-class ones where half of the last 16 or more would be padding (20 classes x
// 256 features: 217 us against 237, 36 x 300: 206 and 202; with 32 lanes a row they lose,
// 24 x 600: 310 and 287, 20 x 1,000: 248 and 230).  At up to 128 features 8-class blocks
// of four rows (400,000 x 100 x 10: 165 us against 184 for 16 classes of two rows,
// 200,000 x 24 x 40: 200 against 224).
static nb_status launch_score_gauss(const GGArgs& a, cudaStream_t st) {
  if (a.C <= 4) {
    if (a.F > 128) return run_score_gauss<16, 4, 4>(a, st);
    return run_score_gauss<8, 4, 4>(a, st);
  }
  if (a.F > 512) return run_score_gauss<32, 4, 16>(a, st);
  if (a.F > 128)
    return (a.C - 1) % 16 < 8 ? run_score_gauss<16, 4, 8>(a, st)   // less padding
                              : run_score_gauss<16, 4, 16>(a, st);
  return run_score_gauss<8, 4, 8>(a, st);
}

// ---------------------------------------------------------------------------
// segmented general scorer: 64-row tiles of a group list, each group scored
// with its own model slot (one launch per batch)
// ---------------------------------------------------------------------------
struct GModel {
  int C, F_pad;
  const float* w;
  const float* bias;
  const float* wmax;
};

struct GSegArgs {
  const SegGroup* groups;
  const SegHeader* hdr;
  GModel md[kSegMaxModels];
  int F, dtype, want_lp, recheck;
  unsigned long long* marks;
  int* status;
};

__global__ void __launch_bounds__(256) k_score_gen_seg(const GSegArgs s) {
  extern __shared__ __align__(16) float gsm[];
  const int n_groups = s.hdr->n_groups;
  const long long tiles = s.hdr->tiles;
  const SegGroup* gr = s.groups;
  const int es = s.dtype == NB_F32 ? 4 : ((s.dtype == NB_U16 || s.dtype == NB_BF16) ? 2 : 1);
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int g = seg_find(n_groups, t, [gr](int i) { return gr[i].tile0; });
    const SegGroup& G = gr[g];
    const GModel& M = s.md[G.model];
    GArgs a{};
    a.X = G.X;
    a.ld = G.ld_bytes / es;
    a.n = G.n;
    a.F = s.F;
    a.F_pad = M.F_pad;
    a.C = M.C;
    a.dtype = s.dtype;
    a.aligned = ((reinterpret_cast<uintptr_t>(G.X) & 15) == 0) && (G.ld_bytes % 16 == 0);
    a.ovf_ptr = G.ovf_ptr;
    a.ovf_col = G.ovf_col;
    a.ovf_add = G.ovf_add;
    a.row_exp = G.row_exp;
    a.w = M.w;
    a.bias = M.bias;
    a.wmax = M.wmax;
    a.label = G.label;
    a.margin = G.margin;
    a.logpost = G.logpost;
    a.want_lp = s.want_lp;
    a.recheck = s.recheck;
    a.marks = s.marks;
    a.status = s.status;
    gen_tile(a, (t - G.tile0) * GBM, gsm);
  }
}

nb_status launch_score_gen_seg(const SegGroup* groups, const SegHeader* hdr,
                               const nb_model* const* models, int n_models, nb_dtype dt, int F,
                               int want_lp, int recheck, unsigned long long* marks, int* status,
                               cudaStream_t st) {
  GSegArgs s{};
  s.marks = marks;
  s.groups = groups;
  s.hdr = hdr;
  int C_max = 2;
  for (int i = 0; i < n_models && i < kSegMaxModels; ++i) {
    const nb_model* m = models[i];
    s.md[i] = GModel{m->C, m->F_pad, m->d.w, m->d.bias, m->d.wmax};
    C_max = m->C > C_max ? m->C : C_max;
  }
  s.F = F;
  s.dtype = dt;
  s.want_lp = want_lp;
  s.recheck = recheck;
  s.status = status;
  const int C_pad = ((C_max + 3) / 4) * 4;
  const int smem =
      (int)sizeof(float) * (GBK * (GBM + 4) + GBK * (GCB + 4) + GBM * C_pad + GBM + GBM * 8);
  if (smem > kSmemOptIn)
    NB_TRY_CUDA(cudaFuncSetAttribute(k_score_gen_seg, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     smem),
                "cudaFuncSetAttribute(gen_seg)");
  int occ = 0;
  NB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_score_gen_seg, 256, smem),
              "occupancy(gen_seg)");
  count_launch();
  k_score_gen_seg<<<num_sms() * (occ > 0 ? occ : 1), 256, smem, st>>>(s);
  NB_TRY_CUDA(cudaGetLastError(), "k_score_gen_seg launch");
  return NB_OK;
}

nb_status launch_score_general(const nb_model* m, const void* X, nb_dtype dt, int64_t n,
                               int64_t ld, const nb_aux* aux, const ScoreOut& o, cudaStream_t st) {
  if (n == 0) return NB_OK;
  if (m->kind == NB_GAUSSIAN) {
    if (dt != NB_F32) {
      set_error("Gaussian models score F32 features");
      return NB_EINVAL;
    }
    GGArgs a{};
    a.X = static_cast<const float*>(X);
    a.ld = ld;
    a.n = n;
    a.F = m->F;
    a.F_pad = m->F_pad;
    a.C = m->C;
    a.nms = m->d.g_nms;
    a.isd = m->d.g_isd;
    a.vec4 = (reinterpret_cast<uintptr_t>(X) & 15) == 0 && (ld & 3) == 0;
    a.kc = m->d.g_const;
    a.label = o.label;
    a.margin = o.margin;
    a.logpost = o.logpost;
    a.want_lp = o.want_lp;
    a.recheck = o.recheck;
    a.marks = o.counted ? reinterpret_cast<unsigned long long*>(o.n_rechecked) : nullptr;
    return launch_score_gauss(a, st);
  }
  const int es = elem_size(dt);
  GArgs a{};
  a.X = static_cast<const char*>(X);
  a.ld = ld;
  a.n = n;
  a.F = m->F;
  a.F_pad = m->F_pad;
  a.C = m->C;
  a.dtype = dt;
  a.aligned = ((reinterpret_cast<uintptr_t>(X) & 15) == 0) && ((ld * es) % 16 == 0);
  a.ovf_ptr = aux ? aux->ovf_ptr : nullptr;
  a.ovf_col = aux ? aux->ovf_col : nullptr;
  a.ovf_add = aux ? aux->ovf_add : nullptr;
  a.row_exp = aux ? aux->row_exp : nullptr;
  a.w = m->d.w;
  a.bias = m->d.bias;
  a.wmax = m->d.wmax;
  a.log_pi = m->d.log_pi;
  a.label = o.label;
  a.margin = o.margin;
  a.logpost = o.logpost;
  a.want_lp = o.want_lp;
  a.recheck = o.recheck;
  a.marks = o.counted ? reinterpret_cast<unsigned long long*>(o.n_rechecked) : nullptr;
  a.status = m->d.sstatus;
  const int C_pad = ((m->C + 3) / 4) * 4;
  const int smem =
      (int)sizeof(float) * (GBK * (GBM + 4) + GBK * (GCB + 4) + GBM * C_pad + GBM + GBM * 8);
  if (smem > kSmemOptIn)   // per device and function: set at every launch
    NB_TRY_CUDA(cudaFuncSetAttribute(k_score_gen, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     smem > 96 * 1024 ? smem : 96 * 1024),
                "cudaFuncSetAttribute");
  int occ = 0;
  NB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_score_gen, 256, smem),
              "occupancy");
  const int64_t tiles = (n + GBM - 1) / GBM;
  const int64_t cap = (int64_t)num_sms() * (occ > 0 ? occ : 1);
  count_launch();
  k_score_gen<<<(unsigned)(tiles < cap ? tiles : cap), 256, smem, st>>>(a);
  NB_TRY_CUDA(cudaGetLastError(), "k_score_gen launch");
  return NB_OK;
}

}  // namespace nbg
