// Two-class multinomial scoring (Sec. 4 posterior and decision rule).
//
// For C = 2 the decision needs only the log-odds
//     d = s_1 - s_0 = b + sum_j x_j Delta_j,
//     b = log pi_1 - log pi_0,  Delta_j = log theta_1j - log theta_0j,
// and the outputs follow from d alone: label = [d > 0] (a tie, d = 0, goes to
// benign), margin = |d|, log P(1|x) = -softplus(-d), log P(0|x) = -softplus(d).
// Each file is read once from HBM with 16-byte streaming loads; the Delta
// table is staged into shared memory by bulk copies (TMA) behind an mbarrier.
//
// Two inner products:
//   * u8 storage: Delta is held as a 22-bit fixed-point integer split into
//     three signed 8-bit limbs; dp4a accumulates x * limb exactly in int32, so
//     the only error is the quantisation of Delta (<= 2^-S / 2 per count).
//     FP8 E4M3 storage takes the same limbs: its values become exact integer
//     counts (row scale 2^0 or 2^1, checked per value, see fp8_biased_pairs)
//     in 16-bit pairs, accumulated with dp2a.
//   * f32 / u16 / bf16 storage: decode to FP32 and FMA against the FP32 Delta
//     table, four accumulators per row per lane.
// Every row also gets a rigorous bound tau on |d_gpu - d_exact|; rows whose
// sign (or whose log posteriors to 1e-5) the bound cannot guarantee are marked
// for the FP64 recheck.
#include <cuda_fp16.h>

#include "score2.cuh"

namespace nbg {

// ---------------------------------------------------------------------------
// u8 storage, fixed-point Delta, exact integer accumulation
// ---------------------------------------------------------------------------
template <int DT, int LPR, int R>
__global__ void __launch_bounds__(256) k_score2_u8(const S2Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t bar;
  if (!stage_table(smem_raw, a.table, a.table_bytes, &bar, a.status, ST_TIMEOUT)) return;
  const uint4* tab = reinterpret_cast<const uint4*>(smem_raw);
  const C2Header h = *a.hdr;

  constexpr int SUBS = 32 / LPR;
  constexpr int RPW = SUBS * R;
  const int lane = threadIdx.x & 31;
  const int sub = lane / LPR, li = lane % LPR;
  const int nv = a.nvec_row, nt = a.nvec_tab;
  const int64_t ntiles = (a.n + RPW - 1) / RPW;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);

  // byte masks of the last (partial) vector
  const int keep = a.F - 16 * (nv - 1);
  uint32_t tm[4];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    int vb = keep - 4 * w;
    vb = vb < 0 ? 0 : (vb > 4 ? 4 : vb);
    tm[w] = vb >= 4 ? 0xFFFFFFFFu : ((1u << (8 * vb)) - 1u);
  }
  const bool has_tail = keep < 16;

  // rows this lane marked for the FP64 recheck, added up once per warp at the
  // end (faster here than an atomic per marked row; the FP kernel below keeps
  // the atomic, which holds no register through its loop)
  unsigned marks = 0;
  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntiles;
       t += nwarps) {
    const int64_t row0 = t * RPW + (int64_t)sub * R;
    int acc0[R], acc1[R], acc2[R];
    uint32_t tot[R], m2[R];
    Fp8Check chk[R];
    const char* rp[R];
    bool ok[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      acc0[r] = acc1[r] = acc2[r] = 0;
      tot[r] = 0;
      ok[r] = row0 + r < a.n;
      rp[r] = a.X + (ok[r] ? row0 + r : 0) * a.ld_bytes;
      m2[r] = DT == NB_FP8E4M3 ? fp8_magic((a.row_exp && ok[r]) ? (int)a.row_exp[row0 + r] : 0)
                               : 0u;
    }
#pragma unroll 2
    for (int v = li; v < nv; v += LPR) {
      const uint4 q0 = tab[v], q1 = tab[nt + v], q2 = tab[2 * nt + v];
      uint4 x[R];
#pragma unroll
      for (int r = 0; r < R; ++r)
        x[r] = ok[r] ? ld_stream16(rp[r] + (int64_t)v * 16) : make_uint4(0, 0, 0, 0);
      if (has_tail && v == nv - 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          x[r].x &= tm[0];
          x[r].y &= tm[1];
          x[r].z &= tm[2];
          x[r].w &= tm[3];
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (DT == NB_FP8E4M3) {
          fp8_vector_limbs(x[r], q0, q1, q2, m2[r], acc0[r], acc1[r], acc2[r], tot[r], chk[r]);
          continue;
        }
        acc0[r] = dp4a_us(x[r].x, q0.x, acc0[r]);
        acc0[r] = dp4a_us(x[r].y, q0.y, acc0[r]);
        acc0[r] = dp4a_us(x[r].z, q0.z, acc0[r]);
        acc0[r] = dp4a_us(x[r].w, q0.w, acc0[r]);
        acc1[r] = dp4a_us(x[r].x, q1.x, acc1[r]);
        acc1[r] = dp4a_us(x[r].y, q1.y, acc1[r]);
        acc1[r] = dp4a_us(x[r].z, q1.z, acc1[r]);
        acc1[r] = dp4a_us(x[r].w, q1.w, acc1[r]);
        acc2[r] = dp4a_us(x[r].x, q2.x, acc2[r]);
        acc2[r] = dp4a_us(x[r].y, q2.y, acc2[r]);
        acc2[r] = dp4a_us(x[r].z, q2.z, acc2[r]);
        acc2[r] = dp4a_us(x[r].w, q2.w, acc2[r]);
        tot[r] = dp4a_uu(x[r].x, 0x01010101u, tot[r]);
        tot[r] = dp4a_uu(x[r].y, 0x01010101u, tot[r]);
        tot[r] = dp4a_uu(x[r].z, 0x01010101u, tot[r]);
        tot[r] = dp4a_uu(x[r].w, 0x01010101u, tot[r]);
      }
    }
    long long D[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      D[r] = ((long long)acc2[r] << 16) + ((long long)acc1[r] << 8) + (long long)acc0[r];
      if (DT == NB_FP8E4M3) tot[r] = fp8_lane_total(tot[r], chk[r], m2[r]);
    }
    if (DT == NB_U8 && a.ovf_ptr) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!ok[r]) continue;
        const int64_t k0 = a.ovf_ptr[row0 + r], k1 = a.ovf_ptr[row0 + r + 1];
        for (int64_t k = k0 + li; k < k1; k += LPR) {
          const uint32_t col = a.ovf_col[k], add = a.ovf_add[k];
          if (col < (uint32_t)a.F) {
            D[r] += (long long)add * (long long)a.delta_q[col];
            tot[r] += add;
          } else {
            atomicOr(a.status, ST_OVF_RANGE);
          }
        }
      }
    }
#pragma unroll
    for (int off = LPR / 2; off > 0; off >>= 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        D[r] += __shfl_xor_sync(0xFFFFFFFFu, D[r], off);
        tot[r] += __shfl_xor_sync(0xFFFFFFFFu, tot[r], off);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!ok[r] || (r % LPR) != li) continue;
      const float Dsum = (float)D[r] * h.inv_scale;
      const float d = Dsum + h.b;
      // quantisation of Delta + int64->f32 and final-add roundings + FP64 slack;
      // +inf past the int32 range of the limb sums
      const float tau = c2_tau_u8((float)tot[r], Dsum, h.b, h.inv_scale, h.maxabs);
      marks += c2_store(a.label, a.margin, a.logpost, a.want_lp, a.recheck, row0 + r, d, tau);
    }
  }
  c2_flush_marks(a, marks);
}

// ---------------------------------------------------------------------------
// FP8 rows of fewer than 32 vectors (F <= 496): five limbs, FP64 outputs
// ---------------------------------------------------------------------------
// Every such row once went to FP64 from the pipelined kernel (a lane without a vector
// failed the count check: 1M files of F = 256 13.3 ms), so what replaces that keeps
// its accuracy: Delta in 37 bits, five limbs instead of three, one rounding of each
// output.  Bound by the decode as k_score2_u8 (1M files of F = 64 45 us, 256 102, 480
// 204; three limbs 39, 110 and 194).
template <int LPR>
__global__ void __launch_bounds__(256, 3) k_score2_fp8(const S2Args a) {
  constexpr int R = 2, SUBS = 32 / LPR, RPW = SUBS * R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t bar;
  if (!stage_table(smem_raw, a.table, a.table_bytes, &bar, a.status, ST_TIMEOUT)) return;
  const uint4* tab = reinterpret_cast<const uint4*>(smem_raw);
  const C2Header h = *a.hdr;
  const int lane = threadIdx.x & 31, sub = lane / LPR, li = lane % LPR;
  const int nv = a.nvec_row, nt = a.nvec_tab;
  const int64_t ntiles = (a.n + RPW - 1) / RPW;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  // byte masks of the last (partial) vector
  const int keep = a.F - 16 * (nv - 1);
  uint32_t tm[4];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    int vb = keep - 4 * w;
    vb = vb < 0 ? 0 : (vb > 4 ? 4 : vb);
    tm[w] = vb >= 4 ? 0xFFFFFFFFu : ((1u << (8 * vb)) - 1u);
  }
  const double step = __hiloint2double((1023 - h.S - 15) << 20, 0);   // 2^-(S+15)
  // the prior's part in whole steps: d is then an integer until it is rounded to FP32.
  // (In FP64 where it does not fit: weights of next to nothing.)
  const double bs = h.b64 * __hiloint2double((1023 + h.S + 15) << 20, 0);
  const bool whole = fabs(bs) < 4.611686018427388e18;
  const long long b = whole ? llrint(bs) : 0ll;
  unsigned marks = 0;
  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntiles;
       t += nwarps) {
    const int64_t row0 = t * RPW + (int64_t)sub * R;
    int acc[R][5];
    uint32_t tot[R], m2[R];
    Fp8Check chk[R];
    const char* rp[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {   // rows past the end repeat the last one and store nothing
      const int64_t row = min(row0 + r, a.n - 1);
#pragma unroll
      for (int l = 0; l < 5; ++l) acc[r][l] = 0;
      tot[r] = 0;
      rp[r] = a.X + row * a.ld_bytes;
      m2[r] = fp8_magic(a.row_exp ? (int)a.row_exp[row] : 0);
    }
#pragma unroll 2
    for (int v = li; v < nv; v += LPR) {
      uint4 x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = ld_stream16(rp[r] + (int64_t)v * 16);
      const uint4 q[5] = {tab[v], tab[nt + v], tab[2 * nt + v], tab[3 * nt + v], tab[4 * nt + v]};
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (v == nv - 1) {
          x[r].x &= tm[0];
          x[r].y &= tm[1];
          x[r].z &= tm[2];
          x[r].w &= tm[3];
        }
        fp8_vector_limbs5(x[r], q, m2[r], acc[r], tot[r], chk[r]);
      }
    }
    long long D[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      // |acc| <= 128 T < 2^31 (c2_tau_u8's limit), |D| < 2^62
      D[r] = ((((long long)acc[r][2] << 16) + ((long long)acc[r][1] << 8) + (long long)acc[r][0]) << 15) +
             ((long long)acc[r][4] << 8) + (long long)acc[r][3];
      tot[r] = fp8_lane_total(tot[r], chk[r], m2[r]);
    }
#pragma unroll
    for (int off = LPR / 2; off > 0; off >>= 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        D[r] += __shfl_xor_sync(0xFFFFFFFFu, D[r], off);
        tot[r] += __shfl_xor_sync(0xFFFFFFFFu, tot[r], off);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (row0 + r >= a.n || r % LPR != li) continue;
      // (|D| < 2^62 and |b| <= 2^62: no wrap)
      const float d = whole ? (float)(D[r] + b) * (float)step : (float)fma((double)D[r], step, h.b64);
      const double d64 = whole ? (double)(D[r] + b) * step : fma((double)D[r], step, h.b64);
      const float T = (float)tot[r];
      // the three-limb kernels' bound: the rows that it does not settle are the
      // recheck's in every kernel
      const float tau = c2_tau_u8(T, d, h.b, h.inv_scale, h.maxabs);
      marks += c2_store64(a.label, a.margin, a.logpost, a.want_lp, a.recheck, row0 + r, d, d64,
                          tau);
    }
  }
  c2_flush_marks(a, marks);
}

template <int DT, int LPR, int R>
__global__ void __launch_bounds__(256) k_score2_fp(const S2Args a) {
  using Dec = Decode<DT>;
  constexpr int EPV = Dec::EPV, QPV = EPV / 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t bar;
  if (!stage_table(smem_raw, a.table, a.table_bytes, &bar, a.status, ST_TIMEOUT)) return;
  const float4* tab = reinterpret_cast<const float4*>(smem_raw);
  const C2Header h = *a.hdr;

  constexpr int SUBS = 32 / LPR;
  constexpr int RPW = SUBS * R;
  const int lane = threadIdx.x & 31;
  const int sub = lane / LPR, li = lane % LPR;
  const int nv = a.nvec_row, nt = a.nvec_tab;
  const int64_t ntiles = (a.n + RPW - 1) / RPW;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const bool has_tail = a.F < nv * EPV;

  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntiles;
       t += nwarps) {
    const int64_t row0 = t * RPW + (int64_t)sub * R;
    float acc[R][4], tot[R];
    const char* rp[R];
    bool ok[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f;
      tot[r] = 0.f;
      ok[r] = row0 + r < a.n;
      rp[r] = a.X + (ok[r] ? row0 + r : 0) * a.ld_bytes;
    }
#pragma unroll 2
    for (int v = li; v < nv; v += LPR) {
      float4 wq[QPV];
#pragma unroll
      for (int q = 0; q < QPV; ++q) wq[q] = tab[q * nt + v];
      uint4 x[R];
#pragma unroll
      for (int r = 0; r < R; ++r)
        x[r] = ok[r] ? ld_stream16(rp[r] + (int64_t)v * 16) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float val[EPV];
        Dec::run(x[r], val);
        if (has_tail && v == nv - 1) {
#pragma unroll
          for (int e = 0; e < EPV; ++e)
            if (v * EPV + e >= a.F) val[e] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < QPV; ++q) {
          acc[r][0] = fmaf(val[4 * q + 0], wq[q].x, acc[r][0]);
          acc[r][1] = fmaf(val[4 * q + 1], wq[q].y, acc[r][1]);
          acc[r][2] = fmaf(val[4 * q + 2], wq[q].z, acc[r][2]);
          acc[r][3] = fmaf(val[4 * q + 3], wq[q].w, acc[r][3]);
          tot[r] += fabsf(val[4 * q + 0]) + fabsf(val[4 * q + 1]) + fabsf(val[4 * q + 2]) +
                    fabsf(val[4 * q + 3]);
        }
      }
    }
    float s[R];
    int nov[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      s[r] = (acc[r][0] + acc[r][1]) + (acc[r][2] + acc[r][3]);
      nov[r] = 0;
    }
    if (DT == NB_U8 && a.ovf_ptr) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!ok[r]) continue;
        const int64_t k0 = a.ovf_ptr[row0 + r], k1 = a.ovf_ptr[row0 + r + 1];
        for (int64_t k = k0 + li; k < k1; k += LPR) {
          const uint32_t col = a.ovf_col[k];
          const float add = (float)a.ovf_add[k];
          if (col < (uint32_t)a.F) {
            s[r] = fmaf(add, a.delta[col], s[r]);
            tot[r] += add;
            ++nov[r];
          } else {
            atomicOr(a.status, ST_OVF_RANGE);
          }
        }
      }
    }
#pragma unroll
    for (int off = LPR / 2; off > 0; off >>= 1) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        s[r] += __shfl_xor_sync(0xFFFFFFFFu, s[r], off);
        tot[r] += __shfl_xor_sync(0xFFFFFFFFu, tot[r], off);
        nov[r] = max(nov[r], __shfl_xor_sync(0xFFFFFFFFu, nov[r], off));
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!ok[r] || (r % LPR) != li) continue;
      float scale = 1.f;
      if (DT == NB_FP8E4M3 && a.row_exp) scale = exp2f((float)a.row_exp[row0 + r]);
      const float sum = s[r] * scale;
      const float d = sum + h.b;
      const float k = (float)(a.k_base + nov[r]);
      const float gam = k * 5.9604645e-8f / (1.f - k * 5.9604645e-8f);
      const float A = tot[r] * scale * h.maxabs * 1.001f;
      const float tau = gam * (A + fabsf(h.b)) * 1.01f + 1e-12f * (A + fabsf(h.b)) + 1e-30f;
      // marked rows are rare: one atomic each, no state carried through the loop
      if (c2_store(a.label, a.margin, a.logpost, a.want_lp, a.recheck, row0 + r, d, tau) && a.marks)
        atomicAdd(a.marks, 1ull);
    }
  }
}

// ---------------------------------------------------------------------------
// F32, U16 and BF16 counts in the log-posterior mode: exact integer sums
// ---------------------------------------------------------------------------
// FP32 sums of rows row0 .. row0 + 3 (rows past the end repeat the last one),
// 32 lanes per row.  Lane k (k < 4) receives row k's sum and |x| total.
template <int DT>
__device__ __forceinline__ void float_rows4(const S2Args& a, int64_t row0, float& s_out,
                                            float& t_out) {
  using Dec = Decode<DT>;
  constexpr int EPV = Dec::EPV;
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int r = 0; r < 4; ++r) {
    const char* rp = a.X + min(row0 + r, a.n - 1) * a.ld_bytes;
    float acc[4] = {0.f, 0.f, 0.f, 0.f}, tf = 0.f;
    for (int v = lane; v < a.nvec_row; v += 32) {
      float val[EPV];
      Dec::run(ld_stream16(rp + (int64_t)v * 16), val);
      const float4* w4 = reinterpret_cast<const float4*>(a.delta) + (int64_t)v * (EPV / 4);
#pragma unroll
      for (int q = 0; q < EPV / 4; ++q) {
        const float4 w = __ldg(w4 + q);
        const float ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x = v * EPV + 4 * q + e < a.F ? val[4 * q + e] : 0.f;
          acc[e] = fmaf(x, ww[e], acc[e]);
          tf += fabsf(x);
        }
      }
    }
    float s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      s += __shfl_xor_sync(0xFFFFFFFFu, s, off);
      tf += __shfl_xor_sync(0xFFFFFFFFu, tf, off);
    }
    if (lane == r) {
      s_out = s;
      t_out = tf;
    }
  }
}

__device__ __forceinline__ void c2_float_store(const S2Args& a, const C2Header& h, int64_t row,
                                               float s, float T) {
  const float d = s + h.b;
  const float k = (float)a.k_base;
  const float gam = k * 5.9604645e-8f / (1.f - k * 5.9604645e-8f);
  const float A = T * h.maxabs * 1.001f;
  const float tau = gam * (A + fabsf(h.b)) * 1.01f + 1e-12f * (A + fabsf(h.b)) + 1e-30f;
  if (c2_store(a.label, a.margin, a.logpost, a.want_lp, a.recheck, row, d, tau) && a.marks)
    atomicAdd(a.marks, 1ull);
}

__device__ __forceinline__ void c2_fix_store(const S2Args& a, const C2Header& h, int64_t row,
                                             long long D, float Rs, float T, int depth) {
  double d;
  float tau;
  fix_result(D, Rs, T, depth, h, d, tau);
  if (c2_store64(a.label, a.margin, a.logpost, a.want_lp, a.recheck, row, (float)d, d, tau) && a.marks)
    atomicAdd(a.marks, 1ull);
}

// The totals T of a group's four rows' counts and R of their residuals, by quarter as in
// sum4_transposed.
template <int LPR>
__device__ __forceinline__ void fix_totals(const FixSum2 (&fix)[2], int li, float& T, float& R) {
  float v[4];
  f32x2_unpack(fix[0].t, v[0], v[1]);
  f32x2_unpack(fix[1].t, v[2], v[3]);
  T = sum4_transposed<LPR>(v[0], v[1], v[2], v[3], li);
  f32x2_unpack(fix[0].r, v[0], v[1]);
  f32x2_unpack(fix[1].r, v[2], v[3]);
  R = sum4_transposed<LPR>(v[0], v[1], v[2], v[3], li);
}

// Short rows of 16-bit values: a group of LPR lanes sums four rows at a time;
// the fixed-point table sits in shared memory.  Only if a row of a group holds
// something else than counts are the group's rows read again for the FP32
// sums.  Bound by about 9 operations a value (F = 128: 2.8 TB/s).
template <int DT, int LPR>
__global__ void __launch_bounds__(256, 3) k_score2_fix(const S2Args a) {
  using Dec = Decode<DT>;
  constexpr int EPV = Dec::EPV, R = 4, SUBS = 32 / LPR, RPW = SUBS * R;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t bar;
  if (!stage_table(smem_raw, a.table, a.table_bytes, &bar, a.status, ST_TIMEOUT)) return;
  const int4* tab = reinterpret_cast<const int4*>(smem_raw);
  const float4* res = reinterpret_cast<const float4*>(smem_raw + a.table_bytes / 2);
  const C2Header h = *a.hdr;
  const int lane = threadIdx.x & 31, sub = lane / LPR, li = lane % LPR;
  const int nv = a.nvec_row;
  const int64_t ntiles = (a.n + RPW - 1) / RPW;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntiles;
       t += nwarps) {
    const int64_t row0 = t * RPW + (int64_t)sub * R;
    const char* rp[R];
    FixSum2 fix[R / 2];
#pragma unroll
    for (int r = 0; r < R; ++r)   // rows past the end repeat the last one and store nothing
      rp[r] = a.X + min(row0 + r, a.n - 1) * a.ld_bytes;
#pragma unroll 2
    for (int v = li; v < nv; v += LPR) {
      uint4 x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = ld_stream16(rp[r] + (int64_t)v * 16);
      int q[EPV];
      float qr[EPV];
#pragma unroll
      for (int k = 0; k < EPV / 4; ++k) {
        const int4 d = tab[v * (EPV / 4) + k];
        const float4 e = res[v * (EPV / 4) + k];
        qr[4 * k] = e.x;
        qr[4 * k + 1] = e.y;
        qr[4 * k + 2] = e.z;
        qr[4 * k + 3] = e.w;
        q[4 * k] = d.x;
        q[4 * k + 1] = d.y;
        q[4 * k + 2] = d.z;
        q[4 * k + 3] = d.w;
      }
#pragma unroll
      for (int r = 0; r < R; r += 2) {
        float v0[EPV], v1[EPV];
        Dec::run(x[r], v0);
        Dec::run(x[r + 1], v1);
        if (v == nv - 1) {
#pragma unroll
          for (int e = 0; e < EPV; ++e)
            if (v * EPV + e >= a.F) v0[e] = v1[e] = 0.f;
        }
#pragma unroll
        for (int e = 0; e < EPV; ++e) fix_add(fix[r / 2], v0[e], v1[e], q[e], qr[e]);
      }
    }
    // per row: the groups whose row is no row of counts
    const unsigned bad[R] = {__ballot_sync(0xFFFFFFFFu, fix[0].bad0()),
                             __ballot_sync(0xFFFFFFFFu, fix[0].bad1()),
                             __ballot_sync(0xFFFFFFFFu, fix[1].bad0()),
                             __ballot_sync(0xFFFFFFFFu, fix[1].bad1())};
    const unsigned any = bad[0] | bad[1] | bad[2] | bad[3];
    const long long D = sum4_transposed<LPR>(fix[0].D0, fix[0].D1, fix[1].D0, fix[1].D1, li);
    float T, Rs;
    fix_totals<LPR>(fix, li, T, Rs);
    const int mr = li / (LPR / 4);   // this lane's quarter holds row mr of the group
    const unsigned gmask = LPR == 32 ? 0xFFFFFFFFu : ((1u << (LPR & 31)) - 1u) << (sub * LPR);
    const unsigned mybad = (mr == 0 ? bad[0] : mr == 1 ? bad[1] : mr == 2 ? bad[2] : bad[3]) & gmask;
    if (li % (LPR / 4) == 0 && row0 + mr < a.n && mybad == 0u)
      c2_fix_store(a, h, row0 + mr, D, Rs, T, EPV * ((nv + LPR - 1) / LPR) + 5);
    if (any) {
#pragma unroll 1
      for (int g = 0; g < SUBS; ++g) {
        const unsigned gm = LPR == 32 ? 0xFFFFFFFFu : ((1u << (LPR & 31)) - 1u) << (g * LPR);
        if (!(any & gm)) continue;
        const int64_t r0 = t * RPW + (int64_t)g * R;
        float s = 0.f, tt = 0.f;
        float_rows4<DT>(a, r0, s, tt);
        const unsigned lb = (lane == 0 ? bad[0] : lane == 1 ? bad[1] : lane == 2 ? bad[2] : bad[3]) & gm;
        if (lane < R && lb && r0 + lane < a.n) c2_float_store(a, h, r0 + lane, s, tt);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// F32, U16 and BF16 rows of any alignment (a row width or a base that is no
// multiple of 16 bytes)
// ---------------------------------------------------------------------------
// A warp takes four rows at a time; lane l reads elements l, l + 32, ... of
// each with element-wise loads (a row's 32 loads cover 64 or 128 consecutive
// bytes), U elements of each row in flight, and each entry of the Delta
// tables, which stay in L1, once for the four rows.  FIX: exact sums, the FP32
// ones only where a row holds something else than counts.  Without FIX (label
// and OFF modes) the FP32 sums.
// 100,003 rows of 1,003 F32 counts (401 MB), log-posterior mode, labels only:
// 76 us for the whole call; 3.57 ms as 2 of the 64 class columns of the general
// scorer's 64 x 64 tiles (1.08 ms) and every row in FP64 on top (2.5 ms).
// 249,252 rows (1 GB): 158 us in the label mode (93% of the measured HBM rate),
// 190 us (78%) in the log-posterior mode.
template <int DT>
__device__ __forceinline__ float any_load(const char* rp, int j) {
  if (DT == NB_F32) {
    float v;
    asm volatile("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(rp + (int64_t)j * 4));
    return v;
  }
  unsigned short h;
  asm volatile("ld.global.nc.L1::no_allocate.u16 %0, [%1];" : "=h"(h) : "l"(rp + (int64_t)j * 2));
  return DT == NB_U16 ? (float)h : __uint_as_float((uint32_t)h << 16);
}

template <int DT, bool FIX>
__global__ void __launch_bounds__(256, 3) k_score2_any(const S2Args a) {
  constexpr int R = 4, U = 8;   // rows, elements in flight per row and lane
  const int lane = threadIdx.x & 31;
  const C2Header h = *a.hdr;
  const int64_t ntiles = (a.n + R - 1) / R;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < ntiles;
       t += nwarps) {
    const char* rp[R];
#pragma unroll
    for (int r = 0; r < R; ++r)   // rows past the end repeat the last one and store nothing
      rp[r] = a.X + min(t * R + r, a.n - 1) * a.ld_bytes;
    // every element once: add(the rows' values, the tables' entry)
    auto sweep = [&](auto&& table, auto&& add) {
      for (int j = lane; j < a.F; j += 32 * U) {
        float x[U][R];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int r = 0; r < R; ++r) x[u][r] = j + 32 * u < a.F ? any_load<DT>(rp[r], j + 32 * u) : 0.f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const auto w = table(j + 32 * u < a.F ? j + 32 * u : 0);
          add(x[u], w);
        }
      }
    };
    const int64_t row = t * R + lane / 8;   // eight lanes hold each row's sums
    bool todo = true;
    if (FIX) {
      FixSum2 fix[R / 2];
      sweep([&](int j) { return __ldg(a.delta_pr + j); },
            [&](const float (&x)[R], int2 q) {
              fix_add(fix[0], x[0], x[1], q.x, __int_as_float(q.y));
              fix_add(fix[1], x[2], x[3], q.x, __int_as_float(q.y));
            });
      // bit r: row r is no row of counts
      const unsigned bad = (__any_sync(0xFFFFFFFFu, fix[0].bad0()) ? 1u : 0u) |
                           (__any_sync(0xFFFFFFFFu, fix[0].bad1()) ? 2u : 0u) |
                           (__any_sync(0xFFFFFFFFu, fix[1].bad0()) ? 4u : 0u) |
                           (__any_sync(0xFFFFFFFFu, fix[1].bad1()) ? 8u : 0u);
      const long long D = sum4_transposed<32>(fix[0].D0, fix[0].D1, fix[1].D0, fix[1].D1, lane);
      float T, Rs;
      fix_totals<32>(fix, lane, T, Rs);
      todo = (bad >> (lane / 8)) & 1u;
      if (lane % 8 == 0 && row < a.n && !todo) c2_fix_store(a, h, row, D, Rs, T, (a.F + 31) / 32 + 5);
      if (!bad) continue;
    }
    float s[R] = {0.f, 0.f, 0.f, 0.f}, tf[R] = {0.f, 0.f, 0.f, 0.f};
    sweep([&](int j) { return __ldg(a.delta + j); },
          [&](const float (&x)[R], float w) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
              s[r] = fmaf(x[r], w, s[r]);
              tf[r] += fabsf(x[r]);
            }
          });
    const float S = sum4_transposed<32>(s[0], s[1], s[2], s[3], lane);
    const float T = sum4_transposed<32>(tf[0], tf[1], tf[2], tf[3], lane);
    if (lane % 8 == 0 && row < a.n && todo) c2_float_store(a, h, row, S, T);
  }
}

// ---------------------------------------------------------------------------
// launcher
// ---------------------------------------------------------------------------
template <typename K>
static nb_status launch_persistent(K kernel, int smem, int64_t ntiles_warp, const S2Args& a,
                                   cudaStream_t st) {
  static thread_local const void* last_k = nullptr;
  static thread_local int last_smem = -1, last_occ = 0;
  if (smem > kSmemOptIn) {
    NB_TRY_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                "cudaFuncSetAttribute");
  }
  int occ;
  if (last_k == (const void*)kernel && last_smem == smem) {
    occ = last_occ;
  } else {
    NB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 256, smem),
                "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    last_k = (const void*)kernel;
    last_smem = smem;
    last_occ = occ;
  }
  if (occ < 1) occ = 1;
  int64_t blocks = (ntiles_warp + 7) / 8;
  const int64_t cap = (int64_t)num_sms() * occ;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  count_launch();
  kernel<<<(unsigned)blocks, 256, smem, st>>>(a);
  NB_TRY_CUDA(cudaGetLastError(), "score2 launch");
  return NB_OK;
}

static int pick_lpr(int nvec_row) {
  int lpr = 1;
  while (lpr < 32 && lpr * 2 < nvec_row) lpr *= 2;
  return lpr;
}

// u8 and FP8 rows: about eight 16-byte vectors per lane and at least two lanes
// per row (measured, 4M files: u8 F = 256 at 89% of HBM against 61% with two
// vectors per lane, F = 64 at 65% against 61%, F = 4096 unchanged at 98%; FP8
// F = 256 at 54% against 36%, F = 1024 at 48% against 37%)
static int pick_lpr_u8(int nvec_row) {
  int lpr = 2;
  while (lpr < 32 && lpr * 8 < nvec_row) lpr *= 2;
  return lpr;
}

static int ilog2(int v) {
  int k = 0;
  while ((1 << k) < v) ++k;
  return k;
}

template <int LPR>
static nb_status dispatch_dt(nb_dtype dt, S2Args& a, int smem, cudaStream_t st) {
  constexpr int R = 4;
  const int64_t rpw = (32 / LPR) * R;
  const int64_t ntiles = (a.n + rpw - 1) / rpw;
  switch (dt) {
    case NB_U8:
      if (a.nvec_row < 16) {   // short rows: two rows per lane group, twice the warps per SM
        const int64_t rpw2 = (32 / LPR) * 2;
        return launch_persistent(k_score2_u8<NB_U8, LPR, 2>, smem, (a.n + rpw2 - 1) / rpw2, a,
                                 st);
      }
      return launch_persistent(k_score2_u8<NB_U8, LPR, R>, smem, ntiles, a, st);
    case NB_F32:
      return launch_persistent(k_score2_fp<NB_F32, LPR, R>, smem, ntiles, a, st);
    case NB_U16:
      return launch_persistent(k_score2_fp<NB_U16, LPR, R>, smem, ntiles, a, st);
    case NB_BF16:
      return launch_persistent(k_score2_fp<NB_BF16, LPR, R>, smem, ntiles, a, st);
    case NB_FP8E4M3:
      if (a.nvec_row < 16) {
        const int64_t rpw2 = (32 / LPR) * 2;
        return launch_persistent(k_score2_u8<NB_FP8E4M3, LPR, 2>, smem, (a.n + rpw2 - 1) / rpw2,
                                 a, st);
      }
      return launch_persistent(k_score2_u8<NB_FP8E4M3, LPR, R>, smem, ntiles, a, st);
  }
  set_error("unknown dtype");
  return NB_EINVAL;
}

// The exact-sum kernel on short rows: 4 or 8 lanes per row, at most 16 vectors.
template <int DT>
static nb_status launch_fix(const S2Args& a, int smem, cudaStream_t st) {
  if (a.nvec_row > 8) return launch_persistent(k_score2_fix<DT, 8>, smem, (a.n + 15) / 16, a, st);
  return launch_persistent(k_score2_fix<DT, 4>, smem, (a.n + 31) / 32, a, st);
}

// Narrow FP8 rows: about eight vectors per lane, at least two lanes per row.
static nb_status launch_fp8(const S2Args& a, int smem, cudaStream_t st) {
  if (a.nvec_row > 16) return launch_persistent(k_score2_fp8<4>, smem, (a.n + 15) / 16, a, st);
  return launch_persistent(k_score2_fp8<2>, smem, (a.n + 31) / 32, a, st);
}

nb_status launch_score2(const nb_model* m, const void* X, nb_dtype dt, int64_t n, int64_t ld,
                        const nb_aux* aux, const ScoreOut& o, cudaStream_t st) {
  const int es = elem_size(dt);
  S2Args a{};
  a.X = static_cast<const char*>(X);
  a.ld_bytes = ld * es;
  a.n = n;
  a.F = m->F;
  a.nvec_row = (m->F * es + 15) / 16;
  a.hdr = m->d.c2;
  a.delta_q = m->d.delta_q;
  a.delta = m->d.delta;
  a.delta_pr = m->d.delta_pr;
  a.ovf_ptr = aux ? aux->ovf_ptr : nullptr;
  a.ovf_col = aux ? aux->ovf_col : nullptr;
  a.ovf_add = aux ? aux->ovf_add : nullptr;
  a.row_exp = aux ? aux->row_exp : nullptr;
  a.label = o.label;
  a.margin = o.margin;
  a.logpost = o.logpost;
  a.want_lp = o.want_lp;
  a.recheck = o.recheck;
  a.marks = o.counted ? reinterpret_cast<unsigned long long*>(o.n_rechecked) : nullptr;
  a.status = m->d.sstatus;
  int smem;
  const bool limbs = dt == NB_U8 || dt == NB_FP8E4M3;   // fixed-point limbs, exact sums
  if (limbs) {
    a.nvec_tab = m->nvec8;
    a.table = m->d.limbs;
    smem = 3 * m->nvec8 * 16;
  } else {
    const int epv = 16 / es;
    a.nvec_tab = m->F_pad / epv;
    a.table = m->d.il[es == 4 ? 0 : (es == 2 ? 1 : 2)];
    smem = m->F_pad * 4;
  }
  a.table_bytes = (uint32_t)smem;
  if (n == 0) return NB_OK;
  const bool fp = dt == NB_F32 || dt == NB_U16 || dt == NB_BF16;
  const bool fix = fp && o.recheck == NB_RECHECK_LP;
  if (!c2_aligned(X, dt, ld)) {   // F32, U16 or BF16 (see score_path)
    a.k_base = (m->F + 31) / 32 + 5 + 2;   // serial FMAs, reduction, weight and final roundings
    const int64_t tiles = (n + 3) / 4;
    switch (dt) {
      case NB_F32:
        return fix ? launch_persistent(k_score2_any<NB_F32, true>, 0, tiles, a, st)
                   : launch_persistent(k_score2_any<NB_F32, false>, 0, tiles, a, st);
      case NB_U16:
        return fix ? launch_persistent(k_score2_any<NB_U16, true>, 0, tiles, a, st)
                   : launch_persistent(k_score2_any<NB_U16, false>, 0, tiles, a, st);
      default:
        return fix ? launch_persistent(k_score2_any<NB_BF16, true>, 0, tiles, a, st)
                   : launch_persistent(k_score2_any<NB_BF16, false>, 0, tiles, a, st);
    }
  }
  const nb_tile_config& cfg = m->tile;
  const bool open = cfg.variant == NB_VARIANT_AUTO && cfg.stages == 0 && cfg.rows_per_stage == 0 &&
                    cfg.rows_per_warp == 0;   // no kernel or shape is asked for
  if (dt == NB_FP8E4M3 && fp8_narrow(m->F) && cfg.variant != NB_VARIANT_REGISTER) {
    a.table = m->d.limbs5;
    smem = 5 * m->nvec8 * 16;
    a.table_bytes = (uint32_t)smem;
    return launch_fp8(a, smem, st);
  }
  // 16-bit rows of at most 16 vectors, which the pipelined kernel spreads over
  // 32 lanes (1M BF16 files: F = 64 52 us against 127, F = 128 93 against 159;
  // at F = 256 175 against 146 and at 1,024 291 against 211, so longer rows
  // stay there).  F32 rows stay with the FP32 sums, which batches share.
  if (fix && es == 2 && fix_rows(m->F) && cfg.variant != NB_VARIANT_REGISTER) {
    a.table = m->d.delta_p;   // and the residuals
    a.table_bytes = 2 * smem;
    a.k_base = (4 / es) + 2 + 5 + 2;   // of the FP32 sums, 32 lanes per row
    return dt == NB_U16 ? launch_fix<NB_U16>(a, 2 * smem, st) : launch_fix<NB_BF16>(a, 2 * smem, st);
  }
  // u8 and wider FP8 rows: the sums are exact, so the kernel and its shape change no
  // result, and the faster one is taken where none is asked for.  Dense rows
  // stream through registers: over F = 64 .. 6,000 that is the fastest or
  // within 4% of it (u8, against the pipelined kernel's default shape: 1M files
  // of F = 64 24 / 121 us, 256 56 / 162, 512 90 / 147; 586,000 of 1,024
  // 102 / 106; 293,000 of 2,048 102 / 139; FP8 from F = 512 on: 167 / 248, 198 / 207,
  // 195 / 238).  With an overflow list the pipelined kernel, whose
  // producer fetches the entries ahead, wins where the row fills its lanes:
  // 16 vectors (two rows per pass: F = 256 127 against 143 us), 32 (512:
  // 163 / 173), 52 to 64 (two rows: 900 148 / 165, 1,024 116 / 143) and up to
  // 128 (1,500 143 / 150, 2,048 103 / 118); elsewhere registers (F = 64
  // 48 / 225, 384 158 / 225, 640 192 / 225, 3,072 117 us).  The default shape
  // took 226 us at F = 256, 144 at 1,024 and 146 at 2,048.  Two stages of 48 rows; shorter ones while the call has fewer than
  // three tiles per block.
  nb_tile_config shape = cfg;
  bool pipe = cfg.variant != NB_VARIANT_REGISTER;
  if (limbs && open) {
    const int nv = a.nvec_row;
    pipe = a.ovf_ptr != nullptr && (nv == 16 || nv == 32 || (nv >= 52 && nv <= 128));
    shape.rows_per_warp = nv == 16 || (nv > 32 && nv <= 64) ? 2 : 1;
    shape.stages = 2;
    const int64_t blocks = (int64_t)num_sms() * 2;
    shape.rows_per_stage = n >= 3 * 48 * blocks ? 48 : (n >= 3 * 24 * blocks ? 24 : 16);
  }
  if (pipe) {
    // overflow slices are staged by bulk copies only from 16-byte aligned arrays
    S2Args ap = a;
    const int epv = 16 / es;
    ap.k_base = ((a.nvec_row + 31) / 32) * (epv / 4) + 2 + 5 + 2;
    const bool side_ok = !a.ovf_ptr || ((reinterpret_cast<uintptr_t>(a.ovf_col) & 15) == 0 &&
                                        (reinterpret_cast<uintptr_t>(a.ovf_add) & 15) == 0);
    const nb_status s =
        launch_score2_pipe(ap, dt, shape.stages, shape.rows_per_stage, shape.rows_per_warp,
                           side_ok ? 1 : 0, st);
    if (s != NB_EUNSUPPORTED || cfg.variant == NB_VARIANT_PIPELINED) return s;
  }
  const int lpr = limbs ? pick_lpr_u8(a.nvec_row) : pick_lpr(a.nvec_row);
  {
    const int epv = 16 / es;
    const int per_lane = (a.nvec_row + lpr - 1) / lpr;
    a.k_base = per_lane * (epv / 4) + 2 + ilog2(lpr) + 2;
  }
  switch (lpr) {
    case 1: return dispatch_dt<1>(dt, a, smem, st);
    case 2: return dispatch_dt<2>(dt, a, smem, st);
    case 4: return dispatch_dt<4>(dt, a, smem, st);
    case 8: return dispatch_dt<8>(dt, a, smem, st);
    case 16: return dispatch_dt<16>(dt, a, smem, st);
    default: return dispatch_dt<32>(dt, a, smem, st);
  }
}

}  // namespace nbg
