// Segmented persistent two-class scorers: one launch scores a whole batch of
// file groups of uneven size (1 .. 50,000 files and more), several resident
// models, under a captured CUDA graph (the paper's groups, Sec. 3 / Sec. 4,
// classified with their group's model).
//
// The launch reads its work list from device memory (header + one descriptor
// per group, see seg.cuh), so a graph captured once serves every batch, and
// every model's Delta table is staged in shared memory once per block.
//
// u8 rows (k_score2_seg_u8) stream through registers as in k_score2_u8: the
// list's 32-row chunks are cut into units of the rows that a warp takes at a
// time, and each warp takes a contiguous range of units, walking the groups.
// The sums are exact integers, so a group gives the same bits alone and inside
// any batch.
//
// F32 rows (k_score2_seg) go through the stage pipeline of pipe.cuh: the grid
// splits the list's tiles (RS rows of one group) into contiguous ranges per
// block; the producer warp walks the groups of its range and streams each
// tile's rows into shared-memory stages; a consumer warp reloads its register
// slice of the table when the stage's group uses another model; finished rows
// keep their group and are finalised 32 at a time.  The per-row arithmetic is
// the single-group kernel's (32 lanes per row).
#include "pipe.cuh"
#include "score2.cuh"
#include "seg.cuh"

namespace nbg {


// tiles of a block's range, walking the group list
struct SegSrc {
  const SegGroup* groups;
  int n_groups;
  long long t0;
  int RS;
  int g;
  TileInfo gi;      // fields of group g
  long long gt0;    // its first tile
  __device__ __forceinline__ void load(int gg) {
    const SegGroup& G = groups[gg];
    g = gg;
    gt0 = G.tile0;
    gi.X = G.X;
    gi.ld_bytes = G.ld_bytes;
    gi.group = gg;
    gi.ovf_ptr = G.ovf_ptr;
    gi.ovf_col = G.ovf_col;
    gi.ovf_add = G.ovf_add;
    gi.E = G.ovf_ptr ? G.ovf_ptr[G.n] : 0;
    gi.y = nullptr;
    gi.sizes = nullptr;
    gi.row0 = G.n;   // holds n until a tile is cut
  }
  __device__ __forceinline__ void init() {
    const SegGroup* gr = groups;
    load(seg_find(n_groups, t0, [gr](int i) { return gr[i].tile0; }));
  }
  __device__ __forceinline__ TileInfo tile(long long k) {
    const long long t = t0 + k;
    while (g + 1 < n_groups && groups[g + 1].tile0 <= t) load(g + 1);
    TileInfo r = gi;
    const long long n = gi.row0;
    r.row0 = (t - gt0) * RS;
    r.nr = (int)min((long long)RS, n - r.row0);
    return r;
  }
};

constexpr int kSegNCW = 8;   // consumer warps (two blocks per SM)

template <int KV>
__global__ void __launch_bounds__((kSegNCW + 1) * 32, 2) k_score2_seg(const SegArgs a, PipeArgs p) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ uint64_t full[kMaxStages], empty[kMaxStages], tabbar;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_groups = a.hdr->n_groups;
  const long long tiles = a.hdr->tiles;
  const long long t0 = tiles * blockIdx.x / gridDim.x;
  const long long t1 = tiles * (blockIdx.x + 1) / gridDim.x;
  const long long ntl = t1 - t0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kSegNCW);
    }
    mbar_init(&tabbar, 1);
  }
  __syncthreads();

  if (warp == kSegNCW) {
    pipe_stage_tables(sm, a.tables, a.n_models, a.table_bytes, a.table_stride, &tabbar);
    if (ntl > 0) {
      SegSrc src{a.groups, n_groups, t0, p.RS, 0, TileInfo{}, 0};
      src.init();
      pipe_produce_tiles(src, p, sm, full, empty, ntl, a.status);
    }
    return;
  }

  // ------------------------------------------------------------- consumers
  if (!mbar_wait_bounded(&tabbar, 0)) {
    if (lane == 0) atomicOr(a.status, ST_TIMEOUT);
    return;
  }
  const int nv = a.nvec_row, nt = a.nvec_tab;
  float4 wq[KV];
  int cur_g = -1, cur_m = -1;
  long long ld_bytes = 0;
  const int tail_v = a.F < nv * 4 ? nv - 1 : -1;

  float rs = 0.f, rtf = 0.f;
  long long rrow = -1;
  int rgrp = 0, nres = 0;
  unsigned marks = 0;

  auto finish = [&]() {
    if (lane < nres) {
      const SegGroup& G = a.groups[rgrp];
      const C2Header& H = *a.chdr[G.model];
      const float d = rs + H.b;
      const float kk = (float)a.k_base;
      const float gam = kk * 5.9604645e-8f / (1.f - kk * 5.9604645e-8f);
      const float A = rtf * H.maxabs * 1.001f;
      const float tau = gam * (A + fabsf(H.b)) * 1.01f + 1e-12f * (A + fabsf(H.b)) + 1e-30f;
      marks += c2_store(G.label, G.margin, G.logpost, a.want_lp, a.recheck, rrow, d, tau);
    }
    nres = 0;
  };

  for (long long k = 0; k < ntl; ++k) {
    const int s = (int)(k % p.S);
    const uint32_t ph = (uint32_t)((k / p.S) & 1);
    if (!mbar_wait_bounded(&full[s], ph)) {
      if (lane == 0) atomicOr(a.status, ST_TIMEOUT);
      return;
    }
    const unsigned char* st = sm + p.stages_off + (size_t)s * p.stage_bytes;
    const StageMeta* mp = reinterpret_cast<const StageMeta*>(st + p.meta_off);
    const int nr = mp->nr;
    const long long row0 = mp->row0;
    const int g = mp->group;
    if (g != cur_g) {
      cur_g = g;
      const SegGroup& G = a.groups[g];
      ld_bytes = G.ld_bytes;
      const int m = G.model;
      if (m != cur_m) {
        cur_m = m;
        const float4* tab = reinterpret_cast<const float4*>(sm + (size_t)m * a.table_stride);
#pragma unroll
        for (int kv = 0; kv < KV; ++kv) {
          const int v = lane + 32 * kv;
          wq[kv] = v < nv ? tab[v] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
    for (int r = warp; r < nr; r += kSegNCW) {
      if (nres == 32) finish();
      const unsigned char* rp = st + (size_t)r * ld_bytes;
      float acc[4] = {0.f, 0.f, 0.f, 0.f}, tf = 0.f;
#pragma unroll
      for (int kv = 0; kv < KV; ++kv) {
        const int v = lane + 32 * kv;
        if (v < nv) {
          const float4 x = *reinterpret_cast<const float4*>(rp + (size_t)v * 16);
          float val[4] = {x.x, x.y, x.z, x.w};
          if (v == tail_v) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (v * 4 + e >= a.F) val[e] = 0.f;
          }
          acc[0] = fmaf(val[0], wq[kv].x, acc[0]);
          acc[1] = fmaf(val[1], wq[kv].y, acc[1]);
          acc[2] = fmaf(val[2], wq[kv].z, acc[2]);
          acc[3] = fmaf(val[3], wq[kv].w, acc[3]);
          tf += fabsf(val[0]) + fabsf(val[1]) + fabsf(val[2]) + fabsf(val[3]);
        }
      }
      float sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
        tf += __shfl_xor_sync(0xFFFFFFFFu, tf, off);
      }
      if (lane == nres) {   // lane j holds the j-th finished row
        rs = sum;
        rtf = tf;
        rrow = row0 + r;
        rgrp = g;
      }
      ++nres;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (nres == 32) finish();
  }
  finish();
  if (marks) atomicAdd(a.marks, (unsigned long long)marks);
}

// ---------------------------------------------------------------------------
// u8 rows: a group of LPR lanes per row, R rows per group
// ---------------------------------------------------------------------------
// Bound by memory latency: a call gives each warp only a few units.  32 groups of
// 62,000 files in all, F = 2,048 (127 MB): 38 us; 53 us through shared-memory
// stages with one block of 12 consumer warps per SM.
template <int LPR, int R>
__global__ void __launch_bounds__(256, 2) k_score2_seg_u8(const SegArgs a) {
  constexpr int RPW = 32 / LPR * R, UPC = 32 / RPW;   // rows per unit, units per 32-row chunk
  static_assert(RPW <= 32, "a unit lies inside a chunk");
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_expect_tx(&bar, a.table_bytes * (uint32_t)a.n_models);
    for (int i = 0; i < a.n_models; ++i)
      for (uint32_t off = 0; off < a.table_bytes; off += 32768)
        bulk_g2s(sm + (size_t)i * a.table_stride + off, static_cast<const char*>(a.tables[i]) + off,
                 a.table_bytes - off < 32768 ? a.table_bytes - off : 32768, &bar);
  }
  __syncthreads();
  const bool ok = mbar_wait_bounded(&bar, 0);
  if (!ok) atomicOr(a.status, ST_TIMEOUT);
  if (__syncthreads_and(ok) == 0) {
    pdl_wait();   // as at the end
    return;
  }

  const int lane = threadIdx.x & 31, sub = lane / LPR, li = lane % LPR;
  const int nv = a.nvec_row, nt = a.nvec_tab, n_groups = a.hdr->n_groups;
  const long long units = a.hdr->chunks * UPC;
  const long long W = (long long)gridDim.x * 8, w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const long long u0 = units * w / W, u1 = units * (w + 1) / W;
  const SegGroup* gr = a.groups;
  // byte masks of the last (partial) vector
  const int keep = a.F - 16 * (nv - 1);
  uint32_t tm[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int vb = keep - 4 * q;
    vb = vb < 0 ? 0 : (vb > 4 ? 4 : vb);
    tm[q] = vb >= 4 ? 0xFFFFFFFFu : ((1u << (8 * vb)) - 1u);
  }
  unsigned marks = 0;
  // the range's first group: the last whose first chunk is not past it (the
  // lanes look at 32 groups at a time: one memory latency, not a search's six)
  int g = -1;
  if (u0 < u1) {
    const long long first = u0 / UPC;
    for (int k = 0; k < n_groups; k += 32) {
      const unsigned m = __ballot_sync(0xFFFFFFFFu, k + lane < n_groups && gr[k + lane].chunk0 <= first);
      g += __popc(m);
      if (m != 0xFFFFFFFFu) break;
    }
  }
  for (long long u = u0; u < u1; ++u) {
    const long long chunk = u / UPC;
    while (g + 1 < n_groups && gr[g + 1].chunk0 <= chunk) ++g;
    const SegGroup& G = gr[g];
    const long long n = G.n, ld = G.ld_bytes;
    const uint4* tab = reinterpret_cast<const uint4*>(sm + (size_t)G.model * a.table_stride);
    const long long row0 = (chunk - G.chunk0) * 32 + (u - chunk * UPC) * RPW + sub * R;
    const char* rp[R];
    int acc0[R], acc1[R], acc2[R];
    uint32_t tot[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {   // rows past the end repeat the last one and store nothing
      rp[r] = G.X + (row0 + r < n ? row0 + r : n - 1) * ld;
      acc0[r] = acc1[r] = acc2[r] = 0;
      tot[r] = 0u;
    }
#pragma unroll 4
    for (int v = li; v < nv; v += LPR) {
      uint4 x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = ld_stream16(rp[r] + (long long)v * 16);
      const uint4 q0 = tab[v], q1 = tab[nt + v], q2 = tab[2 * nt + v];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        uint32_t b[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
        if (v == nv - 1) {
#pragma unroll
          for (int q = 0; q < 4; ++q) b[q] &= tm[q];
        }
        const uint32_t l0[4] = {q0.x, q0.y, q0.z, q0.w}, l1[4] = {q1.x, q1.y, q1.z, q1.w},
                       l2[4] = {q2.x, q2.y, q2.z, q2.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc0[r] = dp4a_us(b[q], l0[q], acc0[r]);
          acc1[r] = dp4a_us(b[q], l1[q], acc1[r]);
          acc2[r] = dp4a_us(b[q], l2[q], acc2[r]);
          tot[r] = dp4a_uu(b[q], 0x01010101u, tot[r]);
        }
      }
    }
    if (G.ovf_ptr) {
      const signed char* limb = reinterpret_cast<const signed char*>(tab);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (row0 + r >= n) continue;
        const int64_t k1 = G.ovf_ptr[row0 + r + 1];
        for (int64_t k = G.ovf_ptr[row0 + r] + li; k < k1; k += LPR) {
          const uint32_t col = G.ovf_col[k];
          const int add = G.ovf_add[k];
          if (col < (uint32_t)a.F) {
            const size_t at = (size_t)(col >> 4) * 16 + (col & 15);
            acc0[r] += add * (int)limb[at];
            acc1[r] += add * (int)limb[(size_t)nt * 16 + at];
            acc2[r] += add * (int)limb[(size_t)nt * 32 + at];
            tot[r] += (uint32_t)add;
          } else {
            atomicOr(a.status, ST_OVF_RANGE);
          }
        }
      }
    }
    const C2Header& H = *a.chdr[G.model];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      long long D = ((long long)acc2[r] << 16) + ((long long)acc1[r] << 8) + (long long)acc0[r];
#pragma unroll
      for (int off = LPR / 2; off > 0; off >>= 1) {
        D += __shfl_xor_sync(0xFFFFFFFFu, D, off);
        tot[r] += __shfl_xor_sync(0xFFFFFFFFu, tot[r], off);
      }
      if (row0 + r < n && r % LPR == li) {
        const float Dsum = (float)D * H.inv_scale;
        const float d = Dsum + H.b;
        const float tau = c2_tau_u8((float)tot[r], Dsum, H.b, H.inv_scale, H.maxabs);
        marks += c2_store(G.label, G.margin, G.logpost, a.want_lp, a.recheck, row0 + r, d, tau);
      }
    }
  }
  if (marks) atomicAdd(a.marks, (unsigned long long)marks);
  // launched programmatically behind the many-class kernel, whose output this
  // one does not read: its completion has to imply that one's
  pdl_wait();
}

// ---------------------------------------------------------------------------
template <int KV>
static nb_status run_seg(const SegArgs& a, const PipeArgs& p, int smem, cudaStream_t st) {
  auto kern = k_score2_seg<KV>;
  if (smem > kSmemOptIn)
    NB_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                "cudaFuncSetAttribute(seg)");
  int occ = 0;
  NB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, (kSegNCW + 1) * 32, smem),
              "occupancy(seg)");
  if (occ < 1) {
    set_error("segmented scorer does not fit on an SM");
    return NB_EUNSUPPORTED;
  }
  count_launch();
  kern<<<num_sms() * occ, (kSegNCW + 1) * 32, smem, st>>>(a, p);
  NB_TRY_CUDA(cudaGetLastError(), "k_score2_seg launch");
  return NB_OK;
}

// behind_tc: the many-class kernel is the launch before this one; it read the lists
// and the cleared counter as this one does, and triggers this one while it runs.  Behind
// anything else (the copy or the memset that settles those) an ordinary launch waits.
template <int LPR, int R>
static nb_status run_seg_u8(const SegArgs& a, bool behind_tc, cudaStream_t st) {
  auto kern = k_score2_seg_u8<LPR, R>;
  const int smem = (int)(a.table_stride * (uint32_t)a.n_models);
  if (smem > kSmemOptIn)
    NB_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                "cudaFuncSetAttribute(seg)");
  int occ = 0;
  NB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 256, smem),
              "occupancy(seg)");
  if (occ < 1) {
    set_error("segmented scorer does not fit on an SM");
    return NB_EUNSUPPORTED;
  }
  count_launch();
  const dim3 grid((unsigned)(num_sms() * occ));
  if (behind_tc) {
    NB_TRY_CUDA(launch_pdl(kern, grid, dim3(256), (size_t)smem, st, a), "k_score2_seg_u8 launch");
  } else {
    kern<<<grid, 256, smem, st>>>(a);
    NB_TRY_CUDA(cudaGetLastError(), "k_score2_seg_u8 launch");
  }
  return NB_OK;
}

// Plan of a segmented two-class launch for rows of at most max_ld_bytes: the
// stages of the F32 kernel, and for both types the rows per tile of the work
// list and the limits of what is accepted (tables and two stages in one
// block's shared memory).
//
// Rows per stage: at most 48 when groups may carry side arrays (the producer's
// lanes hold the overflow pointers of a tile), up to 240 for plain rows, so
// that stages of short rows still move tens of KB.
nb_status seg2_plan(nb_dtype dt, int F, int F_pad, long long max_ld_bytes, int n_models,
                    bool plain_rows, PipeArgs* p, int* kv_out, int* smem_out) {
  const int es = elem_size(dt);
  const int nvec_row = (F * es + 15) / 16;
  const int rpw = dt == NB_U8 ? (nvec_row <= 16 ? 4 : (nvec_row <= 32 ? 2 : 1)) : 1;
  const int lpr = 32 / rpw;
  const int kv = (nvec_row + lpr - 1) / lpr;
  const int kv_max = dt == NB_F32 ? 8 : 4;
  if (kv < 1 || kv > kv_max || max_ld_bytes > 8192) {
    set_error("batched two-class scoring supports rows of at most %d vectors and 8 KB",
              32 * kv_max);
    return NB_EUNSUPPORTED;
  }
  const int ncw = rpw > 1 ? 12 : ((dt == NB_F32 ? kv <= 8 : kv <= 2) ? 8 : 12);
  const uint32_t tab = dt == NB_U8 ? (uint32_t)(3 * F_pad) : (uint32_t)(4 * F_pad);
  const uint32_t stride = (tab + 127) / 128 * 128;
  long long per = 32768 / ((long long)ncw * rpw * max_ld_bytes);
  int rs = ncw * rpw * (int)(per > 0 ? per : 1);
  const int max_rows = plain_rows ? 240 : kMaxStageRows;
  if (rs > max_rows) {
    rs = max_rows - max_rows % (ncw * rpw);   // whole warp passes
    if (rs < 1) rs = max_rows;
  }
  const unsigned budget = ncw == 8 ? 100u * 1024u : 180u * 1024u;
  PipeArgs q{};
  pipe_layout(q, rs, 1, max_ld_bytes, !plain_rows, false, stride * (uint32_t)n_models, 0);
  int S = q.stages_off + q.stage_bytes > budget ? 2 : (int)((budget - q.stages_off) / q.stage_bytes);
  S = S < 2 ? 2 : (S > kMaxStages ? kMaxStages : S);
  pipe_layout(*p, rs, S, max_ld_bytes, !plain_rows, false, stride * (uint32_t)n_models, 0);
  *kv_out = kv;
  *smem_out = (int)(p->stages_off + (uint32_t)p->S * p->stage_bytes);
  if (*smem_out > 220 * 1024) {
    set_error("batched two-class scoring: %d models do not fit in shared memory", n_models);
    return NB_EUNSUPPORTED;
  }
  return NB_OK;
}

nb_status launch_score2_seg(const SegArgs& a, const PipeArgs& p, nb_dtype dt, int kv, int smem,
                            bool behind_tc, cudaStream_t st) {
  if (dt == NB_U8) {   // lanes per row: about eight vectors each (see pick_lpr_u8), rows as there
    const int nv = a.nvec_row;
    if (nv <= 16) return run_seg_u8<2, 2>(a, behind_tc, st);
    if (nv <= 32) return run_seg_u8<4, 4>(a, behind_tc, st);
    if (nv <= 64) return run_seg_u8<8, 4>(a, behind_tc, st);
    return run_seg_u8<16, 4>(a, behind_tc, st);
  }
  if (dt == NB_F32) {
    switch (kv) {
      case 1: return run_seg<1>(a, p, smem, st);
      case 2: return run_seg<2>(a, p, smem, st);
      case 3: return run_seg<3>(a, p, smem, st);
      case 4: return run_seg<4>(a, p, smem, st);
      case 5: return run_seg<5>(a, p, smem, st);
      case 6: return run_seg<6>(a, p, smem, st);
      case 7: return run_seg<7>(a, p, smem, st);
      case 8: return run_seg<8>(a, p, smem, st);
    }
  }
  set_error("batched two-class scoring supports u8 and f32 storage");
  return NB_EUNSUPPORTED;
}

}  // namespace nbg
