// Class counts N_cj = sum_{i : y_i = c} x_ij (exact, uint64) of a multinomial
// fit with any class count; rows of any 4-byte alignment.
//
// A short first kernel sorts the row numbers of each window of up to 1,024 rows
// by class.  A warp then owns a slab of 128 bytes of every row (lane: 4 bytes)
// and a range of windows, sums runs of one class in registers, and adds each
// run to the class's words for its slab in shared memory, each lane its own
// words, without atomics or conflicts.  u8 counts are summed as packed 16-bit
// pairs (even and odd bytes), which hold 256 rows of a class; wider types as
// 32-bit words, 255 rows of values below 2^24 (65,536 of u16).  A warp counts
// its rows per class and moves a class's words to the uint64 counts before they
// could overflow.  At its end it stores its words as they are, and
// k_counts_reduce adds them up.
//
// Bound by HBM latency and issue at 12 warps per SM (the classes' words leave no
// room for more): 64 rows ahead are in flight (8 KB per warp), rows are added
// four at a time where no run ends.  C = 64, F = 8,192, 262,144 u8 rows (2.1
// GB): 434 us (4.95 TB/s) + 9 for the lists + 12 for the reduction; bucketing
// all rows by class and summing 1 KB pieces of 128-row runs, each added to the
// counts with atomics, took 484 + 28 us.  On the way: rows in their stored order
// against shared memory 478 us (bound by its pipe), lists read in the step that
// uses them 981 us (the loads wait for the list), one step ahead 570 us.
#include "device.cuh"
#include "internal.cuh"

namespace nbg {

struct CrArgs {
  const char* X;
  int64_t ld_bytes, n;
  int F, C, slabs, splits, warps;   // warps per block
  int window, per_split;            // rows per window, windows per split
  const uint32_t* list;             // n entries, window by window
  const int* valid;                 // per window: entries of its list
  const int32_t* y;
  const int8_t* row_exp;
  unsigned long long* counts;
  unsigned long long* nc;
  uint32_t* part;                   // per (split, slab): C x 32 x NW words
  int* status;
};

// E features and NW accumulator words of a lane's 4 bytes; LIMIT rows per class
template <int DT>
struct CrType;
template <>
struct CrType<NB_U8> {
  static constexpr int E = 4, NW = 2, LIMIT = 256;
};
template <>
struct CrType<NB_U16> {
  static constexpr int E = 2, NW = 2, LIMIT = 65536;
};
template <>
struct CrType<NB_BF16> {
  static constexpr int E = 2, NW = 2, LIMIT = 255;
};
template <>
struct CrType<NB_F32> {
  static constexpr int E = 1, NW = 1, LIMIT = 255;
};
template <>
struct CrType<NB_FP8E4M3> {
  static constexpr int E = 4, NW = 4, LIMIT = 255;
};

__device__ __forceinline__ uint32_t cr_count(float v, int* status) {
  if (!(v >= 0.f) || v != floorf(v) || v >= 16777216.f) {
    atomicOr(status, ST_BAD_VALUE);
    return 0u;
  }
  return (uint32_t)v;
}

template <int DT>
__device__ __forceinline__ void cr_words(uint32_t w, int8_t ex, int* status,
                                         uint32_t (&v)[CrType<DT>::NW]) {
  if constexpr (DT == NB_U8) {
    v[0] = w & 0x00FF00FFu;
    v[1] = __byte_perm(w, 0u, 0x4341u);
  } else if constexpr (DT == NB_U16) {
    v[0] = w & 0xFFFFu;
    v[1] = w >> 16;
  } else if constexpr (DT == NB_BF16) {
    v[0] = cr_count(__uint_as_float(w << 16), status);
    v[1] = cr_count(__uint_as_float(w & 0xFFFF0000u), status);
  } else if constexpr (DT == NB_F32) {
    v[0] = cr_count(__uint_as_float(w), status);
  } else {
    const float sc = exp2f((float)ex);
    const float2 lo = e4m3x2_to_f32((uint16_t)(w & 0xFFFFu));
    const float2 hi = e4m3x2_to_f32((uint16_t)(w >> 16));
    v[0] = cr_count(lo.x * sc, status);
    v[1] = cr_count(lo.y * sc, status);
    v[2] = cr_count(hi.x * sc, status);
    v[3] = cr_count(hi.y * sc, status);
  }
}

// count of feature e of a lane's words
template <int DT>
__device__ __forceinline__ uint32_t cr_get(const uint32_t (&v)[CrType<DT>::NW], int e) {
  if constexpr (DT == NB_U8) {
    const uint32_t a = v[e & 1];
    return (e >> 1) ? a >> 16 : a & 0xFFFFu;
  } else {
    return v[e];
  }
}

template <int NW>
__device__ __forceinline__ void cr_load(const uint32_t* p, uint32_t (&v)[NW]) {
  if constexpr (NW == 1) {
    v[0] = *p;
  } else if constexpr (NW == 2) {
    const uint2 t = *reinterpret_cast<const uint2*>(p);
    v[0] = t.x;
    v[1] = t.y;
  } else {
    const uint4 t = *reinterpret_cast<const uint4*>(p);
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
  }
}
template <int NW>
__device__ __forceinline__ void cr_store(uint32_t* p, const uint32_t (&v)[NW]) {
  if constexpr (NW == 1) *p = v[0];
  else if constexpr (NW == 2) *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
  else *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
}

constexpr int kCrWarps = 12;       // most warps of a block; one block per SM
constexpr int kCrMaxWindow = 1024;
constexpr int kCrRun = 64;         // most rows of a run (below every LIMIT)

// An entry of a window's list: the row within the window, its class, and
// whether it ends a run of one class.
constexpr uint32_t kCrEnd = 0x80000000u, kCrNone = 0x40000000u;
__device__ __forceinline__ uint32_t cr_entry(int row, int c, bool end) {
  return (uint32_t)row | ((uint32_t)c << 16) | (end ? kCrEnd : 0u);
}

// Lists of the windows (one block each): the rows by class, in order inside a
// class; rows without a valid label are left out.  Also the class sizes.
__global__ void __launch_bounds__(256) k_counts_windows(const int32_t* y, int64_t n, int C, int window,
                                                        uint32_t* list, int* valid,
                                                        unsigned long long* nc, int* status) {
  extern __shared__ uint16_t cw_cnt[];   // [label group][class]
  __shared__ uint16_t off[256];
  __shared__ int wsum[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * window;
  const int nr = r0 < n ? (int)min((int64_t)window, n - r0) : 0;
  const int ng = (nr + 31) / 32;
  for (int k = threadIdx.x; k < ng * C; k += 256) cw_cnt[k] = 0;
  __syncthreads();
  auto label_of = [&](int g) {
    const int r = 32 * g + lane;
    int c = r < nr ? y[r0 + r] : -1;
    if (r < nr && (c < 0 || c >= C)) {
      atomicOr(status, ST_BAD_LABEL);
      c = -1;
    }
    return c;
  };
  for (int g = warp; g < ng; g += 8) {
    const int c = label_of(g);
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    if (c >= 0 && lane == __ffs(peers) - 1) cw_cnt[g * C + c] = (uint16_t)__popc(peers);
  }
  __syncthreads();
  int run = 0;   // rows of class threadIdx.x (C <= 255)
  if (threadIdx.x < C) {
#pragma unroll 4
    for (int g = 0; g < ng; ++g) {
      const int t = cw_cnt[g * C + threadIdx.x];
      cw_cnt[g * C + threadIdx.x] = (uint16_t)run;
      run += t;
    }
    if (run) atomicAdd(&nc[threadIdx.x], (unsigned long long)run);
  }
  int inc = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  int base = 0, total = 0;
  for (int w = 0; w < 8; ++w) {
    if (w < warp) base += wsum[w];
    total += wsum[w];
  }
  off[threadIdx.x] = (uint16_t)(base + inc - run);
  if (threadIdx.x == 0) valid[blockIdx.x] = total;
  __syncthreads();
  for (int g = warp; g < ng; g += 8) {
    const int c = label_of(g);
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    if (c < 0) continue;
    const int k = cw_cnt[g * C + c] + __popc(peers & ((1u << lane) - 1u));   // place in the class
    const int n_c = (c + 1 < 256 && c + 1 < C ? off[c + 1] : total) - off[c];
    list[r0 + off[c] + k] = cr_entry(32 * g + lane, c, k == n_c - 1 || k % kCrRun == kCrRun - 1);
  }
}

// shared bytes of one warp: C rows of words, then the rows per class since the
// last move
template <int DT>
static size_t cr_warp_bytes(int C) {
  return (size_t)C * 32 * CrType<DT>::NW * 4 + ((size_t)C + 3) / 4 * 16;
}

template <int DT>
__global__ void __launch_bounds__(kCrWarps * 32) k_counts_rows(const CrArgs a, uint32_t warp_bytes) {
  using T = CrType<DT>;
  constexpr int E = T::E, NW = T::NW;
  extern __shared__ __align__(16) unsigned char cr_sm[];
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0);   // uniform
  const long long item = (long long)blockIdx.x * a.warps + warp;
  if (item >= (long long)a.slabs * a.splits) return;
  const int C = a.C, slab = (int)(item % a.slabs);
  const long long split = item / a.slabs;
  uint32_t* acc = reinterpret_cast<uint32_t*>(cr_sm + (size_t)warp * warp_bytes);
  uint32_t* cnt = acc + (size_t)C * 32 * NW;   // rows of a class since its last move
  uint32_t* mine = acc + lane * NW;
  {
    const uint32_t z[NW] = {};
    for (int c = 0; c < C; ++c) cr_store<NW>(mine + c * 32 * NW, z);
    for (int c = lane; c < C; c += 32) cnt[c] = 0u;
  }
  __syncwarp();
  pdl_wait();   // the windows' lists
  const int j0 = (slab * 32 + lane) * E;   // this lane's first feature
  const bool on = j0 < a.F;
  // bytes of the features past F in a lane's word count nothing
  const int keep_bytes = (a.F - j0) * (4 / E);
  const uint32_t keep =
      keep_bytes >= 4 ? 0xFFFFFFFFu : (keep_bytes <= 0 ? 0u : (1u << (8 * keep_bytes)) - 1u);
  const bool whole = (slab + 1) * 32 * E <= a.F;   // every lane's features inside the row
  const char* base = a.X + (int64_t)(slab * 32 + lane) * 4;
  const int64_t ld = a.ld_bytes;

  auto flush = [&](int c) {   // class c's words to the uint64 counts
    uint32_t v[NW];
    const uint32_t z[NW] = {};
    cr_load<NW>(mine + c * 32 * NW, v);
    cr_store<NW>(mine + c * 32 * NW, z);
    unsigned long long* out = a.counts + (int64_t)c * a.F + j0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const uint32_t k = cr_get<DT>(v, e);
      if (k && j0 + e < a.F) atomicAdd(out + e, (unsigned long long)k);
    }
  };

  constexpr int U = 32;   // rows per step
  struct Step {
    uint32_t x[U];   // the rows' words
    uint32_t e;      // entry of slot `lane`
    int ex;          // FP8: exponent of slot `lane`'s row
  };
  // The steps of this warp's windows: a step's entries are read a step before
  // its rows, and those a step before they are added.
  struct Next {
    uint32_t e;      // entry of slot `lane`
    int64_t r0;      // first row of the window
    int left;        // rows of the window from this step on; 0: no step is left
  };
  const int w1 = (int)((split + 1) * a.per_split);
  int w = (int)(split * a.per_split), pos = 0, left = 0;
  auto next = [&](Next& x) {
    while (left <= 0 && w < w1) {
      left = a.valid[w];
      pos = 0;
      ++w;
    }
    x.left = left > 0 ? left : 0;
    x.r0 = (int64_t)(w - 1) * a.window;
    x.e = lane < left ? a.list[x.r0 + pos + lane] : kCrNone;
    pos += U;
    left -= U;
  };
  auto fetch = [&](const Next& x, Step& s) {
    s.e = x.e;
    const char* p = base + x.r0 * ld;
    if (DT == NB_FP8E4M3)
      s.ex = a.row_exp && lane < x.left ? (int)a.row_exp[x.r0 + (s.e & 0xFFFFu)] : 0;
    if (whole && x.left >= U) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];"
                     : "=r"(s.x[u])
                     : "l"(p + (int64_t)(__shfl_sync(0xFFFFFFFFu, s.e, u) & 0xFFFFu) * ld));
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t e = __shfl_sync(0xFFFFFFFFu, s.e, u);
        s.x[u] = 0u;
        if (on && !(e & kCrNone))
          s.x[u] = __ldg(reinterpret_cast<const uint32_t*>(p + (int64_t)(e & 0xFFFFu) * ld)) & keep;
      }
    }
  };
  uint32_t t[NW] = {};   // sums of the current run
  auto add = [&](const Step& s) {
    // rows per class of the step; a class that could overflow moves first (the
    // margin of one run: rows counted here may still wait in t)
    const int c = s.e & kCrNone ? -1 : (int)(s.e >> 16 & 0xFFu);
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, c);
    bool over = false;
    if (c >= 0 && lane == __ffs(peers) - 1) {
      const uint32_t q = __popc(peers), k = cnt[c] + q;
      over = k > (uint32_t)(T::LIMIT - kCrRun);
      cnt[c] = over ? q : k;
    }
    __syncwarp();
    for (unsigned m = __ballot_sync(0xFFFFFFFFu, over); m; m &= m - 1)
      flush(__shfl_sync(0xFFFFFFFFu, c, __ffs(m) - 1));
    const unsigned ends = __ballot_sync(0xFFFFFFFFu, (s.e & kCrEnd) != 0u);
    const int off = c * 32 * NW;
#pragma unroll
    for (int g = 0; g < U; g += 4) {
      uint32_t v[4][NW];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int ex = DT == NB_FP8E4M3 ? __shfl_sync(0xFFFFFFFFu, s.ex, g + q) : 0;
        cr_words<DT>(s.x[g + q], (int8_t)ex, a.status, v[q]);
      }
      if (((ends >> g) & 15u) == 0u) {   // no run ends here: the same for the warp
#pragma unroll
        for (int k = 0; k < NW; ++k) t[k] += (v[0][k] + v[1][k]) + (v[2][k] + v[3][k]);
        continue;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int k = 0; k < NW; ++k) t[k] += v[q][k];
        if ((ends >> (g + q)) & 1u) {
          uint32_t* p = mine + __shfl_sync(0xFFFFFFFFu, off, g + q);
          uint32_t o[NW];
          cr_load<NW>(p, o);
#pragma unroll
          for (int k = 0; k < NW; ++k) {
            o[k] += t[k];
            t[k] = 0u;
          }
          cr_store<NW>(p, o);
        }
      }
    }
  };
  // this step's rows, and those of the two that follow
  Step s0, s1, s2;
  Next n0, n1, n2;
  next(n1);
  next(n2);
  if (n1.left) fetch(n1, s1);
  next(n0);
  if (n2.left) fetch(n2, s2);
  while (n1.left > 0) {
    s0 = s1;
    s1 = s2;
    n1 = n2;
    n2 = n0;
    next(n0);
    if (n2.left) fetch(n2, s2);
    add(s0);
  }
  uint32_t* out = a.part + (size_t)item * C * 32 * NW + lane * NW;
  for (int c = 0; c < C; ++c) {
    uint32_t v[NW];
    cr_load<NW>(mine + c * 32 * NW, v);
    cr_store<NW>(out + (size_t)c * 32 * NW, v);
  }
}

// The warps' words of (slab, class) over up to kCrChunk splits, added to the counts.
constexpr int kCrChunk = 32;

template <int DT>
__global__ void __launch_bounds__(256) k_counts_reduce(const CrArgs a, long long nwork) {
  using T = CrType<DT>;
  constexpr int E = T::E, NW = T::NW;
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long wk = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (wk >= nwork) return;
  const int c = (int)(wk % a.C);
  const int slab = (int)(wk / a.C % a.slabs);
  const int k0 = (int)(wk / a.C / a.slabs) * kCrChunk;
  const int k1 = min(k0 + kCrChunk, a.splits);
  unsigned long long s[E] = {};
#pragma unroll 8
  for (int k = k0; k < k1; ++k) {
    uint32_t v[NW];
    cr_load<NW>(a.part + (((size_t)k * a.slabs + slab) * a.C + c) * 32 * NW + lane * NW, v);
#pragma unroll
    for (int e = 0; e < E; ++e) s[e] += cr_get<DT>(v, e);
  }
  const int j0 = (slab * 32 + lane) * E;
  unsigned long long* out = a.counts + (int64_t)c * a.F + j0;
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (s[e] && j0 + e < a.F) atomicAdd(out + e, s[e]);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
constexpr size_t kCrSmem = 216 * 1024;   // shared memory of an SM for the warps' words

template <int DT>
static CrArgs cr_plan(int64_t n, int F, int C, int* per_sm) {
  CrArgs a{};
  a.n = n;
  a.F = F;
  a.C = C;
  a.slabs = (F + 32 * CrType<DT>::E - 1) / (32 * CrType<DT>::E);
  int w = (int)(kCrSmem / cr_warp_bytes<DT>(C));
  w = w > kCrWarps ? kCrWarps : w;
  *per_sm = w;
  if (w < 1) return a;
  a.warps = w;
  // one item per resident warp, at least 64 rows each
  const long long total = (long long)num_sms() * w;
  long long splits = total / a.slabs;
  const long long most = (n + 63) / 64;
  splits = splits > most ? most : splits;
  a.splits = splits < 1 ? 1 : (int)splits;
  // windows of equal size, at most kCrMaxWindow rows
  const long long rows = (n + a.splits - 1) / a.splits;
  a.per_split = (int)((rows + kCrMaxWindow - 1) / kCrMaxWindow);
  a.window = (int)((rows + a.per_split - 1) / a.per_split);
  return a;
}

template <int DT>
static size_t cr_part_bytes(const CrArgs& a) {
  return (size_t)a.slabs * a.splits * a.C * 32 * CrType<DT>::NW * 4;
}

template <int DT>
static nb_status cr_run(CrArgs a, cudaStream_t st) {
  const size_t wb = cr_warp_bytes<DT>(a.C);
  const int smem = (int)(wb * a.warps);
  if (smem > kSmemOptIn)   // per device and function: set at every launch
    NB_TRY_CUDA(cudaFuncSetAttribute(k_counts_rows<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     smem),
                "cudaFuncSetAttribute(k_counts_rows)");
  const long long items = (long long)a.slabs * a.splits;
  const int wsmem = (int)(sizeof(uint16_t) * ((a.window + 31) / 32) * a.C);   // at most 16 KB
  count_launch();
  k_counts_windows<<<(unsigned)(a.splits * a.per_split), 256, wsmem, st>>>(
      a.y, a.n, a.C, a.window, const_cast<uint32_t*>(a.list), const_cast<int*>(a.valid), a.nc,
      a.status);
  NB_TRY_CUDA(cudaGetLastError(), "k_counts_windows");
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_counts_rows<DT>, dim3((unsigned)((items + a.warps - 1) / a.warps)),
                         dim3(a.warps * 32), (size_t)smem, st, a, (uint32_t)wb),
              "k_counts_rows");
  const long long nwork =
      (long long)((a.splits + kCrChunk - 1) / kCrChunk) * a.slabs * a.C;
  count_launch();
  NB_TRY_CUDA(launch_pdl(k_counts_reduce<DT>, dim3((unsigned)((nwork + 7) / 8)), dim3(256), 0, st, a,
                         nwork),
              "k_counts_reduce");
  return NB_OK;
}

template <int DT>
static nb_status cr_launch(nb_model* m, const void* X, int64_t n, int64_t ld, const int32_t* y,
                           const nb_aux* aux, bool aligned, cudaStream_t st) {
  int per_sm = 0;
  CrArgs a = cr_plan<DT>(n, m->F, m->C, &per_sm);
  // fewer than eight warps per SM leave HBM idle: the bucketed kernel then,
  // which takes 16-byte aligned rows (its element-wise form, for other rows, is
  // far slower than even one warp here)
  if (per_sm < (aligned ? 8 : 1)) return NB_EUNSUPPORTED;
  a.X = static_cast<const char*>(X);
  a.ld_bytes = ld * elem_size((nb_dtype)DT);
  a.y = y;
  a.row_exp = aux ? aux->row_exp : nullptr;
  a.counts = reinterpret_cast<unsigned long long*>(m->d.counts);
  a.nc = reinterpret_cast<unsigned long long*>(m->d.nc);
  a.status = m->d.status;
  FitScratch fs(m, st);
  void* p = nullptr;
  const size_t parts = cr_part_bytes<DT>(a), windows = (size_t)a.splits * a.per_split;
  nb_status s = fs.take(parts + windows * a.window * 4 + windows * sizeof(int), &p);
  if (s != NB_OK) return s;
  a.part = static_cast<uint32_t*>(p);
  a.list = reinterpret_cast<uint32_t*>(static_cast<char*>(p) + parts);
  a.valid = reinterpret_cast<const int*>(a.list + windows * a.window);
  s = cr_run<DT>(a, st);
  const nb_status f = fs.release();
  return s != NB_OK ? s : f;
}

// Counts and class sizes of n rows; NB_EUNSUPPORTED when the rows are not
// 4-byte aligned or the classes' words leave too few warps per SM.
nb_status launch_counts_rows(nb_model* m, const void* X, nb_dtype dt, int64_t n, int64_t ld,
                             const int32_t* y, const nb_aux* aux, cudaStream_t st) {
  const int64_t lb = ld * elem_size(dt);
  // a lane reads 4 bytes of a row: rows start on 4 bytes, and the last word of
  // a row ends inside its pitch
  if ((reinterpret_cast<uintptr_t>(X) & 3) != 0 || (lb & 3) != 0) return NB_EUNSUPPORTED;
  const bool aligned = c2_aligned(X, dt, ld);
  switch (dt) {
    case NB_U8: return cr_launch<NB_U8>(m, X, n, ld, y, aux, aligned, st);
    case NB_U16: return cr_launch<NB_U16>(m, X, n, ld, y, aux, aligned, st);
    case NB_F32: return cr_launch<NB_F32>(m, X, n, ld, y, aux, aligned, st);
    case NB_BF16: return cr_launch<NB_BF16>(m, X, n, ld, y, aux, aligned, st);
    case NB_FP8E4M3: return cr_launch<NB_FP8E4M3>(m, X, n, ld, y, aux, aligned, st);
  }
  return NB_EUNSUPPORTED;
}

}  // namespace nbg
