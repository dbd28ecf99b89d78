// K1 (message weights, Eq. (1)) and K2 (stable LSD radix sort of the step's
// row keys) of the GBA aggregate-and-apply step.
//
// The sort follows the onesweep method (Adinets & Merrill 2022): one kernel
// maps the ids to 32-bit keys (global row = table key base + row) and counts
// the digits of every pass, then each pass is a single kernel in which tiles
// rank their keys locally and find their global output offsets by decoupled
// look-back over the per-tile digit counts of earlier tiles (Merrill & Garland
// 2016).  Tiles take tickets from an atomic counter, so a tile only ever waits
// on tiles that are already running; every wait is bounded in time and latches
// ERR_TIMEOUT instead of hanging.  The payload is the global occurrence index.
#include <algorithm>

#include "gba_internal.cuh"

namespace gba {

namespace {

constexpr int SORT_THREADS = 256;
constexpr int SORT_WARPS = SORT_THREADS / 32;
constexpr int OFF_CACHE = 1024;  // message offsets kept in shared memory
constexpr int TAB_CACHE = 64;    // tables whose bounds are kept in shared memory
constexpr uint32_t FULL = 0xffffffffu;

// Look-back status word: [63:32] epoch of the launch, [31:30] flag, [29:0] count.
constexpr unsigned long long FLAG_AGG = 1ull << 30;
constexpr unsigned long long FLAG_INCL = 2ull << 30;
constexpr unsigned long long FLAG_MASK = 3ull << 30;
constexpr unsigned long long COUNT_MASK = (1ull << 30) - 1;

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p) {
  return *(const volatile uint32_t*)p;
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Row of an id in table t (DIRECT ids outside [0, V) latch ERR_ID_RANGE and
// are clamped to row 0; the whole step is then skipped by later kernels).
__device__ __forceinline__ uint64_t row_of_id(const StepArgs& a, const TableInfo& ti, int t,
                                              int64_t id, const ErrSink& err) {
  uint64_t row;
  if (ti.id_mode == 0) {
    row = (uint64_t)id;
    if (id < 0 || id >= ti.V) {
      raise_error(err, ERR_ID_RANGE);
      row = 0;
    }
  } else if (ti.id_mode == 1) {
    row = mod_u64((uint64_t)id, (uint64_t)ti.V, ti.mod_magic);
  } else {  // HASH: the id's slot, inserted on first sight
    if ((unsigned long long)id == HASH_EMPTY) {
      raise_error(err, ERR_ID_RANGE);
      row = 0;
    } else {
      row = hash_find_or_insert(a.hinfo[t], id);
      if (row > a.hinfo[t].mask) {
        raise_error(err, ERR_INTERNAL);
        row = 0;
      }
    }
  }
  return row;
}

// ---------------------------------------------------------------------------
// K1: message weights of Eq. (1), kept-message list, dense staleness counters;
// also clears the per-step sort scratch, and brings the step's description from
// the host: a description of up to META_BY_KERNEL bytes is read from pinned host
// memory here, while the kernel before may still run, instead of by a copy of its
// own in front (about 6 us of a small step, with the gaps around it).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
    k_message_weights(StepArgs a, StepScratch sc, DevStats* st, int n_hist_words,
                      const uint4* host_meta, uint4* dev_meta, int n16) {
  extern __shared__ uint4 s_meta[];
  const int tid = threadIdx.x;
  for (int i = tid; i < n16; i += blockDim.x) {
    uint4 v;  // volatile: the host rewrites this memory between steps
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(host_meta + i)
                 : "memory");
    s_meta[i] = v;
  }
  chain_wait();
  for (int i = tid; i < n16; i += blockDim.x) dev_meta[i] = s_meta[i];
  __syncthreads();  // the tokens are read back below
  for (int i = tid; i < n_hist_words; i += blockDim.x) sc.hist[i] = 0u;
  if (tid < MAX_PASSES) sc.tile_counter[tid] = 0u;
  if (tid == 0) *sc.step_err = 0u;
  if (sc.seg_ticket)
    for (int i = tid; i < 8 * a.T; i += blockDim.x) sc.seg_ticket[i] = 0u;
  if (tid >= 32) return;
  const int lane = tid;
  int kept = 0;
  unsigned long long s_sum = 0, s_max = 0;
  for (int base = 0; base < a.M; base += 32) {
    const int m = base + lane;
    int keep = 0;
    unsigned long long s = 0;
    float f = 0.f;
    if (m < a.M) {
      const int64_t diff = a.k - a.tokens[m];
      s = diff > 0 ? (unsigned long long)diff : 0ull;
      // Eq. (1) (or the decay strategy), and Hop-BW's ignored latest messages
      f = m < a.M - a.drop_latest ? decay_weight(a, s) : 0.f;
      keep = f > 0.f ? 1 : 0;
      sc.keep[m] = keep;
    }
    const uint32_t b = __ballot_sync(0xffffffffu, keep != 0);
    if (keep) {
      const int j = kept + __popc(b & lanemask_lt());
      sc.kept_list[j] = m;
      if (sc.fw) sc.fw[j] = f;
    }
    kept += __popc(b);
    s_sum += s;
    s_max = s > s_max ? s : s_max;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s_sum += __shfl_xor_sync(0xffffffffu, s_sum, o);
    unsigned long long y = __shfl_xor_sync(0xffffffffu, s_max, o);
    s_max = y > s_max ? y : s_max;
  }
  if (lane == 0) {
    *sc.n_kept = kept;
    atomicAdd(&st->steps, 1ull);
    atomicAdd(&st->msgs_kept, (unsigned long long)kept);
    atomicAdd(&st->msgs_dropped, (unsigned long long)(a.M - kept));
    atomicAdd(&st->dense_stale_sum, s_sum);
    atomicMax(&st->dense_stale_max, s_max);
    atomicAdd(&st->occurrences, (unsigned long long)a.N);
  }
}

// ---------------------------------------------------------------------------
// Keys of every occurrence (keys0, the first pass's input) and the digit counts
// of every pass, in one read of the ids.
//
// Latency of the id gathers and, on small steps, the merging of the blocks'
// counts bound this kernel: four ids are in flight per thread, 1,024 occurrences
// within one message are read without looking each one up, and a block takes
// 2,048 keys (1,024 while there are fewer blocks than two per SM) before it adds
// its counts to the step's.  0.85M ids 17 -> 11.5 us, 131M 959 -> 719.
// ---------------------------------------------------------------------------
constexpr int HIST_ITEMS = 4;  // ids in flight per thread

template <int RADIX>
__global__ void __launch_bounds__(SORT_THREADS)
    k_sort_histogram(StepArgs a, SortPlan plan, uint32_t* __restrict__ hist,
                     uint32_t* __restrict__ keys0, ErrSink err) {
  __shared__ uint32_t h[MAX_PASSES][RADIX];
  __shared__ uint32_t s_off[OFF_CACHE];
  __shared__ uint32_t s_nb[TAB_CACHE + 1];
  const int tid = threadIdx.x;
  for (int i = tid; i < MAX_PASSES * RADIX; i += SORT_THREADS) (&h[0][0])[i] = 0u;
  chain_wait();
  const int T = a.T, M = a.M;
  const bool offs_cached = T * (M + 1) <= OFF_CACHE, tabs_cached = T <= TAB_CACHE;
  if (offs_cached)
    for (int i = tid; i < T * (M + 1); i += SORT_THREADS) s_off[i] = a.msg_off[i];
  if (tabs_cached)
    for (int i = tid; i <= T; i += SORT_THREADS) s_nb[i] = (uint32_t)a.nbase[i];
  __syncthreads();
  const uint32_t* offs = offs_cached ? s_off : a.msg_off;
  const uint32_t N = (uint32_t)a.N;  // below 2^30
  auto first_of = [&](int t) { return tabs_cached ? s_nb[t] : (uint32_t)a.nbase[t]; };
  const uint32_t step = (uint32_t)(SORT_THREADS * HIST_ITEMS);
  auto table_at = [&](uint32_t o) {  // the last table that starts at or before o
    int lo = 0, hi = T;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (first_of(mid) <= o)
        lo = mid;
      else
        hi = mid;
    }
    return lo;
  };
  auto message_at = [&](int t, uint32_t& x) {
    const float scale = __fdividef((float)M, (float)(first_of(t + 1) - first_of(t)));
    return message_of(offs + (size_t)t * (M + 1), M, x, scale);
  };
  auto count = [&](const TableInfo& ti, int t, uint32_t o, int64_t id) {
    const uint32_t key = ti.key_base + (uint32_t)row_of_id(a, ti, t, id, err);
    keys0[o] = key;
#pragma unroll
    for (int p = 0; p < MAX_PASSES; ++p)
      if (p < plan.passes) atomicAdd(&h[p][(key >> plan.shift[p]) & plan.mask[p]], 1u);
  };
  for (uint32_t base = blockIdx.x * step; base < N; base += gridDim.x * step) {
    const uint32_t here = min(step, N - base);
    const int t1 = table_at(base);
    uint32_t x1 = base - first_of(t1);
    const int m1 = message_at(t1, x1);
    const uint32_t* off1 = offs + (size_t)t1 * (M + 1) + m1;
    int64_t id[HIST_ITEMS];
    if (off1[1] - off1[0] - x1 >= here) {  // one message holds them all
      const int64_t* src = a.ids_ptr[(size_t)t1 * M + m1] + x1;
#pragma unroll
      for (int e = 0; e < HIST_ITEMS; ++e) {
        const uint32_t i = (uint32_t)(e * SORT_THREADS + tid);
        if (i < here) id[e] = src[i];
      }
      const TableInfo ti = a.tinfo[t1];
#pragma unroll
      for (int e = 0; e < HIST_ITEMS; ++e) {
        const uint32_t i = (uint32_t)(e * SORT_THREADS + tid);
        if (i < here) count(ti, t1, base + i, id[e]);
      }
    } else {
      int tab[HIST_ITEMS];
#pragma unroll
      for (int e = 0; e < HIST_ITEMS; ++e) {
        const uint32_t i = (uint32_t)(e * SORT_THREADS + tid);
        tab[e] = -1;
        if (i >= here) continue;
        const int t = table_at(base + i);
        uint32_t x = base + i - first_of(t);
        const int m = message_at(t, x);
        tab[e] = t;
        id[e] = a.ids_ptr[(size_t)t * M + m][x];
      }
#pragma unroll
      for (int e = 0; e < HIST_ITEMS; ++e)
        if (tab[e] >= 0)
          count(a.tinfo[tab[e]], tab[e], base + (uint32_t)(e * SORT_THREADS + tid), id[e]);
    }
  }
  __syncthreads();
  for (int i = tid; i < plan.passes * RADIX; i += SORT_THREADS) {
    const uint32_t v = (&h[0][0])[i];
    if (v) atomicAdd(hist + i, v);
  }
}

// ---------------------------------------------------------------------------
// One onesweep pass.
//
// Bound by instruction issue and latency: 16 B move per key, and a key costs
// about four warp instructions of 32.  Keys and payloads go to shared memory in
// digit order before the look-back, so that few registers live through it (48
// instead of 80: five blocks per SM instead of three); a short last tile is
// padded with the largest key, which needs no checks.  Lanes of equal digits find
// each other through a shared word of lane bits per digit (a step that CUB's onesweep
// ranks with as well) in the first pass, where digits come in no order (975 us against 1,097 with match.any on 131M keys), and
// by match.any in the later ones, where hot keys come in runs that would meet in
// one word (1,083 us against 824; ballots per bit 1,123).  Above
// SORT_BIG_N keys a tile holds 4,096 of them (5.2M keys: 70 us a pass against 89
// with 2,048).  Digits are 8 bits wide, or up to 9 where that saves a pass: 26-bit
// keys take three passes.  131M keys: 4 x 1.46 -> 1.12 + 2 x 0.83 ms.  The later
// passes with 256 counters spill 12 to 16 bytes a thread, with 512 and large tiles 56.
// ---------------------------------------------------------------------------
template <int ITEMS, int RADIX, bool FIRST>
__global__ void __launch_bounds__(SORT_THREADS, ITEMS == 8 ? 5 : 4)
    k_onesweep(SortPass sp, ErrSink err, int64_t wait_ns) {
  constexpr int TILE = ITEMS * SORT_THREADS;
  constexpr int DPT = RADIX / SORT_THREADS;  // digits per thread: tid * DPT ..
  constexpr int WIN = DPT == 1 ? 8 : 4;      // look-back window
  static_assert(DPT == 1 || DPT == 2, "one or two digits per thread");
  __shared__ __align__(4) uint16_t s_cnt[SORT_WARPS][RADIX];  // per-warp digit counts, then offsets
  __shared__ uint32_t s_out[RADIX];   // output position of tile slot 0 of each digit
  __shared__ uint32_t s_tmp[2][SORT_WARPS];
  __shared__ uint32_t s_kv[2 * TILE];
  uint32_t* const s_keys = s_kv;
  uint32_t* const s_vals = s_kv + TILE;
  static_assert(SORT_WARPS * RADIX <= 2 * TILE, "a word of lane bits per warp and digit");
  __shared__ uint32_t s_tile;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* cnt_words = reinterpret_cast<uint32_t*>(&s_cnt[0][0]);
  for (int i = tid; i < SORT_WARPS * RADIX / 2; i += SORT_THREADS) cnt_words[i] = 0u;
  if (FIRST)
    for (int i = tid; i < SORT_WARPS * RADIX; i += SORT_THREADS) s_kv[i] = 0u;
  chain_wait();
  // the tile's ticket, the step's state and its digit counts in flight together
  uint32_t ticket = 0u;
  if (tid == 0) ticket = atomicAdd(sp.ticket, 1u);
  const uint32_t failed = ld_volatile_u32(err.step) & ERR_ID_RANGE;
  uint32_t hist_d[DPT];
#pragma unroll
  for (int q = 0; q < DPT; ++q) hist_d[q] = sp.hist[tid * DPT + q];
  if (tid == 0) s_tile = ticket;
  // An id range error was latched before this launch (by the histogram):
  // every tile of every pass skips, consistently.
  if (__syncthreads_or(failed != 0u)) return;

  const uint32_t tile = s_tile, N = sp.N;
  const uint32_t base = tile * (uint32_t)TILE;
  const uint32_t n_valid = min(N - base, (uint32_t)TILE);
  const int shift = sp.shift;
  const uint32_t mask = sp.mask;

  // The slots past the end hold the largest key: they are the last of the last
  // digit, so they rank behind every key and are taken off that digit's count.
  uint32_t key[ITEMS], val[ITEMS];
  const uint32_t at = (uint32_t)(warp * (ITEMS * 32) + lane);
  if (n_valid == (uint32_t)TILE) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      key[j] = sp.keys_in[base + at + j * 32];
      val[j] = FIRST ? base + at + j * 32 : sp.vals_in[base + at + j * 32];
    }
  } else {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const bool in = at + j * 32 < n_valid;
      key[j] = in ? sp.keys_in[base + at + j * 32] : 0xFFFFFFFFu;
      val[j] = FIRST ? base + at + j * 32 : (in ? sp.vals_in[base + at + j * 32] : 0u);
    }
  }

  // Warp-level multi-split: stable rank of each key among equal digits.
  const uint32_t lt = lanemask_lt();
  uint32_t rank[ITEMS / 2];  // two 16-bit ranks each
  uint32_t* lanes = s_kv + warp * RADIX;  // the places of the keys are still free
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t d = (key[j] >> shift) & mask;
    uint32_t peers;
    if (FIRST) {
      atomicOr(lanes + d, 1u << lane);
      __syncwarp();
      peers = lanes[d];
    } else {
      peers = __match_any_sync(FULL, d);
    }
    const uint32_t before = s_cnt[warp][d];
    const uint32_t r = before + __popc(peers & lt);
    rank[j / 2] = (j & 1) ? rank[j / 2] | (r << 16) : r;
    __syncwarp();
    if ((peers & lt) == 0u) {
      s_cnt[warp][d] = (uint16_t)(before + __popc(peers));
      if (FIRST) lanes[d] = 0u;
    }
    __syncwarp();
  }
  __syncthreads();

  // This thread's digits: the warps' offsets, the tile's counts, published for
  // the tiles that follow.
  uint32_t count[DPT];
  if constexpr (DPT == 1) {
    uint32_t run = 0u;
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) {
      const uint32_t c = s_cnt[w][tid];
      s_cnt[w][tid] = (uint16_t)run;
      run += c;
    }
    count[0] = run;
  } else {  // both digits in one word: a count is at most TILE < 2^16
    uint32_t run = 0u;
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) {
      uint32_t* word = reinterpret_cast<uint32_t*>(&s_cnt[w][2 * tid]);
      const uint32_t c = *word;
      *word = run;
      run += c;
    }
    count[0] = run & 0xFFFFu;
    count[DPT - 1] = run >> 16;
  }
#pragma unroll
  for (int q = 0; q < DPT; ++q)
    if ((uint32_t)(tid * DPT + q) == mask) count[q] -= (uint32_t)TILE - n_valid;
  unsigned long long* my = sp.status + (size_t)tile * RADIX + tid * DPT;
  const unsigned long long ep = (unsigned long long)sp.epoch << 32;
#pragma unroll
  for (int q = 0; q < DPT; ++q)
    st_relaxed_u64(my + q, ep | (tile == 0 ? FLAG_INCL : FLAG_AGG) | count[q]);

  // Exclusive scans over the digits of the tile's counts and of the step's.
  uint32_t t_sum = 0u, g_sum = 0u;
#pragma unroll
  for (int q = 0; q < DPT; ++q) {
    t_sum += count[q];
    g_sum += hist_d[q];
  }
  uint32_t t_inc = t_sum, g_inc = g_sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(FULL, t_inc, o), z = __shfl_up_sync(FULL, g_inc, o);
    if (lane >= o) {
      t_inc += y;
      g_inc += z;
    }
  }
  if (lane == 31) {
    s_tmp[0][warp] = t_inc;
    s_tmp[1][warp] = g_inc;
  }
  __syncthreads();
  uint32_t t_excl = t_inc - t_sum, g_excl = g_inc - g_sum;
#pragma unroll
  for (int w = 0; w < SORT_WARPS; ++w)
    if (w < warp) {
      t_excl += s_tmp[0][w];
      g_excl += s_tmp[1][w];
    }
  // the warps' offsets within the tile
  if constexpr (DPT == 1) {
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) s_cnt[w][tid] = (uint16_t)(s_cnt[w][tid] + t_excl);
  } else {
    const uint32_t both = t_excl | (t_excl + count[0]) << 16;
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) cnt_words[w * (RADIX / 2) + tid] += both;
  }
  __syncthreads();

  // Keys and payloads in digit order in shared memory.
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t d = (key[j] >> shift) & mask;
    const uint32_t r = (j & 1) ? rank[j / 2] >> 16 : rank[j / 2] & 0xFFFFu;
    const uint32_t pos = s_cnt[warp][d] + r;
    s_keys[pos] = key[j];
    s_vals[pos] = val[j];
  }

  // Decoupled look-back over a window of WIN predecessors at a time: the
  // window's status words are read with independent loads, then consumed from
  // the nearest tile backwards until an inclusive prefix is found.  The words
  // are self-contained (no other data is published with them), so relaxed
  // loads and stores suffice.
  uint32_t prefix[DPT];
#pragma unroll
  for (int q = 0; q < DPT; ++q) prefix[q] = 0u;
  if (tile > 0) {
    int j = (int)tile - 1;
    const uint64_t t0 = globaltimer_ns();
    bool done = false;
    while (!done) {
      unsigned long long v[WIN][DPT];
#pragma unroll
      for (int i = 0; i < WIN; ++i)
#pragma unroll
        for (int q = 0; q < DPT; ++q)
          v[i][q] = j - i >= 0
                        ? ld_relaxed_u64(sp.status + (size_t)(j - i) * RADIX + tid * DPT + q)
                        : 0ull;
      int used = 0;
#pragma unroll
      for (int i = 0; i < WIN; ++i) {
        if (done || used != i) continue;
        // ready once the words carry this launch's epoch and one flag (before
        // tile 0 there are none: zero words are never ready)
        const unsigned long long tag = v[i][0] & ~COUNT_MASK;
        if ((tag >> 32) != (ep >> 32) || (tag & FLAG_MASK) == 0ull ||
            (v[i][DPT - 1] & ~COUNT_MASK) != tag)
          continue;
#pragma unroll
        for (int q = 0; q < DPT; ++q) prefix[q] += (uint32_t)(v[i][q] & COUNT_MASK);
        used = i + 1;
        if (tag & FLAG_INCL) done = true;
      }
      if (done) break;
      j -= used;
      if (j < 0) break;  // cannot happen: tile 0 publishes an inclusive prefix
      if (used == 0) {
        if ((ld_volatile_u32(err.step) & ERR_TIMEOUT) ||
            (int64_t)(globaltimer_ns() - t0) > wait_ns) {
          raise_error(err, ERR_TIMEOUT);
          break;
        }
        __nanosleep(LOOKBACK_SLEEP_NS);
      }
    }
#pragma unroll
    for (int q = 0; q < DPT; ++q)
      st_relaxed_u64(my + q, ep | FLAG_INCL | ((prefix[q] + count[q]) & COUNT_MASK));
  }
  s_out[tid * DPT] = g_excl + prefix[0] - t_excl;
  if constexpr (DPT == 2)
    s_out[tid * DPT + 1] = g_excl + hist_d[0] + prefix[DPT - 1] - (t_excl + count[0]);
  __syncthreads();

  // Runs of equal digits leave in order.
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t i = (uint32_t)(tid + j * SORT_THREADS);
    if (i < n_valid) {
      const uint32_t k = s_keys[i];
      const uint32_t out = s_out[(k >> shift) & mask] + i;
      if (out < N) {
        sp.keys_out[out] = k;
        sp.vals_out[out] = s_vals[i];
      } else {
        raise_error(err, ERR_INTERNAL);
      }
    }
  }
}

template <int ITEMS, int RADIX>
void sweep_as(const SortPass& sp, bool first, ErrSink err, int64_t wait_ns, cudaStream_t s) {
  constexpr int64_t TILE = ITEMS * SORT_THREADS;
  const unsigned tiles = (unsigned)(((int64_t)sp.N + TILE - 1) / TILE);
  if (first)
    launch_chained(sp.N, k_onesweep<ITEMS, RADIX, true>, tiles, SORT_THREADS, 0, s, sp, err, wait_ns);
  else
    launch_chained(sp.N, k_onesweep<ITEMS, RADIX, false>, tiles, SORT_THREADS, 0, s, sp, err, wait_ns);
}

}  // namespace

SortPlan make_sort_plan(int key_bits, int max_digit_bits) {
  SortPlan p{};
  p.passes = (key_bits + max_digit_bits - 1) / max_digit_bits;
  // wider digits only where they save a pass
  const bool wide = p.passes < (key_bits + 7) / 8;
  p.radix = wide ? 512 : 256;
  int shift = 0;
  for (int i = 0; i < p.passes; ++i) {  // an even split of the bits, the wider digits first
    const int bits = (key_bits - shift + p.passes - i - 1) / (p.passes - i);
    p.shift[i] = shift;
    p.mask[i] = (1u << bits) - 1u;
    shift += bits;
  }
  return p;
}

size_t sort_status_words(int64_t N, int radix) {
  const int64_t small = std::min<int64_t>(N, SORT_BIG_N);
  const int64_t tiles = std::max((small + SORT_TILE_KEYS - 1) / SORT_TILE_KEYS,
                                 (N + 2 * SORT_TILE_KEYS - 1) / (2 * SORT_TILE_KEYS));
  return (size_t)tiles * (size_t)radix;
}

void launch_weights(const StepArgs& a, StepScratch sc, DevStats* stats, int n_hist_words,
                    const void* host_meta, void* dev_meta, size_t meta_bytes, cudaStream_t s) {
  launch_chained(a.N, k_message_weights, 1, 256, meta_bytes, s, a, sc, stats, n_hist_words,
                 static_cast<const uint4*>(host_meta), static_cast<uint4*>(dev_meta),
                 (int)(meta_bytes / 16));
}

void launch_sort_histogram(const StepArgs& a, const SortPlan& plan, uint32_t* hist,
                           uint32_t* keys0, ErrSink err, int num_sms, cudaStream_t s) {
  const int64_t grid = std::max<int64_t>(
      1, std::min<int64_t>(std::max<int64_t>((a.N + 2047) / 2048,
                                             std::min<int64_t>((a.N + 1023) / 1024, 2 * num_sms)),
                           (int64_t)num_sms * 6));
  if (plan.radix == 512)
    launch_chained(a.N, k_sort_histogram<512>, (unsigned)grid, SORT_THREADS, 0, s, a, plan, hist, keys0, err);
  else
    launch_chained(a.N, k_sort_histogram<256>, (unsigned)grid, SORT_THREADS, 0, s, a, plan, hist, keys0, err);
}

void launch_onesweep(const SortPlan& plan, int pass, SortPass sp, ErrSink err, int64_t wait_ns,
                     cudaStream_t s) {
  sp.shift = plan.shift[pass];
  sp.mask = plan.mask[pass];
  const bool big = sp.N > SORT_BIG_N;
  if (plan.radix == 512) {
    if (big)
      sweep_as<16, 512>(sp, pass == 0, err, wait_ns, s);
    else
      sweep_as<8, 512>(sp, pass == 0, err, wait_ns, s);
  } else {
    if (big)
      sweep_as<16, 256>(sp, pass == 0, err, wait_ns, s);
    else
      sweep_as<8, 256>(sp, pass == 0, err, wait_ns, s);
  }
}

}  // namespace gba
