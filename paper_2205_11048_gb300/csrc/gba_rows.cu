// K3 + K4 of the GBA aggregate-and-apply step: per unique row of the sorted
// occurrence array, decay each occurrence by the row's step tag against its
// message's token (Eq. (1); Alg. 2, push responding), sum the kept gradient
// rows, divide by the number of messages whose ids include the row, apply the
// optimizer to the row and its state in place, and set the row's tag to k + 1.
//
//  k_seg_scan   One launch over the sorted positions of every table, in tiles
//               of 2048.  Every position's message, tag, staleness and weight
//               are decided here (the tag is read before any row of the step
//               is updated); four counters -- row heads, kept occurrences,
//               (message, row) pairs and kept pairs -- are scanned over the
//               step with a decoupled look-back over epoch-tagged words.  Each
//               row head writes its record (row, prefixes); each kept
//               occurrence writes the address of its gradient row (and its
//               weight) into a list sorted by row.  Rows that cross tiles need
//               no special care: a row's counts are differences of prefixes.
//  k_row_apply  Rows with at most LONG_ROW kept occurrences.  A warp takes a
//               batch of consecutive rows: its lanes read one record and the
//               list entries of one row each, rows with nothing kept drop out,
//               longer ones are listed for k_row_long, and lane groups then
//               sum and apply the rest, the next rows' state and gradients
//               being loaded while the current ones are computed.
//  k_row_long   Rows with more kept occurrences: up to small_limit of them by
//               one lane group each, longer rows in chunks of chunk_entries by
//               one warp each, the warp's lane groups summing contiguous parts
//               that are merged in a fixed order; the warp that completes a
//               row's last chunk merges the chunk sums and applies the row.
//
// The last two run once per range of consecutive tables of one width and
// optimizer.  Every summation order is fixed (sorted order, then fixed parts
// and chunks), so results are bit-identical run to run; no float atomics
// anywhere.  Sums are compensated (TwoSum).
#include <algorithm>
#include <type_traits>

#include "gba_internal.cuh"

namespace gba {

namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr uint32_t NO_KEY = 0xFFFFFFFFu;
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = SCAN_TILE / SCAN_THREADS;
constexpr int SCAN_WARPS = SCAN_THREADS / 32;
static_assert(SCAN_TILE % SCAN_THREADS == 0, "scan tile must fill the block");
constexpr int ROW_THREADS = 256;
constexpr int ROW_WARPS = ROW_THREADS / 32;
// message lookups and tables kept in shared memory by the scan, at most
constexpr size_t SCAN_CACHE_BYTES = 20 * 1024;

// look-back word: [63:32] epoch of the launch, [31:30] flag, [29:0] count
constexpr unsigned long long ST_AGG = 1ull << 30;
constexpr unsigned long long ST_INCL = 2ull << 30;
constexpr unsigned long long ST_FLAGS = 3ull << 30;
constexpr unsigned long long ST_COUNT = (1ull << 30) - 1;

__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p) {
  return *(const volatile uint32_t*)p;
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ld_relaxed_2u64(const unsigned long long* p,
                                                unsigned long long& a, unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_relaxed_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ int32_t token32(int64_t token) {  // tags stay below 2^31
  return token > 0x7FFFFFFFll ? 0x7FFFFFFF : (int32_t)token;
}

// Denominator of a row's weighted sum (Alg. 2: messages whose ids include the
// row; or the messages whose occurrence was kept; or all M messages).
__device__ __forceinline__ float row_denominator(int mode, uint32_t c_all, uint32_t c_kept, int M) {
  const uint32_t den = mode == 0 ? c_all : (mode == 1 ? c_kept : (uint32_t)M);
  return (float)den;
}

// ---------------------------------------------------------------------------
// k_seg_scan
//
// A warp holds 256 consecutive positions as eight rounds of 32, so heads, kept
// occurrences and pairs are counted by ballots, and records and list entries
// leave the registers in order, without staging.  MULTI: more than one table
// (the table of a position is found from its key); CACHED: the message
// lookups fit shared memory; UNIT: every kept weight is 1 and none is written.
// Counters of the step come from the last tile's prefixes, not from atomics.
//
// Bound by instruction issue and by the wait for earlier tiles: 8 B are read
// and at most 28 written per position, about seven warp instructions.  Message
// offsets, addresses and 32-bit tokens sit in shared memory, a message is found
// by an even-split guess and a step or two, a tile within one table uses that
// table's fields throughout, and a round of the look-back only settles how far it
// reaches: the counts are added up per thread and reduced
// once.  0.85M positions 40 -> 18 us, 5.2M (200 MB of tags) 197 -> 100, 131M in
// four tables 3.12 -> 1.4 ms.
// ---------------------------------------------------------------------------
// BIG: four blocks per SM at 64 registers; a step whose tiles are resident with
// three all the same (up to CHAIN_MAX_N positions) is faster with 80 registers
// (0.85M positions: 185.2 -> 181.8 us a step; 131M with 80 registers: 1.2% slower).
// At 64, all but one table with unit weights spill 16 to 152 bytes a thread.
template <bool MULTI, bool CACHED, bool UNIT, bool BIG>
__global__ void __launch_bounds__(SCAN_THREADS, BIG ? 4 : 3)
    k_seg_scan(StepArgs a, SegTable tb0, const SegTable* tabs_g, SegOut so,
               const uint32_t* keys, const uint32_t* vals, DevStats* st, ErrSink err, int64_t wait_ns) {
  extern __shared__ __align__(16) unsigned char s_cache[];
  __shared__ uint32_t s_wsum[4][SCAN_WARPS];
  __shared__ uint32_t s_base[4];
  __shared__ unsigned long long s_stale[2][SCAN_WARPS];
  __shared__ uint32_t s_tile;

  chain_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the step's state, the tile's ticket (by the last warp, which has the least to
  // cache) and the lookups in flight together
  const uint32_t failed = ld_volatile_u32(err.step) & (ERR_ID_RANGE | ERR_TIMEOUT);
  if (tid == SCAN_THREADS - 1) s_tile = atomicAdd(so.ticket, 1u);
  const uint32_t lt = lanemask_lt();
  const int M = a.M, T = MULTI ? a.T : 1;
  const uint32_t* off_all = a.msg_off;            // [T][M + 1]
  const float* const* rowp_all = a.rows_ptr;      // [T][M]
  const int32_t* tok32 = nullptr;                 // [M] tokens, at most 2^31 - 1
  const SegTable* tabs = tabs_g;                  // [T]
  if (CACHED) {
    SegTable* c_tabs = reinterpret_cast<SegTable*>(s_cache);
    const float** c_rowp = reinterpret_cast<const float**>(c_tabs + (MULTI ? T : 0));
    uint32_t* c_off = reinterpret_cast<uint32_t*>(c_rowp + (size_t)T * M);
    int32_t* c_tok = reinterpret_cast<int32_t*>(c_off + (size_t)T * (M + 1));
    for (int i = tid; i < M; i += SCAN_THREADS) c_tok[i] = token32(a.tokens[i]);
    for (int i = tid; i < T * M; i += SCAN_THREADS) c_rowp[i] = a.rows_ptr[i];
    for (int i = tid; i < T * (M + 1); i += SCAN_THREADS) c_off[i] = a.msg_off[i];
    if (MULTI) {
      const uint32_t* src = reinterpret_cast<const uint32_t*>(tabs_g);
      uint32_t* dst = reinterpret_cast<uint32_t*>(c_tabs);
      for (int i = tid; i < (int)(T * sizeof(SegTable) / 4); i += SCAN_THREADS) dst[i] = src[i];
    }
    off_all = c_off;
    rowp_all = c_rowp;
    tok32 = c_tok;
    tabs = c_tabs;
  }
  // block-uniform: another kernel may set the word while this block reads it
  if (__syncthreads_or(failed != 0u)) return;
  const uint32_t tile = s_tile;
  const uint32_t N = (uint32_t)a.N;  // below 2^30
  const uint32_t n_tiles = (N + SCAN_TILE - 1) / SCAN_TILE;
  const uint32_t pw = tile * (uint32_t)SCAN_TILE + (uint32_t)(warp * SCAN_ITEMS * 32);
  const int hop_limit = M - a.drop_latest;  // messages at or past this index are dropped

  // ---- keys and occurrences of this warp's positions (lane l holds position
  // pw + 32 j + l), and the position before them
  uint32_t key[SCAN_ITEMS], val[SCAN_ITEMS];
#pragma unroll
  for (int j = 0; j < SCAN_ITEMS; ++j) {
    const uint32_t p = pw + j * 32 + lane;
    key[j] = p < N ? keys[p] : NO_KEY;
    val[j] = p < N ? vals[p] : 0u;
  }
  uint32_t key_prev = NO_KEY, val_prev = 0u;
  if (pw > 0u && pw < N) {
    key_prev = keys[pw - 1];
    val_prev = vals[pw - 1];
  }
  // The table of the tile's first position, whose fields the whole tile then
  // uses; a tile that runs into the next table (mixed) looks its positions'
  // tables up one by one, each lane moving up from that of its first.
  int t_one = 0;
  if (MULTI) {
    int lo = 0, hi = T;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (tabs[mid].nb <= tile * (uint32_t)SCAN_TILE)
        lo = mid;
      else
        hi = mid;
    }
    t_one = lo;
  }
  const SegTable& tb1 = MULTI ? tabs[t_one] : tb0;
  const bool mixed = MULTI && min((tile + 1u) * (uint32_t)SCAN_TILE, N) > tb1.nb + tb1.n;
  auto advance = [&](int t, uint32_t k) {
    while (t + 1 < T && tabs[t + 1].key_base <= k) ++t;
    return t;
  };
  int32_t tg[SCAN_ITEMS];
  float f_[UNIT ? 1 : SCAN_ITEMS];
  uint32_t flags = 0u;  // bit 4j: head, 4j+1: keep, 4j+2: new (message, row) pair
  uint32_t cnt[4] = {0u, 0u, 0u, 0u};  // the warp's totals
  unsigned long long stale_sum = 0ull;
  uint32_t stale_max = 0u;
  auto decide = [&](auto mixed_tag) {
  constexpr bool MIX = decltype(mixed_tag)::value;
    // the rows' step tags, all loads in flight together (positions of one row
    // read the same tag, so only a row's first read reaches DRAM)
    {
      int t = t_one;
  #pragma unroll
      for (int j = 0; j < SCAN_ITEMS; ++j) {
        tg[j] = (int32_t)a.k;  // message staleness: against the current step
        if (key[j] != NO_KEY) {
          if (MIX) t = advance(t, key[j]);
          const uint32_t x = key[j] - (MIX ? tabs[t] : tb1).key_base;
          if (a.row_staleness == 0 && x < (MIX ? tabs[t] : tb1).rows) tg[j] = (MIX ? tabs[t] : tb1).ver[x];
        }
      }
    }
  
    // ---- pass 1: decide every position
    int m_last = -1;  // message of the position before this round's first
    if (key_prev != NO_KEY) {
      // only compared with positions of the same row, so lane 0's table serves
      const int t0 = MIX ? __shfl_sync(FULL, advance(t_one, key[0]), 0) : t_one;
      const SegTable& tb = MIX ? tabs[t0] : tb1;
      uint32_t o = val_prev - tb.nb;
      if (o < tb.n) m_last = message_of(off_all + (size_t)t0 * (M + 1), M, o, tb.mscale);
    }
    {
      int t = t_one;
  #pragma unroll
      for (int j = 0; j < SCAN_ITEMS; ++j) {
        bool in = key[j] != NO_KEY;
        if (MIX && in) t = advance(t, key[j]);
        const SegTable& tb = (MIX ? tabs[t] : tb1);
        const uint32_t x = key[j] - tb.key_base;
        uint32_t o = val[j] - tb.nb;
        if (in && (o >= tb.n || x >= tb.rows)) {
          raise_error(err, ERR_INTERNAL);  // cannot happen for a correctly sorted array
          in = false;
        }
        int m = -1;
        if (in) m = message_of(off_all + (size_t)t * (M + 1), M, o, tb.mscale);
        // the position before: the lane below, for lane 0 the last of the round before
        const uint32_t kp = __shfl_sync(FULL, lane == 31 ? key_prev : key[j], (lane + 31) & 31);
        const int mp = __shfl_sync(FULL, lane == 31 ? m_last : m, (lane + 31) & 31);
        key_prev = key[j];
        m_last = m;
        bool head = false, keep = false, newp = false;
        float f = 0.f;
        if (in) {
          head = key[j] != kp;
          newp = head || m != mp;
          const int32_t tk = CACHED ? tok32[m] : token32(a.tokens[m]);
          const uint32_t sl = tg[j] > tk ? (uint32_t)(tg[j] - tk) : 0u;
          if (UNIT) {
            keep = sl <= (uint32_t)a.iota && m < hop_limit;
          } else {
            f = m < hop_limit ? decay_weight(a, sl) : 0.f;
            keep = f > 0.f;
          }
          if (newp) {
            stale_sum += sl;
            stale_max = max(stale_max, sl);
          }
        }
        tg[j] = m;  // the tag has served; the message is needed in pass 2,
        val[j] = o;  // and the occurrence's place in it
        if (!UNIT) f_[UNIT ? 0 : j] = f;
        flags |= ((head ? 1u : 0u) | (keep ? 2u : 0u) | (newp ? 4u : 0u)) << (4 * j);
        cnt[0] += __popc(__ballot_sync(FULL, head));
        cnt[1] += __popc(__ballot_sync(FULL, keep));
        cnt[2] += __popc(__ballot_sync(FULL, newp));
        cnt[3] += __popc(__ballot_sync(FULL, newp && keep));
      }
    }
  };
  if constexpr (MULTI) {
    if (mixed)
      decide(std::true_type{});
    else
      decide(std::false_type{});
  } else {
    decide(std::false_type{});
  }

  // ---- the warps' exclusive prefixes within the tile, the tile's totals
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    stale_sum += __shfl_xor_sync(FULL, stale_sum, o);
    stale_max = max(stale_max, __shfl_xor_sync(FULL, stale_max, o));
  }
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < 4; ++c) s_wsum[c][warp] = cnt[c];
    s_stale[0][warp] = stale_sum;
    s_stale[1][warp] = stale_max;
  }
  __syncthreads();
  uint32_t tile_tot[4], run[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t before = 0u, tot = 0u;
#pragma unroll
    for (int w = 0; w < SCAN_WARPS; ++w) {
      const uint32_t y = s_wsum[c][w];
      if (w < warp) before += y;
      tot += y;
    }
    run[c] = before;
    tile_tot[c] = tot;
  }

  // ---- the tile's prefixes: the whole block looks back over earlier tiles,
  // SCAN_THREADS of them at a time (thread i reads tile j - i)
  {
    unsigned long long* my = so.status + (size_t)tile * 4;
    const unsigned long long ep = (unsigned long long)so.epoch << 32;
    if (tid == 0)
      for (int c = 0; c < 4; ++c)
        st_relaxed_u64(my + c, ep | (tile == 0 ? ST_INCL : ST_AGG) | (unsigned long long)tile_tot[c]);
    __shared__ uint32_t s_first_nr[2][SCAN_WARPS], s_first_in[2][SCAN_WARPS];
    __shared__ uint32_t s_part[4][SCAN_WARPS];
    __shared__ int s_give_up[2];
    uint32_t pre[4] = {0u, 0u, 0u, 0u};
    if (tile > 0) {
      uint32_t mine[4] = {0u, 0u, 0u, 0u};  // what this thread's tiles add
      int64_t j = (int64_t)tile - 1;
      const uint64_t t0 = globaltimer_ns();
      for (int b = 0;; b ^= 1) {  // the shared words alternate: one barrier a round
        const int64_t q = j - tid;
        unsigned long long v[4] = {ep | ST_INCL, ep | ST_INCL, ep | ST_INCL, ep | ST_INCL};
        if (q >= 0) {
          ld_relaxed_2u64(so.status + (size_t)q * 4, v[0], v[1]);
          ld_relaxed_2u64(so.status + (size_t)q * 4 + 2, v[2], v[3]);
        }
        // a tile is usable once its four words carry this launch's epoch and
        // the same flag (the writer replaces all four, so a mix is transient)
        const unsigned long long tag = v[0] & ~ST_COUNT;
        const bool ready = (tag >> 32) == (ep >> 32) && (tag & ST_FLAGS) != 0ull &&
                           (v[1] & ~ST_COUNT) == tag && (v[2] & ~ST_COUNT) == tag &&
                           (v[3] & ~ST_COUNT) == tag;
        const bool incl = ready && (tag & ST_INCL) != 0ull;
        const uint32_t rm = __ballot_sync(FULL, ready), im = __ballot_sync(FULL, incl);
        if (lane == 0) {
          s_first_nr[b][warp] = ~rm ? (uint32_t)(warp * 32 + __ffs(~rm) - 1) : (uint32_t)SCAN_THREADS;
          s_first_in[b][warp] = im ? (uint32_t)(warp * 32 + __ffs(im) - 1) : (uint32_t)SCAN_THREADS;
        }
        if (tid == 0) {
          const bool give_up = !ready && ((ld_volatile_u32(err.step) & ERR_TIMEOUT) ||
                                          (int64_t)(globaltimer_ns() - t0) > wait_ns);
          if (give_up) raise_error(err, ERR_TIMEOUT);
          s_give_up[b] = give_up ? 1 : 0;
        }
        __syncthreads();
        uint32_t first_nr = (uint32_t)SCAN_THREADS, first_in = (uint32_t)SCAN_THREADS;
#pragma unroll
        for (int w = 0; w < SCAN_WARPS; ++w) {
          first_nr = min(first_nr, s_first_nr[b][w]);
          first_in = min(first_in, s_first_in[b][w]);
        }
        const bool done = first_in < first_nr || s_give_up[b] != 0;
        const uint32_t take = first_in < first_nr ? first_in + 1 : first_nr;
        if ((uint32_t)tid < take)
#pragma unroll
          for (int c = 0; c < 4; ++c) mine[c] += (uint32_t)(v[c] & ST_COUNT);
        if (done) break;
        if (take == 0u) __nanosleep(LOOKBACK_SLEEP_NS);
        j -= take;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t sum = __reduce_add_sync(FULL, mine[c]);
        if (lane == 0) s_part[c][warp] = sum;
      }
      __syncthreads();
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int w = 0; w < SCAN_WARPS; ++w) pre[c] += s_part[c][w];
      if (tid == 0)
        for (int c = 0; c < 4; ++c)
          st_relaxed_u64(my + c, ep | ST_INCL | (unsigned long long)((pre[c] + tile_tot[c]) & ST_COUNT));
    }
    if (tid == 0) {
      for (int c = 0; c < 4; ++c) s_base[c] = pre[c];
      if (tile == n_tiles - 1) {  // the totals close the record array
        const uint32_t U = pre[0] + tile_tot[0];
        so.rr[U] = make_uint4(0u, pre[1] + tile_tot[1], pre[2] + tile_tot[2], pre[3] + tile_tot[3]);
        so.ustart[T] = U;
        for (int t = T - 1; MULTI && t >= 0 && tabs[t].n == 0u; --t) so.ustart[t] = U;
        // the step's counters of Table 3's kind
        atomicAdd(&st->rows_touched, (unsigned long long)U);
        atomicAdd(&st->occ_kept, (unsigned long long)(pre[1] + tile_tot[1]));
        atomicAdd(&st->pairs, (unsigned long long)(pre[2] + tile_tot[2]));
        atomicAdd(&st->pairs_dropped,
                  (unsigned long long)(pre[2] + tile_tot[2] - pre[3] - tile_tot[3]));
      }
      unsigned long long ss = 0ull, sm = 0ull;
      for (int w = 0; w < SCAN_WARPS; ++w) {
        ss += s_stale[0][w];
        sm = s_stale[1][w] > sm ? s_stale[1][w] : sm;
      }
      if (ss) atomicAdd(&st->row_stale_sum, ss);
      if (sm) atomicMax(&st->row_stale_max, sm);
    }
  }
  __syncthreads();

  // ---- pass 2: row records and the kept list, in order
#pragma unroll
  for (int c = 0; c < 4; ++c) run[c] += s_base[c];
  auto emit = [&](auto mixed_tag) {
    constexpr bool MIX = decltype(mixed_tag)::value;
  {
    int t = t_one;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
      const uint32_t fl = (flags >> (4 * j)) & 7u;
      const bool head = fl & 1u, keep = fl & 2u, newp = fl & 4u;
      const uint32_t hm = __ballot_sync(FULL, head), km = __ballot_sync(FULL, keep),
                     nm = __ballot_sync(FULL, newp);
      if (MIX && key[j] != NO_KEY) t = advance(t, key[j]);
      const SegTable& tb = MIX ? tabs[t] : tb1;
      const uint32_t k_at = run[1] + __popc(km & lt);
      if (head) {
        const uint32_t u = run[0] + __popc(hm & lt);
        so.rr[u] = make_uint4(key[j] - tb.key_base, k_at, run[2] + __popc(nm & lt),
                              run[3] + __popc(nm & km & lt));
        // the first row of a table (and of the empty tables before it)
        if (pw + j * 32 + lane == tb.nb) {
          so.ustart[t] = u;
          for (int e = t - 1; MULTI && e >= 0 && tabs[e].n == 0u; --e) so.ustart[e] = u;
        }
      }
      if (keep) {
        const int m = tg[j];
        so.kl[k_at] = rowp_all[(size_t)t * M + m] + (size_t)val[j] * (size_t)tb.d;
        if (!UNIT) so.kw[k_at] = f_[UNIT ? 0 : j];
      }
      run[0] += __popc(hm);
      run[1] += __popc(km);
      run[2] += __popc(nm);
      run[3] += __popc(nm & km);
    }
  }
  };
  if constexpr (MULTI) {
    if (mixed)
      emit(std::true_type{});
    else
      emit(std::false_type{});
  } else {
    emit(std::false_type{});
  }
}

// ---------------------------------------------------------------------------
// shared pieces of the two row kernels
// ---------------------------------------------------------------------------
// A lane's part of one row: CPL pieces of CH floats; piece q of the row is
// held by lane q mod L as its piece number q / L.
template <int CH, int CPL>
struct Part {
  float v[CH * CPL];
};

template <int CH, int CPL>
__device__ __forceinline__ void load_part(const float* row, int l, int L, int C, Part<CH, CPL>& p) {
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int q = l + c * L;
    if (q < C) {
      if constexpr (CH == 4) {
        const float4 t = *reinterpret_cast<const float4*>(row + 4 * q);
        p.v[4 * c] = t.x;
        p.v[4 * c + 1] = t.y;
        p.v[4 * c + 2] = t.z;
        p.v[4 * c + 3] = t.w;
      } else {
        p.v[c] = row[q];
      }
    }
  }
}

// Brings a row of d floats into L2, for a load that comes later; one lane for
// the whole row.
template <int CH>
__device__ __forceinline__ void prefetch_row(const float* row, int d) {
  if constexpr (CH == 4) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row), "r"(d * 4) : "memory");
  } else {
    for (int i = 0; i < d; i += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + i));
  }
}

// The same past L1, for sums that other blocks of this launch wrote.
template <int CH, int CPL>
__device__ __forceinline__ void load_part_cg(const float* row, int l, int L, int C,
                                             Part<CH, CPL>& p) {
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int q = l + c * L;
    if (q < C) {
      if constexpr (CH == 4) {
        const float4 t = __ldcg(reinterpret_cast<const float4*>(row + 4 * q));
        p.v[4 * c] = t.x;
        p.v[4 * c + 1] = t.y;
        p.v[4 * c + 2] = t.z;
        p.v[4 * c + 3] = t.w;
      } else {
        p.v[c] = __ldcg(row + q);
      }
    }
  }
}

template <int CH, int CPL>
__device__ __forceinline__ void store_part(float* row, int l, int L, int C, const Part<CH, CPL>& p) {
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int q = l + c * L;
    if (q < C) {
      if constexpr (CH == 4) {
        *reinterpret_cast<float4*>(row + 4 * q) =
            make_float4(p.v[4 * c], p.v[4 * c + 1], p.v[4 * c + 2], p.v[4 * c + 3]);
      } else {
        row[q] = p.v[c];
      }
    }
  }
}

// The optimizer step of a row (w and its state at the given addresses) with its
// summed gradient (acc) and denominator.
template <int CH, int CPL, bool ADAM>
__device__ __forceinline__ void finish_row(const OptStep& opt, float* w_at, float* s0_at,
                                           float* s1_at, float den, const CSum (&acc)[CH * CPL],
                                           Part<CH, CPL>& w, Part<CH, CPL>& s0, Part<CH, CPL>& s1,
                                           int l, int L, int C) {
  // den is a whole number: where it is a power of two (most rows: one or two
  // messages), the product with its reciprocal is the quotient
  const uint32_t den_bits = __float_as_uint(den);
  const bool pow2 = (den_bits & 0x007FFFFFu) == 0u;
  const float inv = __uint_as_float(0x7F000000u - den_bits);  // 1 / den, if pow2
  float gr[CH * CPL];
#pragma unroll
  for (int i = 0; i < CH * CPL; ++i) gr[i] = csum_value(acc[i]);
  if (pow2) {
#pragma unroll
    for (int i = 0; i < CH * CPL; ++i) gr[i] = __fmul_rn(gr[i], inv);
  } else {
#pragma unroll
    for (int i = 0; i < CH * CPL; ++i) gr[i] = __fdiv_rn(gr[i], den);
  }
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    if (l + c * L >= C) continue;
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      const int i = c * CH + k;
      float b = ADAM ? s1.v[i] : 0.f;
      opt_update_as<ADAM>(opt, w.v[i], s0.v[i], b, gr[i]);
      s1.v[i] = b;
    }
  }
  store_part<CH, CPL>(w_at, l, L, C, w);
  store_part<CH, CPL>(s0_at, l, L, C, s0);
  if (ADAM) store_part<CH, CPL>(s1_at, l, L, C, s1);
}

// Weight of list entry j (UNIT steps keep no weights: every one is 1).
__device__ __forceinline__ float entry_weight(const SegOut& so, bool unit, uint32_t j) {
  return unit ? 1.f : so.kw[j];
}

template <int CH, int CPL>
__device__ __forceinline__ void add_part(CSum (&acc)[CH * CPL], bool unit, float f,
                                         const Part<CH, CPL>& g) {
#pragma unroll
  for (int i = 0; i < CH * CPL; ++i) csum_add_w(acc[i], unit, f, g.v[i]);
}

constexpr int LONG_WARPS = 16;  // of k_row_long per SM

// Lanes per row (a power of two) and rows per warp of a width of C pieces.
__host__ __device__ inline int row_lanes(int C, int CPL) {
  int L = 1;
  while (L * CPL < C && L < 32) L <<= 1;
  return L;
}

// Kept occurrences per chunk of a row longer than small_limit, for a range of
// tables with n occurrences whose rows take L lanes: 64 for each of the
// warp's lane groups (128 for a group of 32), and fewer, down to 32, while there
// would not be two chunks for every warp that can run: such a step's time is that of
// its longest chunk (steps of 0.33M ids x 256 floats 328 -> 314 us, of 0.85M x 32 199
// -> 195).  Chunks of 8 or 16 a group cost more in claims and partial sums than they
// save (0.17M ids x 18 floats: 398 -> 410 us with 8; 0.03M x 16: 52.4 -> 53.7 with 16).
inline uint32_t chunk_entries(int64_t n, int L, int num_sms) {
  const int64_t G = 32 / L;
  int64_t per = L == 32 ? 128 : 64;  // entries per lane group
  while (per > 32 && n < per * G * 2 * num_sms * LONG_WARPS) per >>= 1;
  return (uint32_t)(per * G);
}

// The longest rows that one lane group of k_row_long takes alone, for a range of
// n occurrences: while all rows fit the machine at once, short ones, so that the
// longest does not decide (32 against 64: 188 us against 192 a step of 0.85M ids);
// otherwise longer ones, which save merging (131M ids: 7.76 -> 7.64 ms).
inline uint32_t small_limit(int64_t n) { return n > (1 << 23) ? SMALL_MAX : SMALL_MAX / 2; }

// The table of row record u among tables [t0, t1).
__device__ __forceinline__ int table_of_row(const uint32_t* ustart, int t0, int t1, uint32_t u) {
  int lo = t0, hi = t1;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (ustart[mid] <= u)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// ---------------------------------------------------------------------------
// k_row_apply
//
// Random accesses to HBM: a row's state and gradients are a few hundred bytes
// at scattered addresses, so what counts is how many warps have how many rows
// in flight.  Each lane of a warp first looks after one row (record, list
// entries, addresses), so that lane groups find the rows that really move
// packed in shared memory.  Rows with nothing kept (30% of the touched rows
// with 40% stale messages) cost no more than their record.  IEEE division and
// square root make up half of the instructions.
// 5.2M ids x 64 floats, 1.6M rows moved, beside the other streams' kernels:
// 505 -> 361 us against one lane group walking its rows through cp.async
// stages (24 warps per SM, 200 instructions per row).
// The register limits below spill in some widths (bytes stored a thread): 12 to 72
// for Adam's rows of up to 128 floats, 28 to 216 for wider ones in float4 pieces,
// 80 to 144 for odd widths of 65 to 128.  Whole steps of 0.16M even ids are faster
// all the same than with the kernels before, which did not spill: 65 floats 199 ->
// 136 us, 127 214 -> 150, Adam's 256 290 -> 219.  Limits without spills were not
// measured.
// ---------------------------------------------------------------------------
// Widths (multiples of 4) up to which k_row_apply loads the next rows into
// registers while it computes; wider rows are prefetched into L2 instead and
// the registers go to more warps (16 floats: 1.08 ms against 1.51 on 11M rows;
// 32 floats: 64 us against 52 on 374K rows).
constexpr int APPLY_AHEAD_DIM = 16;

struct __align__(16) RowSlot {  // one row of a warp's batch
  const float* p[LONG_ROW];  // its kept gradient rows
  float* w;                  // the row and its state
  float* s0;
  float* s1;
  int32_t* ver;
  uint32_t n;                // kept occurrences (1 .. LONG_ROW)
  float den;
  int32_t t;                 // its table
  uint32_t pad;
  float f[LONG_ROW];         // the gradients' weights (unused when every weight is 1)
};

template <int CH, int CPL>
struct RowRegs {
  uint32_t n;  // kept occurrences, 0: no row
  Part<CH, CPL> w, s0, s1, g0;
};

template <int CH, int CPL, bool ADAM, bool MULTI, bool AHEAD>
__global__ void __launch_bounds__(ROW_THREADS, (CH * CPL <= 4 && !AHEAD) ? 4 : (CPL <= 2 ? 3 : 2))
    k_row_apply(StepArgs a, SegTable tb0, const SegTable* tabs, int t0, int t1, uint32_t chunk,
                uint32_t small_max, SegOut so, DevStats* st, ErrSink err) {
  __shared__ RowSlot s_slot[ROW_WARPS][32];
  __shared__ uint4 s_rec[ROW_WARPS][33];  // the next batch's records
  chain_wait();
  // a failed step changes no row (warp-uniform: the warp reduces at the end)
  const uint32_t failed = ld_volatile_u32(err.step);
  const uint32_t us = ld_volatile_u32(so.ustart + t0), ue = ld_volatile_u32(so.ustart + t1);
  if (__any_sync(FULL, failed != 0u)) return;
  constexpr int P = CH * CPL;
  const int d = tb0.d;
  const int C = CH == 4 ? d / 4 : d;  // pieces per row
  const int L = row_lanes(C, CPL);
  const int lg = __ffs(L) - 1;
  const int G = 32 >> lg;  // rows per warp at a time
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> lg, l = lane & (L - 1);
  const uint32_t lt = lanemask_lt();
  const bool unit = a.decay == 0;  // every kept weight is 1
  const int mode = a.sparse_den;
  const int32_t tag = (int32_t)(a.k + 1);
  RowSlot* slot = s_slot[warp];
  uint32_t applied = 0u;

  // batches of 32 rows, smaller ones when there are not enough for every warp
  const uint32_t W = gridDim.x * (uint32_t)ROW_WARPS;
  uint32_t bs = 32u;
  while (bs > (uint32_t)G && ue - us < W * bs) bs >>= 1;
  const uint32_t stride = W * bs;
  uint4* rec = s_rec[warp];
  // records u0 .. u0 + bs (rr[ue] closes the last row), copied while the batch
  // before is worked on
  auto fetch_records = [&](uint32_t u0) {
    for (uint32_t i = (uint32_t)lane; i <= bs; i += 32u)
      if (u0 + i <= ue) cp_async16(rec + i, so.rr + u0 + i);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  uint32_t u0 = us + (blockIdx.x * (uint32_t)ROW_WARPS + (uint32_t)warp) * bs;
  if (u0 < ue) fetch_records(u0);
  for (; u0 < ue; u0 += stride) {
    // ---- one row per lane: its counts, its list entries, its list if long
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    const uint32_t u = u0 + (uint32_t)lane;
    uint4 ra = make_uint4(0u, 0u, 0u, 0u), rb = ra;
    if ((uint32_t)lane < bs && u < ue) {
      ra = rec[lane];
      rb = rec[lane + 1];
    }
    __syncwarp();
    if (u0 + stride < ue) fetch_records(u0 + stride);
    const uint32_t n = rb.y - ra.y, ks = ra.y;
    const float den = row_denominator(mode, rb.z - ra.z, rb.w - ra.w, a.M);
    const uint32_t x = ra.x;
    int t = t0;
    if (MULTI && n > 0u) t = table_of_row(so.ustart, t0, t1, u);
    const bool is_short = n > 0u && n <= (uint32_t)LONG_ROW;
    const float* p[LONG_ROW];
#pragma unroll
    for (int e = 0; e < LONG_ROW; ++e)
      p[e] = is_short && (uint32_t)e < n ? so.kl[ks + e] : nullptr;
    const bool is_small = n > (uint32_t)LONG_ROW && n <= small_max;
    const bool is_long = n > small_max;
    const uint32_t sm = __ballot_sync(FULL, is_small), lm = __ballot_sync(FULL, is_long);
    uint32_t small_at = 0u, long_at = 0u, item_at = 0u, part_at = 0u;
    uint32_t nch = 0u, nparts = 0u;
    if (sm) {
      if (lane == 0) small_at = atomicAdd(so.n_small, (uint32_t)__popc(sm));
    }
    if (lm) {
      nch = is_long ? (n + chunk - 1) / chunk : 0u;
      nparts = nch > 1u ? nch : 0u;
      uint32_t ci = nch, cp = nparts;  // inclusive scans over the lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t yi = __shfl_up_sync(FULL, ci, o), yp = __shfl_up_sync(FULL, cp, o);
        if (lane >= o) {
          ci += yi;
          cp += yp;
        }
      }
      uint32_t b0 = 0u, b1 = 0u, b2 = 0u;
      if (lane == 31) {
        b0 = atomicAdd(so.n_long, (uint32_t)__popc(lm));
        b1 = atomicAdd(so.n_items, ci);
        b2 = cp ? atomicAdd(so.n_parts, cp) : 0u;
      }
      long_at = __shfl_sync(FULL, b0, 31) + __popc(lm & lt);
      item_at = __shfl_sync(FULL, b1, 31) + ci - nch;
      part_at = __shfl_sync(FULL, b2, 31) + cp - nparts;
      if (is_long) {
        so.long_rows[long_at] = make_uint4(u, ks, n, part_at);
        so.long_done[long_at] = 0u;
        for (uint32_t c = 0; c < nch; ++c) so.items[item_at + c] = make_uint2(long_at, c);
      }
    }
    const uint32_t mask = __ballot_sync(FULL, is_short);
    const int cnt = __popc(mask);
    if (is_short) {
      RowSlot& s = slot[__popc(mask & lt)];
      const SegTable& tb = MULTI ? tabs[t] : tb0;
      const size_t base = (size_t)x * (size_t)d;
      s.w = tb.w + base;
      s.s0 = tb.s0 + base;
      if (ADAM) s.s1 = tb.s1 + base;
      s.ver = tb.ver + x;
      *reinterpret_cast<uint4*>(&s.n) = make_uint4(n, __float_as_uint(den), (uint32_t)t, 0u);
#pragma unroll
      for (int e = 0; e < LONG_ROW; ++e) s.p[e] = p[e];
      if (!unit)
#pragma unroll
        for (int e = 0; e < LONG_ROW; ++e) s.f[e] = (uint32_t)e < n ? so.kw[ks + e] : 0.f;
    }
    if (is_small) {  // until its place in the list is known
      RowSlot& s = slot[31 - __popc(sm & lt)];
      *reinterpret_cast<uint4*>(&s.n) =
          make_uint4(x, ks, n | ((uint32_t)t << 8), __float_as_uint(den));
    }
    __syncwarp();

    // ---- the short rows, one per lane group
    auto fetch = [&](int i, RowRegs<CH, CPL>& r) {
      r.n = 0u;
      if (i < cnt) {
        r.n = slot[i].n;
        load_part<CH, CPL>(slot[i].p[0], l, L, C, r.g0);
        load_part<CH, CPL>(slot[i].w, l, L, C, r.w);
        load_part<CH, CPL>(slot[i].s0, l, L, C, r.s0);
        if (ADAM) load_part<CH, CPL>(slot[i].s1, l, L, C, r.s1);
      }
    };
    auto apply = [&](int i, RowRegs<CH, CPL>& r) {
      if (r.n == 0u) return;
      Part<CH, CPL> g1, g2, g3;
      if (r.n > 1u) load_part<CH, CPL>(slot[i].p[1], l, L, C, g1);
      if (r.n > 2u) load_part<CH, CPL>(slot[i].p[2], l, L, C, g2);
      if (r.n > 3u) load_part<CH, CPL>(slot[i].p[3], l, L, C, g3);
      const float f0 = unit ? 1.f : slot[i].f[0];
      CSum acc[P];
#pragma unroll
      for (int e = 0; e < P; ++e) {
        if (f0 == 1.f) {
          // the first term as it is: 0 + g is exact, and its error g - g is 0, or NaN
          // for an infinite g, as in the sums that start from zero
          acc[e] = CSum{r.g0.v[e], __fsub_rn(r.g0.v[e], r.g0.v[e])};
        } else {
          acc[e] = CSum{0.f, 0.f};
          csum_add_prod(acc[e], f0, r.g0.v[e]);
        }
      }
      if (r.n > 1u) add_part<CH, CPL>(acc, unit, unit ? 1.f : slot[i].f[1], g1);
      if (r.n > 2u) add_part<CH, CPL>(acc, unit, unit ? 1.f : slot[i].f[2], g2);
      if (r.n > 3u) add_part<CH, CPL>(acc, unit, unit ? 1.f : slot[i].f[3], g3);
      finish_row<CH, CPL, ADAM>(MULTI ? tabs[slot[i].t].opt : tb0.opt, slot[i].w, slot[i].s0,
                                slot[i].s1, slot[i].den, acc, r.w, r.s0, r.s1, l, L, C);
      if (l == 0) {
        *slot[i].ver = tag;
        ++applied;
      }
    };
    if (AHEAD) {
      RowRegs<CH, CPL> cur, nxt;
      fetch(g, cur);
      for (int i = g; i - g < cnt; i += G) {
        fetch(i + G, nxt);
        apply(i, cur);
        cur = nxt;
      }
    } else {
      auto ahead = [&](int i) {  // row i of the batch into L2
        if (l != 0 || i >= cnt) return;
        prefetch_row<CH>(slot[i].p[0], d);
        prefetch_row<CH>(slot[i].w, d);
        prefetch_row<CH>(slot[i].s0, d);
        if (ADAM) prefetch_row<CH>(slot[i].s1, d);
#pragma unroll
        for (int e = 1; e < LONG_ROW; ++e)
          if ((uint32_t)e < slot[i].n) prefetch_row<CH>(slot[i].p[e], d);
      };
      for (int i = g; i - g < cnt; i += G) {
        ahead(i + G);
        RowRegs<CH, CPL> cur;
        fetch(i, cur);
        apply(i, cur);
      }
    }
    if (sm) {
      small_at = __shfl_sync(FULL, small_at, 0);
      if (lane < __popc(sm))
        so.small_rows[small_at + lane] = *reinterpret_cast<const uint4*>(&slot[31 - lane].n);
    }
    __syncwarp();  // every lane is done with the slots
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) applied += __shfl_xor_sync(FULL, applied, o);
  if (lane == 0 && applied) atomicAdd(&st->rows_applied, (unsigned long long)applied);
}

// ---------------------------------------------------------------------------
// k_row_long
//
// Bound by the latency of the gathers: eight rows in flight per lane group in
// registers, their addresses read one round ahead (16 warps per SM).  More
// warps with fewer rows each were slower (24 warps x 8 rows spill; 32 x 4: 73
// us against 39 on 0.85M ids x 32 floats).  Chunks grow as rows get narrower, so
// that a full one gives every lane group 32 to 128 entries to pipeline
// (chunk_entries), and a row's chunk sums are merged by all lane groups.  Odd
// widths of more than 64 floats spill at 16 warps (96 to 188 bytes stored a thread
// up to 128 floats, 160 to 728 above, most for Adam with several tables); whole
// steps of 0.16M skewed ids are faster than with the kernels before all the same:
// 129 floats 390 -> 277 us, 255 489 -> 354, Adam's 255 501 -> 374.  Fewer rows in
// flight without spills were not measured.  131M ids x 16 floats in four
// tables: 8.95 -> 2.17 ms, 68% of the DRAM bandwidth, against staging in shared
// memory with 8 warps per SM and one lane group merging the chunk sums.
// ---------------------------------------------------------------------------
// Adds list entries [b0, b1) to a lane group's sums in order, UNR gradient rows
// in flight, their addresses read one round ahead.
template <int CH, int CPL, int UNR>
__device__ __forceinline__ void sum_entries(const SegOut& so, bool unit, uint32_t b0, uint32_t b1,
                                            int l, int L, int C, int d,
                                            CSum (&acc)[CH * CPL]) {
  const float* p[UNR];
#pragma unroll
  for (int e = 0; e < UNR; ++e) p[e] = b0 + e < b1 ? so.kl[b0 + e] : nullptr;
  for (uint32_t j = b0; j < b1; j += UNR) {
    // wide rows: the rows of the round after the next into L2
    const uint32_t ja = j + 2 * UNR + (uint32_t)l;
    const float* pf = CH * CPL > 4 && l < UNR && ja < b1 ? so.kl[ja] : nullptr;
    Part<CH, CPL> gr[UNR];
#pragma unroll
    for (int e = 0; e < UNR; ++e)
      if (j + e < b1) load_part<CH, CPL>(p[e], l, L, C, gr[e]);
#pragma unroll
    for (int e = 0; e < UNR; ++e) p[e] = j + UNR + e < b1 ? so.kl[j + UNR + e] : nullptr;
#pragma unroll
    for (int e = 0; e < UNR; ++e)
      if (j + e < b1) add_part<CH, CPL>(acc, unit, entry_weight(so, unit, j + e), gr[e]);
    if (pf) prefetch_row<CH>(pf, d);
  }
}

template <int CH, int CPL, bool ADAM, bool MULTI>
__global__ void __launch_bounds__(ROW_THREADS, 2)
    k_row_long(StepArgs a, SegTable tb0, const SegTable* tabs, int t0, int t1, uint32_t chunk,
               SegOut so, DevStats* st, ErrSink err) {
  chain_wait();
  const uint32_t failed = ld_volatile_u32(err.step);
  const uint32_t n_items = ld_volatile_u32(so.n_items), n_small = ld_volatile_u32(so.n_small);
  if (__any_sync(FULL, failed != 0u)) return;
  constexpr int P = CH * CPL;
  constexpr int UNR = P <= 4 ? 8 : 4;
  const int d = tb0.d;
  const int C = CH == 4 ? d / 4 : d;
  const int L = row_lanes(C, CPL);
  const int lg = __ffs(L) - 1;
  const int G = 32 >> lg;  // lane groups per warp
  const int lane = threadIdx.x & 31;
  const int g = lane >> lg, l = lane & (L - 1);
  const bool unit = a.decay == 0;  // every kept weight is 1
  const int32_t tag = (int32_t)(a.k + 1);
  uint32_t applied = 0u;
  const uint32_t gw = blockIdx.x * (uint32_t)ROW_WARPS + (threadIdx.x >> 5);
  const uint32_t W = gridDim.x * (uint32_t)ROW_WARPS;
  auto claim = [&](uint32_t* ticket, uint32_t n) {
    uint32_t v = 0u;
    if (lane == 0) v = atomicAdd(ticket, n);
    return __shfl_sync(FULL, v, 0);
  };
  // the groups' sums into every group: a tree over the lane groups, so the
  // order is fixed (the sum of two is the same from both sides)
  auto merge_groups = [&](CSum(&acc)[P]) {
    for (int o = L; o < 32; o <<= 1)
#pragma unroll
      for (int i = 0; i < P; ++i) {
        const float hi = __shfl_xor_sync(FULL, acc[i].hi, o);
        const float lo = __shfl_xor_sync(FULL, acc[i].lo, o);
        csum_merge(acc[i], hi, lo);
      }
  };

  // ---- 1. chunks of the longest rows, one warp per chunk; the warp's next
  // item is claimed and read while the current one is summed
  {
    // a warp's first item is the one of its own number, the others are claimed
    // behind those
    uint32_t it = gw;
    uint2 item = it < n_items ? so.items[it] : make_uint2(0u, 0u);
    uint4 lr = it < n_items ? so.long_rows[item.x] : make_uint4(0u, 0u, 0u, 0u);
    while (it < n_items) {
      const uint32_t it_next = W + claim(so.item_ticket, 1u);
      const uint2 item_next = it_next < n_items ? so.items[it_next] : make_uint2(0u, 0u);
      const uint32_t nch = (lr.z + chunk - 1) / chunk;
      const uint32_t e0 = lr.y + item.y * chunk;
      const uint32_t e1 = min(e0 + chunk, lr.y + lr.z);
      const uint32_t per = (e1 - e0 + G - 1) / G;
      const uint32_t b0 = min(e0 + g * per, e1), b1 = min(b0 + per, e1);
      CSum acc[P];
#pragma unroll
      for (int i = 0; i < P; ++i) acc[i] = CSum{0.f, 0.f};
      sum_entries<CH, CPL, UNR>(so, unit, b0, b1, l, L, C, d, acc);
      __syncwarp();
      merge_groups(acc);
      bool finish = nch == 1u;
      if (!finish) {  // one chunk of several: leave its sum; the last chunk finishes the row
        if (g == 0) {
          const size_t pb = (size_t)(lr.w + item.y) * (size_t)d;
          Part<CH, CPL> hi, lo;
#pragma unroll
          for (int i = 0; i < P; ++i) {
            hi.v[i] = acc[i].hi;
            lo.v[i] = acc[i].lo;
          }
          store_part<CH, CPL>(so.part_hi + pb, l, L, C, hi);
          store_part<CH, CPL>(so.part_lo + pb, l, L, C, lo);
        }
        __threadfence();
        __syncwarp();
        uint32_t last = 0u;
        if (lane == 0) last = atomicAdd(so.long_done + item.x, 1u) == nch - 1u;
        finish = __shfl_sync(FULL, last, 0) != 0u;
        if (finish) {  // every chunk's sum is visible: each group merges its share of them in order
          __threadfence();
#pragma unroll
          for (int i = 0; i < P; ++i) acc[i] = CSum{0.f, 0.f};
          const uint32_t share = (nch + G - 1) / G;
          const uint32_t c0 = min(g * share, nch), c1 = min(c0 + share, nch);
          constexpr int MU = P > 4 ? 1 : (CH == 4 ? 2 : 4);  // chunk sums in flight
          for (uint32_t cc = c0; cc < c1; cc += MU) {
            Part<CH, CPL> hi[MU], lo[MU];
#pragma unroll
            for (int e = 0; e < MU; ++e)
              if (cc + e < c1) {
                const size_t qb = (size_t)(lr.w + cc + e) * (size_t)d;
                load_part_cg<CH, CPL>(so.part_hi + qb, l, L, C, hi[e]);
                load_part_cg<CH, CPL>(so.part_lo + qb, l, L, C, lo[e]);
              }
#pragma unroll
            for (int e = 0; e < MU; ++e)
              if (cc + e < c1)
#pragma unroll
                for (int i = 0; i < P; ++i) csum_merge(acc[i], hi[e].v[i], lo[e].v[i]);
          }
          __syncwarp();
          merge_groups(acc);
        }
      }
      if (finish && g == 0) {
        const uint4 ra = so.rr[lr.x], rb = so.rr[lr.x + 1];
        const SegTable& tb = MULTI ? tabs[table_of_row(so.ustart, t0, t1, lr.x)] : tb0;
        const float den = row_denominator(a.sparse_den, rb.z - ra.z, rb.w - ra.w, a.M);
        Part<CH, CPL> w, s0, s1;
        const size_t base = (size_t)ra.x * (size_t)d;
        load_part<CH, CPL>(tb.w + base, l, L, C, w);
        load_part<CH, CPL>(tb.s0 + base, l, L, C, s0);
        if (ADAM) load_part<CH, CPL>(tb.s1 + base, l, L, C, s1);
        finish_row<CH, CPL, ADAM>(tb.opt, tb.w + base, tb.s0 + base, tb.s1 + base, den, acc, w, s0,
                                  s1, l, L, C);
        if (l == 0) {
          tb.ver[ra.x] = tag;
          ++applied;
        }
      }
      __syncwarp();
      it = it_next;
      item = item_next;
      lr = it < n_items ? so.long_rows[item.x] : make_uint4(0u, 0u, 0u, 0u);
    }
  }

  // ---- 2. rows of LONG_ROW + 1 .. small_limit kept occurrences, one lane group each
  {
    uint32_t base = n_small ? claim(so.small_ticket, (uint32_t)G) : 0u;
    uint4 sr = base + g < n_small ? so.small_rows[base + g] : make_uint4(0u, 0u, 0u, 0u);
    while (base < n_small) {
      const uint32_t base_next = claim(so.small_ticket, (uint32_t)G);
      const uint4 sr_next =
          base_next + g < n_small ? so.small_rows[base_next + g] : make_uint4(0u, 0u, 0u, 0u);
      const uint32_t x = sr.x, ks = sr.y, n = sr.z & 255u;  // n = 0: no row for this group
      if (n > 0u) {
        const SegTable& tb = MULTI ? tabs[sr.z >> 8] : tb0;
        Part<CH, CPL> w, s0, s1;
        const size_t rb = (size_t)x * (size_t)d;
        if (l == 0) {
          prefetch_row<CH>(tb.w + rb, d);
          prefetch_row<CH>(tb.s0 + rb, d);
          if (ADAM) prefetch_row<CH>(tb.s1 + rb, d);
        }
        CSum acc[P];
#pragma unroll
        for (int i = 0; i < P; ++i) acc[i] = CSum{0.f, 0.f};
        sum_entries<CH, CPL, UNR>(so, unit, ks, ks + n, l, L, C, d, acc);
        load_part<CH, CPL>(tb.w + rb, l, L, C, w);
        load_part<CH, CPL>(tb.s0 + rb, l, L, C, s0);
        if (ADAM) load_part<CH, CPL>(tb.s1 + rb, l, L, C, s1);
        finish_row<CH, CPL, ADAM>(tb.opt, tb.w + rb, tb.s0 + rb, tb.s1 + rb, __uint_as_float(sr.w),
                                  acc, w, s0, s1, l, L, C);
        if (l == 0) {
          tb.ver[x] = tag;
          ++applied;
        }
      }
      __syncwarp();
      base = base_next;
      sr = sr_next;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) applied += __shfl_xor_sync(FULL, applied, o);
  if (lane == 0 && applied) atomicAdd(&st->rows_applied, (unsigned long long)applied);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename K>
int blocks_per_sm(K kernel, int threads, size_t smem) {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem) != cudaSuccess ||
      b < 1)
    b = 1;
  return b;
}

template <int CH, int CPL, bool ADAM, bool MULTI, bool AHEAD>
void launch_apply_as(const StepArgs& a, const RowRange& r, const SegTable* tabs, const SegOut& so,
                     int64_t G, DevStats* stats, ErrSink err, int num_sms, cudaStream_t s) {
  static const int bps = blocks_per_sm(k_row_apply<CH, CPL, ADAM, MULTI, AHEAD>, ROW_THREADS, 0);
  // every warp has at least the rows that it works on at once
  const int64_t want = (r.n + ROW_WARPS * G - 1) / (ROW_WARPS * G);
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms * bps, want));
  launch_chained(a.N, k_row_apply<CH, CPL, ADAM, MULTI, AHEAD>, (unsigned)grid, ROW_THREADS, 0, s, a,
                 r.first, tabs, r.t0, r.t1, chunk_entries(r.n, (int)(32 / G), num_sms),
                 small_limit(r.n), so, stats, err);
}

template <int CH, int CPL, bool ADAM, bool MULTI>
void launch_rows_as(const StepArgs& a, const RowRange& r, const SegTable* tabs, const SegOut& so,
                    bool longs, DevStats* stats, ErrSink err, int num_sms, cudaStream_t s) {
  const int64_t G = 32 / row_lanes(CH == 4 ? r.first.d / 4 : r.first.d, CPL);
  if (!longs) {
    if constexpr (CH == 1) {
      launch_apply_as<CH, CPL, ADAM, MULTI, CPL == 1>(a, r, tabs, so, G, stats, err, num_sms, s);
    } else {
      if (CPL == 1 && r.first.d <= APPLY_AHEAD_DIM)
        launch_apply_as<CH, CPL, ADAM, MULTI, CPL == 1>(a, r, tabs, so, G, stats, err, num_sms, s);
      else
        launch_apply_as<CH, CPL, ADAM, MULTI, false>(a, r, tabs, so, G, stats, err, num_sms, s);
    }
  } else {
    static const int bps = blocks_per_sm(k_row_long<CH, CPL, ADAM, MULTI>, ROW_THREADS, 0);
    const int64_t warps = r.n / ((LONG_ROW + 1) * G) + r.n / SMALL_MAX + 1;
    const int64_t grid = std::max<int64_t>(
        1, std::min<int64_t>((int64_t)num_sms * std::min(bps, r.long_blocks), (warps + ROW_WARPS - 1) / ROW_WARPS));
    launch_chained(a.N, k_row_long<CH, CPL, ADAM, MULTI>, (unsigned)grid, ROW_THREADS, 0, s, a, r.first,
                   tabs, r.t0, r.t1, chunk_entries(r.n, (int)(32 / G), num_sms), so, stats, err);
  }
}

template <int CH, int CPL>
void launch_rows(const StepArgs& a, const RowRange& r, const SegTable* tabs, const SegOut& so,
                 bool longs, DevStats* stats, ErrSink err, int num_sms, cudaStream_t s) {
  const bool adam = r.first.opt.kind == 1, multi = r.t1 - r.t0 > 1;
  if (adam && multi)
    launch_rows_as<CH, CPL, true, true>(a, r, tabs, so, longs, stats, err, num_sms, s);
  else if (adam)
    launch_rows_as<CH, CPL, true, false>(a, r, tabs, so, longs, stats, err, num_sms, s);
  else if (multi)
    launch_rows_as<CH, CPL, false, true>(a, r, tabs, so, longs, stats, err, num_sms, s);
  else
    launch_rows_as<CH, CPL, false, false>(a, r, tabs, so, longs, stats, err, num_sms, s);
}

template <bool MULTI, bool CACHED, bool UNIT>
void launch_scan_as(const StepArgs& a, const SegTable& tb0, const SegTable* tabs, const SegOut& so,
                    const uint32_t* keys, const uint32_t* vals, DevStats* stats, ErrSink err,
                    int64_t wait_ns, size_t smem, cudaStream_t s) {
  const unsigned tiles = (unsigned)scan_tiles(a.N);
  if (a.N > CHAIN_MAX_N)
    launch_chained(a.N, k_seg_scan<MULTI, CACHED, UNIT, true>, tiles, SCAN_THREADS, smem, s, a, tb0,
                   tabs, so, keys, vals, stats, err, wait_ns);
  else
    launch_chained(a.N, k_seg_scan<MULTI, CACHED, UNIT, false>, tiles, SCAN_THREADS, smem, s, a, tb0,
                   tabs, so, keys, vals, stats, err, wait_ns);
}

}  // namespace

int64_t scan_tiles(int64_t N) { return (N + SCAN_TILE - 1) / SCAN_TILE; }

// Beside one per row, chunks are of at least 32 entries per lane group; full ones,
// or those of a range with fewer than twice what the warps take at a time (twice
// that after the last halving).
int64_t long_items(int64_t n, int num_sms) {
  return std::min(n / 32, n / 128 + 4 * (int64_t)num_sms * LONG_WARPS) + 1;
}

int64_t long_parts(int64_t n, int d, int num_sms) {
  const int CPL = (d & 3) == 0 ? (d <= 128 ? 1 : 2) : (d <= 32 ? 1 : d <= 64 ? 2 : d <= 128 ? 4 : 8);
  const int L = row_lanes((d & 3) == 0 ? d / 4 : d, CPL);
  const int64_t G = 32 / L;
  return 2 * std::min(n / (32 * G), n / (G * (L == 32 ? 128 : 64)) +
                                        4 * (int64_t)num_sms * LONG_WARPS) + 1;
}

void launch_seg_scan(const StepArgs& a, const SegTable& tb0, const SegTable* tabs,
                     const SegOut& so, const uint32_t* keys, const uint32_t* vals,
                     DevStats* stats, ErrSink err, int64_t wait_ns, cudaStream_t s) {
  if (a.N <= 0) return;
  const bool multi = a.T > 1, unit = a.decay == 0;
  const size_t smem = (multi ? (size_t)a.T * sizeof(SegTable) : 0) + (size_t)a.M * 4 +
                      (size_t)a.T * a.M * 8 + (size_t)a.T * (a.M + 1) * 4;
#define GBA_SCAN(MU, CA, UN, SM) \
  launch_scan_as<MU, CA, UN>(a, tb0, tabs, so, keys, vals, stats, err, wait_ns, SM, s)
  if (smem > SCAN_CACHE_BYTES) {
    if (unit)
      GBA_SCAN(true, false, true, 0);
    else
      GBA_SCAN(true, false, false, 0);
  } else if (multi) {
    if (unit)
      GBA_SCAN(true, true, true, smem);
    else
      GBA_SCAN(true, true, false, smem);
  } else {
    if (unit)
      GBA_SCAN(false, true, true, smem);
    else
      GBA_SCAN(false, true, false, smem);
  }
#undef GBA_SCAN
}

#define GBA_ROW_DISPATCH(LONGS)                                                              \
  const int d = r.first.d;                                                                   \
  if ((d & 3) == 0) {                                                                        \
    if (d <= 128) return launch_rows<4, 1>(a, r, tabs, so, LONGS, stats, err, num_sms, s);   \
    return launch_rows<4, 2>(a, r, tabs, so, LONGS, stats, err, num_sms, s);                 \
  }                                                                                          \
  if (d <= 32) return launch_rows<1, 1>(a, r, tabs, so, LONGS, stats, err, num_sms, s);      \
  if (d <= 64) return launch_rows<1, 2>(a, r, tabs, so, LONGS, stats, err, num_sms, s);      \
  if (d <= 128) return launch_rows<1, 4>(a, r, tabs, so, LONGS, stats, err, num_sms, s);     \
  return launch_rows<1, 8>(a, r, tabs, so, LONGS, stats, err, num_sms, s);

void launch_row_apply(const StepArgs& a, const RowRange& r, const SegTable* tabs,
                      const SegOut& so, DevStats* stats, ErrSink err, int num_sms,
                      cudaStream_t s) {
  GBA_ROW_DISPATCH(false)
}

void launch_row_long(const StepArgs& a, const RowRange& r, const SegTable* tabs,
                     const SegOut& so, DevStats* stats, ErrSink err, int num_sms,
                     cudaStream_t s) {
  GBA_ROW_DISPATCH(true)
}

#undef GBA_ROW_DISPATCH

}  // namespace gba
