// Internal declarations shared by the translation units of libgba.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gba {

// ---- device error word bits -------------------------------------------------
constexpr uint32_t ERR_ID_RANGE = 1u;
constexpr uint32_t ERR_TIMEOUT = 2u;
constexpr uint32_t ERR_INTERNAL = 4u;

// Where kernels report a failure: the step's own word (later kernels of the
// same step skip their work when it is set), the handle's word (what the host
// reports), and a flag in mapped pinned host memory the host polls without
// synchronising.
struct ErrSink {
  uint32_t* step;
  uint32_t* dev;
  volatile uint32_t* host;
};

__device__ __forceinline__ void raise_error(const ErrSink& e, uint32_t code) {
  atomicOr(e.step, code);
  atomicOr(e.dev, code);
  *e.host = 1u;
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---- mbarriers and 1-D bulk async copies (shared memory, this CTA) ----------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Waits for the phase with the given parity to complete; the thread may be
// suspended in the instruction for up to the hinted time instead of spinning.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity), "r"(100000u)
      : "memory");
  return ok != 0u;
}

// Bounded wait for the phase with the given parity; false if it gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if ((int64_t)(globaltimer_ns() - t0) > limit_ns) return false;
  }
  return true;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// ---- chained launches -------------------------------------------------------
// The kernels of a step follow one another on a stream, each reading what the
// one before wrote.  They are launched so that a kernel's blocks may be set up
// while the last blocks of the one before still run (programmatic stream
// serialization): chain_wait, first in the kernel, returns once every earlier
// kernel has completed and its writes are visible; it then lets the next kernel
// be set up in turn.  On steps of ten kernels of 3 to 20 us that takes about a
// microsecond off each gap (0.03M ids 61.7 -> 54.5 us a step, 0.85M 209.6 ->
// 200.2); above CHAIN_MAX_N occurrences the waiting blocks' places on the SMs
// are worth more than the gaps where steps overlap (5.2M: 0.7% slower chained) or
// are long (131M: the same), so those steps' kernels start in the plain order.  One
// by one, with the scan's registers that go with it (k_seg_scan), chaining takes
// 278.1 us against 279.6 at 1.3M, 359.8 against 357.0 at 2M, 425 against 430 at 2.6M
// and 688 against 701 at 5.2M occurrences x 32 floats.  Pulls, the copies of pushes and push-time
// dense sums, which come one after another, are always chained (N = 0).
// A block may thus be resident while the kernel before still writes, so memory that
// any kernel writes (parameters, tags, descriptions, a caller's ids and gradients) is
// not read-only for a chained kernel's life: it is read by ordinary loads after
// chain_wait, never by __ldg or through const __restrict__ parameters.
constexpr int64_t CHAIN_MAX_N = 1 << 21;
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_chained(int64_t N, void (*kernel)(P...), unsigned grid, unsigned threads,
                                  size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = N <= CHAIN_MAX_N ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ---- per-table static description (device copy) ----------------------------
struct TableInfo {
  int64_t V;
  uint32_t key_base;  // first global key of the table
  int32_t id_mode;    // 0 DIRECT, 1 MODULO
  uint64_t mod_magic; // floor((2^64 - 1) / V), for mod_u64
};

// x mod V for a 64-bit x and V < 2^32, without a 64-bit division: the
// quotient estimate floor(x * m / 2^64) with m = floor((2^64 - 1) / V) is at
// most 2 below floor(x / V) (division by an invariant integer through a
// precomputed reciprocal, after Granlund and Montgomery 1994), so at most two
// corrections give the exact remainder.
__device__ __forceinline__ uint64_t mod_u64(uint64_t x, uint64_t V, uint64_t m) {
  uint64_t r = x - __umul64hi(x, m) * V;
  if (r >= V) r -= V;
  if (r >= V) r -= V;
  return r;
}

// ---- counter-based initial values (shared by table init and hash inserts) ---
// SplitMix64 (Steele, Lea, Flood 2014): output for state x.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  uint64_t z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Weight of element e of an array: top 24 bits of the hash, centred, times
// 2^-27 (an exact float in [-1/16, 1/16)).
__device__ __forceinline__ float init_weight(uint64_t seed, uint64_t tag, uint64_t e) {
  const uint64_t h = splitmix64(seed ^ tag ^ e);
  const int32_t top = (int32_t)(h >> 40) - 8388608;
  return (float)top * 0x1p-27f;
}

// ---- expandable hash tables of 64-bit ids (id_mode HASH) --------------------
// Open addressing with linear probing over a power-of-two number of slots; the
// row of an id is the slot it occupies, so the embedding arrays are indexed by
// slot.  A new id is inserted by compare-and-swap on its slot's key and its
// row is initialised from the id (element e = id * d + j of the table's
// counter-based stream), so every id starts from the same values whichever
// slot it lands in.
constexpr unsigned long long HASH_EMPTY = 0x8000000000000000ull;  // INT64_MIN: not a valid id
struct HashInfo {
  unsigned long long* keys;  // [slots] id per slot, HASH_EMPTY when free
  uint64_t mask;             // slots - 1
  float* w;
  float* s0;
  float* s1;
  int32_t* ver;
  unsigned long long* count;  // ids inserted so far
  uint64_t seed, tag;
  int32_t d, kind;
  float init_acc;
  int32_t pad;
};

__device__ __forceinline__ void hash_init_row(const HashInfo& hi, uint64_t slot, int64_t id) {
  const float a0 = hi.kind == 0 ? hi.init_acc : 0.f;
  for (int j = 0; j < hi.d; ++j) {
    const size_t e = (size_t)slot * hi.d + j;
    hi.w[e] = init_weight(hi.seed, hi.tag, (uint64_t)id * (uint64_t)hi.d + (uint64_t)j);
    hi.s0[e] = a0;
    if (hi.kind == 1) hi.s1[e] = 0.f;
  }
  hi.ver[slot] = 0;
}

// The slot of id, inserting it when absent; returns mask + 1 when the table
// is full (cannot happen while the host keeps it at most half full).
__device__ __forceinline__ uint64_t hash_find_or_insert(const HashInfo& hi, int64_t id) {
  const unsigned long long key = (unsigned long long)id;
  uint64_t slot = splitmix64(key) & hi.mask;
  for (uint64_t probe = 0; probe <= hi.mask; ++probe, slot = (slot + 1) & hi.mask) {
    const unsigned long long k = *(volatile unsigned long long*)(hi.keys + slot);
    if (k == key) return slot;
    if (k == HASH_EMPTY) {
      const unsigned long long old = atomicCAS(hi.keys + slot, HASH_EMPTY, key);
      if (old == HASH_EMPTY) {
        hash_init_row(hi, slot, id);
        atomicAdd(hi.count, 1ull);
        return slot;
      }
      if (old == key) return slot;
    }
  }
  return hi.mask + 1;
}

// The slot of id, or mask + 1 when it is absent.
__device__ __forceinline__ uint64_t hash_find(const HashInfo& hi, int64_t id) {
  const unsigned long long key = (unsigned long long)id;
  uint64_t slot = splitmix64(key) & hi.mask;
  for (uint64_t probe = 0; probe <= hi.mask; ++probe, slot = (slot + 1) & hi.mask) {
    const unsigned long long k = hi.keys[slot];
    if (k == key) return slot;
    if (k == HASH_EMPTY) break;
  }
  return hi.mask + 1;
}

// ---- optimizer parameters of one parameter group for one step ---------------
struct OptStep {
  int32_t kind;  // 0 Adagrad, 1 Adam
  float lr, b1, b2, eps;
  float c1, c2;    // 1 - b1, 1 - b2 (float arithmetic)
  float bc1, bc2;  // Adam bias corrections of this step
};

// Adagrad and Adam, one IEEE float operation at a time in a fixed order.
template <bool ADAM>
__device__ __forceinline__ void opt_update_as(const OptStep& o, float& w, float& s0, float& s1,
                                              float g) {
  if (!ADAM) {
    float gg = __fmul_rn(g, g);
    float an = __fadd_rn(s0, gg);
    float step = __fmul_rn(o.lr, g);
    float den = __fsqrt_rn(an);
    s0 = an;
    w = __fsub_rn(w, __fdiv_rn(step, den));
  } else {
    float mn = __fadd_rn(__fmul_rn(o.b1, s0), __fmul_rn(o.c1, g));
    float gg = __fmul_rn(g, g);
    float vn = __fadd_rn(__fmul_rn(o.b2, s1), __fmul_rn(o.c2, gg));
    float mhat = __fdiv_rn(mn, o.bc1);
    float vhat = __fdiv_rn(vn, o.bc2);
    float num = __fmul_rn(o.lr, mhat);
    float den = __fadd_rn(__fsqrt_rn(vhat), o.eps);
    s0 = mn;
    s1 = vn;
    w = __fsub_rn(w, __fdiv_rn(num, den));
  }
}
__device__ __forceinline__ void opt_update(const OptStep& o, float& w, float& s0, float& s1,
                                           float g) {
  if (o.kind == 0)
    opt_update_as<false>(o, w, s0, s1, g);
  else
    opt_update_as<true>(o, w, s0, s1, g);
}

// Error-free transformation of a + b (Knuth's TwoSum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  float bp = __fsub_rn(s, a);
  float ap = __fsub_rn(s, bp);
  e = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}

// Compensated accumulator: value = hi + lo.
struct CSum {
  float hi, lo;
};
__device__ __forceinline__ void csum_add(CSum& c, float x) {
  float s, e;
  two_sum(c.hi, x, s, e);
  c.hi = s;
  c.lo = __fadd_rn(c.lo, e);
}
__device__ __forceinline__ void csum_merge(CSum& c, float hi, float lo) {
  float s, e;
  two_sum(c.hi, hi, s, e);
  c.hi = s;
  c.lo = __fadd_rn(__fadd_rn(c.lo, lo), e);
}
__device__ __forceinline__ float csum_value(const CSum& c) { return __fadd_rn(c.hi, c.lo); }

// ---- one global step, as seen by the kernels ---------------------------------
// Passed by value to every kernel of a step; the arrays live in a device
// buffer the host fills before the step.
struct StepArgs {
  int64_t k;
  int32_t M;           // messages popped
  int32_t T;           // tables
  int64_t N;           // id occurrences over all tables
  int32_t iota;
  int32_t row_staleness;
  int32_t sparse_den;
  int32_t decay;        // 0: f in {0, 1} (Eq. (1)); 1: f = lambda^s for s <= iota
  int32_t drop_latest;  // the last drop_latest popped messages are excluded (0: none)
  int32_t n_wtab;       // entries of wtab (decay 1): wtab[s] = lambda^s, s < n_wtab
  const float* wtab;    // [n_wtab] device
  const int64_t* tokens;          // [M]
  const float* const* dense_ptr;  // [M]
  const uint32_t* msg_off;        // [T][M+1] occurrence offsets within the table
  const int64_t* const* ids_ptr;  // [T][M]
  const float* const* rows_ptr;   // [T][M]
  const int64_t* nbase;           // [T+1] first global occurrence of each table
  const TableInfo* tinfo;         // [T]
  const HashInfo* hinfo;          // [T] (tables with id_mode HASH)
};

// Per-step device scratch that K1 clears at the start of a step.
struct StepScratch {
  uint32_t* hist;          // [passes][radix] digit histograms of the key passes
  uint32_t* tile_counter;  // [4] onesweep tile tickets
  int32_t* keep;           // [M] message weights f
  int32_t* kept_list;      // [M] indices of kept messages, in pop order
  int32_t* n_kept;         // [1]
  uint32_t* step_err;      // [1] failures of this step
  uint32_t* seg_ticket;    // [T][8]: word 0 scan tile tickets; words 8 t0 + 1 .. 6, for the
                           // range of tables from t0: long rows, their items, chunk-sum
                           // slots, item tickets, small rows, small-row tickets
  float* fw;               // [M] message weights of the dense sum (decay 1; 1 or 0 otherwise)
};

// Weight of a gradient with staleness s (s >= 0), or 0 when it is excluded:
// Eq. (1) keeps s <= iota; decay 1 scales a kept gradient by lambda^s.
__device__ __forceinline__ float decay_weight(const StepArgs& a, uint64_t s) {
  if (s > (uint64_t)(int64_t)a.iota) return 0.f;
  if (a.decay == 0) return 1.f;
  return s < (uint64_t)a.n_wtab ? __ldg(a.wtab + s) : 0.f;
}

// Compensated accumulation of a product f * g: the product's rounding error
// (from a fused multiply-add) joins the compensation term, so with f = 1 this
// is exactly csum_add.
__device__ __forceinline__ void csum_add_prod(CSum& c, float f, float g) {
  const float p = __fmul_rn(f, g);
  const float e = __fmaf_rn(f, g, -p);
  float s, t;
  two_sum(c.hi, p, s, t);
  c.hi = s;
  c.lo = __fadd_rn(c.lo, __fadd_rn(t, e));
}

// A kept term of a weighted sum.  With decay strategy 0 every kept weight is
// exactly 1 and the term is added by csum_add, which gives what csum_add_prod
// gives for f = 1 (the product and its error are g and 0) with fewer operations.
__device__ __forceinline__ void csum_add_w(CSum& c, bool unit, float f, float g) {
  if (unit)
    csum_add(c, g);
  else
    csum_add_prod(c, f, g);
}

// Pause between two looks at an earlier tile's words: spinning takes issue slots from
// the tiles it waits for.
constexpr unsigned LOOKBACK_SLEEP_NS = 64;

// Accumulated statistics (device).
struct DevStats {
  unsigned long long steps, msgs_kept, msgs_dropped, dense_stale_sum, dense_stale_max, pairs,
      pairs_dropped, row_stale_sum, row_stale_max, occurrences, rows_touched, rows_applied,
      occ_kept;
};

// The message of table-local occurrence x in the offsets off[0..M]: the
// largest m with off[m] <= x (empty messages repeat an offset).
__device__ __forceinline__ int message_of_any(const uint32_t* off, int M, uint32_t x) {
  int lo = 0, hi = M;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= x)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

// The same, starting from the message an even split would give (exact when
// every message holds the same number of ids, as with one-hot fields; scale
// is M over the table's occurrences), then a few neighbours, then the binary
// search.  x becomes the occurrence's index within its message.
__device__ __forceinline__ int message_of(const uint32_t* off, int M, uint32_t& x, float scale) {
  int m = min((int)((float)x * scale), M - 1);
  uint32_t lo = off[m], hi = off[m + 1];
  if (x < lo || x >= hi) {
    for (int s = 0; s < 3 && (x < lo || x >= hi); ++s) {
      if (x < lo) {
        hi = lo;
        lo = off[--m];  // off[0] = 0 <= x: m stays >= 0
      } else {
        lo = hi;
        hi = off[++m + 1];  // x < off[M]: m stays < M
      }
    }
    if (x < lo || x >= hi) {
      m = message_of_any(off, M, x);
      lo = off[m];
    }
  }
  x -= lo;
  return m;
}

// ---- launch wrappers (defined in the kernel translation units) ---------------
// meta_bytes (a multiple of 16, at most META_BY_KERNEL; 0: none) of the step's
// description are brought from host_meta (mapped pinned memory) to dev_meta.
constexpr size_t META_BY_KERNEL = 32 * 1024;
void launch_weights(const StepArgs& a, StepScratch sc, DevStats* stats, int n_hist_words,
                    const void* host_meta, void* dev_meta, size_t meta_bytes, cudaStream_t s);

// ---- the sort of the step's keys
constexpr int MAX_PASSES = 4;
// Keys per onesweep tile, and of more than SORT_BIG_N keys twice as many (a step of
// 1.3M occurrences with either 279 us, 2M 360 with the smaller tiles and 347 with the
// larger, 2.6M 434 and 429, 5.2M 718 and 700).
constexpr int SORT_TILE_KEYS = 2048;
constexpr int64_t SORT_BIG_N = 1 << 21;

// The digits of the passes over keys of so many bits.
struct SortPlan {
  int32_t passes;
  int32_t radix;  // counters per pass: 256 or 512
  int32_t shift[MAX_PASSES];
  uint32_t mask[MAX_PASSES];
};
SortPlan make_sort_plan(int key_bits, int max_digit_bits);
// Look-back words for sorts of up to N keys.
size_t sort_status_words(int64_t N, int radix);

// Digit counts of every pass into hist [passes][radix]; writes each
// occurrence's key to keys0 (the first pass's input).
void launch_sort_histogram(const StepArgs& a, const SortPlan& plan, uint32_t* hist,
                           uint32_t* keys0, ErrSink err, int num_sms, cudaStream_t s);

struct SortPass {
  uint32_t N;
  int32_t shift;  // set by launch_onesweep, as is mask
  uint32_t mask;
  const uint32_t* hist;  // the pass's digit counts
  uint32_t* ticket;
  const uint32_t* keys_in;
  const uint32_t* vals_in;  // unused by the first pass: its payload is the position
  uint32_t* keys_out;
  uint32_t* vals_out;
  unsigned long long* status;
  uint32_t epoch;
};
void launch_onesweep(const SortPlan& plan, int pass, SortPass sp, ErrSink err, int64_t wait_ns,
                     cudaStream_t s);

// One table as the row kernels see it.
struct SegTable {
  float* w;
  float* s0;
  float* s1;
  int32_t* ver;
  int32_t d;
  uint32_t key_base;
  uint32_t rows;  // V of the table
  uint32_t nb;    // first position of its keys in the sorted array, and first occurrence
  uint32_t n;     // how many it has
  float mscale;   // messages over occurrences
  OptStep opt;
  uint32_t pad;
};
static_assert(sizeof(SegTable) % 8 == 0, "copied as words, followed by 8-byte values");

// Consecutive tables of one width and optimizer, handled by one launch of each
// row kernel.
struct RowRange {
  int32_t t0, t1;  // tables [t0, t1)
  int64_t n;       // their occurrences
  // Blocks per SM of the long-row kernel, at most.  As many as fit hold every
  // register of an SM; where steps overlap, one leaves room for the next step's sort
  // and the dense update (2e8 x 64: 932 -> 951 steps/s; steps one by one are slower with one).
  int32_t long_blocks;
  SegTable first;  // table t0
};

// Buffers of the row kernels (one set, used in stream order by the apply
// stream).
//  rr[u]   row u in sorted order over all tables: (row x of its table, and the
//          exclusive prefixes at its head of kept occurrences K, (message, row)
//          pairs C and kept pairs CK); rr[U] holds the totals, so row u's kept
//          occurrences are kl[rr[u].K .. rr[u+1].K), c_x = rr[u+1].C - rr[u].C
//  kl[j]   address of the j-th kept occurrence's gradient row, sorted by row
//  kw[j]   its weight f (not written under Eq. (1), where it is 1)
//  ustart[t]  first row record of table t; ustart[T] = U
// The lists and their counters belong to the range of tables being applied.
struct SegOut {
  uint4* rr;
  const float** kl;
  float* kw;
  unsigned long long* status;  // [tiles][4] look-back words of the scan
  uint32_t epoch;              // tag of this launch's look-back words
  uint32_t* ticket;            // scan tile tickets (cleared by K1)
  uint32_t* ustart;            // [T + 1]
  uint32_t* n_long;            // rows with more than small_limit kept occurrences (cleared by K1)
  uint32_t* n_items;           // chunks of those rows (cleared by K1)
  uint32_t* n_parts;           // chunk-sum slots of rows split into chunks (cleared by K1)
  uint32_t* item_ticket;       // items claimed by warps of the long-row kernel (cleared by K1)
  uint4* long_rows;            // [n_long] (u, first kept, kept count, first chunk-sum slot)
  uint32_t* long_done;         // [n_long] chunks of the row finished
  uint2* items;                // [n_items] (long row, chunk)
  float* part_hi;              // [n_parts][d] compensated chunk sums
  float* part_lo;
  uint4* small_rows;           // [n_small] (row, first kept, table << 8 | kept count, denominator)
  uint32_t* n_small;           // rows of LONG_ROW + 1 .. small_limit kept occurrences (cleared by K1)
  uint32_t* small_ticket;      // small rows claimed by the long-row kernel (cleared by K1)
};

// Rows with at most LONG_ROW kept occurrences are applied by k_row_apply,
// rows of at most small_limit (SMALL_MAX, or half of it in ranges of up to 2^23
// occurrences) by one lane group of k_row_long each, longer ones in chunks.
constexpr int LONG_ROW = 4;
constexpr int SMALL_MAX = 64;
static_assert(SMALL_MAX < 256, "a small row's count shares a word with its table");
constexpr int SCAN_TILE = 2048;  // sorted positions per segment-scan tile

int64_t scan_tiles(int64_t N);
// The most chunks, beside one for each long row, that n occurrences can make, and
// the most chunk-sum slots that they can need at width d.
int64_t long_items(int64_t n, int num_sms);
int64_t long_parts(int64_t n, int d, int num_sms);

// tb0: the first table; tabs: all of them, on the device.
void launch_seg_scan(const StepArgs& a, const SegTable& tb0, const SegTable* tabs,
                     const SegOut& so, const uint32_t* keys, const uint32_t* vals,
                     DevStats* stats, ErrSink err, int64_t wait_ns, cudaStream_t s);

// The range's rows with few kept occurrences; lists the others for
// launch_row_long, which comes next on the stream.
void launch_row_apply(const StepArgs& a, const RowRange& r, const SegTable* tabs,
                      const SegOut& so, DevStats* stats, ErrSink err, int num_sms,
                      cudaStream_t s);
void launch_row_long(const StepArgs& a, const RowRange& r, const SegTable* tabs,
                     const SegOut& so, DevStats* stats, ErrSink err, int num_sms,
                     cudaStream_t s);

struct DenseArgs {
  float* w;
  float* s0;
  float* s1;
  int64_t D;
  int32_t M;
  OptStep opt;
  int32_t withhold = 0;  // test hook: the producer issues no copies, so every
                         // consumer wait runs out and reports ERR_TIMEOUT
};

cudaError_t configure_dense();
void launch_dense(const StepArgs& a, const DenseArgs& da, StepScratch sc, ErrSink err,
                  int64_t wait_ns, int num_sms, cudaStream_t s);

// Arrays copied by one launch: a pushed message's ids, gradient rows and dense
// gradient (at most COPY_MAX of them, each smaller than 2^44 bytes).
constexpr int COPY_MAX = 32;
struct CopyList {
  const void* src[COPY_MAX];
  void* dst[COPY_MAX];
  uint64_t bytes[COPY_MAX];
  uint32_t first[COPY_MAX];  // first chunk of each array (set by launch_push_copy)
  uint32_t chunks;           // chunks of them all (set by launch_push_copy)
  int32_t n;
};
// By at most max_blocks blocks.
constexpr unsigned HOST_BLOCKS = 64;  // fill the link to host memory
cudaError_t launch_push_copy(CopyList cl, unsigned max_blocks, cudaStream_t s);

// Eager dense aggregation: add f * g to a step's accumulator (first: start it;
// reverse: from the last parameter down), and the step's update from the
// accumulator.
void launch_dense_accumulate(float* hi, float* lo, const float* g, int64_t D, float f, bool first,
                             bool reverse, int num_sms, cudaStream_t s);
void launch_dense_eager(const DenseArgs& da, const float* hi, const float* lo, bool has_sum,
                        bool reverse, ErrSink err, int num_sms, cudaStream_t s);

void launch_init_table(float* w, float* s0, float* s1, int32_t* ver, int64_t rows, int32_t d,
                       int32_t kind, float init_acc, uint64_t seed, uint64_t tag,
                       cudaStream_t s);

void launch_init_dense(float* w, float* s0, float* s1, int64_t D, int32_t kind, float init_acc,
                       uint64_t seed, uint64_t tag, cudaStream_t s);

int launch_wait_selftest(int64_t limit_ns, cudaStream_t s, uint32_t* d_word, uint32_t* result);

// Rows of one table for n ids (pull responding), into out[n][d].
void launch_pull_rows(const float* w, int64_t V, int d, int id_mode, uint64_t mod_magic,
                      const HashInfo* hinfo, const int64_t* ids, int64_t n, float* out,
                      ErrSink err, int num_sms, cudaStream_t s);

// Hash tables: fill keys with HASH_EMPTY; move every id of one table into a
// larger one (keys, rows and tags); slots of ids (mask + 1 when absent).
void launch_hash_clear(unsigned long long* keys, uint64_t slots, cudaStream_t s);
void launch_hash_rehash(HashInfo from, HashInfo to, cudaStream_t s);
void launch_hash_lookup(const HashInfo* hinfo, const int64_t* ids, int64_t n, int64_t* slots,
                        cudaStream_t s);

// Compute capability (major * 10 + minor) of the device code the library's
// kernels were loaded from on the current device, or -1.
int kernel_binary_version();

}  // namespace gba
