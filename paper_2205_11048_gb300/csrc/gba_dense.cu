// K5 of the GBA aggregate-and-apply step: the dense parameters.
//
// g = (sum over kept messages m of f_m grad_m) / M  (Alg. 2: weighted sum of the
// dense gradients divided by N_a; Appendix A: v_k = (1/M) sum g), then Adagrad
// or Adam in place -- one pass over HBM: every kept gradient is read once, the
// weights and optimizer state are read and written once.
//
// Each persistent CTA walks every gridDim-th tile of DT parameters.  A
// producer warp streams the tile's slice of every kept message into a ring of
// shared-memory stages with 1-D bulk async copies (cp.async.bulk, completion
// counted on an mbarrier per stage); eight consumer warps sum the slices with
// compensated (TwoSum) float arithmetic, release each stage on an "empty"
// mbarrier, and finish the tile with the optimizer.  Every mbarrier wait is
// bounded in time; a wait that gives up latches ERR_TIMEOUT, the CTA stops
// issuing copies, waits (bounded) for the copies it already issued, and exits.
#include <algorithm>

#include "gba_internal.cuh"

namespace gba {

namespace {

constexpr int DT = 2048;                 // parameters per tile
// Stages of DT floats: as many as help the largest updates, or fewer for updates
// that are short beside the row path (M gradients of D floats of at most DENSE_SHORT
// bytes, all M counted, and more than one CTA per SM).  Steps of 0.85M ids x 32 floats
// and 32 dense gradients, with 8 stages and with 5: 0.13 GB of them 231 and 220 us,
// 0.26 GB 253 and 242, 0.5 GB 298 and 293, 1 GB 376 and 390, 2 GB 542 and 628, 4 GB
// 874 and 1,199.  It is not the room in shared memory that the shorter ring leaves to
// other kernels: three CTAs hold 62,208 of an SM's 65,536 registers, so no block of
// another kernel is beside them with either ring, and asking for the full shared-memory
// split with 5 stages changes nothing.  What is left is that fewer copies in flight (123 KB
// an SM instead of 197) keep the row path's loads waiting less; that was not shown.
constexpr int STAGES_LONG = 8, STAGES_SHORT = 5;
constexpr int64_t DENSE_SHORT = 256ll << 20;
constexpr int CONSUMER_WARPS = 8;        // 256 threads
constexpr int HALF = CONSUMER_WARPS * 32 * 4;  // floats of one float4 per consumer thread
constexpr int PER = DT / HALF;  // thread c owns [h*HALF + 4c, h*HALF + 4c + 4), h < PER
static_assert(DT % HALF == 0, "a tile is a whole number of float4 rows of the consumers");
constexpr int DENSE_THREADS = (CONSUMER_WARPS + 1) * 32;

template <int STAGES>
__global__ void __launch_bounds__(DENSE_THREADS)
    k_dense_apply(StepArgs a, DenseArgs da, StepScratch sc, ErrSink err, int64_t wait_ns) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* stage_buf = reinterpret_cast<float*>(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw + (size_t)STAGES * DT * sizeof(float));
  uint64_t* empty = full + STAGES;
  __shared__ int s_abort;

  // block-uniform: another kernel may set the word while this block reads it
  if (__syncthreads_or((*(volatile uint32_t*)err.step & (ERR_ID_RANGE | ERR_TIMEOUT)) != 0u)) return;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(full + i, 1u);
      mbar_init(empty + i, (uint32_t)CONSUMER_WARPS);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  const int n_kept = *sc.n_kept;
  const int64_t D4 = da.D & ~3ll;  // parameters streamed by bulk copies
  // This CTA's tiles of DT parameters (the last one shorter, a multiple of 4
  // so every copy stays 16-byte aligned): blockIdx.x, blockIdx.x + gridDim.x,
  // ...  At any moment the CTAs work on neighbouring tiles, so the copies from
  // the kept messages' buffers touch few DRAM pages and TLB entries.
  const int64_t t0 = (int64_t)blockIdx.x * DT, tstep = (int64_t)gridDim.x * DT;

  if (warp == CONSUMER_WARPS) {
    // ---- producer
    if (lane == 0) {
      uint32_t q = 0;
      bool ok = da.withhold == 0;
      for (int64_t start = t0; start < D4 && ok; start += tstep) {
        const uint32_t bytes = (uint32_t)((D4 - start < DT ? D4 - start : DT) * sizeof(float));
        for (int j = 0; j < n_kept; ++j, ++q) {
          const int stage = (int)(q % STAGES);
          const uint32_t ph = (q / STAGES) & 1u;
          if (!mbar_wait(empty + stage, ph ^ 1u, wait_ns) || *(volatile int*)&s_abort) {
            raise_error(err, ERR_TIMEOUT);
            s_abort = 1;
            ok = false;
            break;
          }
          const float* src = a.dense_ptr[sc.kept_list[j]] + start;
          mbar_arrive_expect_tx(full + stage, bytes);
          bulk_g2s(stage_buf + (size_t)stage * DT, src, bytes, full + stage);
        }
      }
      // Make sure no copy this CTA issued is still landing when it exits.  The
      // copies read valid memory and land within microseconds; this wait has its
      // own one-second bound, independent of the configurable limit.
      const uint32_t n_drain = q < (uint32_t)STAGES ? q : (uint32_t)STAGES;
      for (uint32_t i = 0; i < n_drain; ++i) {
        const uint32_t qq = q - 1 - i;
        mbar_wait(full + (qq % STAGES), (qq / STAGES) & 1u, 1000000000ll);
      }
    }
  } else {
    // ---- consumers: thread c owns parameters [h*HALF + 4c, h*HALF + 4c + 4)
    // of each tile, h < PER
    const int c = tid;
    const float Mf = (float)da.M;
    uint32_t q = 0;
    for (int64_t start = t0; start < D4; start += tstep) {
      const int64_t n = D4 - start < DT ? D4 - start : DT;
      bool mine[PER];
      int64_t e[PER];
      float4 w[PER], s0[PER], s1[PER];
#pragma unroll
      for (int h = 0; h < PER; ++h) {
        const int64_t off = (int64_t)h * HALF + (int64_t)c * 4;
        mine[h] = off < n;
        e[h] = start + off;
        w[h] = s0[h] = s1[h] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (mine[h]) {
          w[h] = *reinterpret_cast<const float4*>(da.w + e[h]);
          s0[h] = *reinterpret_cast<const float4*>(da.s0 + e[h]);
          if (da.opt.kind == 1) s1[h] = *reinterpret_cast<const float4*>(da.s1 + e[h]);
        }
      }
      CSum acc[4 * PER];
#pragma unroll
      for (int i = 0; i < 4 * PER; ++i) acc[i] = CSum{0.f, 0.f};
      bool aborted = false;
      for (int j = 0; j < n_kept; ++j, ++q) {
        const int stage = (int)(q % STAGES);
        const uint32_t ph = (q / STAGES) & 1u;
        // Every lane waits (acquiring the copied bytes); the outcome is made
        // warp-uniform so the warp leaves the loop together.
        const bool ok = __all_sync(0xffffffffu, mbar_wait(full + stage, ph, wait_ns));
        if (!ok) {
          if (lane == 0) {
            raise_error(err, ERR_TIMEOUT);
            s_abort = 1;
          }
          aborted = true;
          break;
        }
        if (a.decay == 0) {
#pragma unroll
          for (int h = 0; h < PER; ++h) {
            if (mine[h]) {
              const float4 v = *reinterpret_cast<const float4*>(stage_buf + (size_t)stage * DT +
                                                                h * HALF + 4 * c);
              csum_add(acc[4 * h + 0], v.x);
              csum_add(acc[4 * h + 1], v.y);
              csum_add(acc[4 * h + 2], v.z);
              csum_add(acc[4 * h + 3], v.w);
            }
          }
        } else {  // weighted: f_m * g with the product's rounding error kept
          const float f = sc.fw[j];
#pragma unroll
          for (int h = 0; h < PER; ++h) {
            if (mine[h]) {
              const float4 v = *reinterpret_cast<const float4*>(stage_buf + (size_t)stage * DT +
                                                                h * HALF + 4 * c);
              csum_add_prod(acc[4 * h + 0], f, v.x);
              csum_add_prod(acc[4 * h + 1], f, v.y);
              csum_add_prod(acc[4 * h + 2], f, v.z);
              csum_add_prod(acc[4 * h + 3], f, v.w);
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + stage);
      }
      if (aborted || __shfl_sync(0xffffffffu, *(volatile int*)&s_abort, 0) != 0) break;
#pragma unroll
      for (int h = 0; h < PER; ++h) {
        if (!mine[h]) continue;
        float wv[4] = {w[h].x, w[h].y, w[h].z, w[h].w},
              a0[4] = {s0[h].x, s0[h].y, s0[h].z, s0[h].w},
              a1[4] = {s1[h].x, s1[h].y, s1[h].z, s1[h].w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          opt_update(da.opt, wv[i], a0[i], a1[i], __fdiv_rn(csum_value(acc[4 * h + i]), Mf));
        *reinterpret_cast<float4*>(da.w + e[h]) = make_float4(wv[0], wv[1], wv[2], wv[3]);
        *reinterpret_cast<float4*>(da.s0 + e[h]) = make_float4(a0[0], a0[1], a0[2], a0[3]);
        if (da.opt.kind == 1)
          *reinterpret_cast<float4*>(da.s1 + e[h]) = make_float4(a1[0], a1[1], a1[2], a1[3]);
      }
    }
    // The last (D mod 4) parameters: plain loads, CTA 0.
    if (blockIdx.x == 0 && c < (int)(da.D - D4)) {
      const int64_t e = D4 + c;
      CSum acc{0.f, 0.f};
      for (int j = 0; j < n_kept; ++j)
        csum_add_prod(acc, a.decay == 0 ? 1.f : sc.fw[j], a.dense_ptr[sc.kept_list[j]][e]);
      float wv = da.w[e], a0 = da.s0[e], a1 = da.opt.kind == 1 ? da.s1[e] : 0.f;
      opt_update(da.opt, wv, a0, a1, __fdiv_rn(csum_value(acc), Mf));
      da.w[e] = wv;
      da.s0[e] = a0;
      if (da.opt.kind == 1) da.s1[e] = a1;
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Eager aggregation (Alg. 2 discussion: because the tokens fix the weights,
// part of the weighted sum may be formed before the step).  Under the FIFO every pushed
// message belongs to a known future step, so its weight is known at push: its
// dense gradient is added to that step's compensated accumulator (hi, lo)
// right away, in push order -- the order the buffered K5 sums in -- and the
// step then reads D accumulators instead of its kept messages.
//
// Bound by memory: a push moves 4 B of gradient and 16 B of accumulator per
// parameter, 52 us at 16M parameters when all of it goes to HBM (6.1 TB/s).
// Two things keep part of the accumulators in the 129 MB L2 from one push to the
// next: gradients, and accumulators past the first ACC_KEEP4, are loaded and
// stored evict-first, so the first ones stay (42 us); and consecutive pushes
// walk the parameters in opposite directions, so what a push touched last is
// what the next one meets first (36 us together, 8.8 TB/s of those bytes; at
// 64M parameters 201 -> 183 us).  Accumulators that fit in L2 are walked
// forward only (4M parameters: 9.1 us against 10.3 in turns).
// ---------------------------------------------------------------------------
constexpr int64_t ACC_KEEP4 = 2000000;  // float4 of hi and of lo: 32 MB each
constexpr int64_t ACC_TURN = 8000000;   // parameters from which the direction alternates

__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ float4 ld_hint(const float4* a, uint64_t policy) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(a), "l"(policy));
  return v;
}
__device__ __forceinline__ void st_hint(float4* a, float4 v, uint64_t policy) {
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(a), "f"(v.x),
               "f"(v.y), "f"(v.z), "f"(v.w), "l"(policy)
               : "memory");
}

__global__ void __launch_bounds__(256)
    k_dense_accumulate(float* __restrict__ hi, float* __restrict__ lo,
                       const float* g, int64_t D, float f, int first, int reverse) {
  chain_wait();
  const int64_t D4 = D & ~3ll;
  const int64_t n4 = D4 / 4;
  const uint64_t policy = evict_first_policy();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
    const int64_t q = reverse ? n4 - 1 - i : i;
    float4* const hp = reinterpret_cast<float4*>(hi) + q;
    float4* const lp = reinterpret_cast<float4*>(lo) + q;
    const bool stay = q < ACC_KEEP4;
    const float4 v = ld_hint(reinterpret_cast<const float4*>(g) + q, policy);
    const float x[4] = {v.x, v.y, v.z, v.w};
    float4 h4 = make_float4(0.f, 0.f, 0.f, 0.f), l4 = h4;
    if (!first) {
      h4 = stay ? *hp : ld_hint(hp, policy);
      l4 = stay ? *lp : ld_hint(lp, policy);
    }
    float hh[4] = {h4.x, h4.y, h4.z, h4.w}, ll[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      CSum c{hh[j], ll[j]};
      csum_add_prod(c, f, x[j]);
      hh[j] = c.hi;
      ll[j] = c.lo;
    }
    h4 = make_float4(hh[0], hh[1], hh[2], hh[3]);
    l4 = make_float4(ll[0], ll[1], ll[2], ll[3]);
    if (stay) {
      *hp = h4;
      *lp = l4;
    } else {
      st_hint(hp, h4, policy);
      st_hint(lp, l4, policy);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x < (int)(D - D4)) {
    const int64_t e = D4 + threadIdx.x;
    CSum c{first ? 0.f : hi[e], first ? 0.f : lo[e]};
    csum_add_prod(c, f, g[e]);
    hi[e] = c.hi;
    lo[e] = c.lo;
  }
}

// The step's dense update from its accumulator (has_sum 0: no message was
// kept, the gradient is 0), four parameters per thread, in the direction that
// meets the accumulators of the last push first.
__global__ void __launch_bounds__(256)
    k_dense_apply_eager(DenseArgs da, const float* __restrict__ hi, const float* __restrict__ lo,
                        int has_sum, int reverse, ErrSink err) {
  if (__syncthreads_or((*(volatile uint32_t*)err.step & (ERR_ID_RANGE | ERR_TIMEOUT)) != 0u)) return;
  const float Mf = (float)da.M;
  const int64_t n4 = da.D / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const bool adam = da.opt.kind == 1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
    const int64_t q = reverse ? n4 - 1 - i : i;
    float4 h4 = make_float4(0.f, 0.f, 0.f, 0.f), l4 = h4, b4 = h4;
    if (has_sum) {
      h4 = __ldcs(reinterpret_cast<const float4*>(hi) + q);
      l4 = __ldcs(reinterpret_cast<const float4*>(lo) + q);
    }
    const float4 w4 = reinterpret_cast<const float4*>(da.w)[q];
    const float4 a4 = reinterpret_cast<const float4*>(da.s0)[q];
    if (adam) b4 = reinterpret_cast<const float4*>(da.s1)[q];
    const float hh[4] = {h4.x, h4.y, h4.z, h4.w}, ll[4] = {l4.x, l4.y, l4.z, l4.w};
    float wv[4] = {w4.x, w4.y, w4.z, w4.w}, a0[4] = {a4.x, a4.y, a4.z, a4.w},
          a1[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      opt_update(da.opt, wv[j], a0[j], a1[j],
                 __fdiv_rn(has_sum ? __fadd_rn(hh[j], ll[j]) : 0.f, Mf));
    reinterpret_cast<float4*>(da.w)[q] = make_float4(wv[0], wv[1], wv[2], wv[3]);
    reinterpret_cast<float4*>(da.s0)[q] = make_float4(a0[0], a0[1], a0[2], a0[3]);
    if (adam) reinterpret_cast<float4*>(da.s1)[q] = make_float4(a1[0], a1[1], a1[2], a1[3]);
  }
  // the last (D mod 4) parameters
  if (blockIdx.x == 0 && threadIdx.x < (int)(da.D - 4 * n4)) {
    const int64_t e = 4 * n4 + threadIdx.x;
    const float v = has_sum ? __fadd_rn(hi[e], lo[e]) : 0.f;
    float w = da.w[e], s0 = da.s0[e], s1 = adam ? da.s1[e] : 0.f;
    opt_update(da.opt, w, s0, s1, __fdiv_rn(v, Mf));
    da.w[e] = w;
    da.s0[e] = s0;
    if (adam) da.s1[e] = s1;
  }
}

}  // namespace

namespace {

template <int STAGES>
constexpr size_t dense_smem() {
  return (size_t)STAGES * DT * sizeof(float) + 2 * STAGES * sizeof(uint64_t);
}

template <int STAGES>
void dense_as(const StepArgs& a, const DenseArgs& da, StepScratch sc, ErrSink err,
              int64_t wait_ns, int num_sms, int64_t n_tiles, cudaStream_t s) {
  constexpr size_t smem = dense_smem<STAGES>();
  static const int bps = [&]() {  // persistent: as many CTAs as fit on an SM, at most three
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_dense_apply<STAGES>, DENSE_THREADS,
                                                      smem) != cudaSuccess ||
        b < 1)
      b = 1;
    return std::min(b, 3);
  }();
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms * bps, n_tiles));
  k_dense_apply<STAGES><<<(unsigned)grid, DENSE_THREADS, smem, s>>>(a, da, sc, err, wait_ns);
}

}  // namespace

cudaError_t configure_dense() {
  const cudaError_t e =
      cudaFuncSetAttribute(k_dense_apply<STAGES_LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)dense_smem<STAGES_LONG>());
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_dense_apply<STAGES_SHORT>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)dense_smem<STAGES_SHORT>());
}

void launch_dense(const StepArgs& a, const DenseArgs& da, StepScratch sc, ErrSink err,
                  int64_t wait_ns, int num_sms, cudaStream_t s) {
  const int64_t n_tiles = ((da.D & ~3ll) + DT - 1) / DT;
  if (n_tiles > num_sms && da.D * 4 * da.M <= DENSE_SHORT)
    dense_as<STAGES_SHORT>(a, da, sc, err, wait_ns, num_sms, n_tiles, s);
  else
    dense_as<STAGES_LONG>(a, da, sc, err, wait_ns, num_sms, n_tiles, s);
}

void launch_dense_accumulate(float* hi, float* lo, const float* g, int64_t D, float f, bool first,
                             bool reverse, int num_sms, cudaStream_t s) {
  int64_t grid = (D / 4 + 255) / 256;
  if (grid > (int64_t)num_sms * 8) grid = (int64_t)num_sms * 8;
  if (grid < 1) grid = 1;
  launch_chained(0, k_dense_accumulate, (unsigned)grid, 256, 0, s, hi, lo, g, D, f, first ? 1 : 0,
                 reverse && D >= ACC_TURN ? 1 : 0);
}

void launch_dense_eager(const DenseArgs& da, const float* hi, const float* lo, bool has_sum,
                        bool reverse, ErrSink err, int num_sms, cudaStream_t s) {
  int64_t grid = (da.D / 4 + 255) / 256;
  if (grid > (int64_t)num_sms * 8) grid = (int64_t)num_sms * 8;
  if (grid < 1) grid = 1;
  k_dense_apply_eager<<<(unsigned)grid, 256, 0, s>>>(da, hi, lo, has_sum ? 1 : 0,
                                                     reverse && da.D >= ACC_TURN ? 1 : 0, err);
}

}  // namespace gba
