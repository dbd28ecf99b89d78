// Stand-ins for the kernel launchers (see fake_runtime.cpp): they run nothing, but
// check that the buffers they are given are live and large enough (fake_bad counts
// those that are not); the copies of a push are made.
#include <cstring>

#include "gba_internal.cuh"

extern "C" void fake_need(const void* p, size_t bytes);
extern "C" cudaError_t fake_copy_launch();

namespace gba {

SortPlan make_sort_plan(int, int) {
  SortPlan p{};
  p.passes = 2;
  p.radix = 256;
  return p;
}
size_t sort_status_words(int64_t N, int radix) { return (size_t)(N / SORT_TILE_KEYS + 1) * radix; }
int64_t scan_tiles(int64_t N) { return (N + SCAN_TILE - 1) / SCAN_TILE; }
int64_t long_items(int64_t n, int) { return n / 32 + 1; }
int64_t long_parts(int64_t n, int, int) { return n / 16 + 1; }
cudaError_t configure_dense() { return cudaSuccess; }
int kernel_binary_version() { return -1; }

void launch_weights(const StepArgs&, StepScratch, DevStats*, int, const void*, void* dev_meta, size_t n,
                    cudaStream_t) {
  if (n) fake_need(dev_meta, n);
}
void launch_sort_histogram(const StepArgs& a, const SortPlan&, uint32_t*, uint32_t* keys0, ErrSink, int,
                           cudaStream_t) {
  fake_need(keys0, (size_t)a.N * 4);
  for (int t = 0; t < a.T; ++t)  // the tables as the kernel would find them
    if (a.tinfo[t].id_mode == 2) {
      const HashInfo& h = a.hinfo[t];
      fake_need(h.w, (size_t)a.tinfo[t].V * h.d * 4);
      fake_need(h.keys, (size_t)(h.mask + 1) * 8);
    }
}
void launch_onesweep(const SortPlan& plan, int, SortPass sp, ErrSink, int64_t, cudaStream_t) {
  for (const uint32_t* p : {sp.keys_in, (const uint32_t*)sp.keys_out, (const uint32_t*)sp.vals_out})
    fake_need(p, (size_t)sp.N * 4);
  fake_need(sp.status, sort_status_words(sp.N, plan.radix) * 8);
}
void launch_seg_scan(const StepArgs& a, const SegTable&, const SegTable*, const SegOut& so,
                     const uint32_t* keys, const uint32_t* vals, DevStats*, ErrSink, int64_t, cudaStream_t) {
  fake_need(keys, (size_t)a.N * 4);
  fake_need(vals, (size_t)a.N * 4);
  fake_need(so.rr, (size_t)(a.N + 1) * sizeof(uint4));
  fake_need(so.kl, (size_t)a.N * 8);
  if (a.decay) fake_need(so.kw, (size_t)a.N * 4);
  fake_need(so.status, (size_t)scan_tiles(a.N) * 32);
}
void launch_row_apply(const StepArgs&, const RowRange& r, const SegTable*, const SegOut& so, DevStats*,
                      ErrSink, int, cudaStream_t) {
  const size_t rows = (size_t)r.n / (LONG_ROW + 1) + 1;
  fake_need(so.long_rows, rows * sizeof(uint4));
  fake_need(so.long_done, rows * 4);
  fake_need(so.small_rows, rows * sizeof(uint4));
  fake_need(so.items, (size_t)long_items(r.n, 152) * sizeof(uint2));
}
void launch_row_long(const StepArgs&, const RowRange& r, const SegTable*, const SegOut& so, DevStats*,
                     ErrSink, int, cudaStream_t) {
  const size_t floats = (size_t)long_parts(r.n, r.first.d, 152) * r.first.d;
  fake_need(so.part_hi, floats * 4);
  fake_need(so.part_lo, floats * 4);
  fake_need(r.first.w, (size_t)r.first.rows * r.first.d * 4);
  fake_need(r.first.s0, (size_t)r.first.rows * r.first.d * 4);
  fake_need(r.first.ver, (size_t)r.first.rows * 4);
}
void launch_dense(const StepArgs&, const DenseArgs&, StepScratch, ErrSink, int64_t, int, cudaStream_t) {}
cudaError_t launch_push_copy(CopyList cl, unsigned, cudaStream_t) {
  const cudaError_t e = fake_copy_launch();
  if (e != cudaSuccess) return e;
  for (int i = 0; i < cl.n; ++i) {
    fake_need(cl.dst[i], cl.bytes[i]);
    memcpy(cl.dst[i], cl.src[i], cl.bytes[i]);
  }
  return cudaSuccess;
}
void launch_dense_accumulate(float* hi, float*, const float*, int64_t D, float, bool, bool, int,
                             cudaStream_t) {
  fake_need(hi, (size_t)D * 4);
}
void launch_dense_eager(const DenseArgs&, const float*, const float*, bool, bool, ErrSink, int,
                        cudaStream_t) {}
void launch_init_table(float*, float*, float*, int32_t*, int64_t, int32_t, int32_t, float, uint64_t,
                       uint64_t, cudaStream_t) {}
void launch_init_dense(float*, float*, float*, int64_t, int32_t, float, uint64_t, uint64_t,
                       cudaStream_t) {}
int launch_wait_selftest(int64_t, cudaStream_t, uint32_t*, uint32_t*) { return -1; }
void launch_pull_rows(const float*, int64_t, int, int, uint64_t, const HashInfo*, const int64_t*, int64_t,
                      float*, ErrSink, int, cudaStream_t) {}
void launch_hash_clear(unsigned long long* keys, uint64_t slots, cudaStream_t) {
  fake_need(keys, (size_t)slots * 8);
}
void launch_hash_rehash(HashInfo from, HashInfo to, cudaStream_t) {
  for (const HashInfo* h : {&from, &to}) {
    const size_t n = (size_t)(h->mask + 1);
    fake_need(h->w, n * h->d * 4);
    fake_need(h->s0, n * h->d * 4);
    if (h->kind == 1) fake_need(h->s1, n * h->d * 4);
    fake_need(h->ver, n * 4);
    fake_need(h->keys, n * 8);
  }
}
void launch_hash_lookup(const HashInfo*, const int64_t*, int64_t, int64_t*, cudaStream_t) {}

}  // namespace gba
