// The copies of one pushed message (ids and gradient rows of every table, the
// dense gradient) in one launch.
//
// A copying push used to enqueue a memcpy per array, 2 T + 1 of them: on small
// messages the host's cost per call and the copy engine's start-up were the
// whole time (24 messages of three tables, device buffers: 168 copies, 2.5 us
// each on the GPU and 3.4 us each on the host).  Blocks of 256 threads take
// 16 KB each of the concatenated arrays; a block moves its piece with the
// widest loads that the two addresses allow.
// Pinned host memory is read through the link by at most HOST_BLOCKS blocks,
// which fill it (209 GB/s, as the copy engine does in one large copy) and leave the
// SMs to others: 16 messages of 7.6 MB 819 -> 741 us a step against a copy per array.
#include "gba_internal.cuh"

namespace gba {

namespace {

constexpr int COPY_THREADS = 256;
constexpr uint32_t COPY_CHUNK = 16384;  // bytes per block

template <typename W>
__device__ __forceinline__ void copy_piece(const char* src, char* dst, uint32_t bytes) {
  const uint32_t n = bytes / (uint32_t)sizeof(W);
  const W* s = reinterpret_cast<const W*>(src);
  W* d = reinterpret_cast<W*>(dst);
  uint32_t i = threadIdx.x;
  for (; i + 3 * COPY_THREADS < n; i += 4 * COPY_THREADS) {
    const W a = s[i], b = s[i + COPY_THREADS], c = s[i + 2 * COPY_THREADS],
            e = s[i + 3 * COPY_THREADS];
    d[i] = a;
    d[i + COPY_THREADS] = b;
    d[i + 2 * COPY_THREADS] = c;
    d[i + 3 * COPY_THREADS] = e;
  }
  for (; i < n; i += COPY_THREADS) d[i] = s[i];
  const uint32_t done = n * (uint32_t)sizeof(W);
  if (done + threadIdx.x < bytes) dst[done + threadIdx.x] = src[done + threadIdx.x];
}

// LOOP: fewer blocks than chunks, which they take in turn.
template <bool LOOP>
__global__ void __launch_bounds__(COPY_THREADS) k_push_copy(const __grid_constant__ CopyList cl) {
  chain_wait();
  int k = 0;
  for (uint32_t c = blockIdx.x; c < cl.chunks; c += gridDim.x) {
    while (k + 1 < cl.n && c >= cl.first[k + 1]) ++k;
    const uint64_t at = (uint64_t)(c - cl.first[k]) * COPY_CHUNK;
    const uint64_t left = cl.bytes[k] - at;
    const uint32_t bytes = left < COPY_CHUNK ? (uint32_t)left : COPY_CHUNK;
    const char* src = static_cast<const char*>(cl.src[k]) + at;
    char* dst = static_cast<char*>(cl.dst[k]) + at;
    const uint32_t a = (uint32_t)((uintptr_t)src | (uintptr_t)dst);
    if ((a & 15u) == 0u)
      copy_piece<uint4>(src, dst, bytes);
    else if ((a & 7u) == 0u)
      copy_piece<uint2>(src, dst, bytes);
    else if ((a & 3u) == 0u)
      copy_piece<uint32_t>(src, dst, bytes);
    else
      copy_piece<uint8_t>(src, dst, bytes);
    if (!LOOP) break;
  }
}

}  // namespace

cudaError_t launch_push_copy(CopyList cl, unsigned max_blocks, cudaStream_t s) {
  uint64_t blocks = 0;
  for (int k = 0; k < cl.n; ++k) {
    cl.first[k] = (uint32_t)blocks;
    blocks += (cl.bytes[k] + COPY_CHUNK - 1) / COPY_CHUNK;
  }
  if (blocks == 0) return cudaSuccess;
  cl.chunks = (uint32_t)blocks;
  // the launch's own status, not the thread's last error, which may be another's
  if (blocks <= max_blocks)
    return launch_chained(0, k_push_copy<false>, (unsigned)blocks, COPY_THREADS, 0, s, cl);
  return launch_chained(0, k_push_copy<true>, max_blocks, COPY_THREADS, 0, s, cl);
}

}  // namespace gba
