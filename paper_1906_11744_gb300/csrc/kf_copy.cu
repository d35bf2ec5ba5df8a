// Copies of whole calls in one launch: the caller's arrays into the context
// with their checks (kf_load_hits, kf_load_seeds) and the results out of it
// (kf_get_*).  A small event's call is bound by its launches: one copy per
// array, a memset, a check and a flag read back took about 2.5 us of host time
// and 2 us on the device each; a large batch's by HBM (16-byte accesses, as the
// copy engine's).
#include <algorithm>

#include "kf_internal.h"

namespace kfg {

namespace {

// Small blocks: 64 threads of these kernels find room beside the register-capped
// finding kernel of another context (its five blocks leave 4 K registers of an
// SM).  The kernel at the compiler's register count, which launches of up to
// 600,000 candidate places take, fills the register file, and a copy then waits
// for one of its blocks: two contexts in turn take 1,098 us per step of five
// PU-200 events (uploads, graph, downloads) where the graph alone takes 997, the
// serial form 1,205; with copies by the driver and a finding kernel of more
// registers it was 1,554, 1,537 and 1,806.
constexpr int COPY_THREADS = 64;
constexpr int COPY_UNROLL = 4;  // 16-byte words in flight per thread

// bytes of src to dst by the threads (tid of nt) of the grid: 16-byte words
// where both are aligned, else 4-byte words or bytes.
__device__ __forceinline__ void copy_bytes(void* dst, const void* src, size_t bytes, size_t tid, size_t nt) {
  const size_t a = (size_t)dst | (size_t)src;
  size_t done = 0;
  if ((a & 15) == 0) {
    const size_t n = bytes >> 4;
    uint4* d = reinterpret_cast<uint4*>(dst);
    const uint4* s = reinterpret_cast<const uint4*>(src);
    size_t i = tid;
    for (; i + (COPY_UNROLL - 1) * nt < n; i += COPY_UNROLL * nt) {
      uint4 v[COPY_UNROLL];
#pragma unroll
      for (int k = 0; k < COPY_UNROLL; ++k) v[k] = s[i + k * nt];
#pragma unroll
      for (int k = 0; k < COPY_UNROLL; ++k) d[i + k * nt] = v[k];
    }
    for (; i < n; i += nt) d[i] = s[i];
    done = n << 4;
  } else if ((a & 3) == 0) {
    const size_t n = bytes >> 2;
    unsigned* d = reinterpret_cast<unsigned*>(dst);
    const unsigned* s = reinterpret_cast<const unsigned*>(src);
    for (size_t i = tid; i < n; i += nt) d[i] = s[i];
    done = n << 2;
  }
  for (size_t i = done + tid; i < bytes; i += nt)
    reinterpret_cast<unsigned char*>(dst)[i] = reinterpret_cast<const unsigned char*>(src)[i];
}

__global__ void __launch_bounds__(COPY_THREADS) k_copy(const __grid_constant__ CopyList c) {
  const size_t tid = blockIdx.x * (size_t)COPY_THREADS + threadIdx.x, nt = (size_t)gridDim.x * COPY_THREADS;
  for (int k = 0; k < c.n; ++k) copy_bytes(c.dst[k], c.src[k], c.bytes[k], tid, nt);
}

__device__ __forceinline__ void write_offsets(const OffsetArg& o, int* dst) {
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < o.n; i += blockDim.x) dst[i] = o.v[i];
}

// The hit arrays, their offsets (o.n > 0) and the check that every layer index
// lies in [0, n_surf) (bad[0] = 1 otherwise; bad: host memory).
__global__ void __launch_bounds__(COPY_THREADS) k_load_hits(const __grid_constant__ CopyList c, const int* layer, int n,
                                                            int n_surf, const __grid_constant__ OffsetArg o,
                                                            int* hit_off, int* bad) {
  const size_t tid = blockIdx.x * (size_t)COPY_THREADS + threadIdx.x, nt = (size_t)gridDim.x * COPY_THREADS;
  write_offsets(o, hit_off);
  for (int k = 0; k < c.n; ++k) copy_bytes(c.dst[k], c.src[k], c.bytes[k], tid, nt);
  bool out = false;
  for (size_t i = tid; i < (size_t)n; i += nt) out = out || layer[i] < 0 || layer[i] >= n_surf;
  if (out) ((volatile int*)bad)[0] = 1;
}

// The seed arrays, their offsets (o.n > 0, else seed_off holds them), the
// event of every seed (binary search over the offsets), its keep flag, and the
// check of its hits: in range of their event (bad[0] = 1 otherwise) and on
// barrel layers (bad[1] = 1).
__global__ void __launch_bounds__(COPY_THREADS) k_load_seeds(const __grid_constant__ CopyList c, const int* sh, int n,
                                                             int n_events, const __grid_constant__ OffsetArg o,
                                                             int* seed_off, const int* hit_off,
                                                             const int* hlayer, int n_layers, int* seed_event,
                                                             unsigned char* keep, int* bad) {
  const size_t tid = blockIdx.x * (size_t)COPY_THREADS + threadIdx.x, nt = (size_t)gridDim.x * COPY_THREADS;
  write_offsets(o, seed_off);
  for (int k = 0; k < c.n; ++k) copy_bytes(c.dst[k], c.src[k], c.bytes[k], tid, nt);
  bool range = false, layer = false;
  for (size_t s = tid; s < (size_t)n; s += nt) {
    int lo = 0, hi = n_events - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if ((o.n > 0 ? o.v[mid] : seed_off[mid]) <= (int)s) lo = mid; else hi = mid - 1;
    }
    seed_event[s] = lo;
    keep[s] = 1;
    const int h0 = hit_off[lo], nh = hit_off[lo + 1] - h0;
    for (int k = 0; k < 3; ++k) {
      const int h = sh[(size_t)k * n + s];
      if (h < 0 || h >= nh) range = true;
      else if (hlayer[h0 + h] >= n_layers) layer = true;
    }
  }
  if (range) ((volatile int*)bad)[0] = 1;
  if (layer) ((volatile int*)bad)[1] = 1;
}

__global__ void __launch_bounds__(COPY_THREADS) k_find_begin(const FindBegin b) {
  const size_t tid = blockIdx.x * (size_t)COPY_THREADS + threadIdx.x, nt = (size_t)gridDim.x * COPY_THREADS;
  for (size_t i = tid; i < (size_t)b.n_counters; i += nt) b.counters[i] = 0ull;
  for (size_t i = tid; i < (size_t)b.n_queue; i += nt) b.queue[i] = 0u;
  for (size_t i = tid; i < b.n_table; i += nt) b.table[i] = 0u;
  for (size_t i = tid; i < (size_t)b.n_keep; i += nt) b.keep[i] = 1;
}

// Blocks for `bytes` of copies: enough 16-byte words in flight to reach the
// copy bandwidth (32 blocks per SM), one word per thread below that.
int copy_grid(size_t bytes, int num_sms) {
  const size_t want = (bytes / 16 + COPY_THREADS - 1) / COPY_THREADS;
  return (int)std::max<size_t>(1, std::min<size_t>(want, (size_t)num_sms * 32));
}
size_t total(const CopyList& c) {
  size_t b = 0;
  for (int k = 0; k < c.n; ++k) b += c.bytes[k];
  return b;
}

}  // namespace

cudaError_t launch_copy(const CopyList& c, int num_sms, cudaStream_t st) {
  if (c.n == 0) return cudaSuccess;
  k_copy<<<copy_grid(total(c), num_sms), COPY_THREADS, 0, st>>>(c);
  return cudaGetLastError();
}

cudaError_t launch_load_hits(const CopyList& c, const int* layer, int n, int n_surf, const OffsetArg& o, int* hit_off,
                             int* bad, int num_sms, cudaStream_t st) {
  if (n <= 0 && o.n <= 0) return cudaSuccess;
  k_load_hits<<<copy_grid((size_t)n * 16, num_sms), COPY_THREADS, 0, st>>>(c, layer, n, n_surf, o, hit_off, bad);
  return cudaGetLastError();
}

cudaError_t launch_load_seeds(const CopyList& c, const int* sh, int n, int n_events, const OffsetArg& o, int* seed_off,
                              const int* hit_off, const int* hlayer, int n_layers, int* seed_event,
                              unsigned char* keep, int* bad, int num_sms, cudaStream_t st) {
  if (n <= 0 && o.n <= 0) return cudaSuccess;
  k_load_seeds<<<copy_grid((size_t)n * 128, num_sms), COPY_THREADS, 0, st>>>(
      c, sh, n, n_events, o, seed_off, hit_off, hlayer, n_layers, seed_event, keep, bad);
  return cudaGetLastError();
}

cudaError_t launch_find_begin(const FindBegin& b, int num_sms, cudaStream_t st) {
  k_find_begin<<<copy_grid(std::max(b.n_table * 4, (size_t)b.n_keep) * 4, num_sms), COPY_THREADS, 0, st>>>(b);
  return cudaGetLastError();
}

}  // namespace kfg
