// History convolution without device allocation: the sums of
// sbiem_history_sums (Sec. 3.1 window, Sec. 3.3 step (2), midpoint weights)
// on caller-owned device buffers.  It runs the library's warp-per-chunk
// kernel (k_history_t: chunks handed out by an atomic counter, a mode's
// chunk sums added in chunk order by the warp that finishes last), not the
// handle's bulk-async sweep, whose static partition and per-mode finish
// need tables sized per fault.  Its scratch -- chunk table, per-chunk
// partial sums, per-mode counters -- is one fixed static device array
// instead of memory allocated by the library.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#include "kernels.cuh"
#include "sbiem.h"

using namespace sbiem;

namespace {

constexpr int kMaxModes = SBIEM_NOALLOC_MAX_MODES;
constexpr int kMaxChunks = SBIEM_NOALLOC_MAX_CHUNKS;
constexpr int kChunkSlots = 2048;
constexpr int kMaxDevices = 64;

// Layout of the scratch array (byte offsets, each 256-byte aligned).
constexpr size_t align256(size_t b) { return (b + 255) / 256 * 256; }
constexpr size_t kOffHeader = 0;                                    // Header
constexpr size_t kOffChunks = 256;                                  // Chunk[kMaxChunks]
constexpr size_t kOffPartial = kOffChunks + align256(sizeof(Chunk) * kMaxChunks);   // double4[kMaxChunks]
constexpr size_t kOffCounter = kOffPartial + align256(sizeof(double4) * kMaxChunks);  // int[kMaxModes]
constexpr size_t kScratchBytes = kOffCounter + align256(sizeof(int) * kMaxModes);

struct Header {
  int nchunks;
  int overflow;
  int work;
  unsigned status;
};

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

unsigned char* g_addr[kMaxDevices];  // device address of g_scratch, per device

// Inclusive prefix sum over a warp.
__device__ __forceinline__ int warp_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

__device__ __forceinline__ int chunks_of(int32_t r) { return r > 0 ? (r - 1) / kChunkSlots + 1 : 0; }

// Chunk table, mode counters and zeroed sums.  CTA b takes the modes [b T, (b
// + 1) T), one per thread: it counts the chunks of the modes before and after
// them (at most 32 coalesced reads a thread, cheaper than a pass over partial
// counts), scans its own and writes them.  Every CTA thus knows the total; past
// the table it writes nothing and the call is refused.  (One CTA with a serial
// scan took 87 us at 16385 modes, this 6 us.)
constexpr int kChunkThreads = 1024;
__global__ void __launch_bounds__(kChunkThreads)
    k_noalloc_chunks(const int32_t* __restrict__ R, int nmodes, unsigned char* scratch, double* __restrict__ AT,
                     double* __restrict__ AN) {
  Header* hd = reinterpret_cast<Header*>(scratch + kOffHeader);
  Chunk* chunks = reinterpret_cast<Chunk*>(scratch + kOffChunks);
  int* counter = reinterpret_cast<int*>(scratch + kOffCounter);
  __shared__ long long s_before[kChunkThreads / 32], s_after[kChunkThreads / 32], s_own[kChunkThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int n0 = blockIdx.x * kChunkThreads, n = n0 + tid;
  const int r = n < nmodes ? R[n] : 0;
  const int k = chunks_of(r);
  long long before = 0, after = 0;
  for (int q = tid; q < n0; q += kChunkThreads) before += chunks_of(R[q]);
  for (int q = n + kChunkThreads; q < nmodes; q += kChunkThreads) after += chunks_of(R[q]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    before += __shfl_xor_sync(0xffffffffu, before, o);
    after += __shfl_xor_sync(0xffffffffu, after, o);
  }
  const int scan = warp_scan(k);
  if (lane == 0) {
    s_before[wid] = before;
    s_after[wid] = after;
  }
  if (lane == 31) s_own[wid] = scan;
  __syncthreads();
  long long c = scan - k, total = 0;
  for (int w = 0; w < kChunkThreads / 32; ++w) {
    c += s_before[w] + (w < wid ? s_own[w] : 0);
    total += s_before[w] + s_own[w] + s_after[w];
  }
  const bool fits = total <= kMaxChunks;
  if (blockIdx.x == 0 && tid == 0) {
    hd->nchunks = fits ? static_cast<int>(total) : 0;
    hd->overflow = fits ? 0 : 1;
    hd->work = 0;
    hd->status = 0u;
  }
  if (!fits || n >= nmodes) return;
  counter[n] = 0;
  // modes without history keep these zeros; 8 bytes a store, which is all the
  // alignment that a caller's double* has
  for (double* a : {AT + 2 * n, AN + 2 * n}) a[0] = a[1] = 0.0;
  const int64_t first = c;
  for (int q = 0; q < k; ++q, ++c) {
    Chunk ch;
    ch.mode = n;
    ch.first = static_cast<int32_t>(first);
    ch.count = k;
    ch.pad = 0;
    ch.i0 = static_cast<int64_t>(q) * kChunkSlots;
    ch.i1 = min(static_cast<int64_t>(q + 1) * kChunkSlots, static_cast<int64_t>(r));
    chunks[c] = ch;
  }
}

int setup(unsigned char** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SBIEM_ERR_CUDA;
  if (!g_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) return SBIEM_ERR_CUDA;
    g_addr[dev] = static_cast<unsigned char*>(p);
  }
  *out = g_addr[dev];
  return SBIEM_OK;
}

template <class R>
int run(int nmodes, int m, const void* ring, const void* weights, const int64_t* ring_off,
        const int64_t* w_off, const int32_t* Rn, const int32_t* Mn, const int32_t* head, double* AT,
        double* AN, cudaStream_t st) {
  unsigned char* scr = nullptr;
  int rc = setup(&scr);
  if (rc) return rc;
  k_noalloc_chunks<<<(nmodes + kChunkThreads - 1) / kChunkThreads, kChunkThreads, 0, st>>>(
      Rn, nmodes, scr, AT, AN);
  if (cudaGetLastError() != cudaSuccess) return SBIEM_ERR_CUDA;
  Header hd;
  if (cudaMemcpyAsync(&hd, scr + kOffHeader, sizeof(hd), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return SBIEM_ERR_CUDA;
  if (hd.overflow) return SBIEM_ERR_INVALID;
  DevFault<R> f{};
  f.nmodes = nmodes;
  f.ring = static_cast<Slot<R>*>(const_cast<void*>(ring));
  f.w = static_cast<W2<R>*>(const_cast<void*>(weights));
  f.ring_off = ring_off;
  f.w_off = w_off;
  f.Rn = Rn;
  f.Mn = Mn;
  f.head = const_cast<int32_t*>(head);
  f.AT = reinterpret_cast<double2*>(AT);
  f.AN = reinterpret_cast<double2*>(AN);
  Header* dh = reinterpret_cast<Header*>(scr + kOffHeader);
  f.chunks = reinterpret_cast<const Chunk*>(scr + kOffChunks);
  f.partial = reinterpret_cast<double4*>(scr + kOffPartial);
  f.counter = reinterpret_cast<int*>(scr + kOffCounter);
  f.work = &dh->work;
  f.status = &dh->status;
  f.nchunks = hd.nchunks;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int per_sm = history_blocks_per_sm<R>();
  launch_history_atomic<R>(f, m, sms * (per_sm > 0 ? per_sm : 1), st);
  return cudaGetLastError() == cudaSuccess ? SBIEM_OK : SBIEM_ERR_CUDA;
}

}  // namespace

extern "C" int sbiem_history_sums_noalloc(int64_t nmodes, int32_t precision, int64_t m, const void* ring,
                                          const void* weights, const int64_t* ring_off, const int64_t* w_off,
                                          const int32_t* R, const int32_t* M, const int32_t* head, double* AT,
                                          double* AN, void* stream) {
  if (nmodes < 1 || nmodes > kMaxModes || m < 1 || m > (int64_t(1) << 30) ||
      (precision != 0 && precision != 1) || !ring || !weights || !ring_off || !w_off || !R || !M || !head ||
      !AT || !AN)
    return SBIEM_ERR_INVALID;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (precision == 1)
    return run<float>(static_cast<int>(nmodes), static_cast<int>(m), ring, weights, ring_off, w_off, R, M, head,
                      AT, AN, st);
  return run<double>(static_cast<int>(nmodes), static_cast<int>(m), ring, weights, ring_off, w_off, R, M, head,
                     AT, AN, st);
}
