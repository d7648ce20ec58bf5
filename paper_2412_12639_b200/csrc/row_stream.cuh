// A stretch of one fp32 logits row streamed through shared memory by bulk copies: the loop of the
// kernels that scan [rows, vocab] matrices (top-m, acceptance, non-greedy acceptance) where there is
// more data than fits the registers of the CTAs that run at once.  Internal to the library.
//
// What bounds such a scan is bytes in flight: an SM draws about 45 GB/s with 64 KB outstanding, which
// register loads reach only with most of the register file, and every address, predicate and
// register move of the loads is issued by the warps that should be comparing.  Here one thread of an extra
// warp asks for 32 KB at a time and the eight working warps read 16 bytes per lane from shared memory.
//
// Rows start anywhere (4-byte aligned): the copies cover the whole 16-byte units inside the stretch, and
// the up to three entries before and after them are `edge` entries, for the caller to read.
#pragma once

#include "tc_util.cuh"

namespace falcon {

constexpr int kStreamWarps = 8;
constexpr int kStreamThreads = 32 * kStreamWarps;           // working threads; one more warp issues the copies
constexpr int kStreamLane = 32;                             // entries a lane takes per stage
constexpr int kStreamStage = kStreamThreads * kStreamLane;  // 8192 entries, 32 KB
constexpr int kStreamStages = 2;
constexpr uint32_t kStreamBytes = kStreamStages * kStreamStage * 4;
constexpr uint32_t kStreamBytesPair = 78u * 1024u;      // more than a third of an SM's shared memory: two CTAs per SM
constexpr uint32_t kStreamBytesMax = kStreamBytesPair;  // (the attribute the kernels are given once)

// The kernels that scan rows in clusters: places in falcon_ctx::scan_resident.
enum ScanKernel { kScanTopm8, kScanTopm16, kScanTopm32, kScanTopmStream, kScanSample };

// Clusters of `of` CTAs of a kernel that the GPU holds at once (asked once per context; 0 where it cannot say).
inline int clusters_at_once(falcon_ctx* ctx, ScanKernel which, const void* kernel, int threads, uint32_t smem, int of) {
  int& n = ctx->scan_resident[which][of == 1 ? 0 : of == 2 ? 1 : of == 4 ? 2 : 3];
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(of, ctx->sm_count);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = of;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int got = 0;
    if (cudaOccupancyMaxActiveClusters(&got, kernel, &cfg) != cudaSuccess) cudaGetLastError();
    n = got > 0 ? got : -1;
  }
  return n > 0 ? n : 0;
}

// Whether n clusters of `of` CTAs, of which at_once fit, are placed without some of them waiting for others.  Behind an attention
// launch, whose SMs become free one by one, clusters of four and eight need a few places more than they take (us with
// clusters of four, alone and behind one; 104 fit: top-m, 64000 entries, 100 rows 11.3 / 23.9, 101 11.4 / 24.5, 102 11.5 / 25.1, 103 11.7 / 26.6, 105
// 15.0 / 28.0, against 11.9 / 24.1 with clusters of two all along; sample, 32000, 100 rows 9.1 / 21.8, 102 9.1 / 23.0, 105 11.3 / 24.4,
// against 9.3 / 21.9.  Clusters of eight, 48 fit: top-m, 65536, 45 rows 8.2 / 20.9, 46 8.3 / 21.7, 48 9.2 / 24.3, 49 11.9 / 24.9, against 8.2 / 21.3
// with four; sample, 64000, 45 rows 9.2 / 21.9, 46 9.2 / 22.5, 48 9.3 / 24.4, 49 12.1 / 25.0, against 9.6 / 22.5).  Clusters of two fill all
// their 222 places: top-m, 32000, 222 rows 12.0 / 24.3, 223 15.4 / 28.0; sample 12.1 / 24.6, 224 rows 14.3 / 26.8.
inline bool cluster_room(int64_t n, int of, int at_once) {
  return of <= 2 ? n <= at_once : of == 4 ? 26 * n <= 25 * static_cast<int64_t>(at_once) : 16 * n <= 15 * static_cast<int64_t>(at_once);
}

// Dynamic shared memory of a launch of n CTAs in clusters of `of` that take `len` entries each: so much that an SM takes two
// of them at most, where that is enough places.  Behind a kernel whose CTAs end at different times the SMs that become free first
// would be given three each and the last ones none.  Not one per SM, although a launch of no more CTAs than SMs is faster still
// on one stream: a CTA that waits for its turn keeps an SM from the attention launches of other streams, and with one CTA per SM two
// streams that decide at the same time share none.  us with three / two / one per SM allowed: behind an attention launch over four
// sequences on one stream, the same on two streams at once, and two streams with the scans alone:
//   top-m       120 rows of 32000   41.3 / 39.8 / 38.6   55.6 / 56.5 / 60.3   11.6 / 10.7 / 12.1
//               140 of 50000        45.7 / 43.6 / 41.9   60.6 / 60.8 / 64.2   15.5 / 14.2 / 18.1
//   acceptance  100 of 12000        35.5 / 35.0 / 35.0   47.4 / 49.7 / 54.0    6.7 /  6.7 /  6.6
//               148 of 28000        37.8 / 37.3 / 37.4   53.5 / 54.5 / 60.9   10.3 /  9.8 / 11.8
//   sample      148 of 40000        42.8 / 41.5 / 41.0   58.3 / 58.9 / 63.7   14.3 / 13.7 / 17.5
// One stream's scans alone are the same with three and with two.  Not for more than one and a half rows' length of work on some SMs
// and half of it on others (170 rows of 128256 from L2: 13 us with three per SM allowed, 18 with two), nor where clusters might not
// all find their places (sample, 140 rows of 128256 in clusters of two 18.8 and 20.8; top-m behind attention, 60 rows of
// 64000 in clusters of four 7 % slower).
inline uint32_t stream_bytes(int64_t n_ctas, int of, int len, int sm_count) {
  if (of > 2) return kStreamBytes;
  const int64_t slots = of == 2 ? sm_count * 9 / 10 : sm_count;
  const bool even = n_ctas <= slots || (n_ctas <= 2 * slots && (2 * n_ctas > 3 * sm_count || len <= 10 * kStreamStage));
  return even ? kStreamBytesPair : kStreamBytes;
}

struct StreamBars {
  uint64_t full[kStreamStages], empty[kStreamStages];
  int abort;
};

struct RowStream {
  const float* base;  // first entry of the 16-byte aligned part
  int head, body, tail;  // entries before it, in it (a multiple of 4), after it
  uint32_t buf, bars;    // shared-memory addresses
  volatile int* abort;

  __device__ __forceinline__ int stages() const { return (body + kStreamStage - 1) / kStreamStage; }
  // Entries [0, n) of `row`.  Threads 0 .. of any warp call this; one thread calls init().
  __device__ __forceinline__ RowStream(const float* row, int n, void* smem, StreamBars* b) {
    const int mis = static_cast<int>((4 - ((reinterpret_cast<uintptr_t>(row) >> 2) & 3)) & 3);
    head = min(n, mis);
    body = (n - head) & ~3;
    tail = n - head - body;
    base = row + head;
    buf = tc::smem_u32(smem);
    bars = tc::smem_u32(b);
    abort = &b->abort;
  }
  __device__ __forceinline__ static void init(StreamBars* b) {
    for (int i = 0; i < kStreamStages; ++i) {
      tc::mbar_init(tc::smem_u32(&b->full[i]), 1);
      tc::mbar_init(tc::smem_u32(&b->empty[i]), kStreamWarps);
    }
    b->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // The copying thread: stages [i0, i1), in order, without stage `stall` (a test hook: the waits for that one run out).
  __device__ __forceinline__ void produce(int i0, int i1, int stall) const {
    for (int i = i0; i < i1; ++i) {
      const int st = i % kStreamStages;
      const uint32_t full = bars + 8u * st;
      if (i >= kStreamStages && !tc::mbar_wait(bars + 8u * (kStreamStages + st), (i / kStreamStages - 1) & 1, abort)) {
        for (int k = i - kStreamStages; k < i; ++k)
          if (k != stall) tc::mbar_wait_drain(bars + 8u * (k % kStreamStages), (k / kStreamStages) & 1);
        return;
      }
      if (i == stall) continue;
      const uint32_t bytes = static_cast<uint32_t>(min(kStreamStage, body - i * kStreamStage)) * 4u;
      tc::mbar_expect_tx(full, bytes);
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(buf + st * kStreamStage * 4u),
                   "l"(base + static_cast<int64_t>(i) * kStreamStage), "r"(bytes), "r"(full)
                   : "memory");
    }
    // (until the last copies have landed: none may be in flight when the CTA leaves, whatever became of its waits)
    if (i1 == stages())
      for (int k = max(0, i1 - kStreamStages); k < i1; ++k)
        if (k != stall) tc::mbar_wait_drain(bars + 8u * (k % kStreamStages), (k / kStreamStages) & 1);
  }
  // Entry e (0 .. 3) of the lane's j-th 16-byte piece of stage i, counted from `base`.
  __device__ __forceinline__ int index(int i, int j, int e) const {
    return i * kStreamStage + (((threadIdx.x >> 5) * (kStreamLane / 4) + j) * 32 + (threadIdx.x & 31)) * 4 + e;
  }
  // The lane's 32 entries of stage i into registers (beyond the end: -inf).  False when the wait gave up.
  __device__ __forceinline__ bool take(int i, float (&x)[kStreamLane]) const {
    const int st = i % kStreamStages;
    if (!tc::mbar_wait_warp(bars + 8u * st, (i / kStreamStages) & 1, abort)) return false;
    const uint32_t at = buf + st * kStreamStage * 4u + (((threadIdx.x >> 5) * (kStreamLane / 4)) * 32 + (threadIdx.x & 31)) * 16u;
#pragma unroll
    for (int j = 0; j < kStreamLane / 4; ++j)
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[4 * j]), "=f"(x[4 * j + 1]), "=f"(x[4 * j + 2]), "=f"(x[4 * j + 3]) : "r"(at + j * 512) : "memory");
    if (body - i * kStreamStage < kStreamStage) {
#pragma unroll
      for (int j = 0; j < kStreamLane / 4; ++j)
        if (index(i, j, 0) >= body) x[4 * j] = x[4 * j + 1] = x[4 * j + 2] = x[4 * j + 3] = -INFINITY;
    }
    return true;
  }
  // Which of them exist, and one of them (k = 4 j + e) again, until the stage is handed back.
  __device__ __forceinline__ uint32_t live(int i) const {
    const int pieces = min(kStreamStage, body - i * kStreamStage) >> 2, mine = (threadIdx.x >> 5) * (kStreamLane / 4) * 32 + (threadIdx.x & 31);
    const int nj = max(0, min(kStreamLane / 4, (pieces - mine + 31) >> 5));
    return nj >= 8 ? 0xffffffffu : (1u << (4 * nj)) - 1u;
  }
  __device__ __forceinline__ float value(int i, int k) const {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(buf + (i % kStreamStages) * kStreamStage * 4u + (index(i, k >> 2, k & 3) - i * kStreamStage) * 4u));
    return v;
  }
  __device__ __forceinline__ void give_back(int i) const {
    __syncwarp();
    if ((threadIdx.x & 31) == 0) tc::mbar_arrive(bars + 8u * (kStreamStages + i % kStreamStages));
  }
};

}  // namespace falcon
