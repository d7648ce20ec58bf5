// falcon_lm_head_argmax: the greedy token of every tree node straight from the LM head
// (Section 3.1: the LM head turns the aggregated features into the distribution over the
// vocabulary; Eq. 6: p = Softmax(LM(f)); temperature 0, Section 4.1, needs only the position of the
// largest logit).  logit[i, v] = sum_k feat[i, k] * head[v, k] is a dense bf16 contraction whose
// [N, V] fp32 result is never written: the argmax is taken where the accumulator is read.
//
// Up to 128 nodes: the head (V x hidden bf16, 262 MB at 32000 x 4096) is read once and dominates: the kernel is
// bound by HBM, the tensor core is about a third busy.  Every CTA owns a run of vocabulary rows
// (V split evenly over the SMs, in steps of 16, so one launch is one wave) and streams it through a
// TMA ring in chunks of 64 hidden columns together with the matching chunk of the features (L2
// hits after the first CTA).  tcgen05.mma with the nodes on the M side and the CTA's vocabulary rows on the N
// side (up to 256 per instruction) accumulates in TMEM; eight warps then read the accumulators, a thread half a row
// (= half of a node's columns), 32 columns at a time, and keep the first maximum.  A CTA's result for a node
// is one 64-bit atomicMax on a word ordered by (logit, then lower index), so ties go to the lowest
// index whatever the timing; the last CTA to arrive unpacks the words.
//
// More nodes: pairs of CTAs (kPair, cta_group::2): a pair's MMA of 256 rows x up to 256 columns takes half of each operand
// from either CTA's shared memory.  Two arrangements; all of TMEM holds accumulators in both:
//   kLmPair    nodes on the lanes: two node tiles of 256 (up to 512 nodes read the head once) or, up to 256 nodes, two
//              vocabulary tiles (the features are read once for both);
//   kLmLanes   vocabulary rows on the lanes, 256 a pair: up to 256 nodes and two such blocks, or up to 512 nodes in two tiles.
//              The nodes then come in steps of 16 where kLmPair pads them to 256; the launcher says when it is taken.
// What bounds them is the power limit (512 nodes of 5120 x 32000 run at 1.3 PFLOP/s, 1.5 GHz, padding counted; a cuBLAS loop
// holds 1.38), then the round trip of the ring: two stages of up to 96 KB, about 4900 cycles between a stage's MMAs and the
// next ones, 3600 of which are the MMAs'.  32000 x 5120, single CTAs and pairs: 512 nodes 157 -> 130 us, 300 nodes 147 -> 113,
// 256 nodes 78 -> 72.
//
// Warp roles: 0 = TMA producer (one thread), 1 = MMA issuer (one elected thread) and TMEM owner,
// 2-9 = accumulator readers; of a pair, the first CTA's warp 1 issues for both, and each CTA loads its own halves.
// Every wait is bounded; a wait that gives up sets FALCON_DEV_TIMEOUT in the caller's status word and the kernel still leaves in order (loads drained, MMAs finished,
// TMEM freed).

#include <climits>

#include "tc_util.cuh"

namespace falcon {
namespace {
using namespace tc;

constexpr int kLmReaders = 256;
constexpr int kLmThreads = 64 + kLmReaders;
constexpr int kLmKC = 64;             // hidden columns per ring stage: one 128-byte swizzle row of bf16
constexpr int kLmMaxStages = 8;
constexpr int kLmTileMax = 256;       // vocabulary rows per MMA (the N side) at most
constexpr uint32_t kLmSmemMax = 232448;
constexpr uint32_t kLmFeatPad = 64u * kLmKC * 2u;    // see f_rows: what a 64-row feature tile leaves for the MMA to read past

enum LmBar {
  kLmBarFull = 0,                            // [kLmMaxStages] a stage's tiles have landed
  kLmBarEmpty = kLmBarFull + kLmMaxStages,   // [kLmMaxStages] the MMAs that read a stage have finished
  kLmBarAccFull = kLmBarEmpty + kLmMaxStages,
  kLmBarAccEmpty,
  kLmBarDone,
  kLmNumBars
};
constexpr uint32_t kLmResultBytes = 2u * 4u * 256u * 8u;  // (kLmLanes) every reader warp's best for its columns' nodes
constexpr uint32_t kLmSmallBytes = kLmFeatPad + 8u * kLmNumBars + 16u;  // pad, barriers, TMEM base, abort flag, last-CTA flag

struct LmParams {
  int32_t n_rows, vocab;
  int32_t n_kc;       // 64-column chunks of the hidden dimension = ceil(hidden / 64)
  int32_t kch;        // chunks per ring stage
  int32_t f_rows;     // rows of a feature tile as loaded: 128, or with a single tile the number of nodes rounded up
                      // to 8 (64 at least); the MMA still reads 128 rows, and what follows the tile gives
                      // accumulator rows that nobody looks at
  int32_t n_mt;       // node tiles: of 128 rows, of a pair's 256
  int32_t m_res;      // node tiles resident in TMEM at once (1; a pair: 1 or 2)
  int32_t v_res;      // vocabulary tiles resident at once (1; a pair with one node tile: 2)
  int32_t tile_n;     // vocabulary rows per MMA (multiple of 16)
  int32_t span;       // vocabulary rows per CTA or pair (multiple of 16)
  int32_t n_stages;
  int32_t stall_first;  // test hook: the features of ring stage 0 are never requested (a bounded wait then runs out)
  uint32_t stage_bytes, idesc;
  int32_t* argmax_out;
  float* max_out;
  int32_t* status;
  unsigned long long* best;  // [n_rows] the nodes' best (logit, index) so far as one orderable word; zero between calls
  int* ticket;               // zero between calls
};

// (logit, index) as one word whose unsigned order is "larger logit first, then the lower index"; 0 = nothing.
__device__ __forceinline__ unsigned long long lm_pack(float x, int idx) {
  const uint32_t b = __float_as_uint(x + 0.f);  // -0 -> +0
  const uint32_t key = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return (static_cast<unsigned long long>(key) << 32) | static_cast<uint32_t>(~idx);
}
__device__ __forceinline__ float lm_unpack_val(unsigned long long w) {
  const uint32_t k = static_cast<uint32_t>(w >> 32);
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ bool lm_wait_drain(uint32_t bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 20); ++it) {
    uint32_t ok;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    if (ok) return true;
  }
  return false;
}

// The pair's forms of what tc_util.cuh has for one CTA.  A load may signal the other CTA's barrier (`bar`: a
// shared::cluster address); a commit arrives at the same barrier of both CTAs.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5, %5, %5}], "
      "[%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(0)
      : "memory");
}
__device__ __forceinline__ void umma_pair_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_pair_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"(static_cast<uint16_t>(3))
               : "memory");
}
__device__ __forceinline__ uint32_t map_to_leader(uint32_t addr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
  return r;
}
__device__ __forceinline__ void arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// The arrangements: one CTA, nodes on the lanes; pairs of CTAs, nodes on the lanes; pairs, vocabulary rows on the lanes.
constexpr int kLmSingle = 0, kLmPair = 1, kLmLanes = 2;

template <int kMode>
__global__ void __launch_bounds__(kLmThreads, 1)
lm_head_argmax_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_f, const LmParams p) {
  constexpr bool kPair = kMode != kLmSingle;
  extern __shared__ __align__(1024) unsigned char smem_gen[];
  const uint32_t smem_base = smem_u32(smem_gen);
  unsigned char* small = smem_gen + static_cast<uint32_t>(p.n_stages) * p.stage_bytes + kLmFeatPad;
  const uint32_t bars = smem_u32(small);
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(small + 8 * kLmNumBars);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(small + 8 * kLmNumBars + 4);
  volatile int* s_last = reinterpret_cast<volatile int*>(small + 8 * kLmNumBars + 8);
  auto bar = [&](int i) { return bars + 8u * static_cast<uint32_t>(i); };

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int n_cta = gridDim.x;
  const int rank = kPair ? blockIdx.x & 1 : 0, cta = kPair ? blockIdx.x >> 1 : blockIdx.x;  // place in the pair; pair or CTA
  const bool leader = rank == 0;
  const int S = p.n_stages;
  const int v_lo = cta * p.span, v_hi = min(p.vocab, v_lo + p.span);
  const int n_vt = (v_hi - v_lo + p.tile_n - 1) / p.tile_n;  // >= 1 by construction of the grid
  const int m_res = kPair ? p.m_res : 1, v_res = kPair ? p.v_res : 1;
  const int n_vp = (n_vt + v_res - 1) / v_res;                               // passes over the hidden dimension per group
  const uint32_t tmem_cols = kPair ? 512u : 256u;
  const int w_rows = kPair ? p.tile_n >> 1 : p.tile_n;                       // of a head tile in this CTA's shared memory
  const uint32_t w_bytes = static_cast<uint32_t>(w_rows) * (kLmKC * 2u);     // one chunk of it
  const uint32_t f_bytes = static_cast<uint32_t>(p.f_rows) * (kLmKC * 2u);   // one chunk of one feature tile
  const int n_groups = (p.n_mt + m_res - 1) / m_res;
  const int n_ks = (p.n_kc + p.kch - 1) / p.kch;                             // ring stages per accumulator tile
  const int n_iter = n_groups * n_vp * n_ks;                                 // ring stages this CTA goes through
  const int n_pre = min(S, n_iter);
  // CTAs start at different places of the hidden dimension (a sum does not care where it starts), so that at
  // any moment they read different column ranges of their rows instead of all the same one.
  const int rot = static_cast<int>((static_cast<unsigned>(cta) * 11u) % static_cast<unsigned>(n_ks));
  // Ring stage `it` = (node-tile group, vocabulary tile, K step), K fastest.  Its chunks are asked for back to
  // back; a chunk past the hidden size reads as zeros, and so does a node tile past the last one.
  // (a pair: both CTAs' loads signal the first one's barrier, which it arms for both)
  auto full_bar = [&](int st) { return kPair ? map_to_leader(bar(kLmBarFull + st)) : bar(kLmBarFull + st); };
  auto tiles_of = [&](int g) { return kPair ? min(m_res, p.n_mt - g * m_res) : 1; };  // node tiles of a group
  auto arm = [&](int it) {
    if (!leader) return;
    const uint32_t absent = kPair ? static_cast<uint32_t>(p.kch * (m_res - tiles_of(it / (n_ks * n_vp)))) * f_bytes : 0u;
    mbar_expect_tx(bar(kLmBarFull + it % S), (kPair ? 2 : 1) * (p.stage_bytes - absent));
  };
  auto issue_head = [&](int it) {
    const int st = it % S, kq = (it % n_ks + rot) % n_ks, vp = (it / n_ks) % n_vp;
    const uint32_t dst = smem_base + static_cast<uint32_t>(st) * p.stage_bytes;
    for (int c = 0; c < p.kch; ++c) {
      if constexpr (kPair) {
        for (int u = 0; u < v_res; ++u)
          tma_load_pair(dst + (c * v_res + u) * w_bytes, &tm_w, full_bar(st), (kq * p.kch + c) * kLmKC,
                        v_lo + (vp * v_res + u) * p.tile_n + rank * w_rows);
      } else {
        tma_load_5d(dst + c * w_bytes, &tm_w, full_bar(st), (kq * p.kch + c) * kLmKC, v_lo + vp * p.tile_n, 0, 0, 0);
      }
    }
  };
  auto issue_feat = [&](int it) {
    if (it == 0 && p.stall_first) return;
    const int st = it % S, kq = (it % n_ks + rot) % n_ks, g = it / (n_ks * n_vp);
    const uint32_t fdst = smem_base + static_cast<uint32_t>(st) * p.stage_bytes + static_cast<uint32_t>(p.kch * v_res) * w_bytes;
    for (int c = 0; c < p.kch; ++c) {
      if constexpr (kPair) {
        for (int j = 0; j < tiles_of(g); ++j)
          tma_load_pair(fdst + (c * m_res + j) * f_bytes, &tm_f, full_bar(st), (kq * p.kch + c) * kLmKC,
                        kMode == kLmLanes ? ((g * m_res + j) * 2 + rank) * p.f_rows : (g * m_res + j) * 256 + rank * 128);
      } else {
        tma_load_5d(fdst + c * f_bytes, &tm_f, full_bar(st), (kq * p.kch + c) * kLmKC, g * 128, 0, 0, 0);
      }
    }
  };

  if (warp == 0) {
    if (lane == 0) {
      *abort_flag = (smem_base & 1023u) ? 1 : 0;  // the swizzled tiles need a 1 KB aligned base
      *s_last = 0;
      prefetch_tmap(&tm_w);
      prefetch_tmap(&tm_f);
      for (int i = 0; i < kLmNumBars; ++i) mbar_init(bar(i), i == kLmBarAccEmpty ? (kPair ? 2 : 1) * kLmReaders / 32 : 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
  } else if (warp == 1) {
    if constexpr (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem_base)), "r"(tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem_base)), "r"(tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  if constexpr (kPair) cluster_sync_release();  // both CTAs' barriers exist
  // The head is a constant of the model: its first ring fill is asked for before the wait below, while
  // the previous kernel of the stream is still finishing.  The features are that kernel's to write.
  if (warp == 0 && lane == 0 && !*abort_flag)
    for (int it = 0; it < n_pre; ++it) {
      arm(it);
      issue_head(it);
    }
  // Under programmatic dependent launch the grid may start while the previous kernel of the stream
  // drains: the features (and the scratch) are that kernel's business until it has completed.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem_base;

  if (warp == 0) {
    // ================================ TMA producer ================================
    if (lane == 0) {
      bool ok = !*abort_flag;
      int it = ok ? n_pre : 0;
      if (ok)
        for (int i = 0; i < n_pre; ++i) issue_feat(i);
      for (; ok && it < n_iter; ++it) {
        const int st = it % S;
        ok = mbar_wait(bar(kLmBarEmpty + st), (it / S - 1) & 1, abort_flag);
        if (!ok) break;
        arm(it);
        issue_head(it);
        issue_feat(it);
      }
      if (!ok || *abort_flag) {
        // Some wait gave up.  The tiles asked for still arrive: stay until they have, so that no copy
        // is in flight into this CTA's shared memory when it leaves.
        if (leader)
          for (int j = max(0, it - S); j < it; ++j) lm_wait_drain(bar(kLmBarFull + j % S), (j / S) & 1);
        else  // (they signal the other CTA's barriers: leave them a millisecond)
          for (int j = 0; j < 1000; ++j) __nanosleep(1000);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ================================ MMA issuer ================================
    uint32_t elected;
    asm volatile("{ .reg .pred p; elect.sync _|p, 0xffffffff; selp.u32 %0, 1, 0, p; }" : "=r"(elected));
    int it = 0, tile = 0;
    bool ok = leader && !*abort_flag;
    for (int g = 0; ok && g < n_groups; ++g) {
      for (int vp = 0; ok && vp < n_vp; ++vp, ++tile) {
        if (tile > 0) ok = mbar_wait_warp(bar(kLmBarAccEmpty), (tile - 1) & 1, abort_flag);  // the readers are done with TMEM
        if (!ok) break;
        tc_fence_after();
        for (int ks = 0; ok && ks < n_ks; ++ks, ++it) {
          const int st = it % S;
          ok = mbar_wait_warp(bar(kLmBarFull + st), (it / S) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          if (elected) {
            const uint32_t wbase = smem_base + static_cast<uint32_t>(st) * p.stage_bytes;
            const uint32_t fbase = wbase + static_cast<uint32_t>(p.kch * v_res) * w_bytes;
            for (int c = 0; c < p.kch; ++c) {
              for (int j = 0; j < (v_res > 1 ? 2 : tiles_of(g)); ++j) {  // accumulators: node tiles or vocabulary tiles
                const uint32_t fj = fbase + (c * m_res + (m_res > 1 ? j : 0)) * f_bytes, wj = wbase + (c * v_res + (v_res > 1 ? j : 0)) * w_bytes;
#pragma unroll
                for (int kk = 0; kk < kLmKC / 16; ++kk) {
                  // features (A) and head rows (B; kLmLanes: the other way round): both K-major, 16 hidden columns = 32 bytes inside the 128-byte swizzle row
                  const uint64_t fd = smem_desc(fj + kk * 32, 16, 1024), wd = smem_desc(wj + kk * 32, 16, 1024);
                  const uint64_t ad = kMode == kLmLanes ? wd : fd, bd = kMode == kLmLanes ? fd : wd;
                  const uint32_t acc = tmem_base + static_cast<uint32_t>(j) * 256u, more = (ks > 0 || c > 0 || kk > 0) ? 1u : 0u;
                  if constexpr (kPair) umma_pair_ss(acc, ad, bd, p.idesc, more);
                  else umma_bf16_ss(acc, ad, bd, p.idesc, more);
                }
              }
            }
            if constexpr (kPair) umma_pair_commit(bar(kLmBarEmpty + st));
            else umma_commit(bar(kLmBarEmpty + st));
          }
          __syncwarp();
        }
        if (ok && elected) {
          if constexpr (kPair) umma_pair_commit(bar(kLmBarAccFull));
          else umma_commit(bar(kLmBarAccFull));
        }
        __syncwarp();
      }
    }
    // every MMA issued so far has finished before TMEM is given back
    if (elected) {
      if constexpr (kPair) {
        if (leader) umma_pair_commit(bar(kLmBarDone));
      } else {
        umma_commit(bar(kLmBarDone));
      }
      lm_wait_drain(bar(kLmBarDone), 0);
    }
    __syncwarp();
  } else {
    // ================================ accumulator readers ================================
    // Two warps for each TMEM lane quadrant: one for each accumulator of a pair, else one for each half of the columns.
    // The MMAs wait for them wherever another vocabulary tile follows, and the call waits for the last: one thread per row,
    // with a single chain of compares through its columns, took 740 cycles for 32 of them; four chains and the next
    // columns' load under the compares take 150: 60 nodes of 1024 x 100000 42.4 -> 39.3 us, 411 nodes 106 -> 91, of 5120 x 32000
    // 131 -> 126.
    const int q = warp & 3;                 // TMEM lane quadrant this warp can reach
    const int sub = (warp - 2) >> 2;
    const int r = q * 32 + lane;            // accumulator row = node inside its tile
    const int rt = tid - 64;                // 0 .. kLmReaders - 1
    const uint32_t tmem_lane = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + (kPair ? static_cast<uint32_t>(sub) * 256u : 0u);
    int tile = 0;
    bool ok = !*abort_flag;
    if constexpr (kMode == kLmLanes) {
      // A lane is a vocabulary row, a column a node: per column the warp's maximum and the lowest lane that has it, kept by
      // lane (column mod 32).
      unsigned long long* results = reinterpret_cast<unsigned long long*>(small + 8 * kLmNumBars + 16);
      const int n_cols = 2 * p.f_rows;
      for (int g = 0; g < n_groups; ++g) {
        float best[kLmTileMax / 32];
        int idx[kLmTileMax / 32];
#pragma unroll
        for (int k = 0; k < kLmTileMax / 32; ++k) {
          best[k] = -INFINITY;
          idx[k] = INT_MAX;
        }
        for (int vp = 0; ok && vp < n_vp; ++vp, ++tile) {
          ok = mbar_wait_warp(bar(kLmBarAccFull), tile & 1, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const int v0 = v_lo + (v_res > 1 ? vp * 2 + sub : vp) * kLmTileMax + rank * 128 + q * 32;  // lane 0's vocabulary row
          if (v0 < v_hi && (v_res > 1 || sub < tiles_of(g))) {
            const bool exists = v0 + lane < v_hi;
            // The next columns' load runs under these columns' maxima.  It is asked for whether they exist or not: the values of
            // a load under a condition would be merged with older ones before the wait for it.
            uint32_t ring[2][32];
            FALCON_TMEM_LD32(tmem_lane, ring[0]);
#pragma unroll
            for (int k = 0; k < kLmTileMax / 32; ++k) {
              uint32_t(&x)[32] = ring[k & 1];
              tmem_wait_ld(x);
              FALCON_TMEM_LD32(tmem_lane + static_cast<uint32_t>((k + 1) * 32 < n_cols ? (k + 1) * 32 : 0), ring[(k + 1) & 1]);
              if (k * 32 >= n_cols) continue;
              float m_mine = -INFINITY;
              uint32_t who_mine = 0u;
#pragma unroll
              for (int c = 0; c < 32; ++c) {
                const float f = exists ? __uint_as_float(x[c]) : -INFINITY, m = warp_largest(f);
                const uint32_t who = __ballot_sync(0xffffffffu, f == m);
                if (lane == c) {
                  m_mine = m;
                  who_mine = who;
                }
              }
              if (m_mine > best[k]) {  // strict: vocabulary rows ascend over the passes, so the first maximum stays
                best[k] = m_mine;
                idx[k] = v0 + __ffs(static_cast<int>(who_mine)) - 1;
              }
            }
            tmem_wait_ld();
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) arrive_remote(map_to_leader(bar(kLmBarAccEmpty)));
        }
        // one atomic per node and CTA
#pragma unroll
        for (int k = 0; k < kLmTileMax / 32; ++k)
          if (k * 32 < n_cols) results[(sub * 4 + q) * kLmTileMax + k * 32 + lane] = ok && idx[k] != INT_MAX ? lm_pack(best[k], idx[k]) : 0ull;
        asm volatile("bar.sync 1, %0;" ::"n"(kLmReaders) : "memory");
        for (int at = rt; at < m_res * kLmTileMax; at += kLmReaders) {
          const int j = at / kLmTileMax, col = at % kLmTileMax, node = (g * m_res + j) * n_cols + col;
          if (col < n_cols && node < p.n_rows) {
            unsigned long long w = 0ull;
            for (int i = m_res > 1 ? j * 4 : 0; i < (m_res > 1 ? j * 4 + 4 : 8); ++i) w = max(w, results[i * kLmTileMax + col]);
            if (w) atomicMax(p.best + node, w);
          }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kLmReaders) : "memory");
      }
    }
    for (int g = 0; kMode != kLmLanes && g < n_groups; ++g) {
      constexpr int kChains = 4;
      float best[kChains];
      int idx[kChains];
#pragma unroll
      for (int i = 0; i < kChains; ++i) {
        best[i] = -INFINITY;
        idx[i] = INT_MAX;
      }
      for (int vp = 0; ok && vp < n_vp; ++vp, ++tile) {
        ok = mbar_wait_warp(bar(kLmBarAccFull), tile & 1, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const int v0 = v_lo + (v_res > 1 ? vp * 2 + sub : vp) * p.tile_n;
        const int all = v_res > 1 || !kPair || sub < tiles_of(g) ? min(p.tile_n, v_hi - v0) : 0;  // columns with logits
        const int half = kPair ? 0 : ((all >> 1) + 31) & ~31;
        const int begin = kPair || sub == 0 ? 0 : half, end = kPair || sub == 1 ? all : min(all, half);
        auto look = [&](uint32_t (&x)[32], int c0) {
          if (c0 + 32 > end) {  // (columns past the last one hold whatever was there)
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (c0 + c >= end) x[c] = 0xff800000u;
          }
#pragma unroll
          for (int c = 0; c < 32; c += kChains)
#pragma unroll
            for (int i = 0; i < kChains; ++i) {
              const float f = __uint_as_float(x[c + i]);
              if (f > best[i]) {  // strict: a chain's columns ascend, so its first maximum stays; NaN never wins
                best[i] = f;
                idx[i] = v0 + c0 + c + i;
              }
            }
        };
        if (begin < end) {
          // (as above: the loads are unconditional, and take the last columns again behind the end)
          const int last = begin + ((end - begin - 1) & ~31);
          uint32_t x0[32], x1[32];
          FALCON_TMEM_LD32(tmem_lane + static_cast<uint32_t>(begin), x0);
          tmem_wait_ld(x0);
          for (int c0 = begin;; c0 += 64) {
            FALCON_TMEM_LD32(tmem_lane + static_cast<uint32_t>(min(c0 + 32, last)), x1);
            look(x0, c0);
            tmem_wait_ld(x1);
            if (c0 + 32 > last) break;
            FALCON_TMEM_LD32(tmem_lane + static_cast<uint32_t>(min(c0 + 64, last)), x0);
            look(x1, c0 + 32);
            tmem_wait_ld(x0);
            if (c0 + 64 > last) break;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if constexpr (kPair) arrive_remote(map_to_leader(bar(kLmBarAccEmpty)));
          else mbar_arrive(bar(kLmBarAccEmpty));
        }
      }
      // the chains' maxima, ties to the lower index
#pragma unroll
      for (int i = 1; i < kChains; ++i)
        if (best[i] > best[0] || (best[i] == best[0] && idx[i] < idx[0])) {
          best[0] = best[i];
          idx[0] = idx[i];
        }
      const int node = kPair ? (g * m_res + (m_res > 1 ? sub : 0)) * 256 + rank * 128 + r : g * 128 + r;
      // one atomic per node, CTA and warp: the order of arrival does not matter, the word's order decides
      if (node < p.n_rows && ok && idx[0] != INT_MAX) atomicMax(p.best + node, lm_pack(best[0], idx[0]));
    }
    // the last CTA to arrive folds the CTAs' results in vocabulary order
    asm volatile("bar.sync 1, %0;" ::"n"(kLmReaders) : "memory");
    if (rt == 0) {
      if (*abort_flag) dev_status_or(p.status, 0, FALCON_DEV_TIMEOUT);
      *s_last = (arrive_acq_rel(p.ticket) == n_cta - 1) ? 1 : 0;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kLmReaders) : "memory");
    if (*s_last) {
      for (int node = rt; node < p.n_rows; node += kLmReaders) {
        const unsigned long long w = __ldcg(p.best + node);
        p.best[node] = 0ull;  // ready for the next call
        p.argmax_out[node] = w ? static_cast<int>(~static_cast<uint32_t>(w)) : 0;
        if (p.max_out) p.max_out[node] = w ? lm_unpack_val(w) : -INFINITY;
      }
      if (rt == 0) *p.ticket = 0;  // ready for the next call
    }
  }
  tc_fence_before();
  if constexpr (kPair) cluster_sync_release();  // (and neither CTA leaves while the other may still signal it)
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

}  // namespace

cudaError_t set_up_lm_head() {
  cudaError_t e = cudaSuccess;
  for (auto* kernel : {lm_head_argmax_kernel<kLmSingle>, lm_head_argmax_kernel<kLmPair>, lm_head_argmax_kernel<kLmLanes>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kLmSmemMax));
  return e;
}

int launch_lm_head_argmax(falcon_ctx* ctx, const falcon_lm_argmax_args& a, cudaStream_t s) {
  const int N = a.n_rows, V = a.vocab, H = a.hidden;
  const bool pair = N > 128;  // (a single tile has nothing to share: the head's rows bound it)
  int n_mt = pair ? (N + 255) / 256 : 1;
  int m_res = n_mt >= 2 ? 2 : 1, v_res = pair && m_res == 1 ? 2 : 1;
  // One wave: the vocabulary split evenly over the SMs or pairs of them, in tiles of the same multiple of 16 rows.
  const int workers = pair ? ctx->sm_count / 2 : ctx->sm_count;
  const int share = (V + workers - 1) / workers;
  int n_vt = (share + kLmTileMax - 1) / kLmTileMax;
  int tile_n = ((share + n_vt - 1) / n_vt + 15) & ~15;
  int span = tile_n * n_vt;
  if (!pair) {
    span = (share + 15) & ~15;
    tile_n = span < kLmTileMax ? span : kLmTileMax;
  }
  int f_rows = pair ? 128 : (N <= 64 ? 64 : ((N + 7) & ~7));
  uint32_t mma_n = static_cast<uint32_t>(tile_n);
  // Vocabulary rows on the lanes, 256 of them a pair, and the nodes on the side that comes in steps of 16, where that takes
  // so many fewer columns of MMAs (with the nodes on the lanes 300 of them are padded to 512) that it pays for the reading of
  // the accumulators, whose maxima across lanes take longer each time.  What is saved per reading, x = columns of MMAs times
  // chunks of 64 hidden columns, decides; one of them is 2 cycles of the tensor core.  Both arrangements were timed at 80
  // sizes, in bursts of six calls and in loops of half a second (under the power limit, where fewer MMAs count for more).  Bursts
  // alone turn at x = 2200, loops alone at 1000; 1600 is where the two together do: the product of both ratios is 0.999 or more
  // at every size with x >= 1664, and above one at 6 of 24 below.  us, nodes on the lanes -> vocabulary rows (in a loop):
  //   x  768  300 nodes of 1536 x 24000  39.9 -> 42.0 (36.9 -> 39.6)       800 of 512 x 131072    121 -> 142 (134 -> 147)
  //     1024  370 of 1024 x 32000        32.8 -> 34.5 (30.6 -> 32.1)       385 of 2048 x 32000    56.3 -> 59.1 (63.9 -> 63.2)
  //     1280  400 of 2560 x 32000        67.6 -> 70.0 (78.0 both)          430 of 2560 x 50257    103 -> 105 (121 -> 122)
  //     1536  400 of 3072 x 32000        78.8 -> 80.9 (92.8 -> 90.5)       340 of 1024 x 32000    32.6 -> 34.0 (30.1 -> 31.7)
  //     1664  230 of 512 x 16000         13.6 -> 13.1 (12.0 -> 11.7)
  //     1792  400 of 3584 x 32000        90.8 -> 91.5 (107 -> 104)         430 of 3584 x 100000   280 -> 276 (330 -> 326)
  //     1920  280 of 768 x 64000         47.8 -> 48.1 (48.5 -> 45.7)       200 of 512 x 16000     13.5 -> 12.6 (12.0 -> 11.2)
  //     2048  385 of 4096 x 32000        101 -> 103 (122 -> 118), 416 103 both (123 -> 119), 417 (x = 0) 102 -> 106 (123 both)
  //           385 of 2048 x 50000        84.0 -> 85.0 (97.6 -> 95.4), 416 84.3 -> 85.3 (98.7 -> 96.5), 432 (1024) 84.3 -> 88.1 (99.2 -> 99.8)
  //     2560  129 of 1024 x 32000        19.3 -> 19.1 (17.4 -> 17.6)
  //           385 of 5120 x 32000        125 -> 124 (151 -> 145), 411 127 -> 124 (152 -> 146), 417 (0) 127 -> 128 (153 -> 151)
  //     4096  411 of 8192 x 32000        201 -> 192 (241 -> 229)           6400: 352 of 5120 x 32000  124 -> 116 (148 -> 133)
  bool lanes = false;
  if (pair) {
    const int tiles = N <= 256 ? 1 : 2 * ((N + 511) / 512), cols = ((N + tiles - 1) / tiles + 15) & ~15;
    const int blocks = (V + kLmTileMax - 1) / kLmTileMax, per = (blocks + workers - 1) / workers;
    const int two = tiles == 1 && per > 1;  // two vocabulary blocks resident
    const int64_t here = static_cast<int64_t>(tiles) * cols * (two ? (per + 1) / 2 * 2 : per), chunks = (H + kLmKC - 1) / kLmKC;
    const int64_t other = static_cast<int64_t>(n_mt) * tile_n * (v_res > 1 ? (n_vt + 1) / 2 * 2 : n_vt);
    const int64_t reads = static_cast<int64_t>((tiles + 1) / 2) * (two ? (per + 1) / 2 : per);
    lanes = (other - here) * chunks > 1600 * reads;
    if (lanes) {
      n_mt = tiles;
      m_res = tiles > 1 ? 2 : 1;
      v_res = two ? 2 : 1;
      n_vt = per;
      tile_n = kLmTileMax;
      span = per * kLmTileMax;
      f_rows = cols / 2;
      mma_n = static_cast<uint32_t>(cols);
    }
  }
  const int n_cta = (V + span - 1) / span * (pair ? 2 : 1);
  const int w_rows = pair ? tile_n / 2 : tile_n;
  const int n_kc = (H + kLmKC - 1) / kLmKC;
  // Chunks per stage: two where two such stages fit.  Fewer, larger stages mean fewer trips round the ring
  // (32000 x 4096, 60 nodes: 43 us with two chunks in three stages against 53 with one in five and 46 with
  // three in two; in pairs, 512 nodes of 5120: 133 with two chunks in two stages, 158 with one in four; a head stored chunk by chunk so that a tile is contiguous made no difference).
  const uint32_t small_bytes = kLmSmallBytes + (lanes ? kLmResultBytes : 0u);
  const uint32_t chunk_bytes = static_cast<uint32_t>(v_res * w_rows + m_res * f_rows) * (kLmKC * 2u);
  int kch = (2 * 2 * chunk_bytes <= kLmSmemMax - small_bytes) ? 2 : 1;
  if (kch > n_kc) kch = n_kc;
  const uint32_t stage_bytes = static_cast<uint32_t>(kch) * chunk_bytes;
  int n_stages = static_cast<int>((kLmSmemMax - small_bytes) / stage_bytes);
  if (n_stages > kLmMaxStages) n_stages = kLmMaxStages;
  if (n_stages < 2) return FALCON_ERR_CAPACITY;
  const uint32_t smem_bytes = static_cast<uint32_t>(n_stages) * stage_bytes + small_bytes;

  // scratch that is zero between calls: the arrival counter and one 64-bit word per node
  int rc = ensure_tickets(ctx, 2 + 2 * N, s);
  if (rc) return rc;

  // Tensor maps: [hidden, rows] with the hidden index contiguous; a box is 64 columns x the tile's
  // rows, 128-byte swizzled; what lies outside (the hidden tail, rows past the end) reads as zeros.
  CUtensorMap mw, mf;
  {
    const uint64_t hs = static_cast<uint64_t>(a.head_stride) * 2, fs = static_cast<uint64_t>(a.feat_stride) * 2;
    const uint64_t w_dims[5] = {static_cast<uint64_t>(H), static_cast<uint64_t>(V), 1, 1, 1};
    const uint64_t w_strides[4] = {hs, hs * V, hs * V, hs * V};
    const uint32_t w_box[5] = {kLmKC, static_cast<uint32_t>(w_rows), 1, 1, 1};
    const uint64_t f_dims[5] = {static_cast<uint64_t>(H), static_cast<uint64_t>(N), 1, 1, 1};
    const uint64_t f_strides[4] = {fs, fs * N, fs * N, fs * N};
    const uint32_t f_box[5] = {kLmKC, static_cast<uint32_t>(f_rows), 1, 1, 1};
    if (!get_tmap(ctx, a.lm_head, w_dims, w_strides, w_box, &mw) || !get_tmap(ctx, a.features, f_dims, f_strides, f_box, &mf)) {
      ctx->last_error = "cuTensorMapEncodeTiled failed";
      return FALCON_ERR_CUDA;
    }
  }

  LmParams p;
  p.n_rows = N;
  p.vocab = V;
  p.n_kc = n_kc;
  p.kch = kch;
  p.f_rows = f_rows;
  p.n_mt = n_mt;
  p.m_res = m_res;
  p.v_res = v_res;
  p.tile_n = tile_n;
  p.span = span;
  p.n_stages = n_stages;
  p.stall_first = (a.flags & FALCON_LM_TEST_STALL) ? 1 : 0;
  p.stage_bytes = stage_bytes;
  p.idesc = make_idesc(pair ? 256 : 128, mma_n, false, false);
  p.argmax_out = a.argmax_out;
  p.max_out = a.max_out;
  p.status = a.status;
  p.ticket = ctx->tickets;
  p.best = reinterpret_cast<unsigned long long*>(ctx->tickets + 2);

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_cta);
  cfg.blockDim = dim3(kLmThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pair ? 2 : 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, lanes ? lm_head_argmax_kernel<kLmLanes> : pair ? lm_head_argmax_kernel<kLmPair> : lm_head_argmax_kernel<kLmSingle>, mw, mf, p);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "lm_head_argmax_kernel launch");
  return FALCON_OK;
}

}  // namespace falcon
