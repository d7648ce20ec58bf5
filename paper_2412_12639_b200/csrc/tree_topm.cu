// falcon_topm: the m best entries of every logits row, best first (the children a tree
// node gets when the decoding tree is grown, Appendix A).
//
// Order: larger value first, the lower index among equal values; a NaN counts as -inf.
// One thread-block cluster of up to eight CTAs per row (8 warps each); the row is read once (4 V bytes)
// and no intermediate result touches global memory.  A call is a chain of latencies, so it has as few
// hops as the selection allows (one row of 32000: 4.6 us; through scratch lists and an arrival counter
// in global memory it took 7.8):
//   1  every CTA loads the first step of its share into registers (up to 32 entries per lane) and finds
//      the maxima of its groups of lanes, 64 groups in the whole cluster, which go to the shared memory
//      of every CTA; cluster barrier.
//   2  the m-th largest of the 64 group maxima is a threshold that at least m entries of the row reach:
//      everything below it can go, whichever way ties are broken.  On continuous data it leaves little
//      more than m entries of the first steps (about -64 ln(1 - m/64)).
//   3  the survivors go to a list.  Where the share is longer than a step the loads of the next step run
//      under the filtering of this one (two instructions an entry), and after steps 2, 4, 8, ... the
//      threshold is taken afresh from the list, so that each doubling of what has been seen adds
//      about as many survivors as the first step did.
//   4  CTA 0 has or is sent all lists; cluster barrier; it ranks the survivors, a thread each, and
//      writes the first m.
// When a list overflows (many equal values, e.g. a row that is mostly -inf) the cluster takes the exact
// route instead: every warp cuts its entries to at most 64 that contain its m best (threshold from the
// lanes' maxima, or bisection over key and index bits), every CTA its warps', CTA 0 the CTAs'.  Values are
// compared as floats where they are read and become 32-bit keys whose unsigned order is the
// selection order (key 0 = "no entry") only once they have survived.

#include <climits>

#include "row_stream.cuh"

namespace falcon {
namespace {

constexpr int kTopmThreads = 256;
constexpr int kTopmWarps = kTopmThreads / 32;
constexpr int kTopmMaxCluster = 8;
constexpr int kTopmGroups = 64;                                   // group maxima of a row
constexpr int kTopmPerLane = 16;                                  // entries a lane holds in the passes over lists
constexpr int kTopmRowsMax = 32;                                  // entries a lane holds at most in the first pass
constexpr int kTopmCap = 64;                                      // entries a thinning pass leaves at most
constexpr int kList = 512;                                        // survivors a list holds at most
constexpr int kRankMax = 128;                                     // more than these are thinned before they are ranked
static_assert(kTopmMaxCluster * kTopmCap <= 32 * kTopmPerLane, "one warp holds all CTAs' survivors");
static_assert(kTopmWarps * kTopmCap <= 32 * kTopmPerLane, "one warp holds all warps' survivors");
static_assert(kList <= 2 * kTopmThreads, "a thread holds two list entries at most");
static_assert(FALCON_TOPM_MAX <= 32, "the threshold is the m-th largest of 32 lane maxima");
static_assert(FALCON_TOPM_MAX <= kTopmCap, "the exact selection's m entries fit where the survivors go");

struct TopmParams {
  int32_t vocab, m;
  int32_t chunk_len;   // entries per CTA of the cluster
  int32_t steps;       // in which the exact route takes a CTA's share: of 256 x (entries per lane)
  int32_t stall;       // test hook: see RowStream::produce
  int64_t logits_stride;
  const float* logits;
  float* top_val;
  int32_t* top_idx;
};

struct TopmShared {
  uint32_t max[kTopmGroups];            // group maxima (keys; 0 = empty group)
  uint64_t list[kList];                 // survivors
  int cnt;                              // how many there are (also beyond kList)
  uint32_t tau;
  // exact route
  uint32_t key[kTopmWarps * kTopmCap];
  int id[kTopmWarps * kTopmCap];
  uint32_t acc_key[2 * kTopmCap];
  int acc_id[2 * kTopmCap];
  int fill, acc;
};
static_assert(kTopmMaxCluster * kTopmCap <= kList, "CTA 0's list takes every CTA's exact entries");

// float -> key: unsigned order of the keys = order of the values; NaN -> -inf, -0 -> +0; never 0
__device__ __forceinline__ uint32_t to_key(float x) {
  x = (x == x) ? x + 0.f : -INFINITY;
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_key(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// One entry as a 64-bit word whose unsigned order is the selection order: key in the upper half,
// the complemented index in the lower one (so that the lower index is the larger word); 0 = none.
__device__ __forceinline__ uint64_t entry(uint32_t key, int id) {
  return key ? (static_cast<uint64_t>(key) << 32) | static_cast<uint32_t>(~id) : 0ull;
}

// The k-th largest (k = 0: the largest) of one value per lane.  Every lane ranks its value against
// all 32 (equal values in lane order, so the ranks are a permutation); the 32 shuffles are
// independent of one another, unlike the stages of a sorting network.
__device__ __forceinline__ uint32_t warp_kth_largest(uint32_t v, int kth, int lane) {
  int rank = 0;
#pragma unroll 4
  for (int j = 0; j < 32; ++j) {
    const uint32_t o = __shfl_sync(0xffffffffu, v, j);
    rank += (o > v || (o == v && j < lane)) ? 1 : 0;
  }
  const unsigned hit = __ballot_sync(0xffffffffu, rank == kth);
  return __shfl_sync(0xffffffffu, v, __ffs(static_cast<int>(hit)) - 1);
}

// Sum of one int per lane over the warp.
__device__ __forceinline__ int warp_sum(int v) { return static_cast<int>(__reduce_add_sync(0xffffffffu, static_cast<unsigned>(v))); }

// The exact cut for the warp's kLen entries per lane (key 0 = none), of which more than m exist:
// t = the m-th largest key, u = the index up to which the entries equal to t belong to the m best.
// An entry is among the m best iff key > t, or key == t and id <= u.
template <int kLen>
__device__ __noinline__ void exact_cut(const uint32_t (&key)[kLen], const int (&id)[kLen], int m, uint32_t& t_out, int& u_out) {
  uint32_t t = 0u;
  for (int bit = 31; bit >= 0; --bit) {
    const uint32_t cand = t | (1u << bit);
    int c = 0;
#pragma unroll
    for (int k = 0; k < kLen; ++k) c += key[k] >= cand ? 1 : 0;
    if (warp_sum(c) >= m) t = cand;
  }
  int above = 0;
#pragma unroll
  for (int k = 0; k < kLen; ++k) above += key[k] > t ? 1 : 0;
  const int need = m - warp_sum(above);  // >= 1 of the entries equal to t
  int u = 0;
  for (int bit = 30; bit >= 0; --bit) {
    const int test = u | ((1 << bit) - 1);  // this bit 0, all lower bits 1
    int c = 0;
#pragma unroll
    for (int k = 0; k < kLen; ++k) c += (key[k] == t && id[k] <= test) ? 1 : 0;
    if (warp_sum(c) < need) u |= 1 << bit;
  }
  t_out = t;
  u_out = u;
}

// Exclusive prefix sum of one count per lane; total = the warp's sum.
__device__ __forceinline__ int warp_offsets(int cnt, int lane, int& total) {
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - cnt;
}

// Room for `total` entries in a list shared by the CTA's warps: the position of the first.
__device__ __forceinline__ int warp_reserve(int* fill, int total, int lane) {
  int base = 0;
  if (lane == 0 && total > 0) base = atomicAdd(fill, total);
  return __shfl_sync(0xffffffffu, base, 0);
}


// Barrier of the 256 working threads of a CTA (the streaming kernel has a warp more).
__device__ __forceinline__ void worker_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kTopmThreads) : "memory"); }

// Address of this CTA's shared variable in CTA `rank` of the cluster, and accesses to it.
__device__ __forceinline__ uint32_t peer_addr(const void* p, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
  return r;
}
__device__ __forceinline__ void peer_store(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void peer_store64(uint32_t addr, uint64_t v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ int peer_add(uint32_t addr, int v) {
  int old;
  asm volatile("atom.add.shared::cluster.u32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ int peer_load(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
// Barrier of the row's CTAs (its stores to peers' shared memory are visible behind it).
__device__ __forceinline__ void row_arrive(int n_ctas) {
  if (n_ctas > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void row_wait(int n_ctas) {
  if (n_ctas > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  else worker_sync();
}

// Exact route, first pass: the warp's share rowp[0 .. n_w) (lane l: l, l + 32, ..., read again from L2) is
// cut to at most kTopmCap entries that contain its m best, which are appended to the CTA's list.
template <int kRows>
__device__ __noinline__ void warp_cut(const float* rowp, int n_w, int id0, int m, int lane, uint32_t* out_key, int* out_id, int* fill) {
  float x[kRows];
#pragma unroll
  for (int k = 0; k < kRows; ++k) x[k] = (k * 32 + lane < n_w) ? rowp[k * 32 + lane] : -INFINITY;
  const int n_lane = max(0, min(kRows, (n_w - lane + 31) >> 5));
  const uint32_t valid = n_lane >= 32 ? 0xffffffffu : ((1u << n_lane) - 1u);
  float lm = -INFINITY;
#pragma unroll
  for (int k = 0; k < kRows; ++k) lm = fmaxf(lm, x[k]);
  const float tau = from_key(max(1u, warp_kth_largest(valid ? to_key(lm) : 0u, m - 1, lane)));
  uint32_t mask = 0u;
#pragma unroll
  for (int k = 0; k < kRows; ++k)
    if (!(x[k] < tau)) mask |= 1u << k;  // (a NaN passes: whether it belongs is decided on keys)
  mask &= valid;
  if (warp_sum(__popc(mask)) > kTopmCap) {
    uint32_t key[kRows];
    int id[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      key[k] = ((valid >> k) & 1u) ? to_key(x[k]) : 0u;
      id[k] = id0 + k * 32 + lane;
    }
    uint32_t t;
    int u;
    exact_cut<kRows>(key, id, m, t, u);
    mask = 0u;
#pragma unroll
    for (int k = 0; k < kRows; ++k)
      if (key[k] > t || (key[k] == t && id[k] <= u)) mask |= 1u << k;
  }
  int total;
  int off = warp_offsets(__popc(mask), lane, total);
  off += warp_reserve(fill, total, lane);
#pragma unroll
  for (int k = 0; k < kRows; ++k)
    if ((mask >> k) & 1u) {
      out_key[off] = to_key(x[k]);
      out_id[off] = id0 + k * 32 + lane;
      ++off;
    }
}

// The same on entries that are (key, id) pairs in registers (16 per lane: key 0 = none).  The survivors go to out_key / out_id in no particular order: appended to a list shared
// with other warps when `fill` is its fill count, from position 0 when `fill` is null; returns
// their number (the same in every lane).
__device__ __forceinline__ int warp_thin(const uint32_t (&key)[kTopmPerLane], const int (&id)[kTopmPerLane], int m, int lane,
                                         uint32_t* out_key, int* out_id, int* fill) {
  uint32_t lmax = key[0];
#pragma unroll
  for (int k = 1; k < kTopmPerLane; ++k) lmax = max(lmax, key[k]);
  uint32_t tau = warp_kth_largest(lmax, m - 1, lane);
  if (tau == 0u) tau = 1u;  // fewer than m lanes hold anything: keep every entry
  int id_max = INT_MAX;     // entries equal to tau stay if their index is at most this
  int cnt = 0;
#pragma unroll
  for (int k = 0; k < kTopmPerLane; ++k) cnt += key[k] >= tau ? 1 : 0;
  if (warp_sum(cnt) > kTopmCap) {
    exact_cut<kTopmPerLane>(key, id, m, tau, id_max);
    cnt = 0;
#pragma unroll
    for (int k = 0; k < kTopmPerLane; ++k) cnt += (key[k] > tau || (key[k] == tau && id[k] <= id_max)) ? 1 : 0;
  }
  int total;
  int off = warp_offsets(cnt, lane, total);
  if (fill) off += warp_reserve(fill, total, lane);
#pragma unroll
  for (int k = 0; k < kTopmPerLane; ++k) {
    if (key[k] > tau || (key[k] == tau && id[k] <= id_max)) {
      out_key[off] = key[k];
      out_id[off] = id[k];
      ++off;
    }
  }
  return total;
}


// The m-th largest of the 64 group maxima: the smallest of those that fewer than m exceed.  sh.tau must
// read 0xffffffff before; every thread of the CTA calls this and finds it there afterwards.
__device__ __forceinline__ void find_tau(TopmShared& sh, int m, int warp, int lane) {
  const uint32_t mine = sh.max[warp * 8 + (lane & 7)];
  const uint4* seg = reinterpret_cast<const uint4*>(sh.max + (lane >> 3) * 16);
  int above = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint4 v = seg[i];
    above += (v.x > mine) + (v.y > mine) + (v.z > mine) + (v.w > mine);
  }
  above += __shfl_xor_sync(0xffffffffu, above, 8);
  above += __shfl_xor_sync(0xffffffffu, above, 16);
  const uint32_t t = __reduce_min_sync(0xffffffffu, above < m ? mine : 0xffffffffu);
  if (lane == 0) atomicMin(&sh.tau, t);
  worker_sync();
}

// The CTA's list thinned in place by a threshold of its own (64 groups of its entries, dealt out evenly):
// at least m of them stay.  Every thread of the CTA calls this.  Returns the threshold.
__device__ __forceinline__ uint32_t thin_list(TopmShared& sh, int m, int tid) {
  const int warp = warp_index(), lane = tid & 31, n = sh.cnt;
  const uint64_t e0 = tid < n ? sh.list[tid] : 0ull, e1 = tid + kTopmThreads < n ? sh.list[tid + kTopmThreads] : 0ull;
  if (tid < kTopmGroups) sh.max[tid] = 0u;
  if (tid == 0) sh.tau = 0xffffffffu;
  worker_sync();
  if (e0 | e1) atomicMax(&sh.max[tid % kTopmGroups], static_cast<uint32_t>(max(e0, e1) >> 32));
  worker_sync();
  if (tid == 0) sh.cnt = 0;
  find_tau(sh, m, warp, lane);
  const uint32_t tau = max(1u, sh.tau);
  const bool k0 = static_cast<uint32_t>(e0 >> 32) >= tau, k1 = static_cast<uint32_t>(e1 >> 32) >= tau;
  int total;
  int off = warp_offsets((k0 ? 1 : 0) + (k1 ? 1 : 0), lane, total);
  off += warp_reserve(&sh.cnt, total, lane);
  if (k0) sh.list[off++] = e0;
  if (k1) sh.list[off] = e1;
  worker_sync();
  return tau;
}

// Exact route: every CTA leaves its at most kTopmCap entries, key 0 beyond them, in CTA 0's list (64 places
// each).  Every thread of the cluster calls this, with CTA 0's shared memory still there.
template <int kRows>
__device__ __noinline__ void exact_entries(const TopmParams& p, TopmShared& sh, const float* rowp, int n, int c0, int rank) {
  const int warp = warp_index(), lane = threadIdx.x & 31, m = p.m;
  auto from_list = [&](const uint32_t* lk, const int* li, int fill, uint32_t (&key)[kTopmPerLane], int (&id)[kTopmPerLane]) {
#pragma unroll
    for (int k = 0; k < kTopmPerLane; ++k) {
      const int j = k * 32 + lane;
      key[k] = j < fill ? lk[j] : 0u;
      id[k] = j < fill ? li[j] : 0;
    }
  };
  if (threadIdx.x == 0) {
    sh.fill = 0;
    sh.acc = 0;
  }
  worker_sync();
  for (int step = 0; step < p.steps; ++step) {
    const int v0 = (step * kTopmWarps + warp) * 32 * kRows;
    warp_cut<kRows>(rowp + v0, max(0, min(32 * kRows, n - v0)), c0 + v0, m, lane, sh.key, sh.id, &sh.fill);
    worker_sync();
    if (warp == 0) {  // the best so far and this step's
      uint32_t key[kTopmPerLane];
      int id[kTopmPerLane];
      from_list(sh.key, sh.id, sh.fill, key, id);
      const int got = warp_thin(key, id, m, lane, sh.acc_key + sh.acc, sh.acc_id + sh.acc, nullptr);
      __syncwarp();
      if (sh.acc > 0) {
        from_list(sh.acc_key, sh.acc_id, sh.acc + got, key, id);
        __syncwarp();
        const int both = warp_thin(key, id, m, lane, sh.acc_key, sh.acc_id, nullptr);
        __syncwarp();
        if (lane == 0) sh.acc = both;
      } else if (lane == 0) {
        sh.acc = got;
      }
      if (lane == 0) sh.fill = 0;
    }
    worker_sync();
  }
  if (warp == 0)
    for (int j = lane; j < kTopmCap; j += 32)
      peer_store64(peer_addr(&sh.list[rank * kTopmCap + j], 0), j < sh.acc ? entry(sh.acc_key[j], sh.acc_id[j]) : 0ull);
}
// ... and CTA 0 cuts them to at most kTopmCap at the head of its list.
__device__ __noinline__ void exact_finish(TopmShared& sh, int n_ctas, int m) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    uint32_t key[kTopmPerLane];
    int id[kTopmPerLane];
#pragma unroll
    for (int k = 0; k < kTopmPerLane; ++k) {
      const int j = k * 32 + lane;
      const uint64_t e = j < n_ctas * kTopmCap ? sh.list[j] : 0ull;
      key[k] = static_cast<uint32_t>(e >> 32);
      id[k] = static_cast<int>(~static_cast<uint32_t>(e));
    }
    const int got = warp_thin(key, id, m, lane, sh.key, sh.id, nullptr);
    __syncwarp();
    for (int j = lane; j < got; j += 32) sh.list[j] = entry(sh.key[j], sh.id[j]);
    if (lane == 0) sh.cnt = got;
  }
  worker_sync();
}

// Appends the entries of one batch of registers that reach the threshold to a list (the CTA's own, or with
// `remote` CTA 0's).  live: which of x[0 .. kN) are entries; index(k), value(k): vocabulary index and value of
// the lane's entry k, asked for the few survivors only.  A compact loop over them: written out entry by
// entry this was 13 KB of instructions, and fetching those for the first time in a launch took 7000 cycles.
template <int kN, class Index, class Value>
__device__ __forceinline__ void append(TopmShared& sh, const float (&x)[kN], uint32_t tau_key, uint32_t live, bool remote, int lane,
                                       Index index, Value value) {
  const float tau = from_key(tau_key);
  uint32_t mask = 0u;
#pragma unroll
  for (int k = 0; k < kN; ++k) mask |= x[k] >= tau ? 1u << k : 0u;
  if (tau_key <= to_key(-INFINITY)) mask = live;
  const int total = warp_sum(__popc(mask));
  if (total == 0) return;
  int base = 0;
  if (lane == 0) base = remote ? peer_add(peer_addr(&sh.cnt, 0), total) : atomicAdd(&sh.cnt, total);
  base = __shfl_sync(0xffffffffu, base, 0);
  if (base + total > kList) return;  // (the count says so)
#pragma unroll 1
  for (uint32_t left = __ballot_sync(0xffffffffu, mask != 0u); left; left = __ballot_sync(0xffffffffu, mask != 0u)) {
    if (mask) {
      const int k = __ffs(static_cast<int>(mask)) - 1;
      mask &= mask - 1u;
      const int at = base + __popc(left & ((1u << lane) - 1u));
      const uint64_t e = entry(to_key(value(k)), index(k));
      if (remote) peer_store64(peer_addr(&sh.list[at], 0), e);
      else sh.list[at] = e;
    }
    base += __popc(left);
  }
}

// Group maxima to every CTA of the row, and the threshold.  lk: the largest key of this lane's entries (0: it
// has none).  Every working thread calls this.
__device__ __forceinline__ uint32_t first_tau(TopmShared& sh, uint32_t lk, int m, int rank, int n_ctas, int warp, int lane) {
  // 64 groups in the cluster: 8 / n_ctas per warp; lane l sends group l % per to CTA l / per
  const int per = kTopmMaxCluster / n_ctas, width = 32 / per;
  for (int o = width >> 1; o > 0; o >>= 1) lk = max(lk, __shfl_xor_sync(0xffffffffu, lk, o));
  const uint32_t gmax = __shfl_sync(0xffffffffu, lk, (lane % per) * width);
  row_wait(n_ctas);
  if (lane < kTopmMaxCluster) peer_store(peer_addr(&sh.max[(rank * kTopmWarps + warp) * per + lane % per], lane / per), gmax);
  row_arrive(n_ctas);
  row_wait(n_ctas);
  find_tau(sh, m, warp, lane);
  return max(1u, sh.tau);  // (fewer than m groups hold anything: every entry passes)
}

// The end of both kernels: all survivors are in CTA 0's list, or its count says that they are too many.
template <int kRows>
__device__ __forceinline__ void finish_row(const TopmParams& p, TopmShared& sh, const float* rowp, int n, int c0, int rank, int n_ctas, int row) {
  const int tid = threadIdx.x, m = p.m;
  row_arrive(n_ctas);
  row_wait(n_ctas);
  const int cnt = rank == 0 ? sh.cnt : peer_load(peer_addr(&sh.cnt, 0));
  row_arrive(n_ctas);  // CTA 0's shared memory is needed until every CTA has read the count
  if (cnt > kList) {
    row_wait(n_ctas);
    exact_entries<kRows>(p, sh, rowp, n, c0, rank);
    row_arrive(n_ctas);
    row_wait(n_ctas);
    if (rank != 0) return;
    exact_finish(sh, n_ctas, m);
  } else {
    if (rank != 0) return;
    if (n_ctas > 1) row_wait(n_ctas);
    if (cnt > kRankMax) thin_list(sh, m, tid);
  }
  // An entry's place is the number of entries that come before it (they are distinct).
  const int got = sh.cnt;
  for (int t = tid; t < got; t += kTopmThreads) {
    const uint64_t e = sh.list[t];
    int r = 0;
    for (int j = 0; j < got; ++j) r += sh.list[j] > e ? 1 : 0;
    if (r < m) {
      p.top_val[static_cast<int64_t>(row) * m + r] = from_key(static_cast<uint32_t>(e >> 32));
      p.top_idx[static_cast<int64_t>(row) * m + r] = static_cast<int>(~static_cast<uint32_t>(e));
    }
  }
}

// The row in the cluster's registers: kRows entries per lane.
template <int kRows>
__global__ void __launch_bounds__(kTopmThreads, kRows <= 8 ? 6 : (kRows <= 16 ? 4 : 3)) tree_topm_kernel(const __grid_constant__ TopmParams p) {
  __shared__ __align__(16) TopmShared sh;
  const int row = blockIdx.y, rank = blockIdx.x, n_ctas = gridDim.x;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int c0 = rank * p.chunk_len;
  const int n = max(0, min(p.vocab, c0 + p.chunk_len) - c0);
  const float* rowp = p.logits + static_cast<int64_t>(row) * p.logits_stride + c0;
  if (tid == 0) {
    sh.cnt = 0;
    sh.tau = 0xffffffffu;
  }
  row_arrive(n_ctas);  // waited for before the first store to a peer: by then it runs
  // Under programmatic dependent launch the grid may start while the previous kernel of the stream
  // drains: nothing is read or written before that kernel has completed.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // Lane l of a warp holds entries l, l + 32, ... of its share: coalesced 128-byte loads, all in flight at once.
  const int w0 = warp * 32 * kRows + lane;
  float x[kRows];
#pragma unroll
  for (int k = 0; k < kRows; ++k) x[k] = w0 + k * 32 < n ? __ldcs(rowp + w0 + k * 32) : -INFINITY;
  float lm = -INFINITY;
#pragma unroll
  for (int k = 0; k < kRows; ++k) lm = fmaxf(lm, x[k]);
  const uint32_t tau = first_tau(sh, w0 < n ? to_key(lm) : 0u, p.m, rank, n_ctas, warp, lane);
  const int n_lane = max(0, min(kRows, (n - w0 + 31) >> 5));  // the lane's entries are a prefix of its slots
  append<kRows>(sh, x, tau, n_lane >= 32 ? 0xffffffffu : (1u << n_lane) - 1u, n_ctas > 1, lane, [&](int k) { return c0 + w0 + k * 32; },
                [&](int k) {
                  float v = x[0];
#pragma unroll
                  for (int i = 1; i < kRows; ++i) v = k == i ? x[i] : v;
                  return v;
                });
  finish_row<kRows>(p, sh, rowp, n, c0, rank, n_ctas, row);
}

// Whether a CTA's list is thinned behind stage st: when 2, 4, 8, ... stages have been seen and more follow.
__device__ __forceinline__ bool thins_behind(int st, int n_st) { return ((st + 1) & st) == 0 && st > 0 && st + 1 < n_st; }
// For a warp whose wait for stage st gave up: it takes no further stage but comes to the same barriers as the others.
__device__ __noinline__ void thin_with_the_others(TopmShared& sh, int m, int tid, int st, int n_st) {
  for (; st < n_st; ++st)
    if (thins_behind(st, n_st)) {
      worker_sync();
      if (sh.cnt <= kList) thin_list(sh, m, tid);
    }
}

// The row streamed through shared memory, 8192 entries of a CTA at a time.
__global__ void __launch_bounds__(kStreamThreads + 32, 3) tree_topm_stream_kernel(const __grid_constant__ TopmParams p) {
  extern __shared__ __align__(128) unsigned char stream_buf[];
  __shared__ __align__(16) TopmShared sh;
  __shared__ __align__(8) StreamBars bars;
  static_assert(kStreamThreads == kTopmThreads, "the list passes count on 256 working threads");
  const int row = blockIdx.y, rank = blockIdx.x, n_ctas = gridDim.x;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int m = p.m, c0 = rank * p.chunk_len;
  const int n = max(0, min(p.vocab, c0 + p.chunk_len) - c0);
  const float* rowp = p.logits + static_cast<int64_t>(row) * p.logits_stride + c0;
  const RowStream rs(rowp, n, stream_buf, &bars);
  if (tid == kStreamThreads) {
    sh.cnt = 0;
    sh.tau = 0xffffffffu;
    RowStream::init(&bars);
  }
  __syncthreads();
  row_arrive(n_ctas);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int n_st = rs.stages();
  if (warp == kStreamWarps) {
    // The cluster barriers of first_tau() count this warp too: it goes through them once the ring is full, and
    // has left before the next one (all stages are issued by the time the last is taken).
    if (lane == 0) rs.produce(0, min(n_st, kStreamStages), p.stall);
    __syncwarp();
    if (n_ctas > 1) {
      row_wait(n_ctas);
      row_arrive(n_ctas);
      row_wait(n_ctas);
    }
    if (lane == 0) rs.produce(min(n_st, kStreamStages), n_st, p.stall);
    return;
  }
  {
    float x[kStreamLane];
    bool ok = n_st == 0 || rs.take(0, x);
    float lm = -INFINITY;
    if (n_st > 0 && ok) {
#pragma unroll
      for (int k = 0; k < kStreamLane; ++k) lm = fmaxf(lm, x[k]);
    }
    uint32_t tau = first_tau(sh, n_st > 0 && ok && rs.index(0, 0, 0) < rs.body ? to_key(lm) : 0u, m, rank, n_ctas, warp, lane);
    // the up to six entries outside the copies
    if (warp == 0) {
      const bool in = lane < rs.head + rs.tail;
      const int i = lane < rs.head ? lane : lane + rs.body;
      const float xe[1] = {in ? __ldcs(rowp + i) : -INFINITY};
      append<1>(sh, xe, tau, in ? 1u : 0u, false, lane, [&](int) { return c0 + i; }, [&](int) { return xe[0]; });
    }
    int st = 0;
    for (; ok && st < n_st; ++st) {
      if (st > 0) {
        ok = rs.take(st, x);
        if (!ok) break;
        lm = -INFINITY;
#pragma unroll
        for (int k = 0; k < kStreamLane; ++k) lm = fmaxf(lm, x[k]);
      }
      if (tau <= to_key(-INFINITY) || __any_sync(0xffffffffu, to_key(lm) >= tau))
        append<kStreamLane>(sh, x, tau, rs.live(st), false, lane, [&](int k) { return c0 + rs.head + rs.index(st, k >> 2, k & 3); },
                            [&](int k) { return rs.value(st, k); });
      rs.give_back(st);
      if (thins_behind(st, n_st)) {
        worker_sync();
        if (sh.cnt <= kList) tau = max(tau, thin_list(sh, m, tid));  // (beyond: the exact route)
      }
    }
    if (!ok) thin_with_the_others(sh, m, tid, st, n_st);
    if (!ok && lane == 0) atomicAdd(&sh.cnt, kList + 1);  // a wait gave up: the exact route reads the row itself
  }
  worker_sync();
  if (n_ctas > 1) {  // the CTA's own survivors to CTA 0 (which keeps its own where they are)
    const int mine = sh.cnt;
    row_arrive(n_ctas);       // every list is complete: CTA 0's may be appended to
    row_wait(n_ctas);
    if (rank != 0) {
      const uint32_t cnt0 = peer_addr(&sh.cnt, 0), list0 = peer_addr(&sh.list[0], 0);
      for (int j0 = warp * 32; j0 < min(mine, kList); j0 += kStreamThreads) {
        const int some = min(32, mine - j0);
        int base = 0;
        if (lane == 0) base = peer_add(cnt0, some);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (lane < some && base + lane < kList) peer_store64(list0 + 8 * (base + lane), sh.list[j0 + lane]);
      }
      if (mine > kList && tid == 0) peer_add(cnt0, kList + 1);  // overflowed: so does the sum
    }
  }
  finish_row<kStreamLane>(p, sh, rowp, n, c0, rank, n_ctas, row);
}

}  // namespace

cudaError_t set_up_topm() {
  cudaError_t e = prefer_shared(tree_topm_kernel<8>);
  if (e == cudaSuccess) e = prefer_shared(tree_topm_kernel<16>);
  if (e == cudaSuccess) e = prefer_shared(tree_topm_kernel<kTopmRowsMax>);
  if (e == cudaSuccess) e = prefer_shared(tree_topm_stream_kernel);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(tree_topm_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kStreamBytesMax));
  return e;
}

int launch_tree_topm(falcon_ctx* ctx, const falcon_topm_args& a, cudaStream_t s) {
  const int N = a.n_rows;
  if (N > 65535) return FALCON_ERR_CAPACITY;
  TopmParams p;
  p.vocab = a.vocab;
  p.m = a.m;
  p.stall = ctx->test_stall_stage;
  p.logits_stride = a.logits_stride;
  p.logits = a.logits;
  p.top_val = a.top_val;
  p.top_idx = a.top_idx;

  // Rows in registers while the whole grid is resident at once (six CTAs per SM with 8 entries per lane, four with 16,
  // three with 32): the shortest chain.  A cluster costs more than it shares out wherever one CTA's registers hold the row:
  // 1.2 us at once, and more with every cluster the GPU has to place.  So as few CTAs per row as the registers allow,
  // four while there are at most 96 of them, eight below 64 (us with 1 / 2 / 4 / 8: 16 rows of 3000 2.8 / 3.5 / 3.7 /
  // 11.7, 48 of 8000 3.3 / 4.2 / 4.3 / 4.8, 4 of 16000 - / 3.9 / 3.6 / 3.5, 16 of 16000 - / 4.0 / 3.7 / 4.1, 32 of
  // 16000 - / 4.1 / 4.2 / 4.4, 4 of 32000 - / - / 3.9 / 3.7, 48 of 32000 - / - / 4.9 / 5.6).
  // Else streamed, three CTAs per SM: a second wave of the register kernel starts its loads only when a
  // first one has gone through its barriers.
  int ctas = 1, per_lane = 0, chunk = 0;
  auto split = [&](int c) {
    ctas = c;
    chunk = ((a.vocab + c - 1) / c + 3) & ~3;
    per_lane = (chunk + kTopmThreads - 1) / kTopmThreads;
  };
  auto room = [&](int of, ScanKernel which, const void* kernel, int threads, uint32_t smem) {
    return cluster_room(N, of, clusters_at_once(ctx, which, kernel, threads, smem, of));
  };
  auto fits = [&]() {
    return per_lane <= 8    ? room(ctas, kScanTopm8, reinterpret_cast<const void*>(tree_topm_kernel<8>), kTopmThreads, 0)
           : per_lane <= 16 ? room(ctas, kScanTopm16, reinterpret_cast<const void*>(tree_topm_kernel<16>), kTopmThreads, 0)
                            : room(ctas, kScanTopm32, reinterpret_cast<const void*>(tree_topm_kernel<kTopmRowsMax>), kTopmThreads, 0);
  };
  auto streams = [&](int of) {
    return room(of, kScanTopmStream, reinterpret_cast<const void*>(tree_topm_stream_kernel), kStreamThreads + 32, kStreamBytes);
  };
  int c = 1;
  while (c < kTopmMaxCluster && a.vocab > c * kTopmThreads * kTopmRowsMax) c *= 2;
  if (c > 1 && c < 4 && N * 4 <= 96) c = 4;
  if (c > 1 && c < 8 && N * 8 < 64) c = 8;
  // Eight again for the rows at which the SMs would no longer take the clusters of four evenly, as long as the clusters of eight
  // are placed at once, for any length (us with 4 / 8, alone and behind an attention launch; 16385, 24577 and 32768 entries):
  //   50 rows  5.4 / 5.9  18.0 / 17.9      5.8 / 6.2  18.6 / 18.1      6.1 / 6.5  18.9 / 18.4
  //   52       5.4 / 5.9  18.1 / 17.9      5.9 / 6.2  18.6 / 18.1      6.1 / 6.5  18.9 / 18.5
  //   53       6.0 / 5.9  18.1 / 17.9      6.6 / 6.3  18.7 / 18.2      6.9 / 6.5  19.1 / 18.5
  //   61       6.3 / 6.1  18.2 / 18.4      6.8 / 6.5  18.8 / 18.6      7.2 / 6.7  19.1 / 18.8
  //   62       6.3 / 6.2  18.2 / 18.5      6.8 / 6.5  18.8 / 18.9      7.2 / 6.8  19.1 / 19.2
  //   64       6.3 / 6.8  18.2 / 19.4      6.9 / 6.9  18.8 / 19.7      7.2 / 7.1  19.2 / 20.1
  // (below 53 rows the two regimes disagree, and four stay)
  const int64_t rows = N, sm = ctx->sm_count;
  if (c == 4 && 100 * 4 * rows > 142 * sm && 10 * 8 * rows <= 33 * sm) {
    split(8);
    if (fits()) c = 8;
  }
  // (two stages of one CTA against two CTAs' registers: 48 rows of 16000 4.6 and 4.4 us, 64 of 12000 4.6 and 5.0, 120 5.2 and 6.0)
  const bool short_stream = a.vocab > kStreamStage && a.vocab <= 2 * kStreamStage && N >= 56;
  split(c);
  const bool in_regs = !short_stream && per_lane <= kTopmRowsMax && fits();
  if (!in_regs) {
    // CTAs of a cluster where the rows alone leave SMs idle: four and eight wherever they have room (us with 1 / 2 / 4 CTAs: logits in L2,
    // not in L2, and behind an attention launch):
    //   60 rows of 40000  8.2 / 7.9 / 7.6   8.4 / 8.0 / 7.7   20.2 / 19.0 / 17.8    87 of 40000  8.2 / 8.7 / 7.8   9.1 / 9.8 / 9.1  23.7 / 22.7 / 21.8
    //   100 of 49152      9.0 / 8.9 / 8.2   9.9 / 10.2 / 10.0  25.3 / 23.8 / 24.7   100 of 131072  19.2 / 16.1 / 14.4  19.4 / 16.2 / 15.4  35.7 / 29.8 / 30.2
    // Two (1 / 2 CTAs):
    //   up to nine tenths of a row per SM, where the pairs are given two places per SM: rows of more than seven stages
    //     105 of 32768  6.9 / 7.2   7.8 / 8.2  22.8 / 22.0     120 of 57344  9.8 / 10.0  11.2 / 11.7  26.8 / 25.4
    //     120 of 64000 10.6 / 10.3 12.1 / 11.9 27.8 / 25.7     133 of 106496 17.4 / 15.7 17.5 / 15.9  37.9 / 34.2
    //   up to one: more than thirteen
    //     148 of 64000 10.8 / 12.5 12.5 / 14.4 33.5 / 32.9     148 of 106496 17.7 / 18.6 17.7 / 18.7 39.0 / 37.6     131072 20.4 / 20.1  20.5 / 20.1  42.1 / 38.9
    //   beyond: more than ten
    //     149 of 32768  8.4 / 8.2   9.6 / 10.2 28.6 / 28.9     170 of 64000  13.4 / 12.8  14.6 / 15.1  34.1 / 33.8   90112  18.0 / 17.7  18.1 / 17.8  40.5 / 37.0
    //     222 of 64000 15.0 / 16.7 15.1 / 16.8 36.4 / 37.5     222 of 90112  18.7 / 19.8  18.7 / 20.0  42.9 / 40.7
    c = 1;
    while (c < kTopmMaxCluster && streams(2 * c) && a.vocab >= 2 * c * kStreamStage) c *= 2;
    if (c == 2 && a.vocab <= (10 * rows <= 9 * sm ? 7 : rows <= sm ? 13 : 10) * kStreamStage) c = 1;
    split(c);
  }
  p.chunk_len = chunk;

  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas, N);
  cfg.blockDim = dim3(kTopmThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = ctas > 1 ? 2 : 1;
  cudaError_t e;
  if (in_regs) {
    p.steps = 1;
    e = per_lane <= 8    ? cudaLaunchKernelEx(&cfg, tree_topm_kernel<8>, p)
        : per_lane <= 16 ? cudaLaunchKernelEx(&cfg, tree_topm_kernel<16>, p)
                         : cudaLaunchKernelEx(&cfg, tree_topm_kernel<kTopmRowsMax>, p);
  } else {
    p.steps = (chunk + kTopmThreads * kStreamLane - 1) / (kTopmThreads * kStreamLane);
    cfg.blockDim = dim3(kStreamThreads + 32);
    cfg.dynamicSmemBytes = stream_bytes(static_cast<int64_t>(N) * ctas, ctas, chunk, ctx->sm_count);
    e = cudaLaunchKernelEx(&cfg, tree_topm_stream_kernel, p);
  }
  if (e != cudaSuccess) return cuda_fail(ctx, e, "tree_topm_kernel launch");
  return FALCON_OK;
}

}  // namespace falcon
