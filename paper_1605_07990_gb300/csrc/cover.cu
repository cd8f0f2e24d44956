// RR pool counts, greedy Max-Coverage (Algorithm 2), coverage checks (Eq. 1)
// and the Estimate-Inf first-T search (Algorithm 3) on sm_103a.
//
// Counts: cnt[v] = number of sets holding v, one pass over the flat (node,
// sample) entries; sets added later are counted on top.
// Greedy: one persistent kernel for all k picks.  Gains only fall, so the
// nodes of the largest counts hold the next picks; their sets alone are laid
// out per pick (candidate lists) and one block then picks out of its own
// shared memory (see k_greedy).
#include <atomic>
#include <mutex>

#include <cooperative_groups.h>

#include "device.cuh"

namespace ssa {

namespace {

constexpr int TPB = 256;

// samp == nullptr: every entry in [e0, e1) counts; else only samples in [jlo, jhi)
// Hubs appear in a large share of the sets, so the lanes of a
// warp that hold the same node are grouped (labeled_partition) and one of
// them issues the group's atomic: one atomic per distinct node per warp
// instead of one per entry on the hub's counter.
__global__ void k_count_nodes(const int32_t* __restrict__ nodes, const int32_t* __restrict__ samp, int64_t e0,
                              int64_t e1, int64_t jlo, int64_t jhi, int32_t* cnt) {
  namespace cg = cooperative_groups;
  for (int64_t q = e0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < e1; q += (int64_t)gridDim.x * blockDim.x) {
    if (samp) {
      const int64_t s = samp[q];
      if (s < jlo || s >= jhi) continue;
    }
    const int32_t v = nodes[q];
    const cg::coalesced_group same = cg::labeled_partition(cg::coalesced_threads(), v);
    if (same.thread_rank() == 0) atomicAdd(cnt + v, (int)same.size());
  }
}

// ---- block-wide helpers ----
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T x, T* s_warp, T* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  T incl = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const T t = __shfl_up_sync(FULL_MASK, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    T w = lane < nw ? s_warp[lane] : (T)0;
    T wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const T t = __shfl_up_sync(FULL_MASK, wi, d);
      if (lane >= d) wi += t;
    }
    if (lane < nw) s_warp[lane] = wi - w;
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  const T r = s_warp[wid] + incl - x;
  __syncthreads();
  return r;
}

// ---- WRIS prefix sums ----
constexpr int PREFIX_TILE = 4096;  // 1024 threads x 4

__device__ __forceinline__ void load_weights(const uint32_t* w, int64_t n, unsigned long long (&x)[4],
                                             unsigned long long* sum) {
  const int64_t base = (int64_t)blockIdx.x * PREFIX_TILE + (int64_t)threadIdx.x * 4;
  *sum = 0;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    x[t] = base + t < n ? w[base + t] : 0u;
    *sum += x[t];
  }
}

__global__ void __launch_bounds__(1024) k_weight_tiles(const uint32_t* w, int64_t n, unsigned long long* part) {
  __shared__ unsigned long long s_w[32], s_tot;
  unsigned long long x[4], sum;
  load_weights(w, n, x, &sum);
  block_exclusive_scan<unsigned long long>(sum, s_w, &s_tot);
  if (threadIdx.x == 0) part[blockIdx.x] = s_tot;
}

// out[v] = w[0] + ... + w[v - 1], out[n] the total; every block adds up the tiles
// before its own (256 of them at 2^20 nodes, 8,192 at 2^25; quadratic in n)
__global__ void __launch_bounds__(1024) k_weight_prefix(const uint32_t* w, int64_t n, const unsigned long long* part,
                                                        uint64_t* out) {
  __shared__ unsigned long long s_w[32], s_tot, s_before;
  unsigned long long before = 0;
  for (int64_t i = threadIdx.x; i < blockIdx.x; i += blockDim.x) before += part[i];
  block_exclusive_scan<unsigned long long>(before, s_w, &s_tot);
  if (threadIdx.x == 0) s_before = s_tot;
  __syncthreads();
  unsigned long long x[4], sum;
  load_weights(w, n, x, &sum);
  unsigned long long ex = s_before + block_exclusive_scan<unsigned long long>(sum, s_w, &s_tot);
  const int64_t base = (int64_t)blockIdx.x * PREFIX_TILE + (int64_t)threadIdx.x * 4;
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (base + t < n) out[base + t] = ex;
    ex += x[t];
    if (base + t == n - 1) out[n] = ex;
  }
}

// ---- greedy ----

// maximum over the block of x, in every thread
__device__ __forceinline__ unsigned long long block_max(unsigned long long x, unsigned long long* s) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int d = 16; d; d >>= 1) {
    const unsigned long long t = __shfl_xor_sync(FULL_MASK, x, d);
    x = t > x ? t : x;
  }
  if (lane == 0) s[wid] = x;
  __syncthreads();
  if (wid == 0) {
    x = lane < nw ? s[lane] : 0ull;
#pragma unroll
    for (int d = 16; d; d >>= 1) {
      const unsigned long long t = __shfl_xor_sync(FULL_MASK, x, d);
      x = t > x ? t : x;
    }
    if (lane == 0) s[0] = x;
  }
  __syncthreads();
  x = s[0];
  __syncthreads();
  return x;
}

// sync layout: arrival count, release word, error flag and block 0's progress on
// separate 128-byte lines so that polling does not contend with the arrivals.
constexpr int SYNC_COUNT = 0, SYNC_GEN = 32, SYNC_ERR = 64, SYNC_PROGRESS = 96;
constexpr int ARGMAX_STRIDE = 16;  // 64-bit words: argmax slots one 128-byte line apart
constexpr int GCANDS = GREEDY_CANDS;  // candidates of one session: their gains, ids and list offsets fill 192 KB
constexpr int GBITS = 14;          // a candidate's key: gain above, GCANDS - 1 - local id in the low GBITS
constexpr int GMAX = 1 << (32 - GBITS);
constexpr int GBINS = 1024;        // histogram bins
constexpr int SCANDS = 4096;       // candidates and list entries of a session that fits shared memory whole:
constexpr int SENTS = 24576;       // keys, ids, offsets, lengths (12 bytes a candidate), lists (6 an entry)
constexpr int STHREADS = 256;      // threads that make its picks
constexpr int GHISTS = 4;          // histograms in turn, so that one is cleared while another fills
constexpr int GSHARE = 4096;       // sets of a list from which every block covers a share of them (two grid barriers
                                   // and adding up a turn; 820,000 IC sets, k = 300: 3.7 ms alone and from 2,048
                                   // sets on, 3.0 from 4,096 on)
constexpr int GLONG = 256;         // members of a set beyond which its list is made by several warps

// Grid barrier for a cooperative launch.  The last block to arrive runs f()
// (all its threads; f sees every block's writes from before the barrier) and
// publishes the result (< 2^63) in the release word beside a sense bit (bit 0,
// flipped by each release), so every waiter learns it from the poll that
// releases it; all threads get it in `info`.  A wait gives up after `limit`
// polls (about a second by default) without progress, sets sync[SYNC_ERR] and
// returns false; that block then leaves the kernel, and the others give up at
// their next barrier, which it never reaches.  Progress is the word that block 0
// moves while it makes a session's picks alone (every few picks, and every 128 or
// 512 sets of one): a session may take thousands of picks, and the bound has to
// span one step of them, not the session.  Every block passes every barrier in
// the same order, so each keeps the current sense in its shared wait[0] (0 at
// launch, when the release word is zero) instead of reading it back, and in
// wait[1] the progress it saw last.
template <class F>
__device__ __forceinline__ bool grid_barrier(unsigned int* sync, unsigned int* wait, long long limit, F&& f,
                                             unsigned long long& info) {
  __shared__ unsigned long long s_info;
  __shared__ unsigned int s_last, s_ok, s_sense;
  volatile unsigned long long* gw = reinterpret_cast<volatile unsigned long long*>(sync + SYNC_GEN);
  __syncthreads();
  if (threadIdx.x == 0) {
    s_sense = wait[0];
    wait[0] = s_sense ^ 1u;
    s_ok = 1;
    __threadfence();
    const bool last = atomicAdd(sync + SYNC_COUNT, 1u) + 1u == gridDim.x;
    if (last) {
      atomicExch(sync + SYNC_COUNT, 0u);
      __threadfence();
    }
    s_last = last;
  }
  __syncthreads();
  if (s_last) {
    const unsigned long long r = f();
    if (threadIdx.x == 0) {
      atomicExch((unsigned long long*)gw, (r << 1) | (unsigned long long)(s_sense ^ 1u));
      s_info = r;
    }
  } else if (threadIdx.x == 0) {
    unsigned long long w;
    unsigned int ns = 8;
    for (long long spins = 0; (unsigned int)((w = *gw) & 1ull) == s_sense; ++spins) {
      if (spins > limit) {
        const unsigned int p = *(volatile unsigned int*)(sync + SYNC_PROGRESS);
        if (p == wait[1]) {
          atomicExch(sync + SYNC_ERR, 1u);
          s_ok = 0;
          break;
        }
        wait[1] = p;
        spins = 0;
      }
      __nanosleep(ns);
      if (ns < 128) ns <<= 1;
    }
    s_info = w >> 1;
    __threadfence();
  }
  __syncthreads();
  info = s_info;
  return s_ok != 0u;
}

// The greedy's barrier.  GRID: grid_barrier across a cooperative launch.
// CLUSTER: the whole greedy runs in one thread-block cluster, so the barrier is
// the hardware cluster barrier; block 0 then computes f() and the others read
// its result from block 0's shared memory (distributed shared memory) after a
// second cluster barrier.  A cluster barrier always completes (the cluster's
// blocks are scheduled together), so it has no bound to reach.
template <bool CLUSTER, class F>
__device__ __forceinline__ bool greedy_barrier(const GreedyJob& J, unsigned int* wait, F&& f,
                                               unsigned long long& info) {
  if constexpr (!CLUSTER) {
    if (gridDim.x == 1) {  // a single block needs no waits
      __syncthreads();
      info = f();
      __syncthreads();
      return true;
    }
    return grid_barrier(J.sync, wait, J.wait_polls, f, info);
  } else {
    namespace cg = cooperative_groups;
    __shared__ unsigned long long s_res;
    cg::cluster_group cluster = cg::this_cluster();
    __threadfence();  // this block's global writes and atomics before the others look
    cluster.sync();
    if (cluster.block_rank() == 0) {
      const unsigned long long r = f();
      if (threadIdx.x == 0) s_res = r;
    }
    cluster.sync();
    info = *cluster.map_shared_rank(&s_res, 0);
    return true;
  }
}

// Packed key: larger gain first, then smaller id; picked nodes (negative gain)
// key to 0.  With gains below 2^31 - 1 and ids below 2^31, keys stay below 2^62.
__device__ __forceinline__ unsigned long long gain_key(int32_t c, uint32_t v) {
  return c < 0 ? 0ull : (((unsigned long long)(uint32_t)(c + 1)) << 31) | (unsigned long long)(0x7FFFFFFFu - v);
}
__device__ __forceinline__ int32_t key_node(unsigned long long key) {
  return (int32_t)(0x7FFFFFFFu - (uint32_t)(key & 0x7FFFFFFFull));
}
__device__ __forceinline__ int32_t key_gain(unsigned long long key) { return (int32_t)(key >> 31) - 1; }
// the smallest key of gain g (any id)
__device__ __forceinline__ unsigned long long gain_floor_key(int32_t g) {
  return ((unsigned long long)(uint32_t)(g + 1)) << 31;
}

// Histogram bin of a gain: exact below 64, then 32 bins per octave.
__device__ __forceinline__ int gain_bin(int32_t g) {
  if (g < 64) return g;
  const int e = 31 - __clz(g);
  return 64 + (e - 6) * 32 + ((g >> (e - 5)) & 31);
}
// smallest gain of a bin (2^31 - 1 past the last gain)
__device__ __forceinline__ int32_t bin_gain(int b) {
  if (b < 64) return b;
  const int e = 6 + (b - 64) / 32;
  if (e > 30) return 0x7FFFFFFF;
  return (int32_t)((32u + (uint32_t)(b & 31)) << (e - 5));
}

// Sets [0, n_sets) not covered yet, cut into runs of `bs` per warp; each warp
// deals the members of its run's sets to its lanes 32 at a time whatever the
// sets' sizes (median 1, largest 10^4), four rounds in flight.
//   begin(j, start, len): the lane holds set j (len 0: none; it may be set to
//     0 to leave the set out); once per run
//   item(node, owner, base, excl, incl): in round t of four the lane holds
//     member node[t] (-1: none) of the set of lane owner[t]; the run's members
//     count from 0, the round's first is base + 32 t, and the lane's own set
//     holds [excl, incl)
//   finish(j, len)
template <class Begin, class Item, class Finish>
__device__ __forceinline__ void for_live_members(const GreedyJob& J, int64_t warp, int64_t nwarps, int lane,
                                                 Begin&& begin, Item&& item, Finish&& finish) {
  int bs = 32;
  while (bs > 1 && (int64_t)bs * nwarps > J.n_sets) bs >>= 1;
  for (int64_t j0 = warp * bs; j0 < J.n_sets; j0 += nwarps * bs) {
    const int64_t j = j0 + lane;
    int len = 0;
    int64_t start = 0;
    if (lane < bs && j < J.n_sets) {
      const uint8_t was = J.covered[j];
      len = J.set_len[j];
      start = J.set_start[j];
      if (was) len = 0;
    }
    if (!__any_sync(FULL_MASK, len > 0)) continue;
    begin(j, start, len);
    const int incl = warp_inclusive_scan(len, lane);
    const int excl = incl - len;
    const int total = __shfl_sync(FULL_MASK, incl, 31);
    for (int b = 0; b < total; b += 128) {
      int32_t node[4];
      int own[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int q = b + 32 * t + lane;
        int o = 0;
#pragma unroll
        for (int s = 16; s; s >>= 1) {
          const int x = __shfl_sync(FULL_MASK, incl, o + s - 1);
          if (x <= q) o += s;
        }
        o = o > 31 ? 31 : o;
        own[t] = o;
        const int64_t at = __shfl_sync(FULL_MASK, start, o) + (q - __shfl_sync(FULL_MASK, excl, o));
        node[t] = q < total ? __ldg(J.pool_nodes + at) : -1;
      }
      item(node, own, b, excl, incl);
    }
    finish(j, len);
  }
}

// Persistent greedy: all k picks of Algorithm 2 in one launch (a cooperative
// grid, one cluster, or a single block for small pools).
//
// Sessions.  Gains only fall.  A session takes the nodes of key (gain, ~id)
// >= key* -- up to GCANDS of them, key* from a histogram over all n counts --
// as candidates: while the best candidate's key is >= key*, it beats every
// node outside, ties included, so the picks never look outside.  The sets not
// covered yet are read once and written as candidate lists: per set the local
// ids of its candidates, in 16-byte chunks (first {count:16, set:32} and four
// 16-bit ids, then eight per chunk), and per candidate the list of its sets'
// chunks.  This also gives every candidate's exact gain, whatever the counts
// that chose it.  Then block 0 alone makes the picks: gains in its shared
// memory, each thread keeping the best of its candidates, a pick's argmax two
// warp reductions and a block barrier; the pick's sets are read eight lanes to
// a set, their count set to 0 (covered) and their candidates' gains lowered by
// shared-memory atomics.  A pick costs two dependent L2 round trips and two
// block barriers, no grid barrier and no atomic in global memory.  When the
// best candidate falls below key*, the counts of all nodes are taken again
// over the sets left and the next session starts.
//
// The first pick of a large pool goes by a pass over the flat entries instead
// (`bulk`): it covers by far the most members (59% of the entries of 1.15M
// weighted-cascade sets on the 2^25-node R-MAT graph, nearly all of a
// trivalency pool's), which then need no list.  The first session after it
// still chooses candidates by the counts before it: any upper bound on the
// gains outside is a valid key*, and a recount is saved.
//
// Bound: the chain of a pick (two L2 round trips of ~600 clocks, two block
// barriers, the argmax over shared memory), 1.5 us while a pick covers tens of
// sets; picks that cover thousands load the issue slots of the one SM (a member
// is three instructions: chunks hold byte offsets of keys), whose ALU pipe is
// busy for 12% (IC, 1000 picks) to 24% (LT, 500) of a launch.  The blocks of a
// large pool's greedy (SHARE) cover such a pick together.  Measured on
// GB300 against the former design (an inverted index of all entries, a grid
// barrier of ~6 us per pick): 1000 picks over 134,016 sets of the 2^23-node
// R-MAT graph 8.7 -> 2.3 ms, 500 over 131,832 LT sets there 6.0 -> 2.1 ms, 100
// over 1,149,440 sets of the 2^25-node one 3.5 -> 2.0 ms, each with its index
// (0.2, 0.3 and 1.6 ms) gone.  Byte offsets and fewer candidates where few picks
// are left: all rounds of the second 5.6 -> 5.1 ms, of the first 7.7 -> 7.3 ms.
//
// With many picks to go and gains of some hundreds at most, the candidates and
// all their lists fit shared memory (`small`: SCANDS candidates, SENTS entries):
// eight warps then pick without a load from memory.  The 1000 picks above went
// from 1.81 to 1.28 ms a round with it (a session of 1.5 us picks ends after 64
// of them where 192 are left; one that served fewer than 96 is not tried again).
//
// Where the lists of a session do not fit (2^25 chunks are room for every member
// of 17M small sets), the next ones are `tight`: the members are looked at twice
// and only sets that hold a candidate get room.  SSA over 33.7M sets (809M
// entries) of the 2^23-node graph, k = 1000: 244 ms, 3,661 with the best node's
// sets covered by a pass over the pool instead; room for 2^27 chunks: 268 ms.
//
// Gains of 0 go by smallest id.  Barrier waits are bounded (sync[SYNC_ERR] on
// timeout).  Between two barriers block 0 may make up to GCANDS picks, tens of
// milliseconds; it shows its progress, and the bound is on polls that see none.
template <bool CLUSTER, bool SHARE>
__global__ void __launch_bounds__(1024, 1) k_greedy(GreedyJob J) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ unsigned long long s_red[32];
  __shared__ long long s_scan[32], s_scan_tot;
  __shared__ unsigned int s_wait[2];  // sense of the next grid barrier, block 0's progress at the last look
  __shared__ unsigned int s_w[2][32];
  unsigned int* s_key = reinterpret_cast<unsigned int*>(s_dyn);  // block 0 in a session: keys (gain, ~local id),
  unsigned int* s_id = s_key + GCANDS;                           // node ids
  unsigned int* s_off = s_id + GCANDS;                           // and list offsets of the candidates
  unsigned int* s_hist = reinterpret_cast<unsigned int*>(s_dyn);     // otherwise: the histogram
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t gtid = blockIdx.x * (int64_t)blockDim.x + tid;
  const int64_t gthreads = (int64_t)gridDim.x * blockDim.x;
  const int64_t warp = gtid >> 5, nwarps = gthreads >> 5;
  const int64_t n4 = J.n_pad >> 2;
  int n_argmax = 0, n_hist = 0, i = 0;
  bool first = true, bulk = J.bulk_first != 0, flat = false, small_off = false, tight = false;
  if (tid == 0) s_wait[0] = s_wait[1] = 0u;  // the host zeroed the release word (sense 0) and the progress
  unsigned long long info = 0;

  // One pass over the gains: histogram of bin(key) (-1: not counted) merged
  // into the next global histogram, and the largest key into the next argmax
  // slot, which the barrier publishes in `info`.
  // exact_bins: bin(key) is gain_bin of every gain.
  auto scan_gains = [&](const int32_t* cnt, bool exact_bins, auto&& bin, unsigned int** hist) -> bool {
    for (int t = tid; t < GBINS; t += blockDim.x) s_hist[t] = 0u;
    __syncthreads();
    unsigned long long best = 0;
    // most nodes are in no set, one or two: those are counted in registers
    unsigned int ones = 0, twos = 0;
    int32_t one = -1, two = -1;  // the thread's first (smallest) of each
    auto take = [&](int64_t q, const int4& c) {
      const int32_t cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (exact_bins) {
          const bool is1 = cv[u] == 1, is2 = cv[u] == 2;
          ones += is1;
          twos += is2;
          if (is1 && one < 0) one = (int32_t)(q * 4 + u);
          if (is2 && two < 0) two = (int32_t)(q * 4 + u);
        }
        if (cv[u] > (exact_bins ? 2 : 0)) {
          const unsigned long long key = gain_key(cv[u], (uint32_t)(q * 4 + u));
          best = key > best ? key : best;
          const int b = bin(cv[u], key);
          if (b >= 0) atomicAdd(s_hist + b, 1u);
        }
      }
    };
    const int4* c4 = reinterpret_cast<const int4*>(cnt);
    int64_t q = gtid;
    for (; q + 3 * gthreads < n4; q += 4 * gthreads) {  // four loads in flight
      const int4 a = c4[q], b = c4[q + gthreads], c = c4[q + 2 * gthreads], d = c4[q + 3 * gthreads];
      take(q, a);
      take(q + gthreads, b);
      take(q + 2 * gthreads, c);
      take(q + 3 * gthreads, d);
    }
    for (; q < n4; q += gthreads) take(q, c4[q]);
    if (ones) atomicAdd(s_hist + 1, ones);
    if (twos) atomicAdd(s_hist + 2, twos);
    if (best == 0ull && (ones || twos)) best = twos ? gain_key(2, (uint32_t)two) : gain_key(1, (uint32_t)one);
    __syncthreads();
    unsigned int* h = J.hist + (size_t)(n_hist % GHISTS) * GBINS;
    for (int t = tid; t < GBINS; t += blockDim.x)
      if (s_hist[t]) atomicAdd(h + t, s_hist[t]);
    best = block_max(best, s_red);
    unsigned long long* at = J.argmax + (n_argmax % 3) * ARGMAX_STRIDE;
    if (tid == 0 && best) atomicMax(at, best);
    if (!greedy_barrier<CLUSTER>(J, s_wait, [&] { return __ldcg(at); }, info)) return false;
    // clear the slot and the histogram of two scans on: nobody has touched
    // them since the barrier before this one
    if (blockIdx.x == 0) {
      if (tid == 0) J.argmax[((n_argmax + 2) % 3) * ARGMAX_STRIDE] = 0ull;
      unsigned int* z = J.hist + (size_t)((n_hist + 2) % GHISTS) * GBINS;
      for (int t = tid; t < GBINS; t += blockDim.x) z[t] = 0u;
    }
    n_argmax += 1;
    n_hist += 1;
    *hist = h;
    return true;
  };
  // The lowest bin b such that, with `have` nodes of `sum` list entries taken
  // already, the nodes of bins >= b still fit (cap_n nodes, cap_e list entries;
  // top(b): largest gain of bin b).  Returns b, adds what they take to
  // have and sum; *total: nodes in all bins.
  long long cap_n = GCANDS, cap_e = J.ents_cap;
  auto cut = [&](const unsigned int* hist, auto&& top, long long& have, long long& sum, long long* total) -> int {
    const int b = GBINS - 1 - tid;  // 1024 threads: one bin each, from the top
    const long long c = __ldcg(hist + b);
    const long long e = c ? c * (long long)top(b) : 0;
    const long long ic = block_exclusive_scan<long long>(c, s_scan, &s_scan_tot) + c;
    *total = s_scan_tot;
    __syncthreads();
    const long long is = block_exclusive_scan<long long>(e, s_scan, &s_scan_tot) + e;
    const bool fits = have + ic <= cap_n && sum + is <= cap_e;
    // bins fit from the top down to the first that does not
    const unsigned long long n_fit = GBINS - block_max(fits ? 0ull : (unsigned long long)(GBINS - tid), s_red);
    __shared__ long long s_have, s_sum;
    if (n_fit > 0 && tid == (int)n_fit - 1) {
      s_have = ic;
      s_sum = is;
    }
    __syncthreads();
    if (n_fit > 0) {
      have += s_have;
      sum += s_sum;
    }
    __syncthreads();
    return GBINS - (int)n_fit;
  };

  for (;;) {
    // ---- candidates: key* and the best node ----
    const int32_t* cnt = first ? J.cnt0 : J.cnt;
    unsigned int* hist = nullptr;
    if (!scan_gains(cnt, true, [](int32_t c, unsigned long long) { return gain_bin(c); }, &hist)) return;
    const unsigned long long best = info;
    if (best == 0ull) {  // no gain is left
      flat = true;
      break;
    }
    const int32_t vstar = key_node(best);
    const bool wide = key_gain(best) >= GMAX;  // gains that a session's keys cannot hold
    bulk = bulk || wide;
    if (bulk) {
      if (blockIdx.x == 0 && tid == 0) {
        J.seeds[i] = vstar;
        J.gains[i] = key_gain(best);
      }
      i += 1;
      if (i == J.k) break;
      // every set that holds v* is covered (four entries a thread and load)
      const int64_t q4n = J.total_entries >> 2;
      const int4* e4 = reinterpret_cast<const int4*>(J.pool_nodes);
      if (SHARE && !first) {
        // Past the first pick, which covers most members: a warp that comes on such a
        // set takes its members off the gains, and no recount of all that are left
        // follows.  SSA under LT over 20.7M sets (815M entries, 2^20 nodes), k = 50,
        // some of whose picks cover more sets than a key holds: 279 -> 222 ms.
        auto cover_entry = [&](int64_t q, bool mine) {  // warp-uniform call
          int32_t s = mine ? __ldg(J.pool_samp + q) : -1;
          if (mine && (s >= J.n_sets || J.covered[s])) s = -1;
          if (s >= 0) J.covered[s] = 1;
          for (unsigned int m = __ballot_sync(FULL_MASK, s >= 0); m; m &= m - 1u) {
            const int32_t j = __shfl_sync(FULL_MASK, s, __ffs(m) - 1);
            const int64_t start = J.set_start[j];
            const int len = J.set_len[j];
            for (int x = lane; x < len; x += 32) atomicSub(J.cnt + __ldg(J.pool_nodes + start + x), 1);
          }
        };
        for (int64_t q0 = gtid - lane; q0 < q4n; q0 += gthreads) {
          const int64_t q = q0 + lane;
          const int4 e = q < q4n ? __ldg(e4 + q) : make_int4(-1, -1, -1, -1);
          if (!__any_sync(FULL_MASK, e.x == vstar || e.y == vstar || e.z == vstar || e.w == vstar)) continue;
          const int32_t ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) cover_entry(q * 4 + u, ev[u] == vstar);
        }
        if (warp == 0) {  // at most three entries
          const int64_t q = q4n * 4 + lane;
          cover_entry(q, q < (int64_t)J.total_entries && __ldg(J.pool_nodes + q) == vstar);
        }
        if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
        if (blockIdx.x == 0 && tid == 0) J.cnt[vstar] = -1;
        if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
        bulk = false;
        continue;
      }
      for (int64_t q = gtid; q < q4n; q += gthreads) {
        const int4 e = __ldg(e4 + q);
        const int32_t ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (ev[u] == vstar) {
            const int32_t s = __ldg(J.pool_samp + q * 4 + u);
            if (s < J.n_sets) J.covered[s] = 1;
          }
      }
      for (int64_t q = q4n * 4 + gtid; q < (int64_t)J.total_entries; q += gthreads)
        if (__ldg(J.pool_nodes + q) == vstar) {
          const int32_t s = __ldg(J.pool_samp + q);
          if (s < J.n_sets) J.covered[s] = 1;
        }
    }
    const bool session = !bulk || (first && !wide);  // else recount before the next session
    unsigned long long keystar = 0;
    const bool small = session && !first && !small_off && J.k - i >= 64 && key_gain(best) <= SENTS / 64;
    const int i0 = i;
    if (session) {
      // exact counts: some dozens of candidates a pick serve, and the fewer there
      // are, the cheaper an argmax (the counts before a bulk pick need them all)
      const long long few = max(2048ll, 32ll * (J.k - i));
      cap_n = small ? SCANDS : first && bulk ? GCANDS : min((long long)GCANDS, few);
      cap_e = small ? SENTS : (long long)J.ents_cap;
      if (tight) cap_e = min(cap_e, (long long)(J.chunk_cap / 3));  // a set takes 2.5 chunks a candidate at most
      long long have = 0, sum = 0, total = 0;
      int b = cut(hist, [](int x) { return bin_gain(x + 1) - 1; }, have, sum, &total);
      b = max(b, 1);
      keystar = gain_floor_key(bin_gain(b));
      // too few: cut the bin below by key until some of it fits
      unsigned long long lo = b > 1 ? gain_floor_key(bin_gain(b - 1)) : keystar, hi = keystar;
      while (have < 64 && have < total && lo < hi) {
        if ((lo >> 31) == ((hi - 1) >> 31))  // one gain: only ids below n occur
          lo = max(lo, ((lo >> 31) << 31) | (unsigned long long)(0x7FFFFFFFu - (uint32_t)(J.n - 1)));
        const unsigned long long width = (hi - lo + GBINS - 1) / GBINS;
        const int32_t g_hi = key_gain(hi - 1);
        if (!scan_gains(cnt, false, [=](int32_t, unsigned long long key) {
              return key >= lo && key < hi ? (int)((key - lo) / width) : -1;
            }, &hist)) return;
        long long in_range = 0;
        b = cut(hist, [=](int) { return g_hi; }, have, sum, &in_range);
        keystar = min(hi, lo + (unsigned long long)b * width);
        hi = keystar;
        lo = b > 0 && width > 1 ? lo + (unsigned long long)(b - 1) * width : hi;
      }
      // ---- the candidates get local ids and list space ----
      const int4* c4 = reinterpret_cast<const int4*>(cnt);
      const int32_t gmin = key_gain(keystar);
      const int32_t skip = bulk ? vstar : -1;
      // marked first, then numbered in id order, so that of equal gains the
      // smaller local id is the smaller node id.  Block b numbers the mark words
      // [b * per, (b + 1) * per); a warp's 128 nodes are four words of one block.
      // (Counted per block in shared memory first: hubs with neighbouring ids
      // would queue on one global counter.)
      const unsigned int words = (unsigned int)((J.n_pad + 31) >> 5);
      const unsigned int per = (words + 4 * gridDim.x - 1) / (4 * gridDim.x) * 4;
      unsigned int* s_blk = reinterpret_cast<unsigned int*>(s_dyn);
      if (tid < (int)gridDim.x) s_blk[tid] = 0u;
      __syncthreads();
      auto select = [&](int64_t q, const int4& c) {
        const bool any = c.x >= gmin || c.y >= gmin || c.z >= gmin || c.w >= gmin;
        if (!any) return;
        const uint32_t v = (uint32_t)(q * 4);
        const int32_t cv[4] = {c.x, c.y, c.z, c.w};
        unsigned int take = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (cv[u] > 0 && gain_key(cv[u], v + u) >= keystar && (int32_t)(v + u) != skip) take |= 1u << u;
        if (!take) return;
        atomicOr(J.mark + (v >> 5), take << (v & 31u));
        atomicAdd(s_blk + (v >> 5) / per, (unsigned int)__popc(take));
      };
      int64_t q = gtid;
      for (; q + 3 * gthreads < n4; q += 4 * gthreads) {  // four loads in flight
        const int4 a = c4[q], b = c4[q + gthreads], c = c4[q + 2 * gthreads], d = c4[q + 3 * gthreads];
        select(q, a);
        select(q + gthreads, b);
        select(q + 2 * gthreads, c);
        select(q + 3 * gthreads, d);
      }
      for (; q < n4; q += gthreads) select(q, c4[q]);
      __syncthreads();
      if (tid < (int)gridDim.x && s_blk[tid]) atomicAdd(J.blk + tid, s_blk[tid]);
      if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
      int nc;
      {
        const long long own_b = tid < (int)gridDim.x ? (long long)__ldcg(J.blk + tid) : 0ll;
        const long long before = block_exclusive_scan<long long>(own_b, s_scan, &s_scan_tot);
        nc = (int)s_scan_tot;
        __shared__ int s_base;
        if (tid == (int)blockIdx.x) s_base = (int)before;
        __syncthreads();
        // a run of words per thread
        const unsigned int wpt = (per + 1023) >> 10;
        const unsigned int w0 = min(words, blockIdx.x * per + tid * wpt);
        const unsigned int w1 = min(min(words, (blockIdx.x + 1) * per), w0 + wpt);
        int c = 0;
        for (unsigned int w = w0; w < w1; ++w) c += __popc(J.mark[w]);
        int l = s_base + (int)block_exclusive_scan<long long>((long long)c, s_scan, &s_scan_tot);
        if (c)
          for (unsigned int w = w0; w < w1; ++w) {
            for (unsigned int m = J.mark[w]; m; m &= m - 1u) {
              const unsigned int v = (w << 5) + (unsigned int)__ffs(m) - 1u;
              J.cand_id[l] = (int32_t)v;
              J.lid[v] = (uint16_t)(++l);
            }
            J.mark[w] = 0u;
          }
      }
      if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
      // list space, as many entries as the count that chose the candidate
      for (int t0 = (int)blockIdx.x * 1024; t0 < nc; t0 += (int)gridDim.x * 1024) {
        const int t = t0 + tid;
        const long long g = t < nc ? (long long)cnt[J.cand_id[t]] : 0ll;
        const long long at = block_exclusive_scan<long long>(g, s_scan, &s_scan_tot);
        __shared__ unsigned int s_list;
        if (tid == 0) s_list = atomicAdd(J.ncand + 4, (unsigned int)s_scan_tot);
        __syncthreads();
        if (t < nc) {
          J.cand_len[t] = 0;
          J.cand_off[t] = s_list + (unsigned int)at;
        }
        __syncthreads();
      }
      if (blockIdx.x == 0 && tid == 0) J.ncand[0] = (unsigned int)nc;
      if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
      // ---- candidate lists of the sets left ----
      // a member's local id (1 + id, 0: no candidate) goes to its place `r` in
      // the set's chunks at cs, as the byte offset of its key in shared memory, and
      // the chunks to the candidate's list
      auto put = [&](unsigned int l, unsigned int cs, unsigned int off, int pos, int r) {
        reinterpret_cast<uint16_t*>(J.chunks + cs)[4 + r] = (uint16_t)((l - 1u) * 4u);
        J.ents[off + (unsigned int)pos] = cs;
      };
      unsigned int cs = 0;  // this lane's set: its first chunk
      int run = 0;          // and the candidates found so far
      bool over = false;
      for_live_members(
          J, warp, nwarps, lane,
          [&](int64_t j, int64_t start, int& len) {
            // room for every member: chunks are cheap (2 bytes a member) and a counting pass is not
            int room = len;
            if (tight) {  // that did not fit: room for the candidates only
              room = 0;
              if (len <= 32)
                for (int x = 0; x < len; ++x) room += J.lid[__ldg(J.pool_nodes + start + x)] != 0;
              for (unsigned int m = __ballot_sync(FULL_MASK, len > 32); m; m &= m - 1u) {
                const int o = __ffs(m) - 1, end = __shfl_sync(FULL_MASK, len, o);
                const int64_t at = __shfl_sync(FULL_MASK, start, o);
                int c = 0;
                for (int x = lane; x < end; x += 32) c += J.lid[__ldg(J.pool_nodes + at + x)] != 0;
                c = __reduce_add_sync(FULL_MASK, c);
                if (lane == o) room = c;
              }
              if (room == 0) len = 0;
            }
            const int nch = room ? ((room + 19) >> 4) * 2 : 0;
            const int incl = warp_inclusive_scan(nch, lane);
            unsigned long long at = 0;
            if (lane == 31) at = atomicAdd(J.nchunk, (unsigned long long)incl);
            at = __shfl_sync(FULL_MASK, at, 31);
            over = at + (unsigned long long)__shfl_sync(FULL_MASK, incl, 31) > J.chunk_cap;
            cs = (unsigned int)(at + (unsigned long long)(incl - nch));
            run = 0;
            // a long set would keep its warp long after the others: its parts go to the
            // queue (which has a place for every 16 chunks: not where room is tight)
            if (len > GLONG && !over && !tight) {
              const unsigned int parts = (unsigned int)((len + GLONG - 1) / GLONG);
              const unsigned int t0 = atomicAdd(J.ncand + 3, parts);
              *reinterpret_cast<uint2*>(J.chunks + cs) = make_uint2(0u, (unsigned int)j);
              for (unsigned int t = 0; t < parts; ++t) J.tasks[t0 + t] = make_uint4(cs, (unsigned int)j, t * GLONG, 0u);
              len = 0;
            }
          },
          [&](const int32_t* node, const int* own, int b0, int excl, int incl) {
            if (over) return;
            unsigned int l[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) l[t] = node[t] >= 0 ? J.lid[node[t]] : 0u;
            int pos[4];
            unsigned int off[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
              if (l[t]) {
                off[t] = J.cand_off[l[t] - 1u];
                pos[t] = atomicAdd(J.cand_len + (l[t] - 1u), 1);
              }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const int b = b0 + 32 * t;
              const unsigned int m = __ballot_sync(FULL_MASK, l[t] != 0u);
              if (m == 0u) continue;
              const int o = own[t];
              // the owner's members of this round sit in lanes [max(excl - b, 0), min(incl - b, 32))
              const int oex = __shfl_sync(FULL_MASK, excl, o);
              const unsigned int ocs = __shfl_sync(FULL_MASK, cs, o);
              const int orun = __shfl_sync(FULL_MASK, run, o);
              const int f = max(oex - b, 0);
              if (l[t]) {
                const unsigned int below = ((1u << lane) - 1u) & (FULL_MASK << f);
                put(l[t], ocs, off[t], pos[t], orun + __popc(m & below));
              }
              const int s0 = min(max(excl - b, 0), 32), s1 = min(max(incl - b, 0), 32);
              const unsigned int upto = s1 >= 32 ? FULL_MASK : (1u << s1) - 1u;
              const unsigned int from = s0 >= 32 ? 0u : FULL_MASK << s0;
              run += __popc(m & upto & from);
            }
          },
          [&](int64_t j, int len) {
            if (over) {
              if (lane == 0) atomicExch(J.ncand + 1, 1u);
            } else if (len > 0 && run > 0) {
              *reinterpret_cast<uint2*>(J.chunks + cs) = make_uint2((unsigned int)run, (unsigned int)j);
            }
          });
      if (!greedy_barrier<CLUSTER>(J, s_wait, [&] {
            return ((unsigned long long)__ldcg(J.ncand + 1) << 32) | (unsigned long long)__ldcg(J.ncand + 3);
          }, info)) return;
      const unsigned int ntasks = (unsigned int)info;
      if (ntasks > 0u && (info >> 32) == 0ull) {
        // parts of the long sets, a warp each: places in the set's chunks by its running count
        for (int64_t q = warp; q < ntasks; q += nwarps) {
          const uint4 t = J.tasks[q];
          const int64_t start = J.set_start[t.y];
          const int end = min(J.set_len[t.y], (int)t.z + GLONG);
          unsigned int l[GLONG / 32];
          int mine = 0;
#pragma unroll
          for (int u = 0; u < GLONG / 32; ++u) {
            const int x = (int)t.z + u * 32 + lane;
            l[u] = x < end ? (unsigned int)__ldg(J.pool_nodes + start + x) : 0xFFFFFFFFu;
          }
#pragma unroll
          for (int u = 0; u < GLONG / 32; ++u) {
            l[u] = l[u] != 0xFFFFFFFFu ? J.lid[l[u]] : 0u;
            mine += l[u] != 0u;
          }
          const int mi = warp_inclusive_scan(mine, lane);
          int r = 0;
          if (lane == 31 && mi) r = (int)atomicAdd(reinterpret_cast<unsigned int*>(J.chunks + t.x), (unsigned int)mi);
          r = __shfl_sync(FULL_MASK, r, 31) + mi - mine;
#pragma unroll
          for (int u = 0; u < GLONG / 32; ++u)
            if (l[u]) put(l[u], t.x, J.cand_off[l[u] - 1u], atomicAdd(J.cand_len + (l[u] - 1u), 1), r++);
        }
        if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
        info = 0ull;
      } else {
        info >>= 32;
      }
    }
    // lists that did not fit: tight ones next, and if it is not that, the best node's sets first
    const bool retry = session && info != 0ull && !tight;
    bool overflow = session && info != 0ull;
    // ---- the session's picks ----
    if (session) {
      const int nc = (int)__ldcg(J.ncand);
      overflow = overflow || nc == 0;
      // thread 0, at every pick and at every further step of one
      auto progress = [&](unsigned int step) {
        if (!CLUSTER) __stcg(J.sync + SYNC_PROGRESS, (unsigned int)(i + 1) * 0x9E3779B1u + step);
      };
      // Picks out of lists in memory: block 0 picks and covers.  With SHARE it covers
      // the sets of a short list itself; a list of GSHARE sets or more ends its turn: at
      // a barrier the blocks learn the pick, each covers a share of the list and lowers
      // a copy of the keys in its own shared memory (0 at first), and what the others
      // lowered adds up in cand_dec, which block 0 subtracts behind a second barrier.
      const int ncp = (nc + 1023) & ~1023;
      // Slots `slot` and `slot` + 1 of a list of cnt.  Picks that cover thousands
      // of sets load an SM's issue slots: three instructions a member (the pick's
      // own key goes down to gain 0 with the others).
      auto lower = [&](unsigned int pair, int slot, int cnt) {
        if (slot < cnt) atomicSub(reinterpret_cast<unsigned int*>(s_dyn + (pair & 0xFFFFu)), 1u << GBITS);
        if (slot + 1 < cnt) atomicSub(reinterpret_cast<unsigned int*>(s_dyn + (pair >> 16)), 1u << GBITS);
      };
      // the sets of list [off, off + len) from place `base` on in steps of `stride`
      // (warp-uniform; cs: the lane's first), 2^sh lanes a set
      auto cover = [&](const unsigned int off, const int len, int base, const int stride, unsigned int cs, const int sh,
                       const bool own) {
        const int per_set = 1 << sh, r0 = lane & (per_set - 1), first_slots = 8 * per_set - 4;
        for (; base < len; base += stride) {
          if (base > 0 && tid == 0 && own) progress((unsigned int)base);
          const unsigned int c0 = cs;
          if (base + stride < len) cs = __ldcg(J.ents + off + base + stride + (lane >> sh));
          uint4 a = make_uint4(0u, 0u, 0u, 0u);
          if (base + (lane >> sh) < len) a = __ldcg(J.chunks + c0 + r0);  // may run past the list: spare chunks
          const int cnt_l = (int)__shfl_sync(FULL_MASK, a.x, lane & ~(per_set - 1));  // 0: covered
          if (r0 == 0) {
            if (cnt_l) {
              J.covered[a.y] = 1;
              *reinterpret_cast<unsigned int*>(J.chunks + c0) = 0u;
            }
          } else {
            lower(a.x, 8 * r0 - 4, cnt_l);
            lower(a.y, 8 * r0 - 2, cnt_l);
          }
          lower(a.z, 8 * r0, cnt_l);
          lower(a.w, 8 * r0 + 2, cnt_l);
          // what is left of the warp's sets is dealt to the lanes chunk by chunk
          const int rest = r0 == 0 && cnt_l > first_slots ? (cnt_l - first_slots + 7) >> 3 : 0;
          if (!__any_sync(FULL_MASK, rest)) continue;
          const int incl = warp_inclusive_scan(rest, lane);
          const int total = __shfl_sync(FULL_MASK, incl, 31);
          for (int q0 = 0; q0 < total; q0 += 32) {
            const int q = q0 + lane;
            int o = 0;
#pragma unroll
            for (int s = 16; s; s >>= 1) {
              const int x = __shfl_sync(FULL_MASK, incl, o + s - 1);
              if (x <= q) o += s;
            }
            o = o > 31 ? 31 : o;
            const int r = q - (__shfl_sync(FULL_MASK, incl, o) - __shfl_sync(FULL_MASK, rest, o));
            const unsigned int oc = __shfl_sync(FULL_MASK, c0, o);
            const int ocnt = __shfl_sync(FULL_MASK, cnt_l, o);
            if (q < total) {
              const uint4 w = __ldcg(J.chunks + oc + per_set + r);
              lower(w.x, first_slots + 8 * r, ocnt);
              lower(w.y, first_slots + 8 * r + 2, ocnt);
              lower(w.z, first_slots + 8 * r + 4, ocnt);
              lower(w.w, first_slots + 8 * r + 6, ocnt);
            }
          }
        }
      };
      for (bool begun = false;; begun = true) {
        int turn = 0;  // 1 + the pick that ended block 0's turn (0: the session is over)
        if (blockIdx.x == 0 && !overflow && small) {
          // everything into shared memory: the lists of the sets one after the
          // other (count, local ids; count 0: covered), the candidates' lists as
          // places in them
          s_id = s_key + SCANDS;
          unsigned short* s_off16 = reinterpret_cast<unsigned short*>(s_id + SCANDS);
          unsigned short* s_len16 = s_off16 + SCANDS;
          unsigned short* s_ent16 = s_len16 + SCANDS;
          unsigned short* s_mem = s_ent16 + SENTS;
          __shared__ unsigned int s_nmem, s_over;
          if (tid == 0) s_nmem = s_over = 0u;
          const int E = (int)__ldcg(J.ncand + 4);
          for (int t = tid; t < SCANDS; t += 1024) {
            const unsigned int len = t < nc ? (unsigned int)__ldcg(J.cand_len + t) : 0u;
            s_key[t] = t < nc ? (len << GBITS) | (unsigned int)(GCANDS - 1 - t) : 0u;
            s_id[t] = t < nc ? (unsigned int)__ldcg(J.cand_id + t) : 0u;
            s_off16[t] = t < nc ? (unsigned short)__ldcg(J.cand_off + t) : 0;
            s_len16[t] = (unsigned short)len;
          }
          __syncthreads();
          // the first list entry of a set to come (it sets the count's high bit) copies the set
          for (int x0 = tid; x0 < E; x0 += 4096) {
            unsigned int at[4], old[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) at[t] = x0 + 1024 * t < E ? __ldcg(J.ents + x0 + 1024 * t) : 0u;
#pragma unroll
            for (int t = 0; t < 4; ++t)
              old[t] = x0 + 1024 * t < E ? atomicOr(reinterpret_cast<unsigned int*>(J.chunks + at[t]), 0x80000000u)
                                         : 0x80000000u;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              if (old[t] >> 31) continue;
              const unsigned int place = atomicAdd(&s_nmem, old[t] + 1u);
              s_mem[place] = (unsigned short)old[t];
              const unsigned short* ids = reinterpret_cast<const unsigned short*>(J.chunks + at[t]) + 4;
              for (unsigned int y = 0; y < old[t]; ++y) s_mem[place + 1u + y] = __ldcg(ids + y);
              *reinterpret_cast<unsigned int*>(J.chunks + at[t]) = 0x80000000u | place;
            }
          }
          __syncthreads();
          for (int x = tid; x < E; x += 1024)
            s_ent16[x] =
                (unsigned short)__ldcg(reinterpret_cast<const unsigned int*>(J.chunks + __ldcg(J.ents + x)));
          __syncthreads();
          if (tid < STHREADS) {
            // as the picks below, by eight warps and without a load from memory
            auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(STHREADS) : "memory"); };
            unsigned int bk = 0xFFFFFFFFu;
            int par = 0;
            while (i < J.k) {
              if (bk && s_key[(GCANDS - 1 - (bk & (GCANDS - 1))) & (SCANDS - 1)] != bk) {
                bk = 0u;
#pragma unroll
                for (int r = 0; r < SCANDS / STHREADS; ++r) bk = max(bk, s_key[r * STHREADS + tid]);
              }
              const unsigned int wk = __reduce_max_sync(FULL_MASK, bk);
              if (lane == 0) s_w[par][wid] = wk;
              sync();
              const unsigned int top = __reduce_max_sync(FULL_MASK, lane < STHREADS / 32 ? s_w[par][lane] : 0u);
              par ^= 1;
              const int l = GCANDS - 1 - (int)(top & (GCANDS - 1));
              const int g = (int)(top >> GBITS);
              if (top == 0u || gain_key(g, s_id[l]) < keystar) break;
              if (tid == 0) {
                J.seeds[i] = (int32_t)s_id[l];
                J.gains[i] = g;
              }
              const int off = s_off16[l], len = s_len16[l];
              for (int x = tid; x < len; x += STHREADS) {
                const int m = s_ent16[off + x];
                const int c = s_mem[m];
                if (c) s_mem[m] = 0;
                for (int y = 1; y <= c; ++y)
                  atomicSub(reinterpret_cast<unsigned int*>(s_dyn + s_mem[m + y]), 1u << GBITS);
              }
              i += 1;
              sync();
              if (tid == (l & (STHREADS - 1))) s_key[l] = 0u;  // never again
            }
            if (tid == 0) *(volatile unsigned int*)&s_over = 1u;
          } else if (!CLUSTER && tid == STHREADS) {
            // an idle warp shows the progress: every pick lowers the sum of the warps'
            // best keys (a store by the picking warps cost 1% of 1000 picks)
            for (int t = 0; t < (1 << 20) && *(volatile unsigned int*)&s_over == 0u; ++t) {
              unsigned int sum = 0u;
#pragma unroll
              for (int w = 0; w < STHREADS / 32; ++w)
                sum += *(volatile unsigned int*)&s_w[0][w] + *(volatile unsigned int*)&s_w[1][w];
              __stcg(J.sync + SYNC_PROGRESS, sum);
              __nanosleep(1000);
            }
          }
          __syncthreads();
          // the covered flags of the sets whose count is 0 now
          for (int x = tid; x < E; x += 1024)
            if (s_mem[s_ent16[x]] == 0)
              J.covered[__ldcg(reinterpret_cast<const uint2*>(J.chunks + __ldcg(J.ents + x))).y] = 1;
          s_id = s_key + GCANDS;
        } else if (blockIdx.x == 0 && !overflow) {
          if (!begun) {
            for (int t = tid; t < ncp; t += 1024) {
              s_key[t] = t < nc ? ((unsigned int)__ldcg(J.cand_len + t) << GBITS) | (unsigned int)(GCANDS - 1 - t) : 0u;
              s_id[t] = t < nc ? (unsigned int)__ldcg(J.cand_id + t) : 0u;
              s_off[t] = t < nc ? __ldcg(J.cand_off + t) : 0u;
            }
          }
          __syncthreads();
          // best key of the thread's candidates tid, tid + 1024, ...; gains only
          // fall, so it stands until that candidate's own key changes
          unsigned int bk = 0xFFFFFFFFu;
          int par = 0;
          while (i < J.k) {
            if (bk && s_key[GCANDS - 1 - (bk & (GCANDS - 1))] != bk) {
              bk = 0u;
#pragma unroll
              for (int r = 0; r < GCANDS / 1024; ++r)
                if (r * 1024 < ncp) bk = max(bk, s_key[r * 1024 + tid]);
            }
            const unsigned int wk = __reduce_max_sync(FULL_MASK, bk);
            if (lane == 0) s_w[par][wid] = wk;
            __syncthreads();
            const unsigned int top = __reduce_max_sync(FULL_MASK, s_w[par][lane]);
            par ^= 1;
            const int l = GCANDS - 1 - (int)(top & (GCANDS - 1));
            const int g = (int)(top >> GBITS);
            const unsigned int off = s_off[l], v = s_id[l];
            if (top == 0u || gain_key(g, v) < keystar) break;
            // with many picks to go and gains this small, a session out of shared memory is quicker
            if (!small_off && i - i0 >= 64 && J.k - i >= 192 && g <= SENTS / 96) break;
            const int len = __ldcg(J.cand_len + l);
            // lanes per set: eight chunks of each set at once while the sets are few, else two
            const unsigned int spec = __ldcg(J.ents + off + (tid >> 3));  // the buffer has spare entries past the last list
            const int sh = len <= 128 ? 3 : 1;
            const unsigned int cs = sh == 3 ? spec : __ldcg(J.ents + off + (tid >> 1));
            if (tid == 0) {
              J.seeds[i] = (int32_t)v;
              J.gains[i] = g;
              progress(0u);
            }
            if (SHARE && len >= GSHARE) {
              i += 1;
              turn = i < J.k ? l + 1 : 0;  // the last pick's sets need no covering
              break;
            }
            cover(off, len, (tid & ~31) >> sh, 1024 >> sh, cs, sh, true);
            i += 1;
            __syncthreads();
            // never again: its owner, the only thread that reads it, takes it out
            if (tid == (l & 1023)) s_key[l] = 0u;
          }
        }
        if (!begun) {
          // the local ids go back to 0 for the next session
          const int64_t b0 = gridDim.x > 1 ? blockIdx.x - 1 : 0, nb = gridDim.x > 1 ? gridDim.x - 1 : 1;
          if (b0 >= 0)
            for (int64_t t = b0 * 1024 + tid; t < nc; t += nb * 1024) J.lid[__ldcg(J.cand_id + t)] = 0;
          if (SHARE && blockIdx.x != 0 && !overflow && !small)
            for (int t = tid; t < ncp; t += 1024) s_key[t] = 0u;
        }
        if (blockIdx.x == 0 && tid == 0) {
          J.ncand[2] = (unsigned int)i;
          if (SHARE) J.ncand[5] = (unsigned int)turn;
        }
        if (!greedy_barrier<CLUSTER>(J, s_wait, [&] {
              return ((unsigned long long)__ldcg(J.ncand + 2) << 15) | (unsigned long long)__ldcg(J.ncand + 5);
            }, info)) return;
        i = (int)(info >> 15);
        const int l = (int)(info & 0x7FFFull) - 1;
        if (!SHARE || l < 0) break;
        {
          const unsigned int off = __ldcg(J.cand_off + l);
          const int len = __ldcg(J.cand_len + l);
          const int base = (int)blockIdx.x * 512 + ((tid & ~31) >> 1);
          const unsigned int cs = base < len ? __ldcg(J.ents + off + base + (lane >> 1)) : 0u;
          cover(off, len, base, (int)gridDim.x * 512, cs, 1, false);
        }
        __syncthreads();
        if (blockIdx.x != 0)
          for (int t = tid; t < ncp; t += 1024)
            if (s_key[t]) {
              atomicAdd(J.cand_dec + t, (0u - s_key[t]) >> GBITS);
              s_key[t] = 0u;
            }
        if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
        if (blockIdx.x == 0) {
          for (int t = tid; t < ncp; t += 1024) {
            const unsigned int d = __ldcg(J.cand_dec + t);
            if (d) {
              s_key[t] -= d << GBITS;
              __stcg(J.cand_dec + t, 0u);
            }
            if (t == l) s_key[t] = 0u;  // never again
          }
        }
      }
      if (i >= J.k) break;
      if (small && i - i0 < 96) small_off = true;  // it did not pay for its lists
    }
    // ---- gains again over the sets left ----
    for (int64_t q = gtid; q < n4; q += gthreads) reinterpret_cast<int4*>(J.cnt)[q] = make_int4(0, 0, 0, 0);
    if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
    if (blockIdx.x == 0) {
      for (int t = tid; t < i; t += 1024) J.cnt[__ldcg(J.seeds + t)] = -1;  // in no set that is left
      if (tid < (int)gridDim.x) J.blk[tid] = 0u;
      if (tid == 0) {
        J.ncand[1] = J.ncand[3] = J.ncand[4] = 0u;
        *J.nchunk = 0ull;
      }
    }
    for_live_members(
        J, warp, nwarps, lane, [](int64_t, int64_t, int&) {},
        [&](const int32_t* node, const int*, int, int, int) {
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (node[t] >= 0) atomicAdd(J.cnt + node[t], 1);
        },
        [](int64_t, int) {});
    if (!greedy_barrier<CLUSTER>(J, s_wait, [] { return 0ull; }, info)) return;
    bulk = overflow && !retry;
    tight = tight || retry;
    first = false;
  }
  // every gain is 0: the smallest ids not picked yet
  if (flat && blockIdx.x == 0) {
    const int32_t* cnt = first ? J.cnt0 : J.cnt;
    for (int64_t v0 = 0; v0 < J.n && i < J.k; v0 += 1024) {
      const int64_t v = v0 + tid;
      const bool free_v = v < J.n && cnt[v] >= 0;
      const long long at = block_exclusive_scan<long long>(free_v ? 1 : 0, s_scan, &s_scan_tot);
      const long long tot = s_scan_tot;
      __syncthreads();
      if (free_v && i + at < J.k) {
        J.seeds[i + at] = (int32_t)v;
        J.gains[i + at] = 0;
      }
      i = (int)min((long long)J.k, i + tot);
    }
  }
  if constexpr (CLUSTER) {
    // no block may leave while another can still read its shared memory: the
    // payload of the last barrier lives in block 0's
    cooperative_groups::this_cluster().sync();
  }
}

// ---- stare ----
__global__ void k_mark_hits(const int32_t* __restrict__ nodes, const int32_t* __restrict__ samp, int64_t e0,
                            int64_t e1, const uint8_t* __restrict__ in_seed, int64_t j0, int64_t j1, uint8_t* hit) {
  for (int64_t q = e0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < e1;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = samp[q];
    if (s >= j0 && s < j1 && in_seed[nodes[q]]) hit[s - j0] = 1;
  }
}

__global__ void __launch_bounds__(TPB) k_count_flags(const uint8_t* __restrict__ f, int64_t count,
                                                     unsigned long long* out) {
  __shared__ long long s_w[32];
  __shared__ long long s_tot;
  long long c = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    c += f[i];
  block_exclusive_scan<long long>(c, s_w, &s_tot);
  if (threadIdx.x == 0 && s_tot) atomicAdd(out, (unsigned long long)s_tot);
}

constexpr int FR_CHUNK = 4096;

__global__ void __launch_bounds__(1024) k_chunk_counts(const uint8_t* f, int64_t count, long long* part) {
  __shared__ long long s_w[32];
  __shared__ long long s_tot;
  const int64_t base = (int64_t)blockIdx.x * FR_CHUNK;
  long long c = 0;
  for (int i = threadIdx.x; i < FR_CHUNK; i += blockDim.x)
    if (base + i < count) c += f[base + i];
  block_exclusive_scan<long long>(c, s_w, &s_tot);
  if (threadIdx.x == 0) part[blockIdx.x] = s_tot;
}

// Single block: smallest T with prefix(T) >= need (need >= 1).
__global__ void __launch_bounds__(1024) k_find_first(const uint8_t* f, int64_t count, const long long* part,
                                                     int64_t chunks, long long need, long long* out) {
  __shared__ long long s_w[32];
  __shared__ long long s_tot;
  __shared__ long long s_chunk, s_before;
  if (threadIdx.x == 0) {
    s_chunk = -1;
    s_before = 0;
  }
  __syncthreads();
  long long carry = 0;
  for (int64_t b = 0; b < chunks; b += blockDim.x) {
    const int64_t i = b + threadIdx.x;
    const long long x = i < chunks ? part[i] : 0;
    const long long ex = block_exclusive_scan<long long>(x, s_w, &s_tot);
    const long long before = carry + ex;
    if (i < chunks && before < need && before + x >= need) {
      s_chunk = i;
      s_before = before;
    }
    carry += s_tot;
    __syncthreads();
    if (s_chunk >= 0) break;
  }
  const long long total_all = carry;
  const int64_t c = s_chunk;
  long long T = 0;
  if (c >= 0) {
    const int64_t base = c * FR_CHUNK + (int64_t)threadIdx.x * 4;
    long long v[4], loc = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      v[t] = (base + t < count) ? f[base + t] : 0;
      loc += v[t];
    }
    long long ex = s_before + block_exclusive_scan<long long>(loc, s_w, &s_tot);
    __shared__ long long s_T;
    if (threadIdx.x == 0) s_T = 0;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (v[t] && ex < need && ex + 1 >= need) s_T = base + t + 1;
      ex += v[t];
    }
    __syncthreads();
    T = s_T;
  }
  if (threadIdx.x == 0) {
    out[0] = T;
    out[1] = (c >= 0) ? -1 : total_all;  // total only meaningful when not reached
  }
}

// ids outside [0, n) set nothing: a Max-Coverage that gave up at a barrier leaves
// seeds unwritten, and a stare queued behind it reads them before the host knows
__global__ void k_set_bits(const int32_t* ids, int k, int64_t n, uint32_t* bits, uint8_t* bytes) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) {
    const int32_t v = ids[i];
    if (v < 0 || v >= n) continue;
    if (bits) atomicOr(bits + (v >> 5), 1u << (v & 31));
    if (bytes) bytes[v] = 1;
  }
}

__global__ void k_gather_sets(const int32_t* pool_nodes, const int64_t* set_start, const int32_t* set_len,
                              const int64_t* out_off, int64_t first, int64_t count, int32_t* out) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < count; i += nwarps) {
    const int64_t st = set_start[first + i];
    const int32_t len = set_len[first + i];
    const int64_t o = out_off[i];
    for (int t = lane; t < len; t += 32) out[o + t] = pool_nodes[st + t];
  }
}

int grid_stride_blocks(int64_t work, int num_sms, int per_sm = 8) {
  int64_t b = (work + TPB - 1) / TPB;
  if (b > (int64_t)num_sms * per_sm) b = (int64_t)num_sms * per_sm;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st) { return cudaMemsetAsync(p, 0, bytes, st); }

cudaError_t launch_count_nodes(const int32_t* nodes, const int32_t* samp, int64_t e0, int64_t e1, int64_t jlo,
                               int64_t jhi, int32_t* cnt, cudaStream_t st, int num_sms) {
  if (e1 <= e0) return cudaSuccess;
  k_count_nodes<<<grid_stride_blocks(e1 - e0, num_sms), TPB, 0, st>>>(nodes, samp, e0, e1, jlo, jhi, cnt);
  return cudaGetLastError();
}

size_t weight_tmp_words(int64_t n) { return (size_t)((n + PREFIX_TILE - 1) / PREFIX_TILE); }

cudaError_t launch_weight_prefix(const uint32_t* w, int64_t n, uint64_t* out, unsigned long long* tmp,
                                 cudaStream_t st) {
  const unsigned tiles = (unsigned)((n + PREFIX_TILE - 1) / PREFIX_TILE);
  k_weight_tiles<<<tiles, 1024, 0, st>>>(w, n, tmp);
  k_weight_prefix<<<tiles, 1024, 0, st>>>(w, n, tmp, out);
  return cudaGetLastError();
}

namespace {
constexpr int GREEDY_SMEM = GCANDS * 12;  // candidates' gains, ids and list offsets
// Largest cluster of 1024-thread greedy blocks the device can schedule (16 or
// 8), 0 if none; computed once per process.
int greedy_cluster_size() {
  static int size = -1;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  if (size >= 0) return size;
  size = 0;
  for (auto* k : {k_greedy<true, false>, k_greedy<true, true>}) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, GREEDY_SMEM) != cudaSuccess)
      (void)cudaGetLastError();
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      (void)cudaGetLastError();
  }
  for (int c : {16, 8}) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = GREEDY_SMEM;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_greedy<true, true>, &cfg) == cudaSuccess && clusters >= 1) {
      size = c;
      break;
    }
    (void)cudaGetLastError();
  }
  return size;
}
std::atomic<int> g_greedy_mode{0};
}  // namespace

void set_greedy_mode(int mode) { g_greedy_mode.store(mode); }

cudaError_t launch_greedy(const GreedyJob& J, cudaStream_t st, int num_sms, bool shared_gpu) {
  // A solve that shares the GPU with others (serving) runs all picks of a pool
  // of up to GREEDY_CLUSTER_ENTRIES entries in one thread-block cluster: 16 SMs,
  // hardware cluster barriers, and the rest of the GPU free for the other
  // solves.  Otherwise a cooperative grid of one 1024-thread block per SM, or
  // a single block where the passes over counts and entries are too short to
  // share.
  const int mode = g_greedy_mode.load();
  const int csize = mode == 1 ? 0 : greedy_cluster_size();
  const unsigned long long work = (unsigned long long)J.n_pad + J.total_entries;
  const bool share = J.total_entries >= GREEDY_SHARE_ENTRIES;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = GREEDY_SMEM;
  cfg.stream = st;
  cfg.attrs = attr;
  if (mode == 0 && work <= GREEDY_BLOCK_WORK) {
    cfg.gridDim = dim3(1);
  } else if (csize > 0 && (mode == 2 || (shared_gpu && J.total_entries <= GREEDY_CLUSTER_ENTRIES))) {
    cfg.gridDim = dim3(csize);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, share ? k_greedy<true, true> : k_greedy<true, false>, J);
  } else {
    cfg.gridDim = dim3(num_sms);
    // a cooperative launch (all blocks resident at once), also valid inside a stream capture
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.numAttrs = 1;
  }
  auto* k = share ? k_greedy<false, true> : k_greedy<false, false>;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, GREEDY_SMEM);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, k, J);
}

cudaError_t device_code_version(int* binary, int* ptx) {
  cudaFuncAttributes a{};
  const cudaError_t e = cudaFuncGetAttributes(&a, k_greedy<false, false>);
  if (e != cudaSuccess) return e;
  *binary = a.binaryVersion;
  *ptx = a.ptxVersion;
  return cudaSuccess;
}

cudaError_t launch_mark_hits(const int32_t* nodes, const int32_t* samp, int64_t e0, int64_t e1,
                             const uint8_t* in_seed, int64_t j0, int64_t j1, uint8_t* hit, cudaStream_t st,
                             int num_sms) {
  if (e1 <= e0) return cudaSuccess;
  k_mark_hits<<<grid_stride_blocks(e1 - e0, num_sms), TPB, 0, st>>>(nodes, samp, e0, e1, in_seed, j0, j1, hit);
  return cudaGetLastError();
}

cudaError_t launch_count_flags(const uint8_t* flags, int64_t count, unsigned long long* out, cudaStream_t st,
                               int num_sms) {
  if (count <= 0) return cudaSuccess;
  k_count_flags<<<grid_stride_blocks(count, num_sms, 4), TPB, 0, st>>>(flags, count, out);
  return cudaGetLastError();
}

size_t first_reach_tmp_bytes(int64_t count) {
  return sizeof(long long) * (size_t)((count + FR_CHUNK - 1) / FR_CHUNK + 1);
}

cudaError_t launch_first_reach(const uint8_t* flags, int64_t count, long long need, long long* out, void* tmp,
                               cudaStream_t st, int* launches) {
  const int64_t chunks = (count + FR_CHUNK - 1) / FR_CHUNK;
  long long* part = static_cast<long long*>(tmp);
  k_chunk_counts<<<(unsigned)chunks, 1024, 0, st>>>(flags, count, part);
  k_find_first<<<1, 1024, 0, st>>>(flags, count, part, chunks, need, out);
  *launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_set_bits(const int32_t* ids, int k, int64_t n, uint32_t* bits, uint8_t* bytes, cudaStream_t st) {
  if (k <= 0) return cudaSuccess;
  k_set_bits<<<(k + TPB - 1) / TPB, TPB, 0, st>>>(ids, k, n, bits, bytes);
  return cudaGetLastError();
}

cudaError_t launch_gather_sets(const int32_t* pool_nodes, const int64_t* set_start, const int32_t* set_len,
                               const int64_t* out_off, int64_t first, int64_t count, int32_t* out, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  int blocks = (int)((count * 32 + TPB - 1) / TPB);
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_gather_sets<<<blocks, TPB, 0, st>>>(pool_nodes, set_start, set_len, out_off, first, count, out);
  return cudaGetLastError();
}

}  // namespace ssa
