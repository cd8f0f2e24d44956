// RR-set samplers (Definition 2) for IC and LT (Sec. 2.1) on sm_103a.
//
// Tiers share one work list of sample ids:
//   * warp tiers: one warp per sample, visited set as an open-addressing hash
//     (shared memory, or global memory for mid-size sets) or, for weighted
//     cascade, a per-warp n-bit bitmap in global memory; the BFS queue beside
//     it.  Sets that outgrow the queue are handed on (their partial work is
//     dropped).
//   * CTA tier: one CTA per large sample, visited set as an n-bit bitmap
//     (shared memory when it fits, else a per-CTA global slot).
// IC with per-edge thresholds: frontier expansion is edge-balanced inside a
// warp: 32 frontier nodes' in-edge ranges are cut into 4-edge groups (the
// unit of one Philox draw, one aligned 16-byte load of tails) dealt to lanes by
// a warp prefix sum, every group draws its coins, and the live tails are
// visited 32 at a time; the CTA tier shares long in-lists between its warps.
// Bound: integer issue (67% of all issue slots and 60% of the ALU pipe over a
// whole launch of 24,576 trivalency sets; the level barriers are 4% of its
// stalls): 171 instructions per 32 draws, 39 of them Philox.  On the 2^20-node
// R-MAT graph (giant sets of 137,000 nodes) a D-SSA solve went from 366 to 205 ms
// against the form that asked for each tail first, drew for fewer groups (so the
// two forms' draws a second say nothing) and visited slab by slab.
// IC with weighted-cascade weights: every in-edge of a node has the same
// probability, so each lane walks one frontier node's in-list by geometric
// gaps between live edges (the gap form below); the work per node is a
// logarithm per gap and one Philox draw per two, whatever its in-degree.  Bound:
// the three dependent memory round trips of a BFS step.
#include <algorithm>

#include "device.cuh"

namespace ssa {

namespace {

constexpr int WT_WARPS = 8;      // warps per warp-tier block
constexpr int WT_HASH = 1024;    // hash slots per warp (power of two)
constexpr int WT_QCAP = 512;     // largest IC set kept in the warp tier
constexpr int LT_QCAP = 1024;    // largest LT walk kept in the warp tier
constexpr int STAGE = 160;       // live tails waiting for a visit: 31 and those of one slab (32 lanes x 4 edges)
constexpr int CTA_HEAVY_GROUPS = 512;    // the CTA tier splits longer in-lists over all its warps
constexpr int CTA_HEAVY_CAP = 256;       // heavy in-lists per level shared this way
constexpr int SMALL_CTA_THREADS = 128;   // CTAs of the first stage when the visited bitmap is in global memory

// How a sampler kernel learns which edges are live: coins against stored
// thresholds (the LT walk runs in this instantiation too), weighted-cascade
// gaps, or coins against packed trivalency classes.
enum : int { W_COINS = 0, W_GAPS = 1, W_TRI = 2 };
inline int weights_of(const SampleJob& J) {
  if (J.model != 0) return W_COINS;
  return J.wc_implicit ? W_GAPS : J.g.thr ? W_COINS : W_TRI;
}

constexpr uint32_t PHILOX_M0 = 0xD2511F53u, PHILOX_M1 = 0xCD9E8D57u;

// Philox4x32-10 of the counter (x, 0, jlo, cw) with the per-launch round keys
// rk; s0/s1/s2 carry the sample-constant parts of the first round:
// s0 = hi(M1*jlo) ^ rk[0], s1 = lo(M1*jlo), s2 = cw ^ rk[1].
struct SampleConst {
  uint32_t s0, s1, s2;
};

__device__ __forceinline__ SampleConst sample_const(const uint32_t* rk, uint32_t jlo, uint32_t cw) {
  SampleConst c;
  c.s0 = __umulhi(PHILOX_M1, jlo) ^ rk[0];
  c.s1 = PHILOX_M1 * jlo;
  c.s2 = cw ^ rk[1];
  return c;
}

// Rounds 2 to 10.  Both halves of a product come from one 32x32->64 multiply
// (one instruction; asked for as a low and a high product they are two).
__device__ __forceinline__ uint4 philox_rounds(uint4 c, const uint32_t* rk) {
#pragma unroll
  for (int r = 1; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)PHILOX_M0 * c.x, p1 = (uint64_t)PHILOX_M1 * c.z;
    c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ rk[2 * r], (uint32_t)p1,
                   (uint32_t)(p0 >> 32) ^ c.w ^ rk[2 * r + 1], (uint32_t)p0);
  }
  return c;
}

__device__ __forceinline__ uint4 philox_x(uint32_t x, const SampleConst& sc, const uint32_t* rk) {
  // round 1 with c.y = 0 and the sample constants folded in
  const uint64_t p = (uint64_t)PHILOX_M0 * x;
  return philox_rounds(make_uint4(sc.s0, sc.s1, (uint32_t)(p >> 32) ^ sc.s2, (uint32_t)p), rk);
}

// Philox4x32-10 of the counter (x, y, jlo, cw): philox_x with a second
// counter word y, which enters the first round beside the sample constants.
__device__ __forceinline__ uint4 philox_xy(uint32_t x, uint32_t y, const SampleConst& sc, const uint32_t* rk) {
  const uint64_t p = (uint64_t)PHILOX_M0 * x;
  return philox_rounds(make_uint4(sc.s0 ^ y, sc.s1, (uint32_t)(p >> 32) ^ sc.s2, (uint32_t)p), rk);
}

__device__ __forceinline__ int64_t sample_at(const SampleJob& J, unsigned long long idx) {
  return J.work_list ? J.work_list[idx] : J.j0 + (int64_t)idx;
}

__device__ __forceinline__ int32_t pick_root(const SampleJob& J, int64_t j) {
  const uint4 r = keyed_draw(J.seed, PURPOSE_ROOT, J.stream, j, 0);
  const int64_t n = J.g.n;
  if (!J.bprefix) return (int32_t)__umulhi(r.x, (uint32_t)n);
  // WRIS (Sec. 6.3.1): the node whose benefit interval holds a 64-bit target
  const uint64_t W = J.bprefix[n];
  const uint64_t r64 = (uint64_t)r.x | ((uint64_t)r.y << 32);
  const uint64_t target = __umul64hi(r64, W);
  int64_t lo = 0, hi = n - 1;
  while (lo < hi) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (J.bprefix[mid + 1] > target) hi = mid; else lo = mid + 1;
  }
  return (int32_t)lo;
}

// Warp-per-sample tiers: 0 = hash and queue in shared memory (sets up to
// 512 nodes), 1 = per-warp hash and queue in global memory (up to 16384
// nodes).  Larger sets go on to the CTA tier.
template <int TIER>
struct Tier;
template <>
struct Tier<0> {
  static constexpr int HBITS = 10, QCAP = WT_QCAP;
};
template <>
struct Tier<1> {
  static constexpr int HBITS = 15, QCAP = 16384;
};
constexpr int MID_HASH = 1 << Tier<1>::HBITS;
constexpr int MID_QSLOTS = Tier<1>::QCAP + 64;  // queue/slot entries per warp (room for one round past the cap)

template <int HBITS>
__device__ __forceinline__ uint32_t hash_slot(uint32_t u) {
  return (u * 0x9E3779B1u) >> (32 - HBITS);
}

// Insert u into a warp's hash set of 2^HBITS slots; true when u was not
// there, with its slot in *slot.
template <int HBITS>
__device__ __forceinline__ bool hash_insert(uint32_t* H, uint32_t u, uint32_t* slot) {
  const uint32_t key = u + 1u;
  uint32_t h = hash_slot<HBITS>(u);
  for (int probe = 0; probe < (1 << HBITS); ++probe) {
    const uint32_t prev = atomicCAS(H + h, 0u, key);
    if (prev == 0u) {
      *slot = h;
      return true;
    }
    if (prev == key) return false;
    h = (h + 1u) & ((1u << HBITS) - 1u);
  }
  return false;  // not reached: the cap and one round's 64 at most, 576 of 1,024 and 16,448 of 32,768 slots
}

// Threshold of a packed trivalency edge (its class in the two high bits).
__device__ __forceinline__ uint32_t tri_thr(uint32_t s) {
  return (s >> 31) ? TRI_THR2 : (s >> 30) ? TRI_THR1 : TRI_THR0;
}

// Live tails wait in a warp's stage (shared memory: STAGE entries and their
// count) until 32 of them are there, so that the visits -- a look at the visited
// set, an atomic, a queue slot -- run with full warps.  A slab of 32 groups
// gives 4 to 5 live tails under trivalency; visited one slab at a time they
// took longer than the coins.
struct Stage {
  uint32_t* buf;
  unsigned int* cnt;
};

// Visit staged tails, 32 at a time; `all`: also the last ones.  Returns the
// warp-uniform "stop" of visit, after which the stage is empty.
template <class Visit>
__device__ __forceinline__ bool drain(const Stage& st, bool all, int lane, Visit&& visit) {
  __syncwarp();
  int n = (int)*(volatile unsigned int*)st.cnt;
  __syncwarp();  // every lane has read the count before a lane's next push raises it
  if (n < 32 && !(all && n > 0)) return false;
  const unsigned lt_mask = (1u << lane) - 1u;
  bool stop = false;
  do {
    const int take = min(n, 32);
    n -= take;
    const uint32_t u = lane < take ? st.buf[n + lane] : NO_NODE;
    stop = visit(u, lt_mask);
  } while (!stop && (n >= 32 || (all && n > 0)));
  __syncwarp();
  if (lane == 0) *st.cnt = stop ? 0u : (unsigned int)n;
  __syncwarp();
  return stop;
}

// Two 4-edge groups per lane, gA and gB of the in-lists [loA, hiA) and
// [loB, hiB) (when vA, vB): coins for their edges (the tails' loads are in
// flight meanwhile), live tails to the stage, full rounds of visits.  Returns
// visit's "stop".  Whether a tail is in the set already is only asked of live
// ones: asking first saves the draws of 43% of the groups of a trivalency set,
// but a warp draws as long as one lane must.
template <bool TRI, class Visit>
__device__ __forceinline__ bool two_groups(const GraphView& g, bool vA, uint32_t gA, uint32_t loA, uint32_t hiA,
                                           bool vB, uint32_t gB, uint32_t loB, uint32_t hiB, const uint32_t* rk,
                                           const SampleConst& sc, int lane, const Stage& st, Visit&& visit) {
  uint4 sA = make_uint4(0u, 0u, 0u, 0u), sB = sA, tA = sA, tB = sA;
  const uint4* src = reinterpret_cast<const uint4*>(g.src);
  const uint4* thr = reinterpret_cast<const uint4*>(g.thr);
  if (vA) sA = __ldg(src + gA);
  if (vB) sB = __ldg(src + gB);
  if (!TRI) {
    if (vA) tA = __ldg(thr + gA);
    if (vB) tB = __ldg(thr + gB);
  }
  const uint4 rA = philox_x(gA, sc, rk), rB = philox_x(gB, sc, rk);
  // edges 4 grp .. 4 grp + 3 that belong to the in-list
  auto inside = [](bool v, uint32_t grp, uint32_t lo, uint32_t hi) -> uint32_t {
    const uint32_t e = grp * 4u;
    const uint32_t a = lo > e ? lo - e : 0u, b = min(hi - e, 4u);
    return v ? (0xFu << a) & ((1u << b) - 1u) : 0u;
  };
  auto live = [](uint32_t need, const uint4& s, const uint4& t, const uint4& r) -> uint32_t {
    uint32_t m = 0;
    if (edge_live(r.x, TRI ? tri_thr(s.x) : t.x)) m |= 1u;
    if (edge_live(r.y, TRI ? tri_thr(s.y) : t.y)) m |= 2u;
    if (edge_live(r.z, TRI ? tri_thr(s.z) : t.z)) m |= 4u;
    if (edge_live(r.w, TRI ? tri_thr(s.w) : t.w)) m |= 8u;
    return m & need;
  };
  auto push = [&](uint32_t m, const uint4& s) {
    constexpr uint32_t SRC = TRI ? TRI_SRC_MASK : 0xFFFFFFFFu;
    if (m) {
      unsigned int at = atomicAdd(st.cnt, (unsigned int)__popc(m));
      if (m & 1u) st.buf[at++] = s.x & SRC;
      if (m & 2u) st.buf[at++] = s.y & SRC;
      if (m & 4u) st.buf[at++] = s.z & SRC;
      if (m & 8u) st.buf[at] = s.w & SRC;
    }
  };
  push(live(inside(vA, gA, loA, hiA), sA, tA, rA), sA);
  if (drain(st, false, lane, visit)) return true;
  push(live(inside(vB, gB, loB, hiB), sB, tB, rB), sB);
  return drain(st, false, lane, visit);
}

// Edge-balanced expansion of up to 32 frontier nodes (lane i holds node v or
// -1): their in-edge ranges are cut into 4-edge groups dealt to lanes by a
// warp prefix sum.  A node with more than heavy_groups groups is first offered
// to take_heavy(v, lo, hi, ng) (per lane); when it takes the node, the node is
// skipped here.  Returns 0, 1 when visit asked to stop, or 2 when
// take_heavy(...) == HEAVY_ABORT for some lane (the caller hands the sample
// on).  Up to 31 live tails stay in the stage.
constexpr int HEAVY_SKIP = 1, HEAVY_ABORT = 2;

template <bool TRI, class Visit, class Heavy>
__device__ __forceinline__ int expand_ic(const GraphView& g, int32_t v, const uint32_t* rk, const SampleConst& sc,
                                         int lane, const Stage& st, unsigned long long& ev, unsigned long long& draws,
                                         int heavy_groups, Visit&& visit, Heavy&& take_heavy) {
  uint32_t lo = 0, hi = 0;  // edge positions fit 32 bits (m < 2^31)
  if (v >= 0) {
    lo = __ldg(g.off + v);
    hi = __ldg(g.off + v + 1);
  }
  int ng = (hi > lo) ? (int)(((hi + 3) >> 2) - (lo >> 2)) : 0;
  int heavy = 0;
  if (ng > heavy_groups) heavy = take_heavy(v, lo, hi, ng);
  if (__any_sync(FULL_MASK, heavy == HEAVY_ABORT)) return 2;
  ev += hi - lo;
  draws += (unsigned long long)ng;
  if (heavy == HEAVY_SKIP) ng = 0;  // expanded by the taker
  // the nodes with groups go to the low lanes (through the stage's upper part,
  // free while fewer than 32 tails wait)
  const unsigned nz = __ballot_sync(FULL_MASK, ng > 0);
  const int nn = __popc(nz);
  if (nn == 0) return 0;
  if (ng > 0) {
    const int r = __popc(nz & ((1u << lane) - 1u));
    st.buf[64 + r] = lo;
    st.buf[96 + r] = hi;
    st.buf[128 + r] = (uint32_t)ng;
  }
  __syncwarp();
  lo = lane < nn ? st.buf[64 + lane] : 0u;
  hi = lane < nn ? st.buf[96 + lane] : 0u;
  ng = lane < nn ? (int)st.buf[128 + lane] : 0;
  __syncwarp();
  const int incl = warp_inclusive_scan(ng, lane);
  const int excl = incl - ng;
  const int total = __shfl_sync(FULL_MASK, incl, 31);
  const uint32_t g0 = (lo >> 2) - (uint32_t)excl;  // group of item q: q + g0
  const unsigned le_mask = 0xFFFFFFFFu >> (31 - lane);
  int before = 0;  // nodes whose first group lies before the slab
  auto owner = [&](int base) -> int {
    const unsigned d = (unsigned)(excl - base);
    const unsigned starts = __reduce_or_sync(FULL_MASK, lane < nn && d < 32u ? 1u << d : 0u);
    const int o = before + __popc(starts & le_mask) - 1;
    before += __popc(starts);
    return o;
  };
  for (int base = 0; base < total; base += 64) {
    const int qA = base + lane, qB = qA + 32;
    const int oA = owner(base), oB = owner(base + 32);
    const uint32_t gA = (uint32_t)qA + __shfl_sync(FULL_MASK, g0, oA);
    const uint32_t gB = (uint32_t)qB + __shfl_sync(FULL_MASK, g0, oB);
    const uint32_t loA = __shfl_sync(FULL_MASK, lo, oA), hiA = __shfl_sync(FULL_MASK, hi, oA);
    const uint32_t loB = __shfl_sync(FULL_MASK, lo, oB), hiB = __shfl_sync(FULL_MASK, hi, oB);
    if (two_groups<TRI>(g, qA < total, gA, loA, hiA, qB < total, gB, loB, hiB, rk, sc, lane, st, visit))
      return 1;
  }
  return 0;
}

// Weighted-cascade threshold of a node with d in-edges: floor(2^32 / d), and
// 0xFFFFFFFF (probability 1) for d = 1.
__device__ __forceinline__ uint32_t wc_threshold(uint32_t d) {
  return d <= 1u ? 0xFFFFFFFFu : (uint32_t)(0x100000000ull / d);
}

// Gap form of weighted cascade.  All d >= 2 in-edges of a node are live with
// p = t / 2^32 (t = wc_threshold(d)), so the run G of dead edges before the
// next live one has P(G >= g) = q^g, q = 1 - p.  In Q64 integers (x in [0,1)
// as floor(x 2^64), products truncated): Q = (2^32 - t) << 32, P_0 = Q,
// P_(i+1) = hi64(P_i * P_i); G(U) sets bits J-1 .. 0 in turn (J the bit
// length of d, so 2^J - 1 >= d), bit i when U < hi64(A * P_i), A the product
// of the powers already taken (P_i alone for the first), which then becomes
// A.  G(U) is the largest g with U < T(g), T(g) the product along g's bits.
__device__ __noinline__ uint32_t wc_gap_exact(uint32_t d, uint64_t U) {
  uint64_t P[31];
  const int J = 32 - __clz((int)d);
  uint64_t p = (0x100000000ull - wc_threshold(d)) << 32;
  for (int i = 0; i < J; ++i) {
    P[i] = p;
    p = __umul64hi(p, p);
  }
  uint64_t A = 0;
  bool first = true;
  uint32_t gap = 0;
  for (int i = J - 1; i >= 0; --i) {
    const uint64_t cand = first ? P[i] : __umul64hi(A, P[i]);
    if (U < cand) {
      A = cand;
      first = false;
      gap |= 1u << i;
    }
  }
  return gap;
}

// G(U) where it is below `left` (the edges that remain), else some value >=
// left.  Most U lie far from every T(g), and there a logarithm in 32 bits
// decides: with L = log_q(U / 2^64), T(g) lies in [q^g (1 - d 2^-59), q^g] 2^64,
// so when floor(L) = g and L is further than d^2 2^-59 (below 2^-19 for the
// d < 2^20 of the table) from every integer, all T up to T(g) lie above U and
// all others at or below it: G = g.  L = y K with y = -log2(U / 2^64) and
// K = inv[d] = -1 / log2(q).  Errors: __log2f 2^-22 (its stated bound on
// [0.5, 2]), the mantissa cut to 23 bits 1.45 2^-23, the roundings of y, K and
// the product 2^-24 each relative; together below K 4.2e-7 + L 1.8e-7, taken
// as K 4.5e-7 + L 2.5e-7 + 4e-6.  Nearer to an integer than that (about one
// draw in 200 at d = 10,000, one in 12 at 2^17) the exact form decides, so the
// results are its results always.  The exact form is J 64-bit products and
// compares (14 at d = 10,000, ~250 instructions, and a row of powers to read);
// this is one load, one logarithm and a dozen 32-bit operations.  Sampling of a
// whole solve on GB300: 33.1 -> 17.1 ms (SSA, 2^25 nodes, 51.5M visits),
// 12.1 -> 6.7 ms (D-SSA, 2^23), 1.55 -> 0.86 ms (SSA, 2^14).
__device__ __forceinline__ uint32_t wc_gap(float K, uint32_t d, uint32_t left, uint64_t U) {
  const uint32_t hi = (uint32_t)(U >> 32);
  const int lz = __clz((int)hi);
  const uint32_t norm = __funnelshift_l((uint32_t)U, hi, (unsigned)lz);  // bit 31 set when hi != 0
  const float m = __uint_as_float(0x3F800000u | ((norm >> 8) & 0x7FFFFFu));
  const float L = ((float)(lz + 1) - __log2f(m)) * K;
  const float e = fmaf(K, 4.5e-7f, fmaf(L, 2.5e-7f, 4e-6f));
  const float f = floorf(L), r = L - f;
  const bool sure = K > 0.f && hi != 0u;
  if (sure && L - e >= (float)left) return left;
  if (sure && r > e && r < 1.f - e) return (uint32_t)f;
  return wc_gap_exact(d, U);
}

// K of in-degree d: the graph's table below 2^wc_inv_k, 0 (always exact) beyond;
// in-degrees 0 and 1 draw no gaps (a graph of those alone has no table)
__device__ __forceinline__ float wc_inv_of(const GraphView& g, uint32_t d) {
  return d >= 2u && d < (1u << g.wc_inv_k) ? __ldg(g.wc_inv + d) : 0.f;
}

// The gap walk of one weighted-cascade node as a state machine: d = 1 is one
// live edge (probability 1, no draw); otherwise gap c takes the 64-bit uniform
// of words 2(c&1), 2(c&1)+1 of the SKIP draw with counter words (v, c >> 1), the
// next live edge is lo + pos + G, and the walk ends when G reaches past the list.
struct GapWalk {
  uint32_t lo = 0, d = 0;   // the node's in-list
  uint32_t pos = 0, k = 0;  // position in it; draws taken
  float K = 0.f;            // -1 / log2(q)
};

__device__ __forceinline__ void walk_begin(GapWalk& w, const GraphView& g, uint32_t lo, uint32_t d) {
  w.lo = lo;
  w.d = d;
  w.pos = 0;
  w.k = 0;
  w.K = wc_inv_of(g, d);
}

// One step: the two gaps of a draw at once, so that a node with at most one
// live edge (three in four) is done in one round and two edges' loads go out
// together.  e0, e1: CSR positions of the live edges found (NO_NODE: none).
// Returns whether the node may still give live edges.
__device__ __forceinline__ bool walk_step(GapWalk& w, int32_t v, const uint32_t* rk, const SampleConst& skc,
                                          unsigned long long& draws, uint32_t& e0, uint32_t& e1) {
  e0 = e1 = NO_NODE;
  if (w.d < 2u) {
    if (w.d == 1u) e0 = w.lo;
    return false;
  }
  const uint4 r = philox_xy((uint32_t)v, w.k, skc, rk);
  ++draws;
  ++w.k;
  uint32_t left = w.d - w.pos;
  uint32_t G = wc_gap(w.K, w.d, left, (uint64_t)r.x | ((uint64_t)r.y << 32));
  if (G >= left) return false;
  e0 = w.lo + w.pos + G;
  w.pos += G + 1u;
  left -= G + 1u;
  if (left == 0u) return false;
  G = wc_gap(w.K, w.d, left, (uint64_t)r.z | ((uint64_t)r.w << 32));
  if (G >= left) return false;
  e1 = w.lo + w.pos + G;
  w.pos += G + 1u;
  return w.pos < w.d;
}

// The last WRING nodes of a warp's queue with their in-lists, in shared memory:
// entry p of the queue at p mod WRING.  (The queue of the global-memory tiers
// is written in any case: it is the RR set.)
constexpr int WRING = 64;
struct WarpRing {
  int32_t* node;  // null: the queue itself is in shared memory
  uint32_t* lo;
  uint32_t* d;
};

// Weighted-cascade BFS of one sample by one warp over its private queue
// Q[0, tail) (head = 0 at the start; the root's ring entry is set): every lane
// holds at most one node and takes one walk step (two gaps) per round; a lane
// whose node is done takes the next queued node at the start of the next round,
// so the lanes stay busy while the queue holds work.  visit(u, lo, d) with two
// tails and their in-lists per lane (NO_NODE: none) appends the new ones to Q
// and the ring and advances tail (which this function reads through the
// reference); it returns "stop".
//
// Near-critical sets are deep and narrow (5000 nodes: over 100 levels), and a
// batch ends with its largest set, so what counts is the chain of dependent
// loads per level: the edge's tail, then the visited bit together with the
// tail's offsets, which are loaded before it is known to be new and wait in the
// ring.  Sampling of a whole solve on GB300, one gap and its offsets on demand
// before: 17.2 -> 13.5 ms (SSA, 2^25 nodes), 6.7 -> 5.0 ms (D-SSA, 2^23).  (More
// warps per SM at 40 or 48 registers gained nothing: the batches' ends wait on
// single sets.)
template <class Visit>
__device__ __forceinline__ void wc_bfs_warp(const GraphView& g, const int32_t* Q, const WarpRing& ring,
                                            const int& tail, const uint32_t* rk, const SampleConst& skc, int lane,
                                            unsigned long long& ev, unsigned long long& draws, Visit&& visit) {
  const unsigned lt_mask = (1u << lane) - 1u;
  int head = 0;
  int32_t v = -1;
  GapWalk w;
  for (;;) {
    __syncwarp();  // queue entries written by other lanes in the last round
    const bool need = v < 0;
    const unsigned nm = __ballot_sync(FULL_MASK, need);
    const int take = min(__popc(nm), tail - head);
    if (need) {
      const int r = __popc(nm & lt_mask);
      if (r < take) {
        const int h = head + r;
        uint32_t lo, d;
        if (tail - h <= WRING) {
          v = ring.node ? ring.node[h & (WRING - 1)] : Q[h];
          lo = ring.lo[h & (WRING - 1)];
          d = ring.d[h & (WRING - 1)];
        } else {
          v = Q[h];
          lo = __ldg(g.off + v);
          d = __ldg(g.off + v + 1) - lo;
        }
        ev += d;
        walk_begin(w, g, lo, d);
      }
    }
    head += take;
    if (!__any_sync(FULL_MASK, v >= 0)) break;  // queue drained, no lane holds a node
    uint32_t u[2] = {NO_NODE, NO_NODE}, lo[2] = {0u, 0u}, hi[2] = {0u, 0u};
    if (v >= 0) {
      uint32_t e0, e1;
      if (!walk_step(w, v, rk, skc, draws, e0, e1)) v = -1;
      if (e0 != NO_NODE) u[0] = __ldg(g.src + e0);
      if (e1 != NO_NODE) u[1] = __ldg(g.src + e1);
#pragma unroll
      for (int t = 0; t < 2; ++t)
        if (u[t] != NO_NODE) {
          lo[t] = __ldg(g.off + u[t]);
          hi[t] = __ldg(g.off + u[t] + 1);
        }
    }
    const uint32_t d[2] = {hi[0] - lo[0], hi[1] - lo[1]};
    if (visit(u, lo, d, lt_mask)) return;
  }
}

__device__ __forceinline__ void flush_stats(Counters* ctr, unsigned long long ev, unsigned long long nv,
                                            unsigned long long dr, int lane, bool cta_tier) {
  ev = warp_sum(ev);
  nv = warp_sum(nv);
  dr = warp_sum(dr);
  if (lane == 0) {
    if (dr) atomicAdd(&ctr->draws, dr);
    if (ev) atomicAdd(&ctr->edge_visits, ev);
    if (nv) atomicAdd(&ctr->node_visits, nv);
    if (cta_tier && ev) atomicAdd(&ctr->cta_edge_visits, ev);
    if (cta_tier && nv) atomicAdd(&ctr->cta_node_visits, nv);
    if (cta_tier && dr) atomicAdd(&ctr->cta_draws, dr);
  }
}

// Reserve `size` pool entries (one thread).  Reservations are handed out in
// increasing position order, so the ones that fit form a prefix; it ends where
// the first one that did not fit starts (ok_end, the least such position), and
// the rest [ok_end, cursor) are re-run by the host from fail_list.
__device__ __forceinline__ bool reserve(const SampleJob& J, int64_t j, int size, unsigned long long* pos) {
  *pos = atomicAdd(&J.ctr->cursor, (unsigned long long)size);
  if (*pos + (unsigned long long)size <= (unsigned long long)J.pool_cap) return true;
  atomicMin(&J.ctr->ok_end, *pos);
  atomicExch(&J.ctr->pool_overflow, 1u);
  const unsigned long long f = atomicAdd(&J.ctr->fail_count, 1ull);
  J.fail_list[f] = j;
  return false;
}

template <typename QT>
__device__ __forceinline__ void warp_store_set(const SampleJob& J, int64_t j, const QT* Q, int size, int lane) {
  unsigned long long pos = 0;
  int ok = 0;
  if (lane == 0) ok = reserve(J, j, size, &pos);
  ok = __shfl_sync(FULL_MASK, ok, 0);
  pos = __shfl_sync(FULL_MASK, pos, 0);
  if (!ok) return;
  for (int i = lane; i < size; i += 32) {
    J.pool_nodes[pos + i] = Q[i];
    J.pool_samp[pos + i] = (int32_t)j;
  }
  if (lane == 0) {
    J.set_start[j] = (int64_t)pos;
    J.set_len[j] = size;
  }
}

template <int MODE, int TIER, int W>
__global__ void __launch_bounds__(WT_WARPS * 32, 4) k_sample_warp_ic(SampleJob J) {
  constexpr bool WC = W == W_GAPS;
  constexpr int HBITS = Tier<TIER>::HBITS, QCAP = Tier<TIER>::QCAP;
  __shared__ __align__(16) uint32_t s_hash[TIER == 0 ? WT_WARPS : 1][TIER == 0 ? WT_HASH : 4];
  __shared__ int32_t s_q[TIER == 0 ? WT_WARPS : 1][TIER == 0 ? WT_QCAP : 4];
  __shared__ uint32_t s_stage[WT_WARPS][WC ? 1 : STAGE];  // the gap walk needs no staging
  __shared__ unsigned int s_staged[WT_WARPS];
  __shared__ uint32_t s_ring[WT_WARPS][WC ? (TIER == 0 ? 2 : 3) * WRING : 1];  // the gap walk's ring
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const WarpRing ring{TIER == 0 ? nullptr : reinterpret_cast<int32_t*>(s_ring[wid] + 2 * WRING), s_ring[wid],
                      s_ring[wid] + WRING};
  const size_t gwarp = (size_t)blockIdx.x * WT_WARPS + wid;
  uint32_t* H = TIER == 0 ? s_hash[wid] : J.mid_hash + gwarp * MID_HASH;
  int32_t* Q = TIER == 0 ? s_q[wid] : J.mid_queue + gwarp * MID_QSLOTS;
  uint32_t* slots = TIER == 0 ? nullptr : J.mid_slots + gwarp * MID_QSLOTS;
  const Stage stage{s_stage[wid], &s_staged[wid]};
  if (lane == 0) s_staged[wid] = 0u;
  if (TIER == 0) {
    uint4* H4 = reinterpret_cast<uint4*>(H);
    for (int i = lane; i < WT_HASH / 4; i += 32) H4[i] = make_uint4(0, 0, 0, 0);
  }
  __syncwarp();
  // tier 0 takes the batch's samples (or those the lane tier listed), tier 1 the ones tier 0 handed over
  const unsigned long long count =
      TIER == 0 ? (J.lane_tier ? *((volatile unsigned long long*)&J.ctr->lane_count) : (unsigned long long)J.count)
                : *((volatile unsigned long long*)&J.ctr->mid_count);
  unsigned long long* work = TIER == 0 ? &J.ctr->work : &J.ctr->mid_work;
  unsigned long long ev = 0, nv = 0, dr = 0;
  for (;;) {
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(work, 1ull);
    idx = __shfl_sync(FULL_MASK, idx, 0);
    if (idx >= count) break;
    const int64_t j = TIER == 0 ? (J.lane_tier ? J.lane_list[idx] : sample_at(J, idx)) : J.mid_list[idx];
    const SampleConst sc = sample_const(J.rk, (uint32_t)j, ctr_word3(WC ? PURPOSE_SKIP : PURPOSE_IC, J.stream, j));
    const int32_t root = pick_root(J, j);
    if (lane == 0) {
      const uint32_t h0 = hash_slot<HBITS>((uint32_t)root);
      H[h0] = (uint32_t)root + 1u;
      Q[0] = root;
      if (TIER == 1) slots[0] = h0;
      if (WC) {
        ring.lo[0] = __ldg(J.g.off + root);
        ring.d[0] = __ldg(J.g.off + root + 1) - ring.lo[0];
        if (TIER == 1) ring.node[0] = root;
      }
    }
    int tail = 1, head = 0;
    bool overflow = false;
    bool hit = (MODE == MODE_HIT) && test_bit(J.seed_bits, (uint32_t)root);
    // tier 1's hand-over size is tuned at run time (at most its queue capacity)
    const int cap = TIER == 0 ? QCAP : min(QCAP, J.mid_cap);
    __syncwarp();
    auto enter = [&](const uint32_t (&u)[2], const uint32_t (&ulo)[2], const uint32_t (&ud)[2],
                     unsigned lt_mask) -> bool {
      bool h = false;
#pragma unroll
      for (int t = 0; t < (WC ? 2 : 1); ++t) {
        if (t == 1 && !__any_sync(FULL_MASK, u[1] != NO_NODE)) break;
        uint32_t slot = 0;
        const bool is_new = (u[t] != NO_NODE) && hash_insert<HBITS>(H, u[t], &slot);
        const unsigned m = __ballot_sync(FULL_MASK, is_new);
        if (is_new) {
          const int pos = tail + __popc(m & lt_mask);
          if (WC) {
            ring.lo[pos & (WRING - 1)] = ulo[t];
            ring.d[pos & (WRING - 1)] = ud[t];
            if (TIER == 1) ring.node[pos & (WRING - 1)] = (int32_t)u[t];
          }
          if (TIER == 0) {
            if (pos < QCAP) Q[pos] = (int32_t)u[t];
          } else {
            Q[pos] = (int32_t)u[t];  // pos <= cap + 63 < QCAP + 64: room for one round past the cap
            slots[pos] = slot;
          }
          if (MODE == MODE_HIT) h |= test_bit(J.seed_bits, u[t]);
        }
        tail += __popc(m);
      }
      if (MODE == MODE_HIT) hit = __any_sync(FULL_MASK, h) || hit;
      if (tail > cap) overflow = true;
      return overflow || hit;
    };
    auto visit = [&](uint32_t u, unsigned lt_mask) -> bool {
      const uint32_t us[2] = {u, NO_NODE}, none[2] = {0u, 0u};
      return enter(us, none, none, lt_mask);
    };
    // a node with a very long in-list needs many warps: hand the sample to the CTA tier
    // (weighted cascade: no in-list is long, its gap walk costs the same at any degree)
    auto to_cta = [](int32_t, uint32_t, uint32_t, int) { return HEAVY_ABORT; };
    bool handoff = false;
    if constexpr (WC) {
      if (!hit) wc_bfs_warp(J.g, Q, ring, tail, J.rk, sc, lane, ev, dr, enter);
    } else {
      while (head < tail && !overflow && !hit) {
        const int cnt = min(32, tail - head);
        __syncwarp();
        const int32_t v = (lane < cnt) ? Q[head + lane] : -1;
        __syncwarp();
        if (expand_ic<W == W_TRI>(J.g, v, J.rk, sc, lane, stage, ev, dr, J.warp_heavy_groups, visit, to_cta) == 2) {
          handoff = true;
          break;
        }
        if (!overflow && !hit) drain(stage, true, lane, visit);
        head += cnt;
      }
    }
    __syncwarp();
    if (handoff) {
      if (lane == 0) {
        *stage.cnt = 0u;
        const unsigned long long b = atomicAdd(&J.ctr->big_count, 1ull);
        J.big_list[b] = j;
      }
    } else if (overflow) {
      if (lane == 0) {
        if (TIER == 0 && J.mid_cap > 0) {
          const unsigned long long b = atomicAdd(&J.ctr->mid_count, 1ull);
          J.mid_list[b] = j;
        } else {
          const unsigned long long b = atomicAdd(&J.ctr->big_count, 1ull);
          J.big_list[b] = j;
        }
      }
    } else {
      if (MODE == MODE_STORE) warp_store_set(J, j, Q, tail, lane);
      else if (lane == 0) J.hit[j - J.j0] = hit ? 1 : 0;
      if (lane == 0) nv += (unsigned long long)tail;
    }
    __syncwarp();
    if (TIER == 0) {
      uint4* H4 = reinterpret_cast<uint4*>(H);
      for (int i = lane; i < WT_HASH / 4; i += 32) H4[i] = make_uint4(0, 0, 0, 0);
    } else {
      // clear only the slots this sample used (tail <= QCAP + 64 entries recorded)
      for (int i = lane; i < tail; i += 32) H[slots[i]] = 0u;
    }
    __syncwarp();
  }
  flush_stats(J.ctr, ev, nv, dr, lane, false);
}

// Weighted-cascade IC, one warp per sample of up to GQ_CAP nodes (or mid_cap,
// when set), with the visited set as a per-warp n-bit bitmap in global memory
// and the BFS queue in global memory: one tier for every set size up to the
// queue, where the hash tiers stop at 512 and 16384 nodes.  Larger sets go to
// the CTA tier.
constexpr int GQ_CAP = 1 << 16;
constexpr int GQ_SLOTS = GQ_CAP + 64;  // room for one round past the cap

template <int MODE>
__global__ void __launch_bounds__(WT_WARPS * 32, 4) k_sample_warp_wcg(SampleJob J) {
  __shared__ uint32_t s_ring[WT_WARPS][3 * WRING];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const WarpRing ring{reinterpret_cast<int32_t*>(s_ring[wid] + 2 * WRING), s_ring[wid], s_ring[wid] + WRING};
  const size_t gwarp = (size_t)blockIdx.x * WT_WARPS + wid;
  uint32_t* bits = J.wg_bitmap + gwarp * (size_t)J.bitmap_words;
  int32_t* Q = J.wg_queue + gwarp * (size_t)GQ_SLOTS;
  // the batch's samples, or those the lane tier listed
  const unsigned long long count =
      J.lane_tier ? *((volatile unsigned long long*)&J.ctr->lane_count) : (unsigned long long)J.count;
  // sets above mid_cap nodes (when set) go on to the CTA tier, whose warps share a sample
  const int cap = J.mid_cap > 0 ? min(J.mid_cap, GQ_CAP) : GQ_CAP;
  unsigned long long ev = 0, nv = 0, dr = 0;
  for (;;) {
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(&J.ctr->work, 1ull);
    idx = __shfl_sync(FULL_MASK, idx, 0);
    if (idx >= count) break;
    const int64_t j = J.lane_tier ? J.lane_list[idx] : sample_at(J, idx);
    const SampleConst sc = sample_const(J.rk, (uint32_t)j, ctr_word3(PURPOSE_SKIP, J.stream, j));
    const int32_t root = pick_root(J, j);
    if (lane == 0) {
      atomicOr(bits + (root >> 5), 1u << (root & 31));
      Q[0] = root;
      ring.node[0] = root;
      ring.lo[0] = __ldg(J.g.off + root);
      ring.d[0] = __ldg(J.g.off + root + 1) - ring.lo[0];
    }
    int tail = 1;
    bool overflow = false;
    bool hit = (MODE == MODE_HIT) && test_bit(J.seed_bits, (uint32_t)root);
    __syncwarp();
    auto visit = [&](const uint32_t (&u)[2], const uint32_t (&ulo)[2], const uint32_t (&ud)[2],
                     unsigned lt_mask) -> bool {
      uint32_t old[2] = {0u, 0u};
#pragma unroll
      for (int t = 0; t < 2; ++t)
        if (u[t] != NO_NODE) old[t] = atomicOr(bits + (u[t] >> 5), 1u << (u[t] & 31));
      bool h = false;
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const bool is_new = u[t] != NO_NODE && !((old[t] >> (u[t] & 31)) & 1u);
        const unsigned m = __ballot_sync(FULL_MASK, is_new);
        if (is_new) {
          const int pos = tail + __popc(m & lt_mask);
          Q[pos] = (int32_t)u[t];  // tail <= cap <= GQ_CAP before this round: fits GQ_SLOTS
          ring.node[pos & (WRING - 1)] = (int32_t)u[t];
          ring.lo[pos & (WRING - 1)] = ulo[t];
          ring.d[pos & (WRING - 1)] = ud[t];
          if (MODE == MODE_HIT) h |= test_bit(J.seed_bits, u[t]);
        }
        tail += __popc(m);
      }
      if (MODE == MODE_HIT) hit = __any_sync(FULL_MASK, h) || hit;
      if (tail > cap) overflow = true;
      return overflow || hit;
    };
    if (!hit) wc_bfs_warp(J.g, Q, ring, tail, J.rk, sc, lane, ev, dr, visit);
    __syncwarp();
    if (overflow) {
      if (lane == 0) {
        const unsigned long long b = atomicAdd(&J.ctr->big_count, 1ull);
        J.big_list[b] = j;
      }
    } else {
      if (MODE == MODE_STORE) warp_store_set(J, j, Q, tail, lane);
      else if (lane == 0) J.hit[j - J.j0] = hit ? 1 : 0;
      if (lane == 0) nv += (unsigned long long)tail;
    }
    __syncwarp();
    // clear the words of this sample's nodes (every set bit has its queue entry)
    for (int i = lane; i < tail; i += 32) bits[Q[i] >> 5] = 0u;
    __syncwarp();
  }
  flush_stats(J.ctr, ev, nv, dr, lane, false);
}

// Lane tier (weighted-cascade IC): one lane per sample.  Each lane runs the
// whole BFS of its own sample with the gap walk, its queue (up to LANE_Q
// nodes) in thread-local memory and membership tested by scanning that
// queue.  A sample that outgrows the queue is listed in lane_list for the
// warp tiers (its partial work is dropped).  Weighted-cascade sets are mostly
// a handful of nodes (on the 2^25-node R-MAT graph the median is one node and
// nine in ten have at most 18), so 32 independent samples per warp keep far
// more memory requests in flight than one sample per warp.  Lanes claim
// sample indices and store their sets independently of each other.
constexpr int LANE_Q = 32;

template <int MODE>
__global__ void __launch_bounds__(256) k_sample_lane_wc(SampleJob J) {
  const int lane = threadIdx.x & 31;
  int32_t q[LANE_Q];
  uint32_t qlo[LANE_Q], qd[LANE_Q];  // the queued nodes' in-lists, loaded when the node is found
  unsigned long long ev = 0, nv = 0, dr = 0;
  for (;;) {
    // one sample per lane; the lanes that arrive together share one atomic
    const unsigned act = __activemask();
    const int leader = __ffs(act) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd(&J.ctr->lane_work, (unsigned long long)__popc(act));
    base = __shfl_sync(act, base, leader);
    const unsigned long long idx = base + (unsigned long long)__popc(act & ((1u << lane) - 1u));
    if (idx >= (unsigned long long)J.count) break;
    const int64_t j = sample_at(J, idx);
    const SampleConst sc = sample_const(J.rk, (uint32_t)j, ctr_word3(PURPOSE_SKIP, J.stream, j));
    const int32_t root = pick_root(J, j);
    q[0] = root;
    qlo[0] = __ldg(J.g.off + root);
    qd[0] = __ldg(J.g.off + root + 1) - qlo[0];
    int tail = 1;
    bool hit = (MODE == MODE_HIT) && test_bit(J.seed_bits, (uint32_t)root);
    bool overflow = false;
    for (int h = 0; h < tail && !hit && !overflow; ++h) {
      const int32_t v = q[h];
      GapWalk w;
      walk_begin(w, J.g, qlo[h], qd[h]);
      ev += w.d;
      for (bool more = true; more && !hit && !overflow;) {
        uint32_t e[2];
        more = walk_step(w, v, J.rk, sc, dr, e[0], e[1]);
        uint32_t u[2] = {NO_NODE, NO_NODE}, ulo[2] = {0u, 0u}, uhi[2] = {0u, 0u};
#pragma unroll
        for (int t = 0; t < 2; ++t)
          if (e[t] != NO_NODE) u[t] = __ldg(J.g.src + e[t]);
#pragma unroll
        for (int t = 0; t < 2; ++t)
          if (u[t] != NO_NODE) {
            ulo[t] = __ldg(J.g.off + u[t]);
            uhi[t] = __ldg(J.g.off + u[t] + 1);
          }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (u[t] == NO_NODE || hit || overflow) continue;
          bool seen = false;
          for (int i = 0; i < tail; ++i) seen |= q[i] == (int32_t)u[t];
          if (seen) continue;
          if (tail == LANE_Q) {
            overflow = true;
            continue;
          }
          q[tail] = (int32_t)u[t];
          qlo[tail] = ulo[t];
          qd[tail] = uhi[t] - ulo[t];
          ++tail;
          if (MODE == MODE_HIT && test_bit(J.seed_bits, u[t])) hit = true;
        }
      }
    }
    if (overflow) {
      const unsigned long long b = atomicAdd(&J.ctr->lane_count, 1ull);
      J.lane_list[b] = j;
      continue;
    }
    if (MODE == MODE_STORE) {
      unsigned long long at = 0;
      if (reserve(J, j, tail, &at)) {
        for (int i = 0; i < tail; ++i) {
          J.pool_nodes[at + i] = q[i];
          J.pool_samp[at + i] = (int32_t)j;
        }
        J.set_start[j] = (int64_t)at;
        J.set_len[j] = tail;
      }
    } else {
      J.hit[j - J.j0] = hit ? 1 : 0;
    }
    nv += (unsigned long long)tail;
  }
  __syncwarp();
  flush_stats(J.ctr, ev, nv, dr, lane, false);
}

// LT pick of node v with the in-list [lo, lo + d), d > 0, and its draw r: the
// position of the kept in-edge, or NO_NODE when none is kept.  w = 1/d: one of
// the d.  General in-weights: the first whose running threshold sum passes r,
// found among the sums by 8-way search in a lane (seven loads at once) and
// 33-way search in a warp (three round trips up to d = 35,000), where adding up
// 32 thresholds at a time took d / 32 of them and the walks of a power-law
// graph keep coming through hubs: load and D-SSA solve of 1,000,003 nodes and
// 10M edges 8.7 -> 5.0 ms on GB300, its walks 5.6 -> 1.9.  The sums are cut at
// 2^32 - 1, so r = 2^32 - 1 adds up the thresholds themselves.
__device__ __noinline__ uint32_t lt_pick_sum(const GraphView& g, uint32_t lo, uint32_t d, uint32_t r) {
  unsigned long long cum = 0;
  for (uint32_t e = lo; e < lo + d; ++e) {
    cum += g.thr[e];
    if ((unsigned long long)r < cum) return e;
  }
  return NO_NODE;
}

__device__ __forceinline__ uint32_t lt_pick_lane(const SampleJob& J, uint32_t lo, uint32_t d, uint32_t r) {
  if (!J.lt_cumulative) return lo + __umulhi(r, d);
  if (r == 0xFFFFFFFFu) return lt_pick_sum(J.g, lo, d, r);
  uint32_t a = lo, len = d;  // sums before a are <= r; the pick, if any, lies in [a, a + len)
  while (len > 8u) {
    uint32_t at[7];
    int c = 0;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      at[i] = a + (uint32_t)(((uint64_t)len * (uint32_t)(i + 1)) >> 3) - 1u;
      c += __ldg(J.g.lt_cum + at[i]) <= r;
    }
    uint32_t from = a, to = a + len;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      if (i < c) from = at[i] + 1u;
      if (i == c) to = at[i] + 1u;
    }
    a = from;
    len = to - from;
  }
  int c = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) c += (uint32_t)i < len && __ldg(J.g.lt_cum + a + i) <= r;
  return a + (uint32_t)c < lo + d ? a + (uint32_t)c : NO_NODE;
}

__device__ __forceinline__ uint32_t lt_pick_warp(const SampleJob& J, uint32_t lo, uint32_t d, uint32_t r, int lane) {
  if (!J.lt_cumulative) return lo + __umulhi(r, d);
  if (r == 0xFFFFFFFFu) return lt_pick_sum(J.g, lo, d, r);
  uint32_t a = lo, len = d;
  while (len > 32u) {
    auto at = [&](int i) { return a + (uint32_t)((uint64_t)len * (uint32_t)(i + 1) / 33u) - 1u; };
    const int c = __popc(__ballot_sync(FULL_MASK, __ldg(J.g.lt_cum + at(lane)) <= r));
    const uint32_t from = c ? at(c - 1) + 1u : a, to = c < 32 ? at(c) + 1u : a + len;
    a = from;
    len = to - from;
  }
  const unsigned m = __ballot_sync(FULL_MASK, (uint32_t)lane < len && __ldg(J.g.lt_cum + a + lane) > r);
  return m ? a + (uint32_t)__ffs(m) - 1u : NO_NODE;
}

// LT live-edge walk (one keyed in-neighbour per node), warp per sample: every
// lane follows the same walk; membership of the next node is checked by the
// 32 lanes over the walk list in shared memory, while the loads of the next
// step are under way.  Bound: two dependent round trips per node, and the
// longest walk of a batch.  (A tier of one walk per lane in front, for walks of
// up to 64 nodes, was slower: 4.3 -> 4.6 ms of walks in the 2^23-node solve.)
template <int MODE>
__global__ void __launch_bounds__(WT_WARPS * 32) k_sample_warp_lt(SampleJob J) {
  __shared__ int32_t s_q[WT_WARPS][LT_QCAP];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t* Q = s_q[wid];
  unsigned long long ev = 0, nv = 0;
  for (;;) {
    unsigned long long idx = 0;
    if (lane == 0) idx = atomicAdd(&J.ctr->work, 1ull);
    idx = __shfl_sync(FULL_MASK, idx, 0);
    if (idx >= (unsigned long long)J.count) break;
    const int64_t j = sample_at(J, idx);
    const SampleConst sc = sample_const(J.rk, (uint32_t)j, ctr_word3(PURPOSE_LT, J.stream, j));
    const int32_t root = pick_root(J, j);
    if (lane == 0) Q[0] = root;
    int tail = 1;
    bool overflow = false;
    bool hit = (MODE == MODE_HIT) && test_bit(J.seed_bits, (uint32_t)root);
    int32_t cur = root;
    uint32_t lo = __ldg(J.g.off + cur), hi = __ldg(J.g.off + cur + 1);
    __syncwarp();
    while (!hit && hi > lo) {
      const uint4 r = philox_x((uint32_t)cur, sc, J.rk);
      const uint32_t pick = lt_pick_warp(J, lo, hi - lo, r.x, lane);
      if (pick == NO_NODE) break;  // no in-edge kept: the walk ends here
      const int32_t u = (int32_t)__ldg(J.g.src + pick);
      lo = __ldg(J.g.off + u);
      hi = __ldg(J.g.off + u + 1);
      if (MODE == MODE_HIT) hit = test_bit(J.seed_bits, (uint32_t)u);
      if (lane == 0) ev += 1;
      bool found = false;
      for (int i = lane; i < tail; i += 32) found |= (Q[i] == u);
      if (__any_sync(FULL_MASK, found)) {
        hit = false;  // a node seen before was tested then
        break;
      }
      if (tail >= LT_QCAP) {
        overflow = true;
        break;
      }
      if (lane == 0) Q[tail] = u;
      ++tail;
      __syncwarp();
      cur = u;
    }
    __syncwarp();
    if (overflow) {
      if (lane == 0) {
        const unsigned long long b = atomicAdd(&J.ctr->big_count, 1ull);
        J.big_list[b] = j;
      }
    } else {
      if (MODE == MODE_STORE) warp_store_set(J, j, Q, tail, lane);
      else if (lane == 0) J.hit[j - J.j0] = hit ? 1 : 0;
      if (lane == 0) nv += (unsigned long long)tail;
    }
    __syncwarp();
  }
  flush_stats(J.ctr, ev, nv, ev, lane, false);
}

// CTA tier: one CTA per large sample.
// KIND 0: the only CTA stage (bitmap in shared memory, queue of n entries).
// KIND 1: small CTAs (bitmap in global memory, queue of small_qcap entries);
//         a set that outgrows the queue goes on to KIND 2.
// KIND 2: full-size CTAs (global bitmap, queue of n entries) for those sets.
template <int MODE, bool SMEM_BITMAP, int KIND, int W>
__global__ void __launch_bounds__(KIND == 1 ? SMALL_CTA_THREADS : 1024, KIND == 1 ? 1024 / SMALL_CTA_THREADS : 1)
    k_sample_cta(SampleJob J) {
  constexpr bool WC = W == W_GAPS;
  constexpr int WARPS = KIND == 1 ? SMALL_CTA_THREADS / 32 : 32;
  extern __shared__ __align__(16) uint32_t s_bits[];
  __shared__ long long s_item;
  __shared__ int s_tail, s_next, s_hit, s_ok;
  __shared__ unsigned long long s_pos;
  __shared__ uint32_t s_stage[WARPS][WC ? 1 : STAGE];
  __shared__ unsigned int s_staged[WARPS];
  // heavy in-lists of the current level, expanded by all warps together
  __shared__ uint32_t s_hlo[WC ? 1 : CTA_HEAVY_CAP], s_hhi[WC ? 1 : CTA_HEAVY_CAP];
  __shared__ int s_hpref[WC ? 1 : CTA_HEAVY_CAP];
  __shared__ int s_nheavy, s_htotal, s_hnext;
  // weighted cascade: queue head, and nodes queued or being expanded
  __shared__ int s_head, s_pending;
  const int tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x;
  const int64_t n = J.g.n;
  const int64_t qcap = KIND == 1 ? (int64_t)J.small_qcap : n;
  uint32_t* bits = SMEM_BITMAP ? s_bits
                   : (KIND == 1 ? J.small_bitmap : J.slot_bitmap) + (size_t)blockIdx.x * (size_t)J.bitmap_words;
  int32_t* Q = (KIND == 1 ? J.small_queue : J.slot_queue) + (size_t)blockIdx.x * (size_t)qcap;
  const Stage stage{s_stage[tid >> 5], &s_staged[tid >> 5]};
  if (lane == 0) *stage.cnt = 0u;
  if (SMEM_BITMAP)
    for (int64_t i = tid; i < J.bitmap_words; i += nthr) bits[i] = 0u;
  unsigned long long* work = KIND == 2 ? &J.ctr->big2_work : &J.ctr->big_work;
  const int64_t* list = KIND == 2 ? J.big2_list : J.big_list;
  const long long big_count =
      (long long)*((volatile unsigned long long*)(KIND == 2 ? &J.ctr->big2_count : &J.ctr->big_count));
  unsigned long long ev = 0, nv = 0, dr = 0;
  __syncthreads();
  for (;;) {
    if (tid == 0) s_item = (long long)atomicAdd(work, 1ull);
    __syncthreads();
    const long long item = s_item;
    if (item >= big_count) break;
    const int64_t j = list[item];
    const int32_t root = pick_root(J, j);
    if (tid == 0) {
      bits[root >> 5] |= 1u << (root & 31);
      Q[0] = root;
      s_tail = 1;
      s_hit = (MODE == MODE_HIT) && test_bit(J.seed_bits, (uint32_t)root);
    }
    __syncthreads();
    if (J.model == 0) {
      const SampleConst sc = sample_const(J.rk, (uint32_t)j, ctr_word3(WC ? PURPOSE_SKIP : PURPOSE_IC, J.stream, j));
      auto visit = [&](uint32_t u, unsigned lt_mask) -> bool {
        bool is_new = false;
        if (u != NO_NODE) {
          const uint32_t mask = 1u << (u & 31);
          // most live tails are in a large set already: a look is cheaper than the
          // atomic (bits are only ever set during a sample; one in global memory
          // would cost a second round trip)
          if (!SMEM_BITMAP || WC || !(*(volatile uint32_t*)(bits + (u >> 5)) & mask))
            is_new = !(atomicOr(bits + (u >> 5), mask) & mask);
        }
        const unsigned m = __ballot_sync(FULL_MASK, is_new);
        int base = 0;
        if (m) {
          if (lane == 0) {
            if (WC) atomicAdd(&s_pending, __popc(m));  // before the producer's own chunk is retired
            base = atomicAdd(&s_tail, __popc(m));
          }
          base = __shfl_sync(FULL_MASK, base, 0);
          if (is_new) {
            const int pos = base + __popc(m & lt_mask);
            if (KIND != 1 || pos < qcap) Q[pos] = (int32_t)u;
            if (MODE == MODE_HIT && test_bit(J.seed_bits, u)) s_hit = 1;
          }
        }
        if (KIND == 1 && base + __popc(m) > qcap) return true;  // outgrew the small queue
        if (MODE == MODE_HIT) return __any_sync(FULL_MASK, *(volatile int*)&s_hit != 0);
        return false;
      };
      if constexpr (WC) {
        // Weighted cascade without level barriers: any visiting order reaches
        // the same set (the gaps are keyed per node), so the warps pull queued
        // nodes as they appear.  s_pending counts the nodes queued or being walked: a
        // lane's new nodes are added before its node is retired, so s_pending
        // reaches 0 only when nothing is queued and no lane holds a node, and
        // the sample ends there.  A queue slot reads -1 until its node is
        // written, so a claimed slot whose writer has reserved but not yet
        // stored it is waited for.
        auto stopped = [&]() -> bool {
          return (MODE == MODE_HIT && *(volatile int*)&s_hit) || (KIND == 1 && *(volatile int*)&s_tail > qcap);
        };
        if (tid == 0) {
          s_head = 0;
          s_pending = 1;  // the root
        }
        __syncthreads();
        const int qlim = (int)(qcap < 0x7FFFFFFF ? qcap : 0x7FFFFFFF);  // queue slots that can be written
        long long idle = 0;
        // Every lane holds at most one node and takes one walk step per round;
        // lanes without a node claim the next queued ones at the start of a
        // round (one claim per warp, taken by lane 0 and broadcast, so the warp
        // stays converged for the shuffles and ballots below).  A node is
        // retired from s_pending when its walk is done, after the nodes it
        // queued were added.
        const unsigned lt_mask = (1u << lane) - 1u;
        int32_t v = -1;
        GapWalk w;
        for (;;) {
          if (__any_sync(FULL_MASK, stopped())) break;
          const bool need = v < 0;
          const unsigned nm = __ballot_sync(FULL_MASK, need);
          int h = 0, cnt = 0;
          if (lane == 0 && nm) {
            const int want = __popc(nm);
            for (;;) {
              h = *(volatile int*)&s_head;
              const int avail = min(*(volatile int*)&s_tail, qlim) - h;
              cnt = avail < want ? avail : want;
              if (cnt <= 0 || atomicCAS(&s_head, h, h + cnt) == h) break;
            }
          }
          h = __shfl_sync(FULL_MASK, h, 0);
          cnt = __shfl_sync(FULL_MASK, cnt, 0);
          bool empty = false;  // took a node that has no in-edges (or whose slot never arrived)
          if (need) {
            const int r = __popc(nm & lt_mask);
            if (r < cnt) {
              int32_t x;
              // the slot's writer has reserved it; wait (briefly) for its store
              for (long long t = 0; (x = *(volatile int32_t*)&Q[h + r]) < 0; ++t) {
                if (t > (1ll << 22)) {
                  atomicCAS(&J.ctr->error, 0u, SAMPLER_ERR_SLOT);
                  x = -1;
                  break;
                }
              }
              if (x >= 0) {
                const uint32_t lo = __ldg(J.g.off + x);
                walk_begin(w, J.g, lo, __ldg(J.g.off + x + 1) - lo);
                ev += w.d;
              }
              if (x >= 0 && w.d > 0u) v = x;
              else empty = true;
            }
          }
          uint32_t u0 = NO_NODE, u1 = NO_NODE;
          bool fin = false;
          if (v >= 0) {
            uint32_t e0, e1;
            if (!walk_step(w, v, J.rk, sc, dr, e0, e1)) {
              v = -1;
              fin = true;
            }
            if (e0 != NO_NODE) u0 = __ldg(J.g.src + e0);
            if (e1 != NO_NODE) u1 = __ldg(J.g.src + e1);
          }
          if (visit(u0, lt_mask)) break;
          if (__any_sync(FULL_MASK, u1 != NO_NODE) && visit(u1, lt_mask)) break;
          const int nret = __popc(__ballot_sync(FULL_MASK, fin || empty));
          if (lane == 0 && nret) {
            __threadfence_block();  // the nodes they queued before they are retired
            atomicSub(&s_pending, nret);
          }
          if (cnt > 0 || nret > 0 || __any_sync(FULL_MASK, v >= 0)) {
            idle = 0;
            continue;
          }
          // nothing held and nothing to claim: the sample is done once nothing is pending
          if (__any_sync(FULL_MASK, *(volatile int*)&s_pending == 0)) break;
          if (++idle > (1ll << 24)) {  // far longer than any sample: give up and report
            if (lane == 0) atomicCAS(&J.ctr->error, 0u, SAMPLER_ERR_IDLE);
            break;
          }
          __nanosleep(64);
        }
        __syncthreads();
      } else {
      const int wid = tid >> 5;
      auto take_heavy = [&](int32_t, uint32_t lo, uint32_t hi, int) -> int {
        const int slot = atomicAdd(&s_nheavy, 1);
        if (slot >= CTA_HEAVY_CAP) return 0;  // list full: this warp expands it itself
        s_hlo[slot] = lo;
        s_hhi[slot] = hi;
        return HEAVY_SKIP;
      };
      if (tid == 0) s_nheavy = 0;
      int lvl_begin = 0, lvl_end = 1;
      for (;;) {
        // every thread is past the previous barrier and nobody writes s_hit
        // until the next one, so this exit test is uniform across the CTA
        if (lvl_begin >= lvl_end || s_hit || (KIND == 1 && s_tail > qcap)) break;
        if (tid == 0) s_next = lvl_begin;
        __syncthreads();
        for (;;) {
          int b = 0;
          if (lane == 0) b = atomicAdd(&s_next, 32);
          b = __shfl_sync(FULL_MASK, b, 0);
          if (b >= lvl_end) break;
          const int cnt = min(32, lvl_end - b);
          const int32_t v = (lane < cnt) ? Q[b + lane] : -1;
          if (expand_ic<W == W_TRI>(J.g, v, J.rk, sc, lane, stage, ev, dr, CTA_HEAVY_GROUPS, visit, take_heavy))
            break;
        }
        drain(stage, true, lane, visit);
        __syncthreads();
        const int nh = min(s_nheavy, CTA_HEAVY_CAP);
        if (nh > 0 && !s_hit && !(KIND == 1 && s_tail > qcap)) {
          // the heavy in-lists in pieces of 64 groups, dealt to all warps
          if (wid == 0) {
            int carry = 0;
            for (int base = 0; base < nh; base += 32) {
              const int i = base + lane;
              const int np = i < nh ? (int)(((s_hhi[i] + 3) >> 2) - (s_hlo[i] >> 2) + 63) >> 6 : 0;
              const int incl = warp_inclusive_scan(np, lane);
              if (i < nh) s_hpref[i] = carry + incl - np;
              carry += __shfl_sync(FULL_MASK, incl, 31);
            }
            if (lane == 0) {
              s_htotal = carry;
              s_hnext = 0;
            }
          }
          __syncthreads();
          const int htotal = s_htotal;
          for (;;) {
            int c = 0;
            if (lane == 0) c = atomicAdd(&s_hnext, 1);
            c = __shfl_sync(FULL_MASK, c, 0);
            if (c >= htotal) break;
            int it = 0;  // last heavy list whose first piece is <= c
            for (int step = CTA_HEAVY_CAP / 2; step; step >>= 1)
              if (it + step < nh && s_hpref[it + step] <= c) it += step;
            const uint32_t olo = s_hlo[it], ohi = s_hhi[it];
            const uint32_t grp = (olo >> 2) + (uint32_t)(c - s_hpref[it]) * 64u + (uint32_t)lane;
            const uint32_t end = (ohi + 3) >> 2;
            if (two_groups<W == W_TRI>(J.g, grp < end, grp, olo, ohi, grp + 32u < end, grp + 32u, olo, ohi, J.rk, sc,
                                       lane, stage, visit))
              break;
          }
          drain(stage, true, lane, visit);
        }
        __syncthreads();
        if (tid == 0) s_nheavy = 0;
        lvl_begin = lvl_end;
        lvl_end = s_tail;
        __syncthreads();
      }
      }
    } else if (tid == 0) {
      const SampleConst sc = sample_const(J.rk, (uint32_t)j, ctr_word3(PURPOSE_LT, J.stream, j));
      int32_t cur = root;
      int tail = 1;
      bool hit = s_hit != 0;
      while (!hit) {
        const uint32_t lo = J.g.off[cur], d = J.g.off[cur + 1] - lo;
        if (d == 0u) break;
        const uint32_t pick = lt_pick_lane(J, lo, d, philox_x((uint32_t)cur, sc, J.rk).x);
        if (pick == NO_NODE) break;
        const int32_t u = (int32_t)J.g.src[pick];
        ev += 1;
        dr += 1;
        const uint32_t mask = 1u << (u & 31);
        if (bits[u >> 5] & mask) break;
        if (KIND == 1 && tail >= qcap) {
          tail = (int)qcap + 1;  // outgrew the small queue
          break;
        }
        bits[u >> 5] |= mask;
        Q[tail++] = u;
        if (MODE == MODE_HIT) hit = test_bit(J.seed_bits, (uint32_t)u);
        cur = u;
      }
      s_tail = tail;
      s_hit = hit;
    }
    __syncthreads();
    const int tail = s_tail;
    if (KIND == 1 && tail > qcap) {
      // the set outgrew this stage's queue: full-size CTAs redo it; clear the whole bitmap
      if (tid == 0) {
        const unsigned long long b = atomicAdd(&J.ctr->big2_count, 1ull);
        J.big2_list[b] = j;
      }
      for (int64_t i = tid; i < J.bitmap_words; i += nthr) bits[i] = 0u;
      if (WC && J.model == 0)
        for (int64_t i = tid; i < qcap; i += nthr) Q[i] = -1;  // the queue's "not written yet" marks
      __syncthreads();
      continue;
    }
    if (MODE == MODE_STORE) {
      if (tid == 0) {
        unsigned long long pos = 0;
        s_ok = reserve(J, j, tail, &pos);
        s_pos = pos;
      }
      __syncthreads();
      if (s_ok) {
        const unsigned long long pos = s_pos;
        for (int i = tid; i < tail; i += nthr) {
          J.pool_nodes[pos + i] = Q[i];
          J.pool_samp[pos + i] = (int32_t)j;
        }
        if (tid == 0) {
          J.set_start[j] = (int64_t)pos;
          J.set_len[j] = tail;
        }
      }
    } else if (tid == 0) {
      J.hit[j - J.j0] = s_hit ? 1 : 0;
    }
    if (tid == 0) nv += (unsigned long long)tail;
    // reset the visited bits of this sample only (and, for the weighted-cascade
    // IC path, the queue's "not written yet" marks)
    const bool marks = WC && J.model == 0;
    if ((int64_t)tail * 8 < J.bitmap_words) {
      for (int i = tid; i < tail; i += nthr) {
        bits[Q[i] >> 5] = 0u;
        if (marks) Q[i] = -1;
      }
    } else {
      for (int64_t i = tid; i < J.bitmap_words; i += nthr) bits[i] = 0u;
      if (marks)
        for (int i = tid; i < tail; i += nthr) Q[i] = -1;
    }
    __syncthreads();
  }
  flush_stats(J.ctr, ev, nv, dr, lane, true);
}

}  // namespace

constexpr int64_t SMEM_BITMAP_MAX_BYTES = 192 * 1024;

LaunchCfg sampler_config(const GraphView& g, int model, bool wc) {
  LaunchCfg c;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&c.num_sms, cudaDevAttrMultiProcessorCount, dev);
  int per_sm = 0;
  if (model == 0 && wc)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample_warp_ic<MODE_STORE, 0, W_GAPS>, WT_WARPS * 32, 0);
  else if (model == 0)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample_warp_ic<MODE_STORE, 0, W_COINS>, WT_WARPS * 32,
                                                  0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sample_warp_lt<MODE_STORE>, WT_WARPS * 32, 0);
  if (per_sm < 1) per_sm = 1;
  c.warp_blocks = c.num_sms * per_sm;
  const int64_t words = (g.n + 31) / 32;
  c.smem_bitmap_bytes = words * 4;
  c.cta_smem_bitmap = c.smem_bitmap_bytes <= SMEM_BITMAP_MAX_BYTES;
  c.cta_threads = 1024;
  c.cta_blocks = c.num_sms;
  if (!c.cta_smem_bitmap) {
    // global bitmap: many small CTAs first, a few full-size ones for the largest sets
    int small_per_sm = 0;
    if (model == 0 && wc)
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&small_per_sm, k_sample_cta<MODE_STORE, false, 1, W_GAPS>,
                                                    SMALL_CTA_THREADS, 0);
    else
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&small_per_sm, k_sample_cta<MODE_STORE, false, 1, W_COINS>,
                                                    SMALL_CTA_THREADS, 0);
    if (small_per_sm < 1) small_per_sm = 1;
    c.small_blocks = c.num_sms * small_per_sm;
    c.small_qcap = (int)std::min<int64_t>(g.n, 1 << 20);
    c.cta_blocks = std::max(8, c.num_sms / 4);
  }
  c.mid_blocks = c.num_sms * 2;  // 16 warps per SM, each with its own global hash and queue
  // global-bitmap warp tier (weighted-cascade IC, bitmap in global memory): 32
  // warps per SM, each with an n-bit bitmap and a GQ_SLOTS queue, or 16 where
  // the bitmaps would pass 24 GB
  if (model == 0 && wc) {
    int lane_per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lane_per_sm, k_sample_lane_wc<MODE_STORE>, 256, 0);
    c.lane_blocks = c.num_sms * (lane_per_sm < 1 ? 1 : lane_per_sm);
  }
  if (model == 0 && wc && !c.cta_smem_bitmap) {
    const double per_block = (double)words * 4.0 * WT_WARPS;
    c.wg_blocks = c.num_sms * ((double)c.num_sms * 4 * per_block <= 24e9 ? 4 : 2);
  }
  return c;
}

size_t mid_tier_words(const LaunchCfg& c) { return (size_t)c.mid_blocks * WT_WARPS; }
size_t wg_tier_warps(const LaunchCfg& c) { return (size_t)c.wg_blocks * WT_WARPS; }
size_t wg_queue_per_warp() { return GQ_SLOTS; }
int mid_tier_max_cap() { return Tier<1>::QCAP; }
size_t mid_hash_per_warp() { return MID_HASH; }
size_t mid_queue_per_warp() { return MID_QSLOTS; }

size_t sampler_scratch_bytes(const GraphView& g, const LaunchCfg& c) {
  const size_t words = (size_t)((g.n + 31) / 32);
  size_t per_slot = (size_t)g.n * 4 + (c.cta_smem_bitmap ? 0 : words * 4);
  return per_slot * (size_t)c.cta_blocks + ((size_t)c.small_qcap * 4 + words * 4) * (size_t)c.small_blocks;
}

template <int MODE, int W>
static void launch_warp_ic_w(const SampleJob& J, const LaunchCfg& c, cudaStream_t st) {
  const dim3 block(WT_WARPS * 32);
  k_sample_warp_ic<MODE, 0, W><<<c.warp_blocks, block, 0, st>>>(J);
  if (J.mid_cap > 0) k_sample_warp_ic<MODE, 1, W><<<c.mid_blocks, block, 0, st>>>(J);
}

template <int MODE>
static void launch_warp_ic(const SampleJob& J, const LaunchCfg& c, cudaStream_t st) {
  switch (weights_of(J)) {
    case W_GAPS: return launch_warp_ic_w<MODE, W_GAPS>(J, c, st);
    case W_TRI: return launch_warp_ic_w<MODE, W_TRI>(J, c, st);
    default: return launch_warp_ic_w<MODE, W_COINS>(J, c, st);
  }
}

cudaError_t launch_sample_warp(const SampleJob& J, const LaunchCfg& c, cudaStream_t st) {
  const dim3 grid(c.warp_blocks), block(WT_WARPS * 32);
  if (J.model == 0 && J.wc_implicit && J.lane_tier) {
    if (J.mode == MODE_STORE) k_sample_lane_wc<MODE_STORE><<<c.lane_blocks, 256, 0, st>>>(J);
    else k_sample_lane_wc<MODE_HIT><<<c.lane_blocks, 256, 0, st>>>(J);
  }
  if (J.model == 0 && J.wc_implicit && J.warp_global && c.wg_blocks > 0) {
    if (J.mode == MODE_STORE) k_sample_warp_wcg<MODE_STORE><<<c.wg_blocks, block, 0, st>>>(J);
    else k_sample_warp_wcg<MODE_HIT><<<c.wg_blocks, block, 0, st>>>(J);
  } else if (J.model == 0) {
    if (J.mode == MODE_STORE) launch_warp_ic<MODE_STORE>(J, c, st);
    else launch_warp_ic<MODE_HIT>(J, c, st);
  } else {
    if (J.mode == MODE_STORE) k_sample_warp_lt<MODE_STORE><<<grid, block, 0, st>>>(J);
    else k_sample_warp_lt<MODE_HIT><<<grid, block, 0, st>>>(J);
  }
  return cudaGetLastError();
}

template <int MODE, bool SB, int W>
static cudaError_t launch_cta_t(const SampleJob& J, const LaunchCfg& c, cudaStream_t st) {
  if (SB) {
    const size_t smem = (size_t)c.smem_bitmap_bytes;
    cudaError_t e = cudaFuncSetAttribute(k_sample_cta<MODE, true, 0, W>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_sample_cta<MODE, true, 0, W><<<c.cta_blocks, c.cta_threads, smem, st>>>(J);
  } else {
    k_sample_cta<MODE, false, 1, W><<<c.small_blocks, SMALL_CTA_THREADS, 0, st>>>(J);
    k_sample_cta<MODE, false, 2, W><<<c.cta_blocks, c.cta_threads, 0, st>>>(J);
  }
  return cudaGetLastError();
}

template <int MODE, bool SB>
static cudaError_t launch_cta_w(const SampleJob& J, const LaunchCfg& c, cudaStream_t st) {
  switch (weights_of(J)) {
    case W_GAPS: return launch_cta_t<MODE, SB, W_GAPS>(J, c, st);
    case W_TRI: return launch_cta_t<MODE, SB, W_TRI>(J, c, st);
    default: return launch_cta_t<MODE, SB, W_COINS>(J, c, st);
  }
}

cudaError_t launch_sample_cta(const SampleJob& J, const LaunchCfg& c, cudaStream_t st) {
  if (J.mode == MODE_STORE)
    return c.cta_smem_bitmap ? launch_cta_w<MODE_STORE, true>(J, c, st) : launch_cta_w<MODE_STORE, false>(J, c, st);
  return c.cta_smem_bitmap ? launch_cta_w<MODE_HIT, true>(J, c, st) : launch_cta_w<MODE_HIT, false>(J, c, st);
}

}  // namespace ssa
