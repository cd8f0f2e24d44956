// Internal interface between the host driver (api.cpp) and the sm_103a
// kernels (*.cu).  Plain structs of device pointers; no torch types.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

struct ssa_solver;

namespace ssa {

// Device bytes of the RR pool and the greedy lists at the end of the solver's last solve.
int64_t solver_bytes(const ssa_solver* s);

// Sets the calling thread's message returned by ssa_last_error().
void set_last_error(const char* msg);

// Device-resident in-edge CSR (Sec. 2).  Positions fit 32 bits (m < 2^31), and
// what a sampler can do without is not stored beside what it reads: a random
// access moves a 32-byte sector, and what stays in the 129 MB L2 decides the rate.
//   off   n+1 positions
//   src   the tail node of every in-edge.  Weighted cascade stores nothing else:
//         its threshold follows from the in-degree.  Trivalency (n <= 2^30) keeps
//         the edge's class (0.1, 0.01, 0.001) in the two high bits.
//   thr   uint32 live thresholds: explicit weights, and trivalency beyond 2^30 nodes
// A 4-edge group (the unit of one Philox draw) is one aligned 16-byte load of each.
// Against 64-bit offsets and 8-byte {src, thr} records, on GB300: half the graph
// memory (5.3 for 10.5 GB at 1.26e9 edges) at the same speed for weighted
// cascade (latency-bound); trivalency graphs of 16M edges (64 MB) stay in L2
// whole, where the coin kernels read them (hit rate 64 -> 91%).
struct GraphView {
  int64_t n = 0, m = 0;
  const uint32_t* off = nullptr;  // n+1
  const uint32_t* src = nullptr;  // m rounded up to a multiple of 4 (+4)
  const uint32_t* thr = nullptr;  // as src, or null
  // weighted cascade: -1 / log2(q) of the gap form for every in-degree d < 2^wc_inv_k
  // (null / 0 for other weightings)
  const float* wc_inv = nullptr;
  int wc_inv_k = 0;
  // LT with explicit in-weights: running threshold sums of each in-list, at most
  // 2^32 - 1 (m entries; made when the first LT sampler of the graph starts)
  const uint32_t* lt_cum = nullptr;
};

// In-degrees of up to 2^WC_INV_K - 1 have an entry (4 MB at most); for larger
// ones 32 bits would seldom decide, and the exact gap is taken.
constexpr int WC_INV_K = 20;

// That table for a CSR (every in-degree below min(2^WC_INV_K, 2 * max
// in-degree)); *tab stays null when no in-list has 2 edges.
cudaError_t build_wc_inv(const uint32_t* d_off, int64_t n, float** tab, int* k, cudaStream_t st);

// Running sums of every in-list's thresholds, cut at 2^32 - 1 (m entries, allocated here).
cudaError_t build_lt_cum(const uint32_t* d_off, const uint32_t* d_thr, int64_t n, int64_t m, uint32_t** cum,
                         cudaStream_t st);

// Device counters of one sampling batch.
// Bounded waits of the weighted-cascade CTA tier that gave up (Counters::error).
constexpr unsigned SAMPLER_ERR_SLOT = 1;  // a claimed queue slot was never written
constexpr unsigned SAMPLER_ERR_IDLE = 2;  // a warp found no work for far longer than any sample

struct Counters {
  unsigned long long work;         // warp tier: next sample index
  unsigned long long mid_count;    // samples handed from the shared-memory warp tier to the global one
  unsigned long long mid_work;     // global warp tier: next list index
  unsigned long long big_count;    // samples handed to the CTA tier
  unsigned long long big_work;     // CTA tier: next list index
  unsigned long long big2_count;   // samples that outgrew the small CTAs' queue
  unsigned long long big2_work;
  unsigned long long cursor;       // pool entries reserved (absolute)
  unsigned long long edge_visits;  // in-edges examined
  unsigned long long node_visits;  // nodes added to RR sets
  unsigned long long cta_edge_visits;  // the CTA tier's share of the two above
  unsigned long long cta_node_visits;
  unsigned long long cta_draws;    // the CTA tier's share of draws
  unsigned long long draws;        // Philox draws (IC: one per 4-edge group of a visited node, or per two gaps)
  unsigned long long ok_end;        // start of the first pool reservation that did not fit (the
                                    // host sets ~0 before a storing launch): the ones that fit end there
  unsigned long long fail_count;    // samples whose reservation did not fit (listed in fail_list)
  unsigned long long lane_work;    // lane tier: next sample index
  unsigned long long lane_count;   // samples the lane tier handed to the warp tiers
  unsigned int pool_overflow;      // a reservation passed pool_cap
  unsigned int error;              // internal error: 0 none, else SAMPLER_ERR_* of the first wait that gave up
};

enum : int { MODE_STORE = 0, MODE_HIT = 1 };

struct SampleJob {
  GraphView g;
  int model = 0;                 // 0 IC, 1 LT
  int lt_cumulative = 0;         // LT with explicit in-weights: pick by running threshold sums
  int wc_implicit = 0;           // IC with weighted-cascade weights: thresholds from in-degrees,
                                 // records read for live edges only
  int warp_global = 0;           // weighted-cascade IC: every sample through the global-bitmap warp tier
  int lane_tier = 0;             // weighted-cascade IC: the lane tier runs first; the warp tiers take
                                 // only the samples it lists in lane_list (capacity `count`)
  int64_t* lane_list = nullptr;
  uint32_t* wg_bitmap = nullptr; // that tier: per warp bitmap_words words, zero between samples
  int32_t* wg_queue = nullptr;   // that tier: per warp wg_queue_per_warp() entries
  uint64_t seed = 0;
  uint32_t stream = 0;
  int64_t j0 = 0, count = 0;     // samples [j0, j0+count), or work_list[0, count)
  const int64_t* work_list = nullptr;  // explicit sample ids (re-run of pool overflows) or null
  int64_t* fail_list = nullptr;        // samples whose pool reservation did not fit
  uint32_t rk[20] = {};                // Philox round keys: rk[2r], rk[2r+1] = key + r * Weyl
  const uint64_t* bprefix = nullptr;  // WRIS prefix sums (n+1) or null
  int mode = MODE_STORE;
  // MODE_STORE: flat pool entries + per-sample extents
  int32_t* pool_nodes = nullptr;
  int32_t* pool_samp = nullptr;
  int64_t pool_cap = 0;
  int64_t* set_start = nullptr;  // indexed by absolute sample id
  int32_t* set_len = nullptr;
  // MODE_HIT: seed membership bits, per-sample flag (index j - j0)
  const uint32_t* seed_bits = nullptr;
  uint8_t* hit = nullptr;
  // global-memory warp tier: hand-off list and per-warp hash / queue / slot scratch
  int warp_heavy_groups = 0x7FFFFFFF;  // warp tiers hand samples meeting an in-list of more 4-edge
                                       // groups than this to the CTA tier (tuned)
  int mid_cap = 0;               // sets above 512 nodes: 0 = straight to the CTA tier, else the
                                 // global warp tier keeps sets up to mid_cap nodes (<= 16384)
  int64_t* mid_list = nullptr;   // capacity `count`
  uint32_t* mid_hash = nullptr;  // per warp: mid_hash_per_warp() words, zero between samples
  int32_t* mid_queue = nullptr;  // per warp: mid_queue_per_warp()
  uint32_t* mid_slots = nullptr; // per warp: mid_queue_per_warp()
  // CTA tier hand-off and scratch
  int64_t* big_list = nullptr;   // capacity `count`
  uint32_t* slot_bitmap = nullptr;  // per CTA slot: bitmap_words (unused when the bitmap is in smem)
  int32_t* slot_queue = nullptr;    // per CTA slot: n entries
  // small CTAs (global bitmap only): per slot a queue of small_qcap entries and a bitmap
  int small_qcap = 0;
  int32_t* small_queue = nullptr;
  uint32_t* small_bitmap = nullptr;
  int64_t* big2_list = nullptr;     // capacity `count`
  int64_t bitmap_words = 0;
  Counters* ctr = nullptr;
};

// Samples of a batch from which the lane tier runs before the global-bitmap warp
// tier, and before the shared-memory one where sets have at most LANE_TIER_MEAN nodes.
constexpr int64_t LANE_TIER_SAMPLES = 32768, LANE_TIER_SMALL_SETS = 1 << 18, LANE_TIER_MEAN = 6;

struct LaunchCfg {
  int num_sms = 152;
  int warp_blocks = 0;   // grid of the warp tier
  int cta_blocks = 0;    // grid of the CTA tier (= number of scratch slots)
  int mid_blocks = 0;    // grid of the global-memory warp tier
  int cta_threads = 1024;
  int small_blocks = 0;  // small CTAs (256 threads) when the bitmap lives in global memory
  int small_qcap = 0;
  int wg_blocks = 0;     // global-bitmap warp tier (0: not available for this graph)
  int lane_blocks = 0;   // lane tier (weighted-cascade IC)
  bool cta_smem_bitmap = false;
  int64_t smem_bitmap_bytes = 0;
};

// Trivalency classes ride in the two high bits of src up to this many nodes.
constexpr int64_t TRI_PACK_NODES = int64_t(1) << 30;
constexpr uint32_t TRI_SRC_MASK = 0x3FFFFFFFu;
constexpr uint32_t TRI_THR0 = 429496729u, TRI_THR1 = 42949672u, TRI_THR2 = 4294967u;  // floor(2^32 p), p = 0.1, 0.01, 0.001

// ---- graph build -------------------------------------------------------
// Sorts edges by (dst, src, input position), builds off, src and (for weights
// that keep them: d_thr not null) thr.  d_src/d_dst/d_thr_in are device arrays
// of length m.
cudaError_t build_graph(int64_t n, int64_t m, const int32_t* d_src, const int32_t* d_dst,
                        const uint32_t* d_thr_in, int weighting, uint64_t weight_seed,
                        uint32_t* d_off, uint32_t* d_src_out, uint32_t* d_thr, unsigned int* d_err, cudaStream_t st,
                        int* launches);

// Directed R-MAT graph on 2^scale nodes from m_draw SplitMix64-keyed draws
// (quadrant thresholds ta < tab < tabc of a 32-bit draw), self-loops and
// duplicates removed, built straight into the in-edge CSR (allocated here,
// stream-ordered; the caller owns *d_off and *d_src).  *m_out: unique edges.
cudaError_t rmat_graph(int scale, int64_t m_draw, uint32_t ta, uint32_t tab, uint32_t tabc, uint64_t seed,
                       int weighting, uint64_t weight_seed, int64_t* m_out, uint32_t** d_off, uint32_t** d_src,
                       cudaStream_t st, int* launches);

// ---- sampling -----------------------------------------------------------
LaunchCfg sampler_config(const GraphView& g, int model, bool wc_implicit);
size_t sampler_scratch_bytes(const GraphView& g, const LaunchCfg& c);
size_t mid_tier_words(const LaunchCfg& c);  // number of warps of the global-memory tier
size_t wg_tier_warps(const LaunchCfg& c);   // warps of the global-bitmap tier
size_t wg_queue_per_warp();
int mid_tier_max_cap();
size_t mid_hash_per_warp();
size_t mid_queue_per_warp();
cudaError_t launch_sample_warp(const SampleJob& J, const LaunchCfg& c, cudaStream_t st);
cudaError_t launch_sample_cta(const SampleJob& J, const LaunchCfg& c, cudaStream_t st);

// ---- counts, greedy, stare ----------------------------------------------
cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t st);
// entries [e0, e1); with samp non-null only samples in [jlo, jhi) count
cudaError_t launch_count_nodes(const int32_t* nodes, const int32_t* samp, int64_t e0, int64_t e1, int64_t jlo,
                               int64_t jhi, int32_t* cnt, cudaStream_t st, int num_sms);
// WRIS: out[v] = w[0] + ... + w[v - 1] for v <= n (n >= 1); tmp: weight_tmp_words(n) 64-bit words
size_t weight_tmp_words(int64_t n);
cudaError_t launch_weight_prefix(const uint32_t* w, int64_t n, uint64_t* out, unsigned long long* tmp,
                                 cudaStream_t st);

struct GreedyJob {
  const int32_t* cnt0;          // n_pad counts over the sets [0, n_sets); padding 0
  int32_t* cnt;                 // n_pad working gains (written before they are read)
  int64_t n, n_pad;             // nodes; padded to a multiple of 4
  const int32_t* pool_nodes;    // entries [0, total_entries) hold the sets [0, n_sets), maybe others
  const int32_t* pool_samp;
  const int64_t* set_start;
  const int32_t* set_len;
  unsigned long long total_entries;
  int64_t n_sets;               // N: sets [0, N) take part
  int bulk_first;               // the first pick by a pass over the entries
  uint8_t* covered;             // per sample id, zeroed
  int32_t* seeds;               // k (device)
  int32_t* gains;               // k (device)
  int k;
  // control block, zeroed: GREEDY_CTL_BYTES
  unsigned int* sync;           // 128 words: count [0], release word (64-bit) [32], error flag [64], progress [96]
  unsigned long long* argmax;   // 3 slots 16 words apart
  unsigned long long* nchunk;   // chunks handed out
  unsigned int* ncand;          // candidates, chunk overflow, picks made, queued parts, list entries, shared pick
  unsigned int* hist;           // 4 x 1024 bins
  unsigned int* blk;            // 1024: candidates among the nodes that a block numbers
  // candidates of a session
  unsigned int* mark;           // n_pad bits, zero between launches: the candidates
  uint16_t* lid;                // n_pad, zero between launches: 1 + local id
  int32_t* cand_id;             // GREEDY_CANDS node ids
  int32_t* cand_len;            // gain when the lists were made = entries of the list
  unsigned int* cand_off;       // first entry of the candidate's list
  unsigned int* cand_dec;       // what the other blocks' shares of a pick take off the candidate's gain; zero between launches
  unsigned int* ents;           // ents_cap (+ GREEDY_ENTS_SPARE) first chunks of the candidates' sets
  long long ents_cap;
  uint4* chunks;                // chunk_cap (+ GREEDY_CHUNKS_SPARE) chunks of the sets' candidates
  unsigned long long chunk_cap;
  uint4* tasks;                 // parts of long sets (first chunk, set, first member): chunk_cap / 16 + 1
  long long wait_polls;         // polls without progress after which a grid-barrier wait gives up
};
constexpr int GREEDY_CANDS = 16384;
constexpr int GREEDY_ENTS_SPARE = 2048, GREEDY_CHUNKS_SPARE = 16;
// byte offsets in the control block
constexpr size_t GREEDY_CTL_ARGMAX = 512, GREEDY_CTL_NCHUNK = 896, GREEDY_CTL_NCAND = 912, GREEDY_CTL_HIST = 1024,
                 GREEDY_CTL_BLK = 1024 + 4 * 1024 * 4, GREEDY_CTL_BYTES = GREEDY_CTL_BLK + 1024 * 4;
// Pools of more entries make their first pick by a pass over the entries: the
// pass costs a few us, the same pick out of the lists 0.1 us per 100 entries it
// covers (104,000 of 195,660 entries: ~50 us).
constexpr unsigned long long GREEDY_BULK_ENTRIES = 1ull << 18;
// Counts and entries up to this many together are handled by a single block: it
// saves the ~6 us of three grid barriers, but making the lists takes one block
// 17-80 us from 10^4 to 4 x 10^4 entries on, a grid 6-8 us.
constexpr unsigned long long GREEDY_BLOCK_WORK = 1ull << 13;
constexpr long long GREEDY_DEFAULT_WAIT_POLLS = 1ll << 22;  // about a second with the poll back-off
// Process-wide poll limit of the greedy kernel's grid-barrier waits (ssa_set_wait_polls).
long long greedy_wait_polls();
// All k picks in one launch: a cooperative grid (bounded grid barriers), a
// single block for small pools, or, for a solve that shares the GPU with
// others and a pool of up to GREEDY_CLUSTER_ENTRIES entries, one thread-block
// cluster.
constexpr unsigned long long GREEDY_CLUSTER_ENTRIES = 1ull << 26;
// Pools of this many entries and more share the sets of heavy picks between the
// blocks.  max_coverage on GB300, ms, one block's alone / shared: 820,000 LT sets of
// the 2^17-node R-MAT graph (25M entries) k = 20 4.35 / 1.00, k = 100 7.6 / 2.1; 1.9M
// of the 2^20-node one (75M) k = 100 13.1 / 2.7; 820,000 IC sets (12M) k = 100 2.40 /
// 1.68.  Below, few lists are that long, and the turns cost: 130,000 LT sets of the
// 2^22-node graph (5.7M) k = 1000 2.71 / 2.82, 268,000 IC sets (5.9M) 1.65 / 1.67.
constexpr unsigned long long GREEDY_SHARE_ENTRIES = 1ull << 23;
cudaError_t launch_greedy(const GreedyJob& J, cudaStream_t st, int num_sms, bool shared_gpu);
// 0: by the rule above (default); 1: always the cooperative grid; 2: always a cluster (when the device has one)
void set_greedy_mode(int mode);
// SASS and PTX versions (major*10 + minor) of the device code the CUDA runtime loaded for this library
cudaError_t device_code_version(int* binary, int* ptx);

cudaError_t launch_mark_hits(const int32_t* nodes, const int32_t* samp, int64_t e0, int64_t e1,
                             const uint8_t* in_seed, int64_t j0, int64_t j1, uint8_t* hit, cudaStream_t st,
                             int num_sms);
cudaError_t launch_count_flags(const uint8_t* flags, int64_t count, unsigned long long* out,
                               cudaStream_t st, int num_sms);
// First T (1-based) in flags[0, count) where base + prefix hits reaches `need`;
// out[0] = T or 0, out[1] = hits in [0, count).
cudaError_t launch_first_reach(const uint8_t* flags, int64_t count, long long need_minus_base,
                               long long* out, void* tmp, cudaStream_t st, int* launches);
size_t first_reach_tmp_bytes(int64_t count);

// bit / byte of every id in [0, n); others are skipped
cudaError_t launch_set_bits(const int32_t* ids, int k, int64_t n, uint32_t* bits, uint8_t* bytes, cudaStream_t st);
cudaError_t launch_gather_sets(const int32_t* pool_nodes, const int64_t* set_start, const int32_t* set_len,
                               const int64_t* out_off, int64_t first, int64_t count, int32_t* out,
                               cudaStream_t st);

}  // namespace ssa
