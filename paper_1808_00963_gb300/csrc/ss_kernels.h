// Host-side launch interface between the orchestrator (ss_host.cu) and the
// kernel translation units.
#pragma once

#include <cstddef>
#include <cstdint>
#include <functional>

#include <cuda_runtime.h>

#include "ss_internal.cuh"

namespace ss {

// Wraps every kernel launch: counts it and, when profiling is on, brackets it
// with CUDA events on the launching stream.
struct LaunchHook {
  cudaStream_t stream;
  void run(const char* name, const std::function<void()>& launch) const;
};

// Plan of one round of multi-block steps: its task table and geometry.
struct BigPlan {
  GenTask* gt;            // the round's subsets
  uint32_t G;             // how many (0: the loop ends)
  uint32_t tiles;         // tiles over them
  uint32_t R;             // tile = 256 * R records
  uint32_t list;          // big list they came from; their big children go to the other one
  uint64_t ncounters;
  uint32_t next_tile;     // work counter: blocks take the next tile from it, so that uneven tiles balance out
};

// Control block of the multi-block steps in device memory.  The host fills
// the first part once per sort (and the first round's plan, if it knows it:
// a single set is one subset); the last block of each round's k_big_emit
// writes the plan of the next round from the list of big subsets this round
// leaves (a planning kernel before each round took 6-8 us), so rounds follow
// one another with no host in between (Section 4.2.8: the fully parallel levels need no sequential
// coordinator).  k_scan_down copies the plan to `mv`, which k_big_emit and the
// scatter read: no block may read what another block of its kernel replaces.
struct BigCtl {
  SortCtx c;
  GenTask* gtbuf[2];      // cap_big tasks each, for two successive rounds
  void* splitters;        // cap_big * big_splitters_bytes(logv)
  uint32_t* counters;     // [task][bucket][tile] counters of the round
  uint32_t* partials;     // ncounters_max / 4096 + 2
  uint32_t* gstart;       // cap_big * KP bucket starts
  uint32_t* gdesc;        // cap_big * KP bucket descriptors
  uint64_t ncounters_max;
  uint32_t cap_big;
  uint32_t R_fixed;       // tile rounds; 0: chosen per round from the strings in big subsets
  uint32_t sms;
  uint32_t K;             // buckets per step, 2^(logv + 1) - 1
  uint32_t round;
  uint32_t emitted;       // blocks of the round's k_big_emit that are done
  BigPlan cur;            // the round's plan, for its kernels before k_big_emit
  BigPlan mv;             // the same from k_big_emit on, which puts the next round's into cur
};

// Rounds of 256 strings in a tile of a round over `total` strings in G
// subsets: kTilesPerSm tiles per SM where there are that many strings (three or
// four blocks of an SM take tiles as they finish; with two per SM half of the
// slots had none: 1 M records under a 200-character prefix 572 us, with 6 per SM
// 531, 9 487, 12 487; 4 M DNA suffixes 1047 / 1044 / 1012 / 1007; 2 M URLs from
// host memory 1602 / 1545 / 1557 / 1569), at least kMinTileRounds (a tile's
// fixed work is its 2^(logv + 1) counters; with a minimum of 8, 100 k strings
// filled 49 of 152 SMs: classification 17.3 -> 12.8 us, scatter 22.9 -> 15.4
// us), at most kMaxTileRounds, and more where the tiles' counters would not
// fit.  With at most 16 the scatter's shared memory lets three blocks share an
// SM instead of two; with 8 there are twice the counters (at most 8 / 16 / 32:
// 20 M URLs 4065 / 4020 / 4255 us, 512 sets 1992 / 1973 / 2016, 4 M DNA suffixes
// 940 / 948 / 954, 10 M random strings 1579 / 1600 / 1704).
constexpr uint32_t kMinTileRounds = 2, kMaxTileRounds = 16, kTilesPerSm = 9;
__host__ __device__ inline uint32_t tile_rounds(uint64_t total, uint64_t G, uint32_t sms, uint32_t K,
                                                uint64_t ncounters_max, uint32_t fixed) {
  if (fixed) return fixed;
  const uint64_t per = total / ((uint64_t)sms * kTilesPerSm * 256) + 1;
  uint32_t R = (uint32_t)(per < kMinTileRounds ? kMinTileRounds : (per > kMaxTileRounds ? kMaxTileRounds : per));
  while (R < 8 && K * (total / (256ull * R) + G) > ncounters_max) ++R;
  return R;
}

// Most rounds of multi-block steps one sort may take (each advances every big
// subset by at least one character; a subset sharing more than about 2^20
// characters is reported as SS_ERR_TOO_LARGE).
constexpr uint32_t kMaxBigRounds = 1u << 20;

// Kernel launches of one multi-block round: sample, classify, the two
// prefix-sum kernels, emit and scatter.
constexpr uint32_t kBigRoundKernels = 6;

// The dynamic shared memory that the kernels of a translation unit may have, at
// its largest, on the current device (a kernel's limit belongs to a device):
// called once per device, before the first launch there.
cudaError_t set_big_limits();
cudaError_t set_queue_limits();
cudaError_t set_small_limits();

size_t big_splitters_bytes(int logv);
size_t big_scatter_smem(int logv, uint32_t R);
// The plan of the first round from list 0 (for several sets; a single set's
// is written by the host).
cudaError_t launch_big_plan(BigCtl* ctl, cudaStream_t st, const LaunchHook& hook);
// The kernels of one round (they do nothing when its plan holds no subset);
// with use_cond it also sets the loop graph's condition (1 while big subsets
// remain).
cudaError_t launch_big_round(int logv, bool dna, BigCtl* ctl, uint32_t R_max, uint32_t sms, uint64_t cond_handle,
                             bool use_cond, cudaStream_t st, const LaunchHook& hook);
// Kernels the loop graphs of this device have launched so far (their plan
// kernels count them on the device; reading the count waits for the device).
uint64_t graph_launch_count();

// Persistent work-queue kernel (single-block S^5 steps).
cudaError_t queue_occupancy(int logv, int* blocks_per_sm);
cudaError_t launch_queue(int logv, const SortCtx& c, uint32_t grid, cudaStream_t st, const LaunchHook& hook);

// Small subsets, set-up and LCP fix-up.
struct BeginArgs {
  uint32_t* ctrl;
  uint32_t* ready;
  uint32_t* wide;
  uint32_t ctrl_words, ready_words, num_sets;
  SetDesc* set;   // where the set descriptor goes, or null
  SetDesc sd;
  BigCtl* ctl;    // where the multi-block loop's control block goes, or null
  BigCtl v;
  GenTask root;   // the first round's task, where the host knows it (v.cur.G)
};
// Sets of kRankMin..kRankMax strings are ranked by counting (ss_rank.cu).
constexpr uint32_t kRankMin = 33, kRankMax = 4096;
struct RankArgs {
  ulonglong2* keys;   // [n][2]: the first 4 keys of each string
  uint32_t* rank;     // [n]
};
cudaError_t launch_rank(const BeginArgs& a, const RankArgs& r, const SortCtx& c, cudaStream_t st,
                        const LaunchHook& hook);

constexpr uint32_t kSmallCutoffMax = 4096;  // largest small_cutoff
size_t small_cta_smem(uint32_t pmax);
cudaError_t launch_begin(const BeginArgs& a, cudaStream_t st, const LaunchHook& hook);
cudaError_t launch_init(const SortCtx& c, cudaStream_t st, const LaunchHook& hook);
// With `last`, the warp sorts are the sort's last kernel and do what
// launch_lcp_fix does otherwise (there are no marks to resolve then).
cudaError_t launch_small(const SortCtx& c, uint32_t pmax, uint32_t sms, bool last, cudaStream_t st,
                         const LaunchHook& hook);
cudaError_t launch_lcp_fix(const SortCtx& c, uint32_t grid, cudaStream_t st, const LaunchHook& hook);
// Zeroes a few words with a kernel.
cudaError_t launch_zero(uint32_t* dst, uint32_t words, cudaStream_t st, const LaunchHook& hook);
// Packs bytes over {A, C, G, T, 0} into 3-bit codes (dna_key's layout).
cudaError_t launch_pack_dna(const uint8_t* chars, uint64_t len, uint64_t* out, uint64_t words, uint32_t* bad,
                            uint32_t grid, cudaStream_t st, const LaunchHook& hook);
cudaError_t launch_distinguishing(const uint8_t* chars, const uint64_t* offsets, uint32_t n, uint32_t cap,
                                  const uint32_t* perm, const uint32_t* lcp, uint8_t* dchar, uint32_t* dprefix,
                                  unsigned long long* sum_d, uint32_t grid, cudaStream_t st, const LaunchHook& hook);

// K-way LCP merge of sorted runs (ss_merge.cu): ceil(log2 K) rounds of
// pairwise LCP merges over 32-byte records.
constexpr uint32_t kMergeMaxRuns = 64;
constexpr uint32_t kMergeBlock = 128, kMergeBlocksPerSm = 8;
constexpr uint32_t kMergeLanesPerSm = kMergeBlock * kMergeBlocksPerSm;

struct alignas(32) MergeRec {
  uint64_t w0, w1;   // the string's characters [h, h + 16), first one most significant
  uint64_t off;      // string offset
  uint32_t idx;      // string index
  uint32_t h;        // LCP with the preceding string of its run
};

// Records of all runs, run k at [start[k], start[k + 1]).
struct MergePrepArgs {
  const uint8_t* chars;
  const uint64_t* offsets;
  uint32_t cap;
  uint32_t K;
  uint32_t total;
  MergeRec* dst;
  uint32_t start[kMergeMaxRuns + 1];
  const uint32_t* perm[kMergeMaxRuns];
  const uint32_t* lcp[kMergeMaxRuns];
  uint32_t ibase[kMergeMaxRuns];  // added to run k's entries (runs sorted with local indices)
};

// One round: current run c at [start[c], start[c + 1]); runs 2p and 2p + 1
// are merged into the same range; every S-th record of a run is a sample,
// the samples of run c being [sbase[c], sbase[c + 1]).
struct MergeRoundArgs {
  const uint8_t* chars;
  const uint64_t* offsets;
  uint32_t cap;
  uint32_t ncur;
  uint32_t S;
  uint32_t nsamples;
  const MergeRec* src;
  MergeRec* dst;            // null in the last round
  uint32_t* cut;            // per sample: records of the partner run before it
  uint32_t* cut_lcp;        // ... and its LCP with the one after them
  uint32_t* out_perm;       // last round
  uint32_t* out_lcp;        // last round, may be null
  uint32_t* counter;        // piece counter, zero at launch
  uint32_t start[kMergeMaxRuns + 1];
  uint32_t sbase[kMergeMaxRuns + 1];
};

cudaError_t launch_merge_prep(const MergePrepArgs& a, uint32_t sms, cudaStream_t st, const LaunchHook& hook);
cudaError_t launch_merge_round(const MergeRoundArgs& a, uint32_t sms, cudaStream_t st, const LaunchHook& hook);
cudaError_t launch_merge_copy(const uint32_t* perm, const uint32_t* lcp, uint32_t n, uint32_t* out_perm,
                              uint32_t* out_lcp, uint32_t sms, cudaStream_t st, const LaunchHook& hook);
// Sets *bad unless every string i lies in [offsets[i], offsets[i + 1]) with
// its terminator at offsets[i + 1] - 1 (the last one ending at end - 1).  If
// *bad is set, by this call or before it, all offsets become `empty`.
cudaError_t launch_layout_check(const uint8_t* chars, uint64_t end, uint64_t* offsets, uint32_t n, uint64_t empty,
                                uint32_t* bad, uint32_t sms, cudaStream_t st, const LaunchHook& hook);

// Suffix array by prefix doubling (ss_sa.cu).
enum class SaKernel { kIota, kNameFirst, kEncode, kNamePairs, kGroups, kLcp };
constexpr uint32_t kSaScanBlocks = 1024;  // most blocks of the naming passes (one total each)

// Name arrays of the suffixes after each round (ISA^{h0 2^k}, k = 0..count-1),
// kept for the LCPs above h0.
constexpr uint32_t kSaMaxSnaps = 40;
struct SaSnaps {
  const uint32_t* p[kSaMaxSnaps];
  uint32_t count;
};

struct SaArgs {
  const uint8_t* text = nullptr;
  uint64_t n = 0;                 // suffixes
  uint32_t h = 0;                 // current depth (h0 for kNameFirst / kLcp)
  uint32_t M = 0;                 // members of unfinished groups
  uint64_t* off = nullptr;
  uint32_t* sa = nullptr;
  const uint32_t* lcp = nullptr;  // capped LCPs of the first sort
  uint32_t* lcp_out = nullptr;    // final LCP array (holds the capped LCPs on entry)
  uint32_t* isa = nullptr;
  const uint32_t* cpos = nullptr;   // suffix array positions of the members, and their groups
  const uint32_t* group = nullptr;
  uint32_t* out = nullptr;          // the same for the next round (out: the long LCPs' positions for kLcp)
  uint32_t* group_out = nullptr;
  uint2* totals = nullptr;          // kSaScanBlocks
  uint32_t* result = nullptr;       // host memory: members left, 1 if a group is large
  uint32_t* listed = nullptr;       // kLcp: how many long LCPs
  uint32_t* member = nullptr;
  uint32_t* second = nullptr;
  uint32_t* new_group = nullptr;
  uint8_t* enc = nullptr;
  uint64_t* eoff = nullptr;
  const uint32_t* perm2 = nullptr;
  const uint32_t* lcp2 = nullptr;
  SaSnaps snaps{};
};

cudaError_t sa_launch(SaKernel k, const SaArgs& x, uint32_t sms, cudaStream_t st, const LaunchHook& hook);

}  // namespace ss
