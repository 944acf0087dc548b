// Small subsets, initial set-up and the final LCP fix-up.
//
// A subset of at most small_cutoff strings with a common prefix of `depth`
// characters is finished by one block (33..cutoff strings) or one warp (2..32)
// without further distribution steps.  A block splits the subset once by a
// sample of its caches and ranks every string by counting within its bucket; a
// warp sorts its strings by (segment, cache, index) with a network in
// registers.  Runs of equal caches without a terminator are refined by
// reloading their caches deeper and sorting again (the recursion of the
// equality buckets of Section 4.2.2, done in place).  This replaces the paper's
// sequential base cases (caching multikey quicksort and insertion sort,
// Section 4.2.8).  LCPs between neighbours are computed from the caches as they
// are separated (Section 4.2.3, "LCP via XOR").
#include "ss_kernels.h"
#include "ss_step.cuh"

namespace ss {

namespace {

__device__ __forceinline__ uint32_t find_set(const SortCtx& c, uint32_t r) {
  uint32_t lo = 0, hi = c.num_sets - 1;  // last set with base <= r
  while (lo < hi) {
    uint32_t mid = (lo + hi + 1) >> 1;
    if (c.sets[mid].base <= r) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Prepares a sort's workspace: zeroes the control words, the work queue's
// flags and the sets' wide flags, and writes the set descriptor and the
// multi-block loop's control block where they are given (kernel parameters, so
// the host stages and waits for nothing).  One launch for what took three
// memsets and two or three kernels (with the status word in host memory, 1000
// URLs 151 -> 124 us, 100 k random strings 140 -> 128 us).
__global__ void __launch_bounds__(kBlock) k_begin(BeginArgs a) {
  const uint32_t i0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint32_t i = i0; i < a.ctrl_words; i += stride) a.ctrl[i] = 0;
  for (uint32_t i = i0; i < a.ready_words; i += stride) a.ready[i] = 0;
  for (uint32_t i = i0; i < a.num_sets; i += stride) a.wide[i] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (a.set) *a.set = a.sd;
    if (a.ctl) {
      *a.ctl = a.v;
      if (a.v.cur.G) a.v.cur.gt[0] = a.root;
    }
  }
}

// Records of every set at depth 0, in index order (the stable starting point),
// and one root task per set.
__global__ void __launch_bounds__(kBlock) k_init(SortCtx c) {
  const uint32_t stride = gridDim.x * blockDim.x;
  unsigned long long bytes = 0;
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < c.num_sets; s += stride) {
    const SetDesc sd = c.sets[s];
    if (sd.n == 0) continue;
    if (sd.lcp) sd.lcp[0] = 0;
    if (sd.n == 1) sd.perm[0] = 0;
    else if (c.num_sets > 1 || sd.n <= c.wide_threshold)  // (the host has planned a single set's first round)
      route_task(c, Task{sd.base, sd.n, 0, make_meta(s, 0)}, c.big_cur);
  }
  __syncwarp();
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < c.total; r += stride) {
    const uint32_t s = c.num_sets == 1 ? 0 : find_set(c, r);
    const SetDesc sd = c.sets[s];
    const uint32_t i = r - sd.base;
    const uint64_t off = sd.offsets[i];
    if ((off >> 32) && !c.wide[s]) atomicOr(c.wide + s, 1u);
    if (sd.n > c.wide_threshold) {  // a multi-block root: wide records
      store_wkey(c.rec[0] + r, load_key128(sd.chars, off, 0, sd.cap, sd.dna));
      c.wid[0][r] = make_uint2(i, (uint32_t)off);
      bytes += 48;  // offset 8 + 16 characters read, wide record 24 written
    } else {
      store_rec(c.rec[0] + r, load_key(sd.chars, off, 0, sd.cap, sd.dna), i, (uint32_t)off);
      bytes += 32;  // offset 8 + 8 characters read, record 16 written
    }
  }
  account(c, kKInit, bytes);
}

// What the last kernel of a sort does about its status: it goes into the
// stream's status word, and if a device-side error stopped the sort part way,
// positions it did not reach hold whatever the output buffers held, so every
// set gets the identity permutation and zero LCPs instead and no later kernel
// (this one, or a caller's) follows an index that is out of range.  Called by
// `stride` threads numbered by `thread`; returns whether there was an error.
__device__ __forceinline__ bool end_sort(const SortCtx& c, uint32_t status, uint32_t thread, uint32_t stride) {
  if (!status) return false;
  if (c.fold_status && thread == 0) atomicOr_system(c.fold_status, status);
  for (uint32_t r = thread; r < c.total; r += stride) {
    const SetDesc sd = c.sets[c.num_sets == 1 ? 0 : find_set(c, r)];
    sd.perm[r - sd.base] = r - sd.base;
    if (sd.lcp) sd.lcp[r - sd.base] = 0;
  }
  return true;
}

// ---- warp-level refinement ----------------------------------------------------

constexpr uint32_t kFull = 0xFFFFFFFFu;

// Order of the warp sort: (segment, key, source lane); tag = segment << 5 |
// source lane, segment 32 for idle lanes.  Evaluated without branches.
__device__ __forceinline__ bool wtag_less(uint64_t ka, uint32_t ta, uint64_t kb, uint32_t tb) {
  const uint32_t sa = ta >> 5, sb = tb >> 5;
  return (sa < sb) | ((sa == sb) & ((ka < kb) | ((ka == kb) & (ta < tb))));
}

// Bitonic sort of one (key, tag) per lane, ascending in lane order.
__device__ __forceinline__ void warp_sort(uint32_t& tag, uint64_t& key) {
  const uint32_t lane = lane_id();
#pragma unroll
  for (uint32_t k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      const uint32_t ot = __shfl_xor_sync(kFull, tag, j);
      const uint64_t ok = __shfl_xor_sync(kFull, key, j);
      const bool up = (lane & k) == 0;
      const bool lower = (lane & j) == 0;
      const bool take = (lower == up) ? wtag_less(ok, ot, key, tag) : wtag_less(key, tag, ok, ot);
      tag = take ? ot : tag;
      key = take ? ok : key;
    }
  }
}

// Finishes the subsets ("groups") held by a warp, one string per lane.  Lanes
// [g0, g0 + glen) hold one group: strings with a common prefix of their
// `depth` characters, in ascending index order, with key = their cache at that
// depth.  Lane-static (they do not move): active, g0, chars/cap of the group's
// set and lcp_g, the LCP output at the group's first position.  Sorting by
// (segment, cache, index) splits a group into runs of equal caches; a run of
// one string or of equal strings (cache holds the terminator) is finished;
// every other run jumps over the characters all its members share, found with
// a 64-character look-ahead, and is sorted again.  Writes lcp_g[j] for every
// position j > 0 of each group and returns the index at the lane's position.
// With max_jumps > 0, runs still open after that many look-aheads are handed
// to defer(position in group, run's first position, run length, cache, index,
// offset, depth) on each of their lanes and left unfinished: a few long
// common prefixes would otherwise keep whole warps busy while most of their
// lanes idle (their lcp_g entries after the run's first one stay unwritten).
template <typename Defer>
__device__ uint32_t warp_refine(bool active, uint32_t g0, uint32_t nact, uint64_t key, uint32_t idx,
                                uint64_t off, uint32_t depth, uint32_t cap, const uint8_t* chars, uint32_t dna,
                                uint32_t* lcp_g, uint32_t* status, unsigned long long& bytes, uint32_t max_jumps,
                                Defer&& defer) {
  const uint32_t lane = lane_id();
  uint32_t seg = active ? g0 : 0xFFFFFFFFu;
  uint32_t open = active ? 1u : 0u;
  uint32_t jumps = 0;
  if (!active) { key = ~0ull; idx = 0xFFFFFFFFu; off = 0; depth = 0; }
  const uint32_t upto = (lane == 31) ? kFull : ((2u << lane) - 1);
  while (true) {
    // sort only if some run is out of (cache, index) order: after a look-ahead
    // jump over characters all members share, the runs often still are
    {
      const uint32_t ps0 = __shfl_up_sync(kFull, seg, 1);
      const uint64_t pk0 = __shfl_up_sync(kFull, key, 1);
      const uint32_t pi0 = __shfl_up_sync(kFull, idx, 1);
      const bool disorder = active && lane > 0 && seg == ps0 && (key < pk0 || (key == pk0 && idx < pi0));
      if (__any_sync(kFull, disorder)) {
        // Segments occupy fixed lanes, and depth and open are the same for
        // every member of a segment, so only the key and the source lane
        // move; ties go by source lane, which within a segment is index
        // order.  Index and offset follow from the source lane.
        uint32_t tag = ((active ? seg : 32u) << 5) | lane;
        warp_sort(tag, key);
        const uint32_t src = tag & 31u;
        idx = __shfl_sync(kFull, idx, src);
        off = __shfl_sync(kFull, off, src);
      }
    }
    const uint32_t ps = __shfl_up_sync(kFull, seg, 1);
    const uint64_t pk = __shfl_up_sync(kFull, key, 1);
    const bool start = lane == 0 || seg != ps || key != pk;
    if (active && open && lane > g0 && seg == ps && key != pk && lcp_g) lcp_g[lane - g0] = depth + key_lcp(pk, key, dna);
    const uint32_t starts = __ballot_sync(kFull, active && start);
    const uint32_t my_start = 31 - __clz(starts & upto);
    const uint32_t above = starts & ~upto;
    const uint32_t next = above ? (uint32_t)(__ffs(above) - 1) : nact;
    if (active && open) {
      if (next - my_start == 1) {
        open = 0;
      } else if (key_end(key, dna)) {
        open = 0;
        if (lane != my_start && lcp_g) lcp_g[lane - g0] = depth + key_nnz(key, dna);
      }
    }
    if (active) seg = my_start;
    if (!__any_sync(kFull, active && open)) break;
    if (max_jumps && jumps == max_jumps) {
      if (active && open) defer(lane - g0, my_start - g0, next - my_start, key, idx, off, depth);
      break;
    }
    ++jumps;
    // look-ahead: the first window (8, 16, ... characters deeper) where the
    // members of the run differ or end; the run continues there
    uint64_t w[kLookWindows];
    uint32_t nwin = 0;
    const uint32_t kw = key_width(dna);
    if (active && open) nwin = load_key_windows_block<kLookWindows>(chars, off, depth + kw, cap, dna, w);
    const uint32_t segmask = (next >= 32 ? kFull : ((1u << next) - 1)) & ~((1u << my_start) - 1);
    uint32_t jstop = kLookWindows - 1;
    bool found = false;
#pragma unroll
    for (int j = 0; j < kLookWindows; ++j) {
      const uint64_t lw = __shfl_sync(kFull, w[j], my_start);
      const bool stop = active && open && ((uint32_t)j >= nwin || w[j] != lw || key_end(w[j], dna));
      const uint32_t b = __ballot_sync(kFull, stop) & segmask;
      if (!found && b) { jstop = (uint32_t)j; found = true; }
    }
    if (active && open) {
      const uint32_t nd = depth + kw * (jstop + 1);
      if (nd > kMaxDepth) {
        latch_status(status, kStTooDeep);
        open = 0;
      } else {
        uint64_t k = w[0];
#pragma unroll
        for (int j = 1; j < kLookWindows; ++j) if ((uint32_t)j == jstop) k = w[j];
        key = jstop < nwin ? k : load_key(chars, off, nd, cap, dna);
        depth = nd;
        bytes += 8ull * (jstop + 1);
      }
    }
  }
  return idx;
}

// Packs up to 16 items (lane k < nt holds item k's length, 1..32) into rounds
// of whole items that fit into 32 lanes, in order.  For each round calls
// round(active, g0, nact, k): the lane belongs to item k, whose first lane is
// g0; nact lanes are in use.
template <typename Round>
__device__ __forceinline__ void pack_rounds(uint32_t nt, uint32_t my_len, Round&& round) {
  const uint32_t lane = lane_id();
  const uint32_t upto = (lane == 31) ? kFull : ((2u << lane) - 1);
  uint32_t a = 0;
  while (a < nt) {
    const uint32_t mine = (lane < nt && lane >= a) ? my_len : 0u;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, incl, o);
      if (lane >= (uint32_t)o) incl += t;
    }
    const uint32_t fits = __ballot_sync(kFull, lane >= a && lane < nt && incl <= 32);
    const uint32_t b = 32 - __clz(fits);
    const uint32_t excl = incl - mine;
    const uint32_t startbits = __reduce_or_sync(kFull, (lane >= a && lane < b) ? (1u << excl) : 0u);
    const uint32_t nact = __shfl_sync(kFull, incl, b - 1);
    const uint32_t k = a + __popc(startbits & upto) - 1;
    const uint32_t g0 = 31 - __clz(startbits & upto);
    round(lane < nact, g0, nact, k);
    a = b;
  }
}

// Warps take runs of up to 16 consecutive small tasks and pack as many whole
// tasks as fit into 32 lanes per round.
constexpr uint32_t kPackChunk = 16;
// Look-aheads (64 characters each) a run may take in the first of the two
// passes over the warp tasks; then it is left to the second one.
constexpr uint32_t kFirstPassJumps = 1;

// One pass over a list of warp tasks.  With max_jumps > 0, runs with long
// common prefixes are deferred to the list `out`: their records go back to
// the record buffer at their current positions, and each run becomes a task.
// Last: this is the sort's last kernel.  DNA: the character encoding (with it
// fixed and at 64 registers, four blocks fit an SM).
template <bool Last, bool DNA>
__global__ void __launch_bounds__(kBlock, 4) k_small_warp(SortCtx c, TaskList list, TaskList out, uint32_t max_jumps) {
  constexpr uint32_t dna = DNA ? 1u : 0u;
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t count = min(*list.count, list.cap);
  const uint32_t lane = lane_id();
  unsigned long long bytes = 0;
  // few tasks: one per warp (parallelism); many: up to 16 per warp (packing)
  const uint32_t chunk = min(kPackChunk, max(1u, (count + nwarps - 1) / nwarps));
  for (uint32_t c0 = warp * chunk; c0 < count; c0 += nwarps * chunk) {
    const uint32_t nt = min(chunk, count - c0);
    Task mt{0, 0, 0, 0};
    if (lane < nt) mt = list.items[c0 + lane];
    pack_rounds(nt, mt.len, [&](bool active, uint32_t g0, uint32_t nact, uint32_t k) {
      const uint32_t tb = __shfl_sync(kFull, mt.begin, k & 31);
      const uint32_t tdepth = __shfl_sync(kFull, mt.depth, k & 31);
      const uint32_t tmeta = __shfl_sync(kFull, mt.meta, k & 31);
      uint64_t key = 0, off = 0;
      uint32_t id = 0, cap = kNoCap;
      const uint8_t* chars = nullptr;
      uint32_t* lcp_g = nullptr;
      uint32_t* perm = nullptr;
      const uint32_t par = tmeta >> 31;
      if (active) {
        const SetDesc sd = c.sets[tmeta & 0x7FFFFFFFu];
        const uint32_t e = lane - g0;
        const Rec r = load_rec(c.rec[par] + tb + e);
        key = r.key;
        id = r.idx;
        off = rec_offset(sd, c.wide[tmeta & 0x7FFFFFFFu], r.idx, r.off);
        cap = sd.cap;
        chars = sd.chars;
        lcp_g = sd.lcp ? sd.lcp + (tb - sd.base) : nullptr;
        perm = sd.perm + (tb - sd.base);
      }
      const uint32_t fin = warp_refine(
          active, g0, nact, key, id, off, tdepth, cap, chars, dna, lcp_g, c.status, bytes, max_jumps,
          [&](uint32_t e, uint32_t rs, uint32_t rl, uint64_t k, uint32_t ix, uint64_t o, uint32_t d) {
            store_rec(c.rec[par] + tb + e, k, ix, (uint32_t)o);
            bytes += 16;
            if (e == rs) list_push(out, Task{tb + rs, rl, d, tmeta}, c.status);
          });
      if (active) {
        perm[lane - g0] = fin;
        bytes += lcp_g ? 24 : 20;  // record 16 read; perm 4 (+ lcp 4) written
      }
    });
  }
  account(c, kKSmallWarp, bytes);
  if constexpr (Last) {  // the last block ends the sort
    __shared__ uint32_t s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(c.done, 1u) == gridDim.x - 1 ? 1u : 0u;
    __syncthreads();
    if (s_last) end_sort(c, __ldcg(c.status), threadIdx.x, kBlock);
  }
}

// ---- block-level refinement -------------------------------------------------------
//
// A subset of 33..small_cutoff strings is sorted by one block in shared memory.
// These sorts are bound by instruction issue (their data is on chip), so the
// design minimises the instructions per string: one more splitting by 32 or 64
// sampled keys, after which a string finds its rank by comparing itself with
// the few others of its bucket.  Both launches, 20 M URLs 700 -> 571 us, 1 M
// URLs 190 -> 139, batch of 512 sets 930 -> 700, 4 M DNA suffixes 171 -> 126
// against a block merge sort (runs of 32 by warp networks, merge paths) in 64-
// and 256-thread blocks; merging by binary searches in the partner run took as
// many instructions as the merge paths (794 us on 20 M URLs), one-warp blocks
// for the small subsets 570 / 220 / 834 / 124 us, 128-thread ones 713 / 168 /
// 789 / 173.

constexpr uint32_t kSmallNarrowThreads = 64, kSmallWideThreads = 256;

// Sampled keys, all of them splitters: 2 * S + 1 buckets (bucket 2r + 1: the
// keys equal to splitter r; bucket 2r: those between splitters r - 1 and r).
constexpr uint32_t kNarrowSample = 32, kWideSample = 64;
// Subsets of more than kManySampleAbove strings (a small_cutoff above 1024)
// take more splitters: a string is compared with its bucket, of 2 n / S strings
// on average.  60 sets of 4096 strings with 64 splitters 237 us, with 256 124
// (merge sort before: 133); 2048 strings 110 / 87 (104).
constexpr uint32_t kManySample = 256, kManySampleAbove = 1024;

// Equality buckets of more strings than this get their places in string order
// right away instead of a rank by comparing positions.
constexpr uint32_t kSmallEqual = 64;

template <uint32_t SMAX>
struct SmallSplit {
  uint64_t drawn[SMAX];         // the sample
  uint64_t key[SMAX];           // ... sorted
  uint32_t first[2 * SMAX + 2]; // bucket sizes, then bucket starts
  uint8_t big[2 * SMAX + 2];    // number of a large equality bucket, kNotBig for the others
  uint32_t nbig;
};
constexpr uint32_t kNotBig = 255;

struct SmallSmem {    // carved from dynamic shared memory, for subsets of up to pmax strings
  uint64_t* key;      // cache: in the order before a sort, in sorted order after it
  uint64_t* gkey;     // cache, grouped by bucket
  uint2* open;        // ranges still to be sorted deeper: (start | length << 16, depth)
  uint32_t* idx;      // index, by original position
  uint32_t* off;      // low offset word, by original position
  uint32_t* tmp;      // bucket | place in it << 16; after the sort: runs to hand on, start | length << 16
  uint32_t* heads;    // bit i of word w: sorted position lo + 32 w + i starts a run of equal caches
  uint16_t* pos[2];   // original position, in sorted order (two buffers)
  uint16_t* gpos;     // position before the sort, grouped by bucket
};

__host__ __device__ inline uint32_t small_words(uint32_t pmax) { return pmax / 32 + 1; }

__device__ __forceinline__ SmallSmem small_smem(uint8_t* smem, uint32_t pmax) {
  SmallSmem m;
  m.key = reinterpret_cast<uint64_t*>(smem);
  m.gkey = m.key + pmax;
  m.open = reinterpret_cast<uint2*>(m.gkey + pmax);
  m.idx = reinterpret_cast<uint32_t*>(m.open + small_words(pmax));
  m.off = m.idx + pmax;
  m.tmp = m.off + pmax;
  m.heads = m.tmp + pmax;
  m.pos[0] = reinterpret_cast<uint16_t*>(m.heads + small_words(pmax));
  m.pos[1] = m.pos[0] + pmax;
  m.gpos = m.pos[1] + pmax;
  return m;
}

// Sorts the n elements whose caches are key[0, n) by (cache, place before the
// sort): key becomes sorted, pos_out[i] is pos_in[place of the i-th] (null: the
// place itself).  pos_out must not be pos_in.  Ends with a barrier; the caller
// has written key before a barrier.
// The sample is drawn at pseudo-random places, one from each of S equal
// stretches.  (Evenly spaced places can all hold one key, where the order of
// the strings has a period: with every 16th of 1024 strings the same key, all
// other strings shared one bucket.)
template <uint32_t NT, uint32_t SMAX>
__device__ void small_sort(const SmallSmem& m, SmallSplit<SMAX>& sp, uint64_t* key, uint32_t n, const uint16_t* pos_in,
                           uint16_t* pos_out, uint32_t seed) {
  static_assert(SMAX <= NT, "a sampled key per thread");
  const uint32_t S = SMAX > kWideSample && n <= kManySampleAbove ? kWideSample : SMAX;
  const uint32_t tid = threadIdx.x, lane = lane_id();
  // the sample, put in order by counting
  for (uint32_t b = tid; b < 2 * S + 2; b += NT) sp.first[b] = 0;
  if (tid == 0) sp.nbig = 0;
  uint64_t mine = 0;
  if (tid < S) {
    const uint32_t stretch = 0xFFFFFFFFu / S + 1;  // 2^32 / S
    mine = key[__umulhi(tid * stretch + ((uint32_t)mix64(seed + tid) & (stretch - 1)), n)];
    sp.drawn[tid] = mine;
  }
  __syncthreads();
  if (tid < S) {
    uint32_t r = 0;
#pragma unroll 8
    for (uint32_t i = 0; i < S; ++i) {
      const uint64_t o = sp.drawn[i];  // the same word for every lane
      r += (o < mine || (o == mine && i < tid)) ? 1u : 0u;
    }
    sp.key[r] = mine;
  }
  __syncthreads();
  // bucket of every element, and its place in the bucket (in no particular order)
  for (uint32_t j = tid; j < n; j += NT) {
    const uint64_t k = key[j];
    uint32_t a = 0;
#pragma unroll
    for (uint32_t half = S / 2; half > 0; half >>= 1) a += sp.key[a + half - 1] < k ? half : 0u;
    a += sp.key[a] < k ? 1u : 0u;
    const uint32_t b = 2 * a + ((a < S && sp.key[a] == k) ? 1u : 0u);
    m.tmp[j] = b | atomicAdd(&sp.first[b], 1u) << 16;
  }
  __syncthreads();
  if (tid < 32) {  // bucket starts
    constexpr uint32_t kPer = (2 * SMAX + 2 + 31) / 32;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      const uint32_t b = lane * kPer + u;
      v[u] = b < 2 * S + 2 ? sp.first[b] : 0u;
      sum += v[u];
    }
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, inc, o);
      if (lane >= (uint32_t)o) inc += t;
    }
    uint32_t run = inc - sum;
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      const uint32_t b = lane * kPer + u;
      if (b < 2 * S + 2) {
        sp.first[b] = run;
        sp.big[b] = (b & 1u) && v[u] > kSmallEqual ? (uint8_t)atomicAdd(&sp.nbig, 1u) : (uint8_t)kNotBig;
      }
      run += v[u];
    }
  }
  __syncthreads();
  const uint32_t nbig = sp.nbig;
  if (nbig) {
    // stable places in the large equality buckets: the strings of each in every
    // 32 consecutive ones, by ballots, and the sums of these counts before them
    uint16_t* cnt = reinterpret_cast<uint16_t*>(m.gkey);  // nbig * chunks <= n / 65 * (n / 32 + 1) counts
    const uint32_t chunks = (n + 31) / 32;
    for (uint32_t c0 = tid >> 5; c0 < chunks; c0 += NT / 32) {
      const uint32_t j = 32 * c0 + lane;
      const uint32_t t = j < n ? m.tmp[j] : 0u;
      const uint32_t id = j < n ? sp.big[t & 0xFFFFu] : kNotBig;
      uint32_t place = t >> 16;
      for (uint32_t g = 0; g < nbig; ++g) {
        const uint32_t mask = __ballot_sync(kFull, id == g);
        if (id == g) place = __popc(mask & lanemask_lt());
        if (lane == 0) cnt[g * chunks + c0] = (uint16_t)__popc(mask);
      }
      if (j < n) m.tmp[j] = (t & 0xFFFFu) | place << 16;
    }
    __syncthreads();
    for (uint32_t g = tid; g < nbig; g += NT) {
      uint32_t run = 0;
      for (uint32_t c0 = 0; c0 < chunks; ++c0) {
        const uint32_t v = cnt[g * chunks + c0];
        cnt[g * chunks + c0] = (uint16_t)run;
        run += v;
      }
    }
    __syncthreads();
    for (uint32_t j = tid; j < n; j += NT) {
      const uint32_t id = sp.big[m.tmp[j] & 0xFFFFu];
      if (id != kNotBig) m.tmp[j] += (uint32_t)cnt[id * chunks + j / 32] << 16;
    }
    __syncthreads();
  }
  for (uint32_t j = tid; j < n; j += NT) {
    const uint32_t t = m.tmp[j];
    const uint32_t q = sp.first[t & 0xFFFFu] + (t >> 16);
    m.gkey[q] = key[j];
    m.gpos[q] = (uint16_t)j;
  }
  __syncthreads();
  for (uint32_t q = tid; q < n; q += NT) {
    const uint64_t k = m.gkey[q];
    const uint32_t j = m.gpos[q];
    const uint32_t b = m.tmp[j] & 0xFFFFu;
    const uint32_t s = sp.first[b], e = sp.first[b + 1];
    uint32_t r = s;
    if (b & 1u) {  // equal keys
      if (e - s > kSmallEqual) r = q;  // in string order already
      else
        for (uint32_t i = s; i < e; ++i) r += m.gpos[i] < j ? 1u : 0u;
    } else {
      for (uint32_t i = s; i < e; ++i) {
        const uint64_t o = m.gkey[i];
        r += (o < k || (o == k && m.gpos[i] < j)) ? 1u : 0u;
      }
    }
    __syncwarp(__activemask());
    key[r] = k;  // the unsorted keys are not needed any more
    pos_out[r] = pos_in ? pos_in[j] : (uint16_t)j;
  }
  __syncthreads();
}

// Sorts the subsets of one list: c.small_cta (64-thread blocks) or
// c.small_cta_wide (256 threads; it runs first, and passes runs that the
// 64-thread blocks can take on to them).  While there are fewer than min_count
// subsets in all, the wide launch takes both lists and passes nothing on: a
// larger block is done with a subset sooner, and the GPU is not full anyway.
// Each block claims one subset at a time from its launch's counter (subset sizes vary several-fold, so a fixed share
// per block left many SMs idle at the end); the next subset is claimed, and
// its task read, while the current one sorts.
template <uint32_t NT, uint32_t SMAX, bool DNA>
__global__ void __launch_bounds__(NT) k_small_cta(SortCtx c, uint32_t pmax, uint32_t min_count) {
  constexpr uint32_t dna = DNA ? 1u : 0u;  // the character encoding, fixed per instance
  constexpr uint32_t NW = NT / 32;
  constexpr bool kWide = NT == kSmallWideThreads;
  extern __shared__ __align__(16) uint8_t smem[];
  const SmallSmem m = small_smem(smem, pmax);
  __shared__ SmallSplit<SMAX> split;
  __shared__ uint32_t s_ti, s_open, s_jstop, s_neq, s_runs, s_base;
  __shared__ Task s_task;
  __shared__ uint64_t s_lead[kLookWindows];
  const uint32_t tid = threadIdx.x, lane = lane_id(), w = tid >> 5;
  unsigned long long bytes = 0;
  // Subsets passed on while this launch runs only raise n_narrow from at
  // least min_count - n_wide, so every block of both launches finds the same `few`.
  const uint32_t n_narrow = min(*c.small_cta.count, c.small_cta.cap);
  const uint32_t n_wide = min(*c.small_cta_wide.count, c.small_cta_wide.cap);
  const bool few = n_narrow + n_wide < min_count;
  if (!kWide && few) return;
  // this launch's subsets: the first na of the narrow list, then the wide list
  const uint32_t na = !kWide || few ? n_narrow : 0u;
  const uint32_t count = kWide ? na + n_wide : na;
  const uint32_t hand_max = kWide && !few ? kSmallCtaNarrowMax : 32u;
  auto task_of = [&](uint32_t i) { return i < na ? c.small_cta.items[i] : c.small_cta_wide.items[i - na]; };
  uint32_t* claim = c.small_claim + (kWide ? 1 : 0);
  uint32_t next = 0;  // thread 0: the claimed subset, kept in registers until it is needed
  Task next_task{0, 0, 0, 0};
  if (tid == 0) {
    next = atomicAdd(claim, 1u);
    if (next < count) next_task = task_of(next);
  }
  while (true) {
    if (tid == 0) {
      s_ti = next;
      s_task = next_task;
      s_open = 0;
      s_neq = 0;
      s_runs = 0;
    }
    __syncthreads();
    if (s_ti >= count) break;
    const Task t = s_task;
    if (tid == 0) next = atomicAdd(claim, 1u);
    __syncwarp();  // lane 0 would run on by itself, and every shuffle below would wait for it
    if (t.len > pmax) {  // cannot happen: a list holds only sizes its launch's shared arrays take
      if (tid == 0) latch_status(c.status, kStQueueFull);
      break;
    }
    const SetDesc sd = c.sets[task_set(t)];
    const uint32_t kw = key_width(dna);  // characters per key
    Rec* recs = c.rec[task_par(t)] + t.begin;
    uint32_t* lcp = sd.lcp ? sd.lcp + (t.begin - sd.base) : nullptr;
    uint32_t* perm = sd.perm + (t.begin - sd.base);
    const uint32_t wide = c.wide[task_set(t)];
    uint32_t lo = 0, n = t.len, depth = t.depth;
    // the range being sorted: the whole subset first, then runs of more than
    // 32 strings whose caches were equal (rare), one at a time
    const uint64_t k0 = recs[0].key;
    bool neq = false;
    for (uint32_t j = tid; j < n; j += NT) {
      const Rec r = load_rec(recs + j);
      m.idx[j] = r.idx;
      m.off[j] = r.off;
      m.key[j] = r.key;
      neq = neq || r.key != k0;
    }
    if (neq) s_neq = 1;
    __syncthreads();
    auto off_at = [&](uint32_t j) {  // string offset of the element at sorted position j
      const uint32_t q = m.pos[0][j];
      return rec_offset(sd, wide, m.idx[q], m.off[q]);
    };
    // one run: jump over the prefix all its strings share
    bool sorted = s_neq || key_end(k0, dna);
    if (s_neq) {
      small_sort<NT, SMAX>(m, split, m.key, n, nullptr, m.pos[0], t.begin);
    } else {
      for (uint32_t j = tid; j < n; j += NT) m.pos[0][j] = (uint16_t)j;
      if (tid == 0 && !sorted) {
        m.open[0] = make_uint2(n << 16, depth);
        s_open = 1;
      }
      __syncthreads();
    }
    if (tid == 0 && next < count) next_task = task_of(next);
    __syncwarp();
    while (true) {
      if (sorted) {
        // LCPs between neighbours with different caches, run starts
        const uint64_t* key = m.key;
        const uint32_t nw = (n + 31) / 32;
        for (uint32_t q = w; q < nw; q += NW) {
          const uint32_t j = lo + 32 * q + lane;
          const bool in = 32 * q + lane < n;
          const uint64_t k = in ? key[j] : 0ull;
          const uint64_t pk = in && j > lo ? key[j - 1] : 0ull;
          const bool differs = in && j > lo && k != pk;
          if (differs && lcp) lcp[j] = depth + key_lcp(pk, k, dna);
          const uint32_t hb = __ballot_sync(kFull, differs || j == lo);
          if (lane == 0) m.heads[q] = hb;
        }
        __syncthreads();
        // Runs of one string or of equal strings are finished; runs of at most
        // 32 strings go back to the record buffer as new warp tasks (a warp
        // finishes them without holding this block); larger ones are sorted
        // deeper here.
        for (uint32_t q = w; q < nw; q += NW) {
          const uint32_t j = lo + 32 * q + lane;
          const bool in = 32 * q + lane < n;
          const uint32_t own = m.heads[q];
          uint32_t ws = q, hs = own & ((2u << lane) - 1);  // lane 31: all bits
          while (!hs) hs = m.heads[--ws];                  // position lo starts a run
          const uint32_t s0 = lo + 32 * ws + 31 - __clz(hs);
          uint32_t wn = q, hn = own & ~((2u << lane) - 1);
          while (!hn && ++wn < nw) hn = m.heads[wn];
          const uint32_t size = (hn ? lo + 32 * wn + __ffs(hn) - 1 : lo + n) - s0;
          const uint64_t k = in ? key[j] : 0ull;
          const bool ended = key_end(k, dna);
          const bool fin = in && (size == 1 || ended);
          const bool hand = in && !fin && size <= hand_max;
          const uint32_t src = in ? m.pos[0][j] : 0u;
          const uint32_t id = m.idx[src];
          if (fin) {
            perm[j] = id;
            if (lcp && j != s0) lcp[j] = depth + key_nnz(k, dna);
          } else if (hand) {
            store_rec(recs + j, k, id, m.off[src]);
            bytes += 16;
          }
          if (in && !fin && j == s0) {
            if (size <= 32) m.tmp[atomicAdd(&s_runs, 1u)] = j | size << 16;
            else if (hand) list_push(c.small_cta, Task{t.begin + j, size, depth, t.meta}, c.status);
            else m.open[atomicAdd(&s_open, 1u)] = make_uint2(s0 | size << 16, depth);
          }
          __syncwarp();
        }
        __syncthreads();
        // the runs for the warp list, with one counter update for all of them:
        // every block of the launch appends to the same counter
        const uint32_t runs = s_runs;
        if (runs) {
          if (tid == 0) s_base = atomicAdd(c.small_warp.count, runs);
          __syncthreads();
          for (uint32_t q = tid; q < runs; q += NT) {
            const uint32_t r = m.tmp[q], slot = s_base + q;
            if (slot < c.small_warp.cap) c.small_warp.items[slot] = Task{t.begin + (r & 0xFFFFu), r >> 16, depth, t.meta};
            else latch_status(c.status, kStQueueFull);
          }
          __syncthreads();
          if (tid == 0) s_runs = 0;
        }
      }
      sorted = true;
      const uint32_t left = s_open;
      if (left == 0) break;
      // the next open range: all its caches are equal and hold no terminator;
      // compare each string's next 64 characters with the first one's and
      // continue at the first window where some string differs or ends
      const uint2 r = m.open[left - 1];
      lo = r.x & 0xFFFFu;
      n = r.x >> 16;
      depth = r.y;
      const bool look = depth + kw * kLookWindows <= kMaxDepth;  // else one window only
      __syncthreads();
      if (tid == 0) {
        s_open = left - 1;
        s_jstop = look ? kLookWindows - 1 : 0u;
      }
      uint64_t x[kLookWindows];
      for (uint32_t j0 = 0; j0 < n; j0 += NT) {  // the same code for the leader and the others: it is
        const uint32_t j = j0 + tid;             // run rarely, so fetching it is part of what it costs
        if (look && j < n) load_key_windows<kLookWindows>(sd.chars, off_at(lo + j), depth + kw, sd.cap, dna, x);
        __syncwarp();
        if (j == 0) {
#pragma unroll
          for (int q = 0; q < kLookWindows; ++q) s_lead[q] = x[q];
        }
        if (j0 == 0) __syncthreads();
        uint32_t js = kLookWindows;
        if (look && j < n) {
#pragma unroll
          for (int q = kLookWindows - 1; q >= 0; --q)
            if (x[q] != s_lead[q] || key_end(x[q], dna)) js = (uint32_t)q;
        }
        js = __reduce_min_sync(kFull, js);
        if (lane == 0 && js < kLookWindows) atomicMin(&s_jstop, js);
      }
      __syncthreads();
      const uint32_t jstop = s_jstop;
      depth += kw * (jstop + 1);
      if (depth > kMaxDepth) {
        if (tid == 0) latch_status(c.status, kStTooDeep);
        break;
      }
      for (uint32_t j = tid; j < n; j += NT) {
        if (n <= NT && look) {  // the windows are still at hand
          uint64_t k = x[0];
#pragma unroll
          for (int q = 1; q < kLookWindows; ++q) k = (uint32_t)q == jstop ? x[q] : k;
          m.key[lo + j] = k;
        } else {
          m.key[lo + j] = load_key(sd.chars, off_at(lo + j), depth, sd.cap, dna);
        }
        bytes += 8ull * (jstop + 1);
      }
      __syncthreads();
      small_sort<NT, SMAX>(m, split, m.key + lo, n, m.pos[0] + lo, m.pos[1] + lo, t.begin + lo + depth);
      for (uint32_t j = tid; j < n; j += NT) m.pos[0][lo + j] = m.pos[1][lo + j];
      __syncthreads();
    }
    for (uint32_t j = tid; j < t.len; j += NT) bytes += sd.lcp ? 24 : 20;  // record 16 read; perm 4 (+ lcp 4) written
    __syncthreads();
  }
  account(c, kKSmallCta, bytes);
}

// Resolves the boundary marks left by the multi-block steps (listed in
// c.marks): out_lcp[j] = mark | h means the strings at j-1 and j share exactly
// their first h characters plus the common prefix of their wide keys at depth h.
// (The single-block steps write their boundary LCPs themselves.)
__global__ void __launch_bounds__(kBlock) k_lcp_fix(SortCtx c) {
  const uint32_t stride = gridDim.x * blockDim.x;
  unsigned long long bytes = 0;
  // every other kernel of the sort has finished, so its status is final
  if (end_sort(c, *c.status, blockIdx.x * blockDim.x + threadIdx.x, stride)) return;
  const uint32_t nm = min(*c.marks_count, c.marks_cap);
  for (uint32_t m = blockIdx.x * blockDim.x + threadIdx.x; m < nm; m += stride) {
    const uint32_t r = c.marks[m];
    const uint32_t s = c.num_sets == 1 ? 0 : find_set(c, r);
    const SetDesc sd = c.sets[s];
    const uint32_t j = r - sd.base;
    const uint32_t v = sd.lcp[j];
    bytes += 8;  // list entry and LCP entry read
    if (j == 0 || !(v & kLcpMark)) continue;
    const uint32_t h = v & ~kLcpMark;
    const uint32_t pa = sd.perm[j - 1], pb = sd.perm[j];
    if (pa >= sd.n || pb >= sd.n) continue;  // cannot happen after a sort without errors
    const u128 a = load_key128(sd.chars, sd.offsets[pa], h, sd.cap, sd.dna);
    const u128 b = load_key128(sd.chars, sd.offsets[pb], h, sd.cap, sd.dna);
    sd.lcp[j] = h + KeyOps<u128>::lcp(a, b, sd.dna);
    bytes += 60;  // lcp 4 written; per string: perm 4 + offset 8 + 16 characters read
  }
  account(c, kKLcpFix, bytes);
}

// Distinguishing characters and prefix lengths of a sorted set (Section
// 4.3.4, proof of Lemma 2.1): c^_j = s_j[h_j] and d_j = max(h_j, h_{j+1}) + 1,
// h_0 = h_n = 0; optionally the sum of d_j (= D) into *sum_d.
__global__ void __launch_bounds__(kBlock) k_distinguishing(const uint8_t* __restrict__ chars,
                                                           const uint64_t* __restrict__ offsets, uint32_t n,
                                                           uint32_t cap, const uint32_t* __restrict__ perm,
                                                           const uint32_t* __restrict__ lcp, uint8_t* dchar,
                                                           uint32_t* dprefix, unsigned long long* sum_d) {
  unsigned long long acc = 0;
  const uint32_t stride = gridDim.x * blockDim.x;
  const uint32_t lim = (n + 31) / 32 * 32;
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < lim; j += stride) {
    if (j < n) {
      const uint32_t h = j == 0 ? 0u : lcp[j];
      const uint32_t next = j + 1 < n ? lcp[j + 1] : 0u;
      const uint32_t d = max(h, next) + 1;
      if (dprefix) dprefix[j] = d;
      if (dchar) dchar[j] = h < cap ? chars[offsets[perm[j]] + h] : 0;
      acc += d;
    }
    if (sum_d) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
      if (lane_id() == 0 && acc) atomicAdd(sum_d, acc);
      acc = 0;
    }
  }
}

}  // namespace

// Packs a byte buffer over {A, C, G, T, terminator} into 3-bit codes (0 =
// terminator, 1..4 = A, C, G, T), most significant first, character p at
// bits [3p, 3p + 3) of the word stream; sets *bad if another byte occurs.
__global__ void k_pack_dna(const uint8_t* __restrict__ chars, uint64_t len, uint64_t* __restrict__ out,
                           uint64_t words, uint32_t* bad) {
  for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words;
       w += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t g0 = 64 * w;
    uint64_t v = 0;
    bool invalid = false;
    for (uint64_t p = g0 / 3; p <= (g0 + 63) / 3; ++p) {
      uint64_t code = 0;
      if (p < len) {
        const uint8_t ch = chars[p];
        code = ch == 'A' ? 1 : ch == 'C' ? 2 : ch == 'G' ? 3 : ch == 'T' ? 4 : 0;
        invalid = invalid || (ch != 0 && code == 0);
      }
      const int64_t s = (int64_t)(3 * p) - (int64_t)g0;  // first bit of the code, from the word's top
      v |= s <= 61 ? code << (61 - s) : code >> (s - 61);
    }
    out[w] = v;
    if (invalid) atomicOr(bad, 1u);
  }
}

// Blocks per SM of the two block-sort launches.
constexpr uint32_t kSmallNarrowBlocks = 16, kSmallWideBlocks = 4;

size_t small_cta_smem(uint32_t pmax) {
  return (size_t)pmax * (8 + 8 + 4 + 4 + 4 + 2 + 2 + 2) + (size_t)small_words(pmax) * (8 + 4);
}

cudaError_t launch_begin(const BeginArgs& a, cudaStream_t st, const LaunchHook& hook) {
  const uint32_t words = max(a.ready_words, a.ctrl_words);
  hook.run("init", [&] { k_begin<<<min((words + kBlock - 1) / kBlock, 152u * 2u), kBlock, 0, st>>>(a); });
  return cudaGetLastError();
}

cudaError_t launch_init(const SortCtx& c, cudaStream_t st, const LaunchHook& hook) {
  const uint32_t grid = max(1u, min((max(c.total, c.num_sets) + kBlock - 1) / kBlock, 152u * 16u));
  hook.run("init", [&] { k_init<<<grid, kBlock, 0, st>>>(c); });
  return cudaGetLastError();
}

cudaError_t set_small_limits() {
  constexpr cudaFuncAttribute kLimit = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int wide = (int)small_cta_smem(kSmallCutoffMax);
  constexpr uint32_t kNT = kSmallWideThreads;
  cudaError_t e = cudaFuncSetAttribute(k_small_cta<kNT, kWideSample, false>, kLimit, wide);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small_cta<kNT, kWideSample, true>, kLimit, wide);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small_cta<kNT, kManySample, false>, kLimit, wide);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small_cta<kNT, kManySample, true>, kLimit, wide);
  return e;
}

template <bool DNA>
static cudaError_t launch_small_t(const SortCtx& c, uint32_t pmax, uint32_t sms, bool last, cudaStream_t st,
                                  const LaunchHook& hook) {
  // subsets of more than kSmallCtaNarrowMax strings, then smaller ones
  const uint32_t min_count = 2 * sms * kSmallWideBlocks;
  if (pmax > kSmallCtaNarrowMax) {
    const auto wide = pmax > kManySampleAbove ? k_small_cta<kSmallWideThreads, kManySample, DNA>
                                              : k_small_cta<kSmallWideThreads, kWideSample, DNA>;
    hook.run("small_cta", [&] {
      wide<<<sms * kSmallWideBlocks, kSmallWideThreads, small_cta_smem(pmax), st>>>(c, pmax, min_count);
    });
  }
  const uint32_t narrow_max = min(pmax, kSmallCtaNarrowMax);
  // (so few strings that the wide launch has taken them all: see k_small_cta)
  const bool few = pmax > kSmallCtaNarrowMax && c.total / 33 < min_count;
  if (!few) hook.run("small_cta", [&] {
    k_small_cta<kSmallNarrowThreads, kNarrowSample, DNA>
        <<<sms * kSmallNarrowBlocks, kSmallNarrowThreads, small_cta_smem(narrow_max), st>>>(
            c, narrow_max, pmax > kSmallCtaNarrowMax ? min_count : 0u);
  });
  const uint32_t grid = max(1u, min(sms * 8, (c.total / 2 + kWarps - 1) / kWarps));  // tasks hold at least 2 strings
  if (last) {  // few strings: one pass, there is nothing to gain from packing deferred runs
    hook.run("small_warp", [&] { k_small_warp<true, DNA><<<grid, kBlock, 0, st>>>(c, c.small_warp, c.small_deep, 0u); });
    return cudaGetLastError();
  }
  // the second pass takes what the first one has deferred, and defers nothing
  hook.run("small_warp", [&] {
    k_small_warp<false, DNA><<<grid, kBlock, 0, st>>>(c, c.small_warp, c.small_deep, kFirstPassJumps);
  });
  hook.run("small_warp", [&] { k_small_warp<false, DNA><<<grid, kBlock, 0, st>>>(c, c.small_deep, c.small_warp, 0u); });
  return cudaGetLastError();
}

cudaError_t launch_small(const SortCtx& c, uint32_t pmax, uint32_t sms, bool last, cudaStream_t st,
                         const LaunchHook& hook) {
  return c.dna ? launch_small_t<true>(c, pmax, sms, last, st, hook)
               : launch_small_t<false>(c, pmax, sms, last, st, hook);
}

cudaError_t launch_pack_dna(const uint8_t* chars, uint64_t len, uint64_t* out, uint64_t words, uint32_t* bad,
                            uint32_t grid, cudaStream_t st, const LaunchHook& hook) {
  hook.run("init", [&] { k_pack_dna<<<grid, kBlock, 0, st>>>(chars, len, out, words, bad); });
  return cudaGetLastError();
}

// A few zero words written by a kernel: a copy engine that works on a large
// copy queued on another stream would hold a memset up for milliseconds.
__global__ void k_zero(uint32_t* dst, uint32_t words) {
  for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) dst[i] = 0u;
}

cudaError_t launch_zero(uint32_t* dst, uint32_t words, cudaStream_t st, const LaunchHook& hook) {
  hook.run("zero", [&] { k_zero<<<1, 32, 0, st>>>(dst, words); });
  return cudaGetLastError();
}

cudaError_t launch_distinguishing(const uint8_t* chars, const uint64_t* offsets, uint32_t n, uint32_t cap,
                                  const uint32_t* perm, const uint32_t* lcp, uint8_t* dchar, uint32_t* dprefix,
                                  unsigned long long* sum_d, uint32_t grid, cudaStream_t st, const LaunchHook& hook) {
  hook.run("distinguishing", [&] {
    k_distinguishing<<<grid, kBlock, 0, st>>>(chars, offsets, n, cap, perm, lcp, dchar, dprefix, sum_d);
  });
  return cudaGetLastError();
}

cudaError_t launch_lcp_fix(const SortCtx& c, uint32_t grid, cudaStream_t st, const LaunchHook& hook) {
  hook.run("lcp_fix", [&] { k_lcp_fix<<<grid, kBlock, 0, st>>>(c); });
  return cudaGetLastError();
}

}  // namespace ss
