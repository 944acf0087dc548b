// Persistent work-queue kernel: the GPU counterpart of the job queue of
// Section 4.2.8.  Each block repeatedly claims a subset from a device queue
// and runs one complete S^5 step on it (Algorithm 4.1: sample, splitter tree,
// classification, counting, prefix sum, stable redistribution).  Buckets that
// are still unsorted and larger than the small-sort cutoff are pushed back
// onto the same queue (an equality bucket whose splitter has no terminator is
// requeued at depth + 8); smaller ones go to the small-sort lists.
//
// Termination: `pending` counts tasks pushed and not yet finished; a block
// that finds its claimed slot empty exits once pending is 0.  Every wait is
// bounded (SortCtx::wait_ns of wall-clock time), after which the status word
// is latched and the block exits.
#include "ss_kernels.h"
#include "ss_step.cuh"

namespace ss {

namespace {

// Threads of a block.  Most subsets are a few thousand strings and the last
// ones to be split decide when the kernel ends (blocks of the 1 M URL sort
// were idle for 4/5 of it), so a step is built for latency: 16 warps at 64
// registers, two blocks per SM.  Cycles of an average step (2600 strings, 20 M
// URLs) with three 256-thread blocks per SM / now: sample and splitters
// 24.5k / 12.7k, classification 13.6k / 11.5k, scatter 53k / 29k.  1 M URLs 788
// -> 726 us, suffix array of 4 M characters 1791 -> 1742, 20 M URLs 4370 -> 4281;
// four records per lane and move batch spill: 740 / 1809 / 4355 us.
constexpr uint32_t kQueueThreads = 512;
constexpr uint32_t kQueueWarps = kQueueThreads / 32;
constexpr uint32_t kQueueBlocks = 2;                      // per SM
constexpr uint32_t kQueueRounds = kMaxTile / kQueueThreads;  // tile = kQueueThreads * rounds records
constexpr int kQueueMoveBatch = 2;                        // records per lane moved together

template <int LOGV>
struct QueueSmem {
  SampleSmem<LOGV, uint64_t> sm;
  uint32_t hist[Geo<LOGV>::KP];    // bucket sizes, then running destinations
  uint32_t bstart[Geo<LOGV>::KP];  // bucket starts relative to the task (KP >= K + 1)
  uint32_t desc[Geo<LOGV>::KP];
  union {
    struct {
      // largest LCP of an even bucket's keys with the splitter below / above it
      uint32_t below[Geo<LOGV>::V + 1];
      uint32_t above[Geo<LOGV>::V + 1];
      uint32_t used[64];           // bit i of word w: bucket 32 w + i is not empty
    } lc;
    uint16_t cntw[kQueueWarps * Geo<LOGV>::KP];
  } u;
  uint16_t tb[kMaxTile];           // bucket of each record of a tile
  u128 lead[kLookWindows / 2];     // look-ahead of a subset's first string
  uint32_t jstop;
  Task task;
  uint32_t got;
};

// Claims the next task: waits (bounded) until it has been pushed, or until all
// work is done (no task pending: nothing can be pushed any more).
__device__ bool claim_task(const WorkQueue& q, Task* out, uint32_t* status, uint64_t wait_ns) {
  const uint32_t k = atomicAdd(q.head, 1u);
  const uint32_t slot = k % q.cap, lap = k / q.cap;
  const uint64_t t0 = globaltimer_ns();
  uint32_t ns = 64;
  volatile uint32_t* pending = q.pending;
  while (true) {
    if (load_acquire(q.ready + slot) == 2 * lap + 1) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(q.items + slot));
      *out = Task{v.x, v.y, v.z, v.w};
      store_release(q.ready + slot, 2 * lap + 2);  // the task is read before the slot goes to the next lap
      return true;
    }
    if (*pending == 0) return false;
    if (globaltimer_ns() - t0 > wait_ns) {
      latch_status(status, kStTimeout);
      return false;
    }
    __nanosleep(ns);
    ns = ns < 2048 ? ns * 2 : ns;
  }
}

// Exclusive scan of n counters in shared memory.
__device__ void block_excl_scan_smem(const uint32_t* in, uint32_t* out, uint32_t n) {
  __shared__ uint32_t wsum[kQueueWarps];
  const uint32_t per = (n + kQueueThreads - 1) / kQueueThreads;
  const uint32_t b0 = min(n, threadIdx.x * per), b1 = min(n, b0 + per);
  uint32_t s = 0;
  for (uint32_t j = b0; j < b1; ++j) s += in[j];
  uint32_t inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane_id() >= (uint32_t)o) inc += t;
  }
  const uint32_t w = threadIdx.x >> 5;
  if (lane_id() == 31) wsum[w] = inc;
  __syncthreads();
  uint32_t run = inc - s;
#pragma unroll
  for (uint32_t k = 0; k < kQueueWarps; ++k) run += k < w ? wsum[k] : 0u;
  for (uint32_t j = b0; j < b1; ++j) {
    const uint32_t v = in[j];
    out[j] = run;
    run += v;
  }
  __syncthreads();
}

// Prefix jump of a subset whose keys at `depth` are all equal and hold no end:
// every string's next 64 characters are compared with the first one's, and the
// subset goes on, in place, at the first window where some string differs or
// ends.  Without it a subset sharing a long prefix was moved once for every 8
// characters of it (6000 strings sharing 200 characters 683 -> 242 us; the
// queue of 1 M URLs 125 -> 100 us, of the suffix array of 4 M characters, whose
// steps pay for the registers, 360 -> 373).  Returns the new depth, with the
// records' keys reloaded; the task's depth if some key differs.  Two keys at a
// time in a loop that is not unrolled: the look-ahead of the block sorts, eight
// at once, took more registers than the step has to spare (20 M URLs: the
// queue 455 -> 530 us, inline or as a call).
template <int LOGV, bool DNA>
__device__ __forceinline__ uint32_t queue_jump(const SortCtx& c, QueueSmem<LOGV>& s) {
  constexpr uint32_t NT = kQueueThreads, kDna = DNA ? 1u : 0u;
  const Task t = s.task;
  const SetDesc sd = c.sets[task_set(t)];
  Rec* recs = c.rec[task_par(t)] + t.begin;
  const uint32_t kw = key_width(kDna);
  if (t.depth + kw * kLookWindows > kMaxDepth) return t.depth;
  const uint64_t key = s.sm.sample[0];
  bool differs = false;
  for (uint32_t p = threadIdx.x; p < t.len; p += NT) differs = differs || recs[p].key != key;
  if (threadIdx.x == 0) s.jstop = kLookWindows - 1;
  if (__syncthreads_or(differs)) return t.depth;
  const uint32_t wide = c.wide[task_set(t)];
  // (the first string of the subset is its own first lead: it agrees with itself)
  for (int lead = 1; lead >= 0; --lead) {
    const uint32_t end = lead ? 1u : t.len;
    for (uint32_t p = threadIdx.x; p < end; p += NT) {
      const uint64_t off = rec_offset(sd, wide, recs[p].idx, recs[p].off);
#pragma unroll 1
      for (uint32_t q = 0; q < (uint32_t)kLookWindows / 2; ++q) {
        const u128 k = load_key128(sd.chars, off, t.depth + kw * (2 * q + 1), sd.cap, kDna);
        if (lead) s.lead[q] = k;
        const u128 l = s.lead[q];
        if (k != l || KeyOps<u128>::end(k, kDna)) {
          const bool first = k_hi(k) != k_hi(l) || key_end(k_hi(k), kDna);
          atomicMin(&s.jstop, 2 * q + (first ? 0u : 1u));
          break;
        }
      }
    }
    __syncthreads();
  }
  const uint32_t nd = t.depth + kw * (s.jstop + 1);
  for (uint32_t p = threadIdx.x; p < t.len; p += NT)
    recs[p].key = load_key(sd.chars, rec_offset(sd, wide, recs[p].idx, recs[p].off), nd, sd.cap, kDna);
  __syncthreads();
  return nd;
}

// The sampling of the step on the block's task (and the zeroing of its
// counters); returns whether the whole sample is one key without an end.
template <int LOGV, bool DNA>
__device__ __forceinline__ bool queue_sample(const SortCtx& c, QueueSmem<LOGV>& s) {
  using Gm = Geo<LOGV>;
  const Task t = s.task;
  constexpr uint32_t dna = DNA ? 1u : 0u;
  for (uint32_t b = threadIdx.x; b < Gm::KP; b += kQueueThreads) {
    s.hist[b] = 0;
    if (b <= Gm::V) s.u.lc.below[b] = s.u.lc.above[b] = 0;
  }
  const Rec* recs = c.rec[task_par(t)] + t.begin;
  build_splitters<LOGV, uint64_t, kQueueThreads>([&](uint32_t pos) { return recs[pos].key; }, t.len,
                                                 mix64(c.seed ^ ((uint64_t)t.begin << 20) ^ t.depth), s.sm, dna);
  const uint64_t k0 = s.sm.sample[0];  // the sorted sample
  return k0 == s.sm.sample[Gm::S - 1] && !key_end(k0, dna);
}

// The rest of the S^5 step on task t by this block, after its sampling.
// Returns this thread's share of the step's algorithmic bytes: the sample,
// cache 8 read + bucket index 2 written per record while classifying, and the
// bytes of each record's move.
template <int LOGV, bool DNA>
__device__ unsigned long long queue_step(const SortCtx& c, const Task& t, QueueSmem<LOGV>& s) {
  using Gm = Geo<LOGV>;
  constexpr uint32_t NT = kQueueThreads, kDna = DNA ? 1u : 0u;
  const SetDesc sd = c.sets[task_set(t)];
  const uint32_t par = task_par(t);
  const Rec* recs = c.rec[par] + t.begin;
  const uint32_t wide = c.wide[task_set(t)];
  Splitters<LOGV>& sp = s.sm.sp;
  const bool with_lcp = sd.lcp != nullptr;
  unsigned long long bytes = threadIdx.x == 0 ? Gm::S * 8ull : 0ull;

  // classification (Algorithm 4.1): classify into the array o and count.  With
  // an LCP output also how far each even bucket's keys agree with the
  // splitters around it: its smallest key x has the largest LCP with the
  // splitter below, its largest key with the one above.  These are small
  // numbers, raised with 32-bit atomics where they grow (minima and maxima of
  // the 64-bit keys themselves took a compare-and-swap loop per key).
  // A subset of at most one tile keeps its bucket indices in shared memory.
  const bool one_tile = t.len <= kMaxTile;
  uint16_t* bo = one_tile ? s.tb : c.bucket_of + t.begin;
  bytes += 10ull * classify_count_k<LOGV, uint64_t, NT>(
      [&](uint32_t p) { return recs[p].key; }, bo, t.len, sp.tree, sp.x, s.hist, c.classifier, nullptr,
      [&](uint32_t b, uint64_t k) {
        if (!with_lcp || (b & 1u)) return;
        const uint32_t r = b >> 1;
        if (r > 0) {
          const uint32_t l = key_lcp(k, sp.x[r - 1], kDna);
          if (l > s.u.lc.below[r]) atomicMax(&s.u.lc.below[r], l);
        }
        if (r < Gm::V) {
          const uint32_t l = key_lcp(k, sp.x[r], kDna);
          if (l > s.u.lc.above[r]) atomicMax(&s.u.lc.above[r], l);
        }
      });
  __syncthreads();

  // prefix sum over the bucket sizes; bucket outcomes
  for (uint32_t b = threadIdx.x; b < Gm::KP; b += NT) {  // whole warps: KP is a multiple of 32
    const uint32_t used = __ballot_sync(0xFFFFFFFFu, b < Gm::K && s.hist[b] != 0);
    if (lane_id() == 0) s.u.lc.used[b >> 5] = used;
  }
  block_excl_scan_smem(s.hist, s.bstart, Gm::KP);  // bstart[K] = len (hist[K] is 0)
  if (with_lcp) {
    // LCP at each bucket boundary (Section 4.2.3 "LCP via XOR", Section 4.2.8
    // "LCP Calculation"): between the last string of the previous non-empty
    // bucket and the first string of this one lie the splitters x_a <= ... <=
    // x_b, and for keys u <= v <= w lcp(u, w) is the smaller of lcp(u, v) and
    // lcp(v, w).  An equality bucket's key is its splitter.
    const uint64_t some = nonzero_words(s.u.lc.used, Gm::KP / 32);
    for (uint32_t b = threadIdx.x; b < Gm::K; b += NT) {
      if (!s.hist[b]) continue;
      const uint32_t pb = last_set_before(s.u.lc.used, some, b);
      if (pb == kNone) continue;
      const uint32_t ra = pb >> 1, rb = (b & 1u) ? b >> 1 : (b >> 1) - 1;
      uint32_t l = key_lcp(sp.x[ra], sp.x[rb], kDna);
      if (!(pb & 1u)) l = min(l, s.u.lc.above[ra]);
      if (!(b & 1u)) l = min(l, s.u.lc.below[b >> 1]);
      sd.lcp[t.begin + s.bstart[b] - sd.base] = t.depth + l;
    }
    __syncthreads();  // hist is overwritten below
  }
  for (uint32_t b = threadIdx.x; b < Gm::K; b += NT) {
    const uint32_t size = s.hist[b];
    s.desc[b] = size ? bucket_desc<LOGV>(b, size, t.depth, sp, kDna) : kFin;
    s.hist[b] = t.begin + s.bstart[b];
  }
  __syncthreads();

  // redistribution: stable and out of place, tile by tile; a subset that fits
  // one tile is spread over all warps (each warp owns 32 * R consecutive
  // records of a tile)
  const uint32_t R = min(kQueueRounds, (t.len + NT - 1) / NT);
  const uint32_t T = NT * R;
  for (uint32_t t0 = 0; t0 < t.len; t0 += T) {
    const uint32_t tl = min(T, t.len - t0);
    if (!one_tile) {
      for (uint32_t p = threadIdx.x; p < tl; p += NT) s.tb[p] = bo[t0 + p];
      __syncthreads();
    }
    const uint32_t src0 = t.begin + t0;
    tile_scatter<LOGV, NT, kQueueMoveBatch>(
        s.tb, tl, R, s.hist, s.u.cntw,
        [&](const uint32_t(&pp)[kQueueMoveBatch], const uint32_t(&bb)[kQueueMoveBatch],
            const uint32_t(&dd)[kQueueMoveBatch]) {
          bytes += move_batch<kQueueMoveBatch, DNA>(c, sd, wide, par, src0, t.depth, s.desc,
                                               [&](uint32_t b) { return t.begin + s.bstart[b]; }, pp, bb, dd);
        });
  }
  __syncthreads();

  // new subsets become visible only after their records have been moved (the
  // push releases what the block wrote before the barrier)
  for (uint32_t b = threadIdx.x; b < Gm::K; b += NT) {
    const uint32_t start = s.bstart[b];
    const uint32_t size = s.bstart[b + 1] - start;
    if (size) emit_bucket(c, sd, t, start, size, s.desc[b], 0, false);  // boundary LCPs are written already
  }
  return bytes;
}

// (the character encoding is fixed per instance: at 64 registers the branches on
// it cost spills, 372 -> 357 us in the suffix array of 4 M characters)
template <int LOGV, bool DNA>
__global__ void __launch_bounds__(kQueueThreads, kQueueBlocks) k_queue(SortCtx c) {
  extern __shared__ __align__(16) uint8_t smem[];
  QueueSmem<LOGV>& s = *reinterpret_cast<QueueSmem<LOGV>*>(smem);
  unsigned long long bytes = 0;
  while (true) {
    if (threadIdx.x == 0) s.got = claim_task(c.mq, &s.task, c.status, c.wait_ns) ? 1u : 0u;
    __syncthreads();
    if (!s.got) break;
    while (queue_sample<LOGV, DNA>(c, s)) {
      const uint32_t nd = queue_jump<LOGV, DNA>(c, s);
      if (nd == s.task.depth) break;
      __syncthreads();
      if (threadIdx.x == 0) s.task.depth = nd;
      __syncthreads();
    }
    const Task t = s.task;
    bytes += queue_step<LOGV, DNA>(c, t, s);
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicSub(c.mq.pending, 1u);
    }
  }
  account(c, kKQueue, bytes);
}

template <int LOGV>
cudaError_t set_limits_t() {
  constexpr cudaFuncAttribute kLimit = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(k_queue<LOGV, false>, kLimit, (int)sizeof(QueueSmem<LOGV>));
  return e == cudaSuccess ? cudaFuncSetAttribute(k_queue<LOGV, true>, kLimit, (int)sizeof(QueueSmem<LOGV>)) : e;
}

template <int LOGV>
cudaError_t occupancy_t(int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_queue<LOGV, false>, kQueueThreads,
                                                       sizeof(QueueSmem<LOGV>));
}

template <int LOGV, bool DNA>
cudaError_t launch_queue_t(const SortCtx& c, uint32_t grid, cudaStream_t st, const LaunchHook& hook) {
  hook.run("queue", [&] { k_queue<LOGV, DNA><<<grid, kQueueThreads, sizeof(QueueSmem<LOGV>), st>>>(c); });
  return cudaGetLastError();
}

template <bool DNA>
cudaError_t launch_queue_d(int logv, const SortCtx& c, uint32_t grid, cudaStream_t st, const LaunchHook& hook) {
  switch (logv) {
    case 7: return launch_queue_t<7, DNA>(c, grid, st, hook);
    case 8: return launch_queue_t<8, DNA>(c, grid, st, hook);
    case 9: return launch_queue_t<9, DNA>(c, grid, st, hook);
    default: return launch_queue_t<10, DNA>(c, grid, st, hook);
  }
}

}  // namespace

cudaError_t set_queue_limits() {
  cudaError_t e = set_limits_t<7>();
  if (e == cudaSuccess) e = set_limits_t<8>();
  if (e == cudaSuccess) e = set_limits_t<9>();
  if (e == cudaSuccess) e = set_limits_t<10>();
  return e;
}

cudaError_t queue_occupancy(int logv, int* blocks_per_sm) {
  switch (logv) {
    case 7: return occupancy_t<7>(blocks_per_sm);
    case 8: return occupancy_t<8>(blocks_per_sm);
    case 9: return occupancy_t<9>(blocks_per_sm);
    default: return occupancy_t<10>(blocks_per_sm);
  }
}

cudaError_t launch_queue(int logv, const SortCtx& c, uint32_t grid, cudaStream_t st, const LaunchHook& hook) {
  return c.dna ? launch_queue_d<true>(logv, c, grid, st, hook) : launch_queue_d<false>(logv, c, grid, st, hook);
}

}  // namespace ss
