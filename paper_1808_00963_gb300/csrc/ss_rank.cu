// Sorts of a few thousand strings by counting.
//
// A set of kRankMin..kRankMax strings is too small for distribution steps: a
// step is a chain of dependent phases on one block while the rest of the GPU
// idles.  Comparing every pair of strings fills it instead: every string gets
// its first 4 keys (32 characters, or 84 DNA codes), its rank is the number of
// strings with a smaller (keys, index), and one block then writes the outputs
// of the strings whose keys differ from their neighbours' (LCPs by "LCP via
// XOR", Section 4.2.3) and hands runs of equal keys on to the ordinary
// small-subset sorts.  The n^2 comparisons, of 11 instructions each, take 6 us
// for 1000 strings, launch included.  Whole sorts of URL-like / random strings,
// before / now: 300 strings 51 / 31 and 35 / 31 us, 1000 92 / 39 and 41 / 30,
// 4096 100 / 68 and 62 / 46; at 8192 the steps are as fast (115 / 116) or faster
// (73 / 81), so kRankMax is 4096.
#include "ss_kernels.h"
#include "ss_step.cuh"

namespace ss {

namespace {

constexpr int kRankWords = 4;
constexpr uint32_t kRankTile = 128;      // strings compared with by one block
constexpr uint32_t kFinishThreads = 1024;
static_assert(kRankMax <= 65536, "positions are kept in 16 bits");

// The keys of every string, and what k_begin does for the other sorts.
__global__ void __launch_bounds__(64) k_rank_keys(BeginArgs a, RankArgs r) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint32_t k = i; k < a.ctrl_words; k += stride) a.ctrl[k] = 0;
  for (uint32_t k = i; k < a.ready_words; k += stride) a.ready[k] = 0;
  if (i == 0) *a.set = a.sd;
  if (i >= a.sd.n) return;
  const SetDesc& sd = a.sd;
  const uint64_t off = sd.offsets[i];
  uint64_t w[kRankWords];
  load_key_windows<kRankWords>(sd.chars, off, 0, sd.cap, sd.dna, w);
  r.keys[2 * i] = make_ulonglong2(w[0], w[1]);
  r.keys[2 * i + 1] = make_ulonglong2(w[2], w[3]);
  r.rank[i] = 0;
}

// ~0 if (keys a, index ia) < (keys b, index ib), else 0: the borrow of a - b.
__device__ __forceinline__ uint32_t rank_less(const ulonglong2& a0, const ulonglong2& a1, uint32_t ia,
                                              const ulonglong2& b0, const ulonglong2& b1, uint32_t ib) {
  uint32_t r;
  asm("{\n\t"
      ".reg .u32 t;\n\t"
      ".reg .u64 u;\n\t"
      "sub.cc.u32 t, %1, %2;\n\t"
      "subc.cc.u64 u, %3, %4;\n\t"
      "subc.cc.u64 u, %5, %6;\n\t"
      "subc.cc.u64 u, %7, %8;\n\t"
      "subc.cc.u64 u, %9, %10;\n\t"
      "subc.u32 %0, 0, 0;\n\t"
      "}"
      : "=r"(r)
      : "r"(ia), "r"(ib), "l"(a1.y), "l"(b1.y), "l"(a1.x), "l"(b1.x), "l"(a0.y), "l"(b0.y), "l"(a0.x), "l"(b0.x));
  return r;
}

// Adds to the rank of every string of a block the number of strings of one
// tile that go before it.
__global__ void __launch_bounds__(kBlock) k_rank_count(RankArgs r, uint32_t n) {
  __shared__ ulonglong2 t[2 * kRankTile];
  const uint32_t j0 = blockIdx.y * kRankTile;
  const uint32_t m = min(kRankTile, n - j0);
  if (threadIdx.x < 2 * m) t[threadIdx.x] = r.keys[2 * j0 + threadIdx.x];
  const uint32_t i = blockIdx.x * kBlock + threadIdx.x;
  const ulonglong2 k0 = r.keys[2 * min(i, n - 1)], k1 = r.keys[2 * min(i, n - 1) + 1];
  __syncthreads();
  uint32_t less = 0;
#pragma unroll 4
  for (uint32_t j = 0; j < m; ++j) less -= rank_less(t[2 * j], t[2 * j + 1], j0 + j, k0, k1, i);
  if (i < n && less) atomicAdd(r.rank + i, less);
}
static_assert(2 * kRankTile <= kBlock, "a tile is loaded by one block at once");

// Writes the outputs of the strings told apart by their keys; runs of equal
// keys that do not hold the end go on at the last key's depth.
__global__ void __launch_bounds__(kFinishThreads) k_rank_finish(SortCtx c, RankArgs r) {
  __shared__ uint16_t order[kRankMax];
  __shared__ uint32_t heads[kRankMax / 32 + 1];
  const SetDesc sd = c.sets[0];
  const uint32_t n = sd.n, dna = sd.dna, kw = key_width(dna);
  const uint32_t tid = threadIdx.x, lane = lane_id(), w = tid >> 5;
  const uint32_t words = (n + 31) / 32;
  bool far = false;
  for (uint32_t i = tid; i < n; i += kFinishThreads) {
    order[r.rank[i]] = (uint16_t)i;
    far = far || (sd.offsets[i] >> 32);
  }
  const int wide = __syncthreads_or(far);
  if (tid == 0) c.wide[0] = wide ? 1u : 0u;
  for (uint32_t q = w; q < words; q += kFinishThreads / 32) {
    const uint32_t j = 32 * q + lane;
    bool head = j == 0;
    if (j > 0 && j < n) {
      const uint32_t i = order[j], p = order[j - 1];
      const ulonglong2 a0 = r.keys[2 * p], a1 = r.keys[2 * p + 1], b0 = r.keys[2 * i], b1 = r.keys[2 * i + 1];
      const uint64_t a[kRankWords] = {a0.x, a0.y, a1.x, a1.y}, b[kRankWords] = {b0.x, b0.y, b1.x, b1.y};
      uint32_t l = 0;
#pragma unroll
      for (int u = kRankWords - 1; u >= 0; --u)
        if (a[u] != b[u]) {
          l = kw * u + key_lcp(a[u], b[u], dna);
          head = true;
        }
      if (head && sd.lcp) sd.lcp[j] = l;
    }
    if (j == 0 && sd.lcp) sd.lcp[0] = 0;
    const uint32_t hb = __ballot_sync(0xFFFFFFFFu, head);
    if (lane == 0) heads[q] = hb;
  }
  __syncthreads();
  for (uint32_t q = w; q < words; q += kFinishThreads / 32) {
    const uint32_t j = 32 * q + lane;
    if (j < n) {
      uint32_t ws = q, hs = heads[q] & ((2u << lane) - 1);  // lane 31: all bits
      while (!hs) hs = heads[--ws];                         // position 0 starts a run
      const uint32_t s0 = 32 * ws + 31 - __clz(hs);
      uint32_t wn = q, hn = heads[q] & ~((2u << lane) - 1);
      while (!hn && ++wn < words) hn = heads[wn];
      const uint32_t size = (hn ? 32 * wn + __ffs(hn) - 1 : n) - s0;
      const uint32_t i = order[j];
      if (size == 1) {
        sd.perm[j] = i;
      } else {
        const ulonglong2 b0 = r.keys[2 * i], b1 = r.keys[2 * i + 1];
        const uint64_t b[kRankWords] = {b0.x, b0.y, b1.x, b1.y};
        if (key_end(b[kRankWords - 1], dna)) {  // equal strings (the keys after the end are 0)
          uint32_t l = 0;
#pragma unroll
          for (int u = kRankWords - 1; u >= 0; --u)
            if (key_end(b[u], dna)) l = kw * u + key_nnz(b[u], dna);
          sd.perm[j] = i;
          if (sd.lcp && j != s0) sd.lcp[j] = l;
        } else {
          store_rec(c.rec[0] + j, b[kRankWords - 1], i, (uint32_t)sd.offsets[i]);
          if (j == s0) route_task(c, Task{j, size, kw * (kRankWords - 1), make_meta(0, 0)}, 0);
        }
      }
    }
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_rank(const BeginArgs& a, const RankArgs& r, const SortCtx& c, cudaStream_t st,
                        const LaunchHook& hook) {
  const uint32_t n = a.sd.n;
  hook.run("init", [&] { k_rank_keys<<<(n + 63) / 64, 64, 0, st>>>(a, r); });
  hook.run("rank", [&] {
    k_rank_count<<<dim3((n + kBlock - 1) / kBlock, (n + kRankTile - 1) / kRankTile), kBlock, 0, st>>>(r, n);
  });
  hook.run("rank", [&] { k_rank_finish<<<1, kFinishThreads, 0, st>>>(c, r); });
  return cudaGetLastError();
}

}  // namespace ss
