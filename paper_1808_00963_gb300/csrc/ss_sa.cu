// Suffix array construction by prefix doubling (Section 8.2, Observation 8.1,
// Algorithms 8.1 and 8.3) on top of the string sort.
//
// Round 0 sorts all suffixes by their first h0 characters with the string
// sort (a cap of h0) and names every suffix by the smallest rank of its
// h0-group (ISA^{h0}, names stored + 1 so that 0 stands for "past the end of
// the text").  Each following round takes only the suffixes of unfinished
// groups (those with more than one member; finished groups are discarded, as
// in Larsson and Sadakane's scheme).  The members of a group lie side by side
// in the suffix array and share ISA^h[i], so only ISA^h[i + h] orders them: if
// every group is small (at most kSmallGroup members), each member finds its
// place and new name by comparing itself with the others of its group.
// Otherwise the round encodes the name pair (ISA^h[i], ISA^h[i + h]) of each
// member as a 10-byte string of base-255 digits 1..255 (no zero byte, same
// order as the pair), sorts those strings with the string sort, writes them
// back into their groups' ranges of the suffix array and renames: a new
// 2h-group starts where the pair changes (LCP of the encoded strings below
// 10), its name is the suffix array position of its first member.
#include "ss_kernels.h"

namespace ss {

namespace {

constexpr uint32_t kPairBytes = 10;   // two names of 5 base-255 digits
constexpr uint32_t kPairStride = 11;  // + terminator
constexpr uint32_t kSmallGroup = 256;  // members of a group that are compared with one another (see k_sa_groups)
constexpr uint32_t kNoGroup = 0xFFFFFFFFu;

// ---- naming and compaction in two passes -------------------------------------------------
//
// After a sort every position p of it either starts a group or not.  One pass
// over the positions needs two scans: the last group start up to p (the group,
// hence the name) and the number of unfinished members up to p (their place in
// the next round's list).  k_sa_reduce takes the totals of each block's
// stretch, k_sa_down adds the totals before its stretch and does everything
// else at once.  (As separate kernels, with the flags and starts in memory:
// 9 launches and 106 us for 4 M suffixes; as two: 61 us, 51 of them in
// k_sa_down, whose 4-byte stores to the names go everywhere.)

constexpr uint32_t kScanBlock = 1024;
constexpr uint32_t kScanItems = 4;
constexpr uint32_t kScanTile = kScanBlock * kScanItems;

// A source gives for position p whether it starts a group (start: the group) and
// belongs to an unfinished one (open), and its item: the suffix and its suffix
// array position; name() takes the item and its group.

// The sorted suffixes after round 0 (LCPs capped at h0).
struct SaFirst {
  const uint32_t* sa;
  const uint32_t* lcp;
  uint32_t h;
  uint32_t* isa;
  __device__ __forceinline__ void at(uint32_t p, uint32_t n, uint32_t& start, uint32_t& open) const {
    const bool head = p == 0 || lcp[p] < h;
    const bool next_same = p + 1 < n && lcp[p + 1] >= h;
    start = head ? p : 0u;
    open = !head || next_same ? 1u : 0u;
  }
  __device__ __forceinline__ uint2 item(uint32_t p) const { return make_uint2(sa[p], p); }
  __device__ __forceinline__ void name(uint2 x, uint32_t group) const { isa[x.x] = group + 1; }
};

// The members of unfinished groups after a round's sort of their name pairs.
struct SaPairs {
  const uint32_t* cpos;
  const uint32_t* member;
  const uint32_t* perm;
  const uint32_t* lcp;
  uint32_t* sa;
  uint32_t* isa;
  __device__ __forceinline__ void at(uint32_t p, uint32_t n, uint32_t& start, uint32_t& open) const {
    const bool head = p == 0 || lcp[p] < kPairBytes;
    const bool next_same = p + 1 < n && lcp[p + 1] >= kPairBytes;
    start = head ? cpos[p] : 0u;
    open = !head || next_same ? 1u : 0u;
  }
  __device__ __forceinline__ uint2 item(uint32_t p) const { return make_uint2(member[perm[p]], cpos[p]); }
  __device__ __forceinline__ void name(uint2 x, uint32_t group) const {
    sa[x.y] = x.x;
    isa[x.x] = group + 1;
  }
};

// The same after k_sa_groups, which has named them (group[p]: the new group of
// the member at p, kNoGroup if it is finished).
struct SaGroups {
  const uint32_t* cpos;
  const uint32_t* group;
  __device__ __forceinline__ void at(uint32_t p, uint32_t, uint32_t& start, uint32_t& open) const {
    const uint32_t g = group[p];
    open = g != kNoGroup ? 1u : 0u;
    start = open ? g : 0u;  // (not decreasing over the unfinished members)
  }
  __device__ __forceinline__ uint2 item(uint32_t p) const { return make_uint2(0, cpos[p]); }
  __device__ __forceinline__ void name(uint2, uint32_t) const {}
};

// Maximum and sum over the block, for every thread.
__device__ __forceinline__ void block_max_sum(uint32_t& mx, uint32_t& sum) {
  __shared__ uint32_t wm[kScanBlock / 32], ws[kScanBlock / 32];
  const uint32_t w = threadIdx.x >> 5, lane = lane_id();
  mx = __reduce_max_sync(0xFFFFFFFFu, mx);
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if (lane == 0) {
    wm[w] = mx;
    ws[w] = sum;
  }
  __syncthreads();
  mx = __reduce_max_sync(0xFFFFFFFFu, wm[lane]);
  sum = __reduce_add_sync(0xFFFFFFFFu, ws[lane]);
  __syncthreads();
}
static_assert(kScanBlock == 1024, "block_max_sum: one total per lane");

__device__ __forceinline__ uint32_t sa_stretch(uint32_t n) {  // positions per block, whole tiles
  const uint32_t tiles = (uint32_t)(((uint64_t)n + kScanTile - 1) / kScanTile);
  return (tiles + gridDim.x - 1) / gridDim.x * kScanTile;
}

template <class Src>
__global__ void __launch_bounds__(kScanBlock) k_sa_reduce(Src s, uint32_t n, uint2* totals) {
  const uint64_t per = sa_stretch(n), lo = blockIdx.x * per, hi = min((uint64_t)n, lo + per);
  uint32_t mx = 0, sum = 0;
  for (uint64_t p = lo + threadIdx.x; p < hi; p += kScanBlock) {
    uint32_t start, open;
    s.at((uint32_t)p, n, start, open);
    mx = max(mx, start);
    sum += open;
  }
  block_max_sum(mx, sum);
  if (threadIdx.x == 0) totals[blockIdx.x] = make_uint2(mx, sum);
}

// out / group_out: the suffix array positions of the unfinished members and
// their groups, in order.  result[0] = how many, result[1] set if one of their
// groups has more than kSmallGroup members (host memory, zero at launch).
template <class Src>
__global__ void __launch_bounds__(kScanBlock) k_sa_down(Src s, uint32_t n, const uint2* __restrict__ totals,
                                                        uint32_t* out, uint32_t* group_out,
                                                        volatile uint32_t* result) {
  __shared__ uint32_t wm[kScanItems * 32], ws[kScanItems * 32];
  const uint32_t w = threadIdx.x >> 5, lane = lane_id();
  const uint64_t per = sa_stretch(n), lo = blockIdx.x * per, hi = min((uint64_t)n, lo + per);
  uint32_t mx = 0, sum = 0;  // of everything before the tile
  for (uint32_t b = threadIdx.x; b < blockIdx.x; b += kScanBlock) {
    const uint2 t = totals[b];
    mx = max(mx, t.x);
    sum += t.y;
  }
  block_max_sum(mx, sum);
  bool big = false;
  for (uint64_t t0 = lo; t0 < hi; t0 += kScanTile) {
    uint32_t start[kScanItems], open[kScanItems], im[kScanItems], is[kScanItems];
    uint2 item[kScanItems];
#pragma unroll
    for (uint32_t u = 0; u < kScanItems; ++u) {
      const uint64_t p = t0 + u * kScanBlock + threadIdx.x;
      start[u] = open[u] = 0;
      if (p < hi) {
        s.at((uint32_t)p, n, start[u], open[u]);
        item[u] = s.item((uint32_t)p);  // loaded with the rest, not after the scan
      }
    }
#pragma unroll
    for (uint32_t u = 0; u < kScanItems; ++u) {  // inclusive over the warp
      uint32_t m = start[u];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, m, d);
        if (lane >= (uint32_t)d) m = max(m, o);
      }
      const uint32_t bits = __ballot_sync(0xFFFFFFFFu, open[u] != 0);
      im[u] = m;
      is[u] = __popc(bits & lanemask_lt()) + open[u];
      if (lane == 31) {
        wm[u * 32 + w] = m;
        ws[u * 32 + w] = is[u];
      }
    }
    __syncthreads();
    // the warps' totals in order: the sub-tiles u one after the other
    if (w == 0) {
      uint32_t cm = mx, cs = sum;
#pragma unroll
      for (uint32_t u = 0; u < kScanItems; ++u) {
        uint32_t m = wm[u * 32 + lane], c = ws[u * 32 + lane];
        const uint32_t own = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t om = __shfl_up_sync(0xFFFFFFFFu, m, d), oc = __shfl_up_sync(0xFFFFFFFFu, c, d);
          if (lane >= (uint32_t)d) {
            m = max(m, om);
            c += oc;
          }
        }
        uint32_t before = __shfl_up_sync(0xFFFFFFFFu, m, 1);
        if (lane == 0) before = 0;
        wm[u * 32 + lane] = max(cm, before);
        ws[u * 32 + lane] = cs + c - own;
        cm = max(cm, __shfl_sync(0xFFFFFFFFu, m, 31));
        cs += __shfl_sync(0xFFFFFFFFu, c, 31);
      }
      mx = cm;
      sum = cs;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t u = 0; u < kScanItems; ++u) {
      const uint64_t p = t0 + u * kScanBlock + threadIdx.x;
      if (p < hi) {
        const uint32_t g = max(im[u], wm[u * 32 + w]);
        s.name(item[u], g);
        if (open[u]) {
          const uint32_t at = item[u].y, c = ws[u * 32 + w] + is[u] - 1;
          out[c] = at;
          group_out[c] = g;
          big = big || at - g >= kSmallGroup;
        }
      }
    }
    __syncthreads();
  }
  if (__syncthreads_or(big) && threadIdx.x == 0) result[1] = 1;
  if (hi == n && lo < hi && threadIdx.x == 0) result[0] = sum;  // thread 0 carries the running sum
}

template <class Src>
cudaError_t name_and_compact(const Src& s, uint32_t n, uint2* totals, uint32_t* out, uint32_t* group_out,
                             uint32_t* result, uint32_t sms, cudaStream_t st, const LaunchHook& hook) {
  const uint32_t tiles = (uint32_t)(((uint64_t)n + kScanTile - 1) / kScanTile);
  const uint32_t grid = std::min(std::min(tiles, sms * 2), kSaScanBlocks);
  hook.run("sa_name", [&] { k_sa_reduce<Src><<<grid, kScanBlock, 0, st>>>(s, n, totals); });
  hook.run("sa_name", [&] { k_sa_down<Src><<<grid, kScanBlock, 0, st>>>(s, n, totals, out, group_out, result); });
  return cudaGetLastError();
}

// ---- rounds ------------------------------------------------------------------------

__global__ void k_sa_iota(uint64_t* off, uint64_t n) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    off[i] = i;
}

__device__ __forceinline__ void put_digits(uint8_t* p, uint32_t v) {
#pragma unroll
  for (int k = 4; k >= 0; --k) {
    p[k] = (uint8_t)(v % 255u + 1u);
    v /= 255u;
  }
}

// Name pairs of the unfinished members as 10-byte strings (+ terminator).
__global__ void k_sa_encode(const uint32_t* cpos, uint32_t M, const uint32_t* sa, const uint32_t* isa, uint32_t n,
                            uint32_t h, uint32_t* member, uint8_t* enc, uint64_t* eoff) {
  for (uint64_t at = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; at < M; at += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t m = (uint32_t)at;
    const uint32_t i = sa[cpos[m]];
    member[m] = i;
    const uint32_t k1 = isa[i];
    const uint32_t k2 = (uint64_t)i + h < n ? isa[i + h] : 0u;
    uint8_t* p = enc + (uint64_t)m * kPairStride;
    put_digits(p, k1);
    put_digits(p + 5, k2);
    p[kPairBytes] = 0;
    eoff[m] = (uint64_t)m * kPairStride;
  }
}

// The members of a round with small groups, and the name that orders them.
__global__ void k_sa_second(const uint32_t* cpos, uint32_t M, const uint32_t* sa, const uint32_t* isa, uint32_t n,
                            uint32_t h, uint32_t* member, uint32_t* second) {
  for (uint64_t at = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; at < M; at += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t m = (uint32_t)at;
    const uint32_t i = sa[cpos[m]];
    member[m] = i;
    second[m] = (uint64_t)i + h < n ? isa[i + h] : 0u;
  }
}

// Sorts every group by its members' second names (ties keep their order): the
// place of a member is the number of members before it.  group[m] is the
// suffix array position of the group's first member, and the members of a
// group are consecutive, so the group starts at m - (cpos[m] - group[m]).  284 k
// members in groups of a few take 12 us with k_sa_second.  The work grows with
// the group's size, the sort of the encoded pairs does not: suffix arrays of
// 2 M characters whose groups all have k members take, compared / sorted,
//   k = 2: 599 / 1265 us, 32: 608 / 1198, 128: 728 / 1202, 256: 943 / 1223,
//   512: 1391 / 1274, 1024: 2134 / 1270,
// hence kSmallGroup.
__global__ void k_sa_groups(const uint32_t* __restrict__ cpos, const uint32_t* __restrict__ group, uint32_t M,
                            const uint32_t* __restrict__ member, const uint32_t* __restrict__ second, uint32_t* sa,
                            uint32_t* isa, uint32_t* new_group) {
  for (uint64_t at = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; at < M; at += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t m = (uint32_t)at;
    const uint32_t g = group[m], first = m - (cpos[m] - g), k = second[m], i = member[m];
    uint32_t less = 0, equal = 0, equal_before = 0;
    for (uint32_t q = first; q < M && group[q] == g; ++q) {
      const uint32_t o = second[q];
      less += o < k ? 1u : 0u;
      equal += o == k ? 1u : 0u;
      equal_before += (o == k && q < m) ? 1u : 0u;
    }
    sa[g + less + equal_before] = i;
    isa[i] = g + less + 1;
    new_group[first + less + equal_before] = equal > 1 ? g + less : kNoGroup;
  }
}

// Final LCP array.  Entries below h0 come from the first sort (they sit at the
// starts of h0-groups, whose members were only permuted inside the group);
// k_sa_long lists the others (j >= 1 with lcp >= h0) and k_sa_lcp gives each of
// them one warp.  Its first lane climbs down the name
// arrays of the rounds: suffixes a and b share their first h0 2^k characters
// from t on iff their names after round k at a + t and b + t agree, so taking
// each k from the last round down whenever they agree gives the largest
// multiple t of h0 with a and b equal in their first t characters (names do
// not agree past the end of the text).  The warp then compares the two
// suffixes from t on, 256 characters per step: lane k compares the
// 8-character windows at h + 8k, and the first lane that sees a difference
// (or the end of the shorter suffix) gives the LCP, fewer than h0 characters
// on.  The work per entry is O(rounds + h0 / 256) however long the LCP (a
// direct comparison from h0 took seconds on periodic texts).  A suffix at a
// has n - a characters, so no lane reads past the text.
// (A warp of k_sa_long takes 256 positions for one update of the counter:
// 16 us for 4 M suffixes; with 32 the updates alone took 60 us.)
__global__ void k_sa_long(const uint32_t* lcp, uint32_t n, uint32_t h0, uint32_t* pos, uint32_t* count) {
  constexpr uint32_t kPer = 8;
  const uint64_t warps = (uint64_t)gridDim.x * blockDim.x / 32;
  const uint64_t w0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  for (uint64_t j0 = w0 * 32 * kPer; j0 < n; j0 += warps * 32 * kPer) {
    uint32_t bits[kPer], total = 0;
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      const uint64_t j = j0 + 32 * u + lane_id();
      bits[u] = __ballot_sync(0xFFFFFFFFu, j > 0 && j < n && lcp[j] >= h0);
    }
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) total += __popc(bits[u]);
    uint32_t k = 0;
    if (lane_id() == 0 && total) k = atomicAdd(count, total);
    k = __shfl_sync(0xFFFFFFFFu, k, 0);
#pragma unroll
    for (uint32_t u = 0; u < kPer; ++u) {
      if ((bits[u] >> lane_id()) & 1u) pos[k + __popc(bits[u] & lanemask_lt())] = (uint32_t)(j0 + 32 * u + lane_id());
      k += __popc(bits[u]);
    }
  }
}

__global__ void k_sa_lcp(const uint8_t* text, const uint32_t* sa, uint32_t n, uint32_t h0, const uint32_t* pos,
                         const uint32_t* listed, uint32_t* lcp, SaSnaps sn) {
  const uint32_t count = *listed;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
  for (uint64_t w = (uint64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); w < count; w += warps) {
    const uint32_t j = pos[w];
    const uint64_t a = sa[j - 1], b = sa[j];
    const uint64_t la = n - a, lb = n - b;
    const uint64_t lmin = la < lb ? la : lb;
    unsigned long long t = h0;
    if (lane == 0 && sn.count) {
      t = 0;
      for (int k = (int)sn.count - 1; k >= 0; --k) {
        const uint32_t* nm = sn.p[k];
        if (a + t < n && b + t < n && nm[a + t] == nm[b + t]) t += (unsigned long long)h0 << k;
      }
    }
    t = __shfl_sync(0xFFFFFFFFu, t, 0);
    uint64_t h = t;
    uint64_t result = 0;
    while (true) {
      const uint64_t d = h + 8ull * lane;
      uint32_t stop = 8;  // characters that agree in this lane's window (8 = all)
      if (d >= lmin) {
        stop = 0;
      } else {
        const uint64_t ca = load_cache(text, a, (uint32_t)d, kNoCap);
        const uint64_t cb = load_cache(text, b, (uint32_t)d, kNoCap);
        if (ca != cb) stop = lcp8(ca, cb);
        else if (has_nul(ca)) stop = nnz_prefix(ca);
      }
      const uint32_t done = __ballot_sync(0xFFFFFFFFu, stop < 8);
      if (done) {
        const uint32_t first = __ffs(done) - 1;
        const uint32_t s_first = __shfl_sync(0xFFFFFFFFu, stop, first);
        result = h + 8ull * first + s_first;
        break;
      }
      h += 256;
    }
    if (lane == 0) lcp[j] = (uint32_t)result;
  }
}

}  // namespace

cudaError_t sa_launch(SaKernel k, const SaArgs& x, uint32_t sms, cudaStream_t st, const LaunchHook& hook) {
  auto grid = [&](uint64_t m) {
    return (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((m + 255) / 256, (uint64_t)sms * 32));
  };
  switch (k) {
    case SaKernel::kIota:
      hook.run("sa_iota", [&] { k_sa_iota<<<grid(x.n), 256, 0, st>>>(x.off, x.n); });
      break;
    case SaKernel::kNameFirst:
      return name_and_compact(SaFirst{x.sa, x.lcp, x.h, x.isa}, (uint32_t)x.n, x.totals, x.out, x.group_out, x.result,
                              sms, st, hook);
    case SaKernel::kEncode:
      hook.run("sa_encode", [&] {
        k_sa_encode<<<grid(x.M), 256, 0, st>>>(x.cpos, x.M, x.sa, x.isa, (uint32_t)x.n, x.h, x.member, x.enc, x.eoff);
      });
      break;
    case SaKernel::kNamePairs:
      return name_and_compact(SaPairs{x.cpos, x.member, x.perm2, x.lcp2, x.sa, x.isa}, x.M, x.totals, x.out,
                              x.group_out, x.result, sms, st, hook);
    case SaKernel::kGroups:
      hook.run("sa_groups", [&] {
        k_sa_second<<<grid(x.M), 256, 0, st>>>(x.cpos, x.M, x.sa, x.isa, (uint32_t)x.n, x.h, x.member, x.second);
      });
      hook.run("sa_groups", [&] {
        k_sa_groups<<<grid(x.M), 256, 0, st>>>(x.cpos, x.group, x.M, x.member, x.second, x.sa, x.isa, x.new_group);
      });
      if (const cudaError_t e = cudaGetLastError()) return e;
      return name_and_compact(SaGroups{x.cpos, x.new_group}, x.M, x.totals, x.out, x.group_out, x.result, sms, st,
                              hook);
    case SaKernel::kLcp:
      if (const cudaError_t e = cudaMemsetAsync(x.listed, 0, 4, st)) return e;
      hook.run("sa_lcp", [&] { k_sa_long<<<grid(x.n / 8 + 1), 256, 0, st>>>(x.lcp_out, (uint32_t)x.n, x.h, x.out, x.listed); });
      hook.run("sa_lcp", [&] {
        k_sa_lcp<<<grid(32ull * x.n), 256, 0, st>>>(x.text, x.sa, (uint32_t)x.n, x.h, x.out, x.listed, x.lcp_out,
                                                    x.snaps);
      });
      break;
  }
  return cudaGetLastError();
}

}  // namespace ss
