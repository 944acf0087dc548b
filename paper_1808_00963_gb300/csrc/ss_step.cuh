// Building blocks of one Super Scalar String Sample Sort step (Algorithm 4.1),
// by one block (of 256 threads unless a template argument says otherwise).
// Used by the multi-block step kernels and by the persistent single-block
// kernel.
#pragma once

#include "ss_internal.cuh"

namespace ss {

constexpr uint32_t kBlock = 256;
constexpr uint32_t kWarps = kBlock / 32;
constexpr uint32_t kMaxRounds = 32;                  // tile = 256 * rounds records
constexpr uint32_t kMaxTile = kBlock * kMaxRounds;
constexpr uint32_t kFin = 1u << 31;                  // bucket descriptor: finished
constexpr uint32_t kNulEq = 1u << 30;                // ... all members equal strings
constexpr uint32_t kLow30 = (1u << 30) - 1;

// v = 2^LOGV - 1 splitters x_0..x_{v-1}, k = 2v + 1 buckets (Section 4.2.2).
template <int LOGV>
struct Geo {
  static constexpr uint32_t V = (1u << LOGV) - 1;
  static constexpr uint32_t K = 2 * V + 1;
  static constexpr uint32_t KP = 2u << LOGV;        // K rounded up to a power of two
  static constexpr uint32_t S = 2u << LOGV;         // sample size alpha * (v + 1), alpha = 2
};

// Splitters of one step (K: uint64_t for narrow keys, u128 for wide ones).
template <int LOGV, typename K = uint64_t>
struct Splitters {
  K tree[Geo<LOGV>::V + 1];  // t[1..v], level order (t[0] unused)
  K x[Geo<LOGV>::V + 1];     // x_0..x_{v-1} sorted; x[v] unused
  uint8_t hp[Geo<LOGV>::V + 1];     // h'_0..h'_v: lcp of neighbouring splitters
};

// Shared memory of the splitter construction.  The merge alternates between
// `sample` and the room of the splitters, which are only written once it is
// done.
template <int LOGV, typename K>
struct SampleSmem {
  static_assert(sizeof(K) * Geo<LOGV>::S <= sizeof(Splitters<LOGV, K>), "the merge's second buffer");
  union {
    Splitters<LOGV, K> sp;
    K merge[Geo<LOGV>::S];
  };
  K sample[Geo<LOGV>::S];
  uint16_t lo[Geo<LOGV>::S];   // first sample position with a key >= sample[i]
  uint16_t hi[Geo<LOGV>::S];   // first sample position with a key >  sample[i]
  uint32_t heads[64];          // bit i of word w: position 32 w + i starts a run of equal keys
};

// Which of a bitmap's up to 64 words hold a set bit (bit w: word w); every
// lane of the warp calls it.
__device__ __forceinline__ uint64_t nonzero_words(const uint32_t* words, uint32_t nw) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t b0 = __ballot_sync(0xFFFFFFFFu, lane < nw && words[lane] != 0);
  const uint32_t b1 = __ballot_sync(0xFFFFFFFFu, lane + 32 < nw && words[lane + 32] != 0);
  return (uint64_t)b1 << 32 | b0;
}

// The last set bit before / the first one after position p of such a bitmap
// (kNone: there is none); some: its nonzero_words.
constexpr uint32_t kNone = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t last_set_before(const uint32_t* words, uint64_t some, uint32_t p) {
  const uint32_t w = p >> 5;
  const uint32_t own = words[w] & ((1u << (p & 31u)) - 1);
  if (own) return w * 32 + 31 - __clz(own);
  const uint64_t below = some & ((1ull << w) - 1);
  if (!below) return kNone;
  const uint32_t v = 63 - __clzll((long long)below);
  return v * 32 + 31 - __clz(words[v]);
}

__device__ __forceinline__ uint32_t first_set_after(const uint32_t* words, uint64_t some, uint32_t p) {
  const uint32_t w = p >> 5;
  const uint32_t own = words[w] & ~((2u << (p & 31u)) - 1);  // bit 31: none above
  if (own) return w * 32 + __ffs(own) - 1;
  const uint64_t above = w == 63 ? 0ull : some & ~((2ull << w) - 1);
  if (!above) return kNone;
  const uint32_t v = __ffsll((long long)above) - 1;
  return v * 32 + __ffs(words[v]) - 1;
}

// Ascending bitonic sort of the 32 keys a warp holds, one per lane.
template <typename K>
__device__ __forceinline__ K warp_bitonic(K v) {
  const uint32_t lane = threadIdx.x & 31;
#pragma unroll
  for (uint32_t k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (uint32_t j = k >> 1; j > 0; j >>= 1) {
      const K o = KeyOps<K>::shfl_xor(v, (int)j);
      const bool take_min = ((lane & j) == 0) == ((lane & k) == 0);
      v = take_min ? (o < v ? o : v) : (o > v ? o : v);
    }
  }
  return v;
}

// The sampling steps of Algorithm 4.1 for a subset of len keys, by a block of
// NT threads: draw a sample of alpha * (v + 1) keys at pseudo-random positions,
// sort it, select the splitters with the recursive duplicate-skipping rule of
// Section 4.2.3 ("Sampling"): the middle sample of a range becomes the
// splitter, the ranges left and right of the run of samples equal to it are
// split recursively.  A node whose range is empty takes the sample just above
// its range (the nearest splitter on the right among its ancestors), or
// all-ones past the end, which keeps t a search tree.  Finally h'_i =
// lcp(x_{i-1}, x_i) with h'_0 = h'_v = 0, the splitter LCPs of Algorithm 4.1.
//
// A step waits for its sample, so this is built for latency: warps sort runs
// of 32 keys in registers, the runs are merged pairwise, each key finding its
// place with a binary search in the partner run (30 dependent shared loads
// for 512 keys; ranking every key in every other warp's run took 84 in
// a 256-thread block, then 36 more to find the runs of equal keys, which now
// come from a bitmap of run starts).  With the run of equal keys around every
// sample position known, each tree node finds its range by walking from the
// root along its level-order index, so the recursion needs no step-by-step
// synchronisation.  Ends with __syncthreads().
// key_at(pos) gives the key of the subset's record pos.
template <int LOGV, typename K, uint32_t NT, typename KeyAt>
__device__ void build_splitters(KeyAt&& key_at, uint32_t len, uint64_t hseed, SampleSmem<LOGV, K>& sm, uint32_t dna) {
  using G = Geo<LOGV>;
  constexpr uint32_t S = G::S;
  constexpr int kLevels = LOGV + 1 - 5;  // merge levels from runs of 32 to S
  const uint32_t tid = threadIdx.x;
  K* src = (kLevels & 1) ? sm.merge : sm.sample;  // the last level writes sample
  K* dst = (kLevels & 1) ? sm.sample : sm.merge;
  for (uint32_t p = tid; p < S; p += NT) {  // whole warps: S is a multiple of 32
    const uint64_t h = mix64(hseed + p);
    src[p] = warp_bitonic<K>(key_at((uint32_t)(((h >> 32) * (uint64_t)len) >> 32)));
  }
  __syncthreads();
#pragma unroll 1
  for (uint32_t run = 32; run < S; run <<= 1) {
    // each key's place in the merged pair of runs: its own index plus the
    // partner's keys before it (a left key goes before an equal right one)
    for (uint32_t p = tid; p < S; p += NT) {
      const K k = src[p];
      const uint32_t i = p & (run - 1);
      const K* other = src + (p ^ i ^ run);
      const bool right = (p & run) != 0;
      uint32_t a = 0;
      for (uint32_t half = run >> 1; half > 0; half >>= 1) {
        const K o = other[a + half - 1];
        a += (right ? o <= k : o < k) ? half : 0u;
      }
      const K o = other[a];
      a += (right ? o <= k : o < k) ? 1u : 0u;
      dst[(p & ~(2 * run - 1)) + i + a] = k;
    }
    __syncthreads();
    K* t = src;
    src = dst;
    dst = t;
  }
  const K* s = sm.sample;
  // runs of equal keys, from one bit per position that starts one
  for (uint32_t p = tid; p < S; p += NT) {
    const uint32_t hb = __ballot_sync(0xFFFFFFFFu, p == 0 || s[p - 1] != s[p]);
    if ((tid & 31u) == 0) sm.heads[p >> 5] = hb;
  }
  __syncthreads();
  const uint64_t some = nonzero_words(sm.heads, S / 32);
  for (uint32_t p = tid; p < S; p += NT) {
    const bool head = (sm.heads[p >> 5] >> (p & 31u)) & 1u;
    sm.lo[p] = (uint16_t)(head ? p : last_set_before(sm.heads, some, p));  // position 0 starts a run
    sm.hi[p] = (uint16_t)min(S, first_set_after(sm.heads, some, p));
  }
  __syncthreads();
  for (uint32_t q = tid; q < G::V; q += NT) {
    const uint32_t i = q + 1;               // level-order index
    const int l = 31 - __clz(i);            // its level
    uint32_t a = 0, b = S;                  // its range of the sorted sample
    for (int d = l - 1; d >= 0; --d) {
      if (a < b) {
        const uint32_t m = (a + b) >> 1;
        if (((i >> d) & 1u) == 0) {
          const uint32_t le = sm.lo[m];
          b = le > a ? le : a;              // left of the run of keys equal to s[m]
        } else {
          const uint32_t rs = sm.hi[m];
          a = rs < b ? rs : b;              // right of that run
        }
      } else {
        a = b;
      }
    }
    const K val = a < b ? s[(a + b) >> 1] : (b < S ? s[b] : KeyOps<K>::ones());
    sm.sp.tree[i] = val;
    sm.sp.x[(2 * (i - (1u << l)) + 1) * (1u << (LOGV - 1 - l)) - 1] = val;
  }
  if (tid == 0) {
    sm.sp.tree[0] = 0;
    sm.sp.x[G::V] = 0;
  }
  __syncthreads();
  for (uint32_t r = tid; r <= G::V; r += NT)
    sm.sp.hp[r] = (r == 0 || r == G::V) ? 0 : (uint8_t)KeyOps<K>::lcp(sm.sp.x[r - 1], sm.sp.x[r], dna);
  __syncthreads();
}

// Lemma 4.1: one-based level-order index l <-> one-based pre-order index p
// (the position of the vertex's splitter in sorted order) of a perfect binary
// tree with w levels, by rotating the bits around the first (resp. last) one
// bit.
__device__ __forceinline__ uint32_t level_to_pre(uint32_t l, uint32_t w) {
  const uint32_t s = 31 - __clz(l);  // bits after the first one bit
  const uint32_t x = w - s;          // position of the first one bit, from the top
  return ((l & ((1u << s) - 1)) << x) | (1u << (x - 1));
}

__device__ __forceinline__ uint32_t pre_to_level(uint32_t p, uint32_t w) {
  const uint32_t t = (uint32_t)__ffs(p) - 1;  // bits after the last one bit
  const uint32_t y = w - t;                    // position of the last one bit, from the top
  return (1u << (y - 1)) | (p >> (t + 1));
}

// Classification variants of Section 4.2.3 (they give the same buckets up to
// the numbering of empty ones, hence the same output).
constexpr uint32_t kClassifyUI = 0;   // unrolled <=-descent, equality test on the sorted copy x
constexpr uint32_t kClassifyUIC = 1;  // same descent, equality test in t via Lemma 4.1 (no copy needed)
constexpr uint32_t kClassifyE = 2;    // equality test at every node of the descent
constexpr uint32_t kClassifyUIJ = 3;  // UI entered through a jump table over the key's top bits

// Jump tables (Section 4.4, "Jump tables"): for every value p of a key's top
// kJumpBits bits, the first node of the descent whose splitter does not
// decide by those bits alone (its top bits equal p), or the leaf reached
// (>= 2^LOGV) when every splitter on the way decides.  Keys with top bits p
// take the same path down to that node, so the descent can start there.
constexpr int kJumpBits = 12;
constexpr uint32_t kJumpSize = 1u << kJumpBits;

template <int LOGV, typename K>
__device__ __forceinline__ uint32_t jump_entry(uint32_t p, const K* tree) {
  uint32_t i = 1;
  while (i < (1u << LOGV)) {
    const uint32_t tp = KeyOps<K>::top(tree[i], kJumpBits);
    if (p == tp) break;
    i = 2 * i + (p > tp ? 1u : 0u);
  }
  return i;
}

// The UI classification entered at the jump table's node: the remaining
// levels are predicated off for keys already at a leaf.
template <int LOGV, typename K>
__device__ __forceinline__ uint32_t classify_jump(K c, const K* tree, const K* x, const uint16_t* jump) {
  uint32_t i = jump[KeyOps<K>::top(c, kJumpBits)];
#pragma unroll
  for (int l = 0; l < LOGV; ++l)
    if (i < (1u << LOGV)) i = 2 * i + (c > tree[i] ? 1u : 0u);
  const uint32_t r = i - (1u << LOGV);
  const bool eq = r < Geo<LOGV>::V && x[r] == c;
  return 2 * r + (eq ? 1u : 0u);
}

// The classification of one key in Algorithm 4.1: branch-free descent of the level-order tree,
// i := 2i + [c > t_i] (the reading of its descent step under which bucket b_{2r} holds
// x_{r-1} < c < x_r), then the single equality test with x_r.
template <int LOGV, typename K>
__device__ __forceinline__ uint32_t classify(K c, const K* tree, const K* x, uint32_t variant = kClassifyUI) {
  uint32_t i = 1;
  if (variant == kClassifyE) {
    uint32_t eq = 0;
#pragma unroll
    for (int l = 0; l < LOGV; ++l) {
      const K t = tree[i];
      if (!eq && c == t) eq = i;
      i = 2 * i + (c > t ? 1u : 0u);
    }
    if (eq) return 2 * (level_to_pre(eq, LOGV) - 1) + 1;
    return 2 * (i - (1u << LOGV));
  }
#pragma unroll
  for (int l = 0; l < LOGV; ++l) i = 2 * i + (c > tree[i] ? 1u : 0u);
  const uint32_t r = i - (1u << LOGV);
  bool eq = false;
  if (r < Geo<LOGV>::V) eq = (variant == kClassifyUIC) ? tree[pre_to_level(r + 1, LOGV)] == c : x[r] == c;
  return 2 * r + (eq ? 1u : 0u);
}

// Buckets of U keys.  For S5-UI the U descents advance one tree level at a
// time together, so that U independent shared-memory loads are in flight per
// level rather than one (20 M URL strings: the classification 0.64 -> 0.55 ms).
template <int LOGV, int U, typename K>
__device__ __forceinline__ void classify_batch(const K (&k)[U], uint32_t (&b)[U], const K* tree, const K* x,
                                               uint32_t variant, const uint16_t* jump) {
  if (variant == kClassifyUI) {
    uint32_t i[U];
#pragma unroll
    for (int u = 0; u < U; ++u) i[u] = 1;
#pragma unroll
    for (int l = 0; l < LOGV; ++l) {
#pragma unroll
      for (int u = 0; u < U; ++u) i[u] = 2 * i[u] + (k[u] > tree[i[u]] ? 1u : 0u);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t r = i[u] - (1u << LOGV);
      b[u] = 2 * r + ((r < Geo<LOGV>::V && x[r] == k[u]) ? 1u : 0u);
    }
    return;
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    b[u] = (variant == kClassifyUIJ && jump) ? classify_jump<LOGV, K>(k[u], tree, x, jump)
                                             : classify<LOGV, K>(k[u], tree, x, variant);
}

// Classifies n keys (the classification loop of Algorithm 4.1): writes the bucket of
// keys[p] to bo[p] and counts it in hist (one shared-memory atomic per key:
// cheaper than grouping a warp's equal buckets with __match_any_sync first).  Each thread loads 8 keys before descending the tree for them,
// so that the loads of a batch overlap.  seen(b, key) is called for every key
// after its bucket is known.  Returns this thread's records.
struct NothingSeen {
  template <typename K>
  __device__ __forceinline__ void operator()(uint32_t, K) const {}
};
template <int LOGV, typename K, uint32_t NT, int U, typename KeyAt, typename Seen>
__device__ __forceinline__ void classify_some(KeyAt&& key_at, uint16_t* __restrict__ bo, uint32_t p0, uint32_t n,
                                              const K* tree, const K* x, uint32_t* hist, uint32_t variant,
                                              const uint16_t* jump, Seen&& seen) {
  K k[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const uint32_t p = p0 + u * NT;
    k[u] = p < n ? key_at(p) : (K)0;
  }
  uint32_t bb[U];
  classify_batch<LOGV, U, K>(k, bb, tree, x, variant, jump);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const uint32_t p = p0 + u * NT;
    if (p < n) {
      bo[p] = (uint16_t)bb[u];
      atomicAdd(&hist[bb[u]], 1u);
      seen(bb[u], k[u]);
    }
  }
}

template <int LOGV, typename K, uint32_t NT, typename KeyAt, typename Seen = NothingSeen>
__device__ __forceinline__ uint32_t classify_count_k(KeyAt&& key_at, uint16_t* __restrict__ bo, uint32_t n,
                                                     const K* tree, const K* x, uint32_t* hist, uint32_t variant,
                                                     const uint16_t* jump, Seen&& seen = NothingSeen()) {
  constexpr int U = sizeof(K) == 8 ? 8 : 4;  // keys per thread in flight (wide keys take 4 registers)
  uint32_t p0 = threadIdx.x, left = (n + NT - 1) / NT;  // keys per thread
  for (; left > U / 2; left -= min(left, (uint32_t)U), p0 += U * NT)
    classify_some<LOGV, K, NT, U>(key_at, bo, p0, n, tree, x, hist, variant, jump, seen);
  // the rest (or a subset of few keys per thread) without idle descents
  if (left) classify_some<LOGV, K, NT, U / 2>(key_at, bo, p0, n, tree, x, hist, variant, jump, seen);
  return threadIdx.x < n ? (n - 1 - threadIdx.x) / NT + 1 : 0u;
}

// What happens to bucket b of a step at depth h (Output of Algorithm 4.1 and
// Section 4.2.3): an even bucket b_{2r} continues at depth h + h'_r, an
// equality bucket at h + 8, unless its splitter holds the terminator (then all
// members are equal strings and the bucket is finished; their LCP is their
// length); a single string is finished.
template <int LOGV, typename K>
__device__ __forceinline__ uint32_t bucket_desc(uint32_t b, uint32_t size, uint32_t depth,
                                                const Splitters<LOGV, K>& sp, uint32_t dna) {
  const uint32_t r = b >> 1;
  if (b & 1) {
    const K xr = sp.x[r];
    if (KeyOps<K>::end(xr, dna)) return kFin | kNulEq | (depth + KeyOps<K>::nnz(xr, dna));
    if (size == 1) return kFin;
    return depth + KeyOps<K>::width(dna);
  }
  if (size == 1) return kFin;
  return depth + sp.hp[r];
}

constexpr uint32_t kInvalid = 0xFFFFFFFFu;

// The lanes of the warp whose record falls into the same bucket b as this
// lane's (valid lanes only; every lane of the warp calls it): the mask of
// valid lanes narrowed by one ballot per bit of the bucket index.  Cheaper to
// issue than __match_any_sync (measured on the distribution) and stable in
// lane order like it.
template <int LOGV>
__device__ __forceinline__ uint32_t bucket_peers(uint32_t b, bool valid) {
  uint32_t m = __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
  for (int i = 0; i <= LOGV; ++i) {  // bucket indices have LOGV + 1 bits
    const bool bit = (b >> i) & 1u;
    const uint32_t v = __ballot_sync(0xFFFFFFFFu, bit);
    m &= bit ? v : ~v;
  }
  return m;
}

// Stable distribution of one tile of records (the redistribution of Algorithm 4.1 with the
// per-processor bucket arrays of Theorem 4.4, one per warp).
//   tb[0..tl)    bucket of each record of the tile (shared memory)
//   base[b]      in: destination of the tile's first record of bucket b;
//                out: base[b] + number of the tile's records in bucket b
//   cntw         shared scratch, NT / 32 * KP uint16 (4-byte aligned)
// Warp w owns records [w * 32R, (w + 1) * 32R) of the tile; inside a warp
// ranks come from the lanes with the same bucket (bucket_peers), so equal
// buckets keep input order.
// move(p[], b[], dest[]) is called with MB rounds of one warp at a time
// (p = kInvalid for lanes without a record).  Ends with __syncthreads().
// cntw holds what is still to come of a bucket from this warp on, so that 16
// bits are enough (a record goes to base[b] - left): half the shared memory
// leaves the multi-block kernel 124 KB of L1 instead of 60.
static_assert(kMaxTile <= 0xFFFF, "counts within a tile have 16 bits");
template <int LOGV, uint32_t NT, int MB, typename Move>
__device__ void tile_scatter(const uint16_t* tb, uint32_t tl, uint32_t R, uint32_t* base,
                             uint16_t* cntw, Move&& move) {
  using G = Geo<LOGV>;
  constexpr uint32_t kWarps = NT / 32;
  const uint32_t w = threadIdx.x >> 5, lane = lane_id();
  for (uint32_t i = threadIdx.x; i < kWarps * G::KP / 2; i += NT) reinterpret_cast<uint32_t*>(cntw)[i] = 0;
  __syncthreads();
  uint16_t* mine = cntw + w * G::KP;
  const uint32_t p0 = w * 32 * R;
  for (uint32_t r = 0; r < R; ++r) {
    const uint32_t p = p0 + r * 32 + lane;
    if (p < tl) {  // counts only: no need to group equal buckets
      const uint32_t b = tb[p];
      atomicAdd(reinterpret_cast<uint32_t*>(mine) + (b >> 1), 1u << (16 * (b & 1u)));
    }
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < G::K; b += NT) {
    uint32_t run = 0;
#pragma unroll
    for (uint32_t ww = kWarps; ww-- > 0;) {
      run += cntw[ww * G::KP + b];
      cntw[ww * G::KP + b] = (uint16_t)run;
    }
    base[b] += run;
  }
  __syncthreads();
  const uint32_t lt = lanemask_lt();
  for (uint32_t r0 = 0; r0 < R; r0 += MB) {
    uint32_t pp[MB], bb[MB], dd[MB];
#pragma unroll
    for (int u = 0; u < MB; ++u) {
      const uint32_t r = r0 + u;
      const uint32_t p = p0 + r * 32 + lane;
      const bool valid = r < R && p < tl;
      const uint32_t b = valid ? tb[p] : 0u;
      const uint32_t peers = bucket_peers<LOGV>(b, valid);
      uint32_t dest = 0;
      const uint32_t left = mine[b];  // records of the bucket not yet placed, this warp's and the later ones'
      if (valid) dest = base[b] - left + __popc(peers & lt);
      __syncwarp();
      if (valid && lane == (uint32_t)(__ffs(peers) - 1)) mine[b] = (uint16_t)(left - __popc(peers));
      __syncwarp();
      pp[u] = valid ? p : kInvalid;
      bb[u] = b;
      dd[u] = dest;
    }
    move(pp, bb, dd);
  }
  __syncthreads();
}

// Moves a batch of records to their buckets (the body of the redistribution): a finished
// record writes its final index (and, inside a bucket of equal strings, its
// LCP); an open one is copied to the other buffer with its cache reloaded at
// the bucket's new depth (fused character gather).  All loads of the batch
// are issued before any of them is used.  bucket_first(b) is the position of
// the first record of bucket b.  Returns the algorithmic bytes: bucket index 2
// + record 16 read (the record carries the string's offset); finished: perm 4
// (+ lcp 4) written; open: record 16 written, plus 8 characters read when the
// cache is reloaded.
template <int MB, bool DNA, typename First>
__device__ __forceinline__ uint32_t move_batch(const SortCtx& c, const SetDesc& sd, uint32_t wide, uint32_t par,
                                               uint32_t src0, uint32_t depth, const uint32_t* desc,
                                               First&& bucket_first, const uint32_t (&pp)[MB],
                                               const uint32_t (&bb)[MB], const uint32_t (&dd)[MB]) {
  uint32_t id[MB], ds[MB], o32[MB];
  uint64_t key[MB], off[MB];
  uint32_t bytes = 0;
#pragma unroll
  for (int u = 0; u < MB; ++u) {
    id[u] = 0;
    o32[u] = 0;
    ds[u] = kFin;
    key[u] = 0;
    if (pp[u] != kInvalid) {
      ds[u] = desc[bb[u]];
      const Rec r = load_rec(c.rec[par] + src0 + pp[u]);
      id[u] = r.idx;
      key[u] = r.key;
      o32[u] = r.off;
    }
  }
  // the characters of every byte-string reload are requested before any of
  // them is used (one memory round trip for the batch)
  CharWords ww[MB];
#pragma unroll
  for (int u = 0; u < MB; ++u) {
    off[u] = 0;
    if (pp[u] != kInvalid && !(ds[u] & kFin) && (ds[u] & kLow30) != depth) {
      off[u] = rec_offset(sd, wide, id[u], o32[u]);
      if (!DNA) issue_chars(sd.chars, off[u], ds[u] & kLow30, sd.cap, 8, ww[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < MB; ++u) {
    if (pp[u] == kInvalid) continue;
    const uint32_t d = ds[u];
    const uint32_t dest = dd[u];
    if (d & kFin) {
      sd.perm[dest - sd.base] = id[u];
      bytes += 22;
      if (sd.lcp && (d & kNulEq) && dest != bucket_first(bb[u])) {
        sd.lcp[dest - sd.base] = d & kLow30;
        bytes += 4;
      }
      continue;
    }
    const uint32_t nd = d & kLow30;
    uint64_t k = key[u];
    bytes += 34;
    if (nd != depth) {
      k = DNA ? dna_key(sd.chars, off[u], nd, sd.cap) : finish_chars8(ww[u], sd.chars, off[u], nd, sd.cap);
      bytes += 8;
    }
    store_rec(c.rec[par ^ 1] + dest, k, id[u], o32[u]);
  }
  return bytes;
}

// move_batch for records of a multi-block subset, held in the wide form (wide
// key in the record slot, (idx, off) in wid[]).  A record whose new bucket is
// itself a multi-block subset stays wide (key reloaded at the new depth unless
// the depth is unchanged); otherwise it becomes a narrow record, whose key is
// cut out of the wide one when the new depth is at most 8 characters deeper
// (bytes), or is the first or second half of it (DNA codes, 0 or 21 deeper),
// and gathered from the string otherwise.  bucket_first(b) is the position of
// bucket b's first record (bucket_first(b + 1) - bucket_first(b) its size).
// load(key, wi) gives the batch's wide keys and (idx, off).
// Returns the algorithmic bytes: bucket index 2 + wide record 24 read;
// finished: perm 4 (+ lcp 4) written; open: 24 (wide) or 16 (narrow) written,
// plus 16 (wide) or 8 (narrow) characters read when gathered.
template <int MB, bool DNA, typename Load, typename First>
__device__ __forceinline__ uint32_t move_batch_wide(const SortCtx& c, const SetDesc& sd, uint32_t wide,
                                                    uint32_t par, uint32_t depth, const uint32_t* desc, Load&& load,
                                                    First&& bucket_first, const uint32_t (&pp)[MB],
                                                    const uint32_t (&bb)[MB], const uint32_t (&dd)[MB]) {
  constexpr uint32_t kSkip = 0, kFinal = 1, kKeep = 2, kGather = 3;  // what a record needs
  uint32_t ds[MB], how[MB];
  bool to_wide[MB];
  uint2 wi[MB];
  u128 key[MB];
  uint32_t bytes = 0;
#pragma unroll
  for (int u = 0; u < MB; ++u) {
    ds[u] = pp[u] != kInvalid ? desc[bb[u]] : kFin;
    wi[u] = make_uint2(0, 0);
    key[u] = 0;
  }
  load(key, wi);
  // what each record needs; the characters of every byte-string gather are
  // requested before any of them is used (one memory round trip for the batch)
  CharWords ww[MB];
#pragma unroll
  for (int u = 0; u < MB; ++u) {
    how[u] = kSkip;
    to_wide[u] = false;
    if (pp[u] == kInvalid) continue;
    const uint32_t d = ds[u];
    if (d & kFin) {
      how[u] = kFinal;
      continue;
    }
    const uint32_t adv = (d & kLow30) - depth;
    const uint32_t size = bucket_first(bb[u] + 1) - bucket_first(bb[u]);
    to_wide[u] = c.big_enabled && size > c.big_threshold;
    const bool derive = to_wide[u] ? adv == 0 : (DNA ? (adv == 0 || adv == kDnaWidth) : adv <= 8);
    how[u] = derive ? kKeep : kGather;
    if (!derive && !DNA)
      issue_chars(sd.chars, rec_offset(sd, wide, wi[u].x, wi[u].y), d & kLow30, sd.cap, to_wide[u] ? 16 : 8, ww[u]);
  }
#pragma unroll
  for (int u = 0; u < MB; ++u) {
    if (how[u] == kSkip) continue;
    const uint32_t dest = dd[u];
    if (how[u] == kFinal) {
      sd.perm[dest - sd.base] = wi[u].x;
      bytes += 30;
      if (sd.lcp && (ds[u] & kNulEq) && dest != bucket_first(bb[u])) {
        sd.lcp[dest - sd.base] = ds[u] & kLow30;
        bytes += 4;
      }
      continue;
    }
    const uint32_t nd = ds[u] & kLow30;
    const uint32_t adv = nd - depth;
    u128 k = key[u];
    if (how[u] == kGather) {
      if (DNA) {
        const uint64_t o = rec_offset(sd, wide, wi[u].x, wi[u].y);
        k = to_wide[u] ? load_key128(sd.chars, o, nd, sd.cap, 1u) : make_k(dna_key(sd.chars, o, nd, sd.cap), 0);
      } else {
        const uint64_t o = rec_offset(sd, wide, wi[u].x, wi[u].y);
        uint64_t hi, lo = 0;
        if (to_wide[u]) finish_chars16(ww[u], sd.chars, o, nd, sd.cap, hi, lo);
        else hi = finish_chars8(ww[u], sd.chars, o, nd, sd.cap);
        k = make_k(hi, lo);
      }
      bytes += to_wide[u] ? 16 : 8;
    }
    if (to_wide[u]) {
      bytes += 50;
      store_wkey(c.rec[par ^ 1] + dest, k);
      c.wid[par ^ 1][dest] = wi[u];
    } else {
      bytes += 42;
      // a gathered narrow key is the first half; a kept one is cut out of the wide key
      const uint64_t nk = how[u] == kGather ? k_hi(k) : (DNA ? (adv ? k_lo(k) : k_hi(k)) : narrow_at(k, adv));
      store_rec(c.rec[par ^ 1] + dest, nk, wi[u].x, wi[u].y);
    }
  }
  return bytes;
}

// Emits the outcome of one non-empty bucket: its boundary LCP mark, if asked
// for (resolved at the end, Section 4.2.8 "LCP Calculation": the LCP with the
// previous bucket is depth + lcp of the two strings' wide keys at this depth)
// and, if it is not finished, a new task.
__device__ __forceinline__ void emit_bucket(const SortCtx& c, const SetDesc& sd, const Task& t,
                                            uint32_t start, uint32_t size, uint32_t desc,
                                            uint32_t next_big, bool mark) {
  if (mark && start > 0 && sd.lcp) sd.lcp[t.begin + start - sd.base] = kLcpMark | t.depth;
  if (!(desc & kFin)) {
    Task ch{t.begin + start, size, desc & kLow30, make_meta(task_set(t), task_par(t) ^ 1)};
    route_task(c, ch, next_big);
  }
}

}  // namespace ss
