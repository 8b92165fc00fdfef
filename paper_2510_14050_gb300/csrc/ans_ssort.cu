// Segmented sample sort of 64-bit link keys.
//
// Grouping equal (src, dst) pairs (Table I caption: A(i, j) = #packets i -> j)
// needs the packed keys src << 32 | dst of every window, or of a whole batch,
// in order (Sec. IV-B: rows ascending, columns ascending within a row).  Equal
// keys are indistinguishable, so the sort need not be stable, and it works
// from the most significant end:
//
//   sample   one CTA per segment sorts ~16 sampled keys per bucket on chip and
//            takes every 16th as a splitter; a key that fills several buckets
//            gets one of its own (its copies need no sorting at all);
//   count    every key's bucket by a search tree of splitters in shared
//            memory (ids kept as 16-bit words), bucket sizes;
//   scatter  keys moved to their buckets: ranks by one shared-memory atomic
//            per key, space by one global atomic per bucket and tile -- no
//            chain of tiles waiting for one another;
//   local    every bucket (~1366 keys, up to 2048 in segments of 1.4 to 2.1
//            million) sorted by one CTA on chip: 16 keys per thread in
//            registers, then merge-path rounds in shared memory; one of more
//            than 2048 keys (16 samples a bucket misjudge about one in forty;
//            half of them at 2^21) in pieces merged through global memory.
//
// Buckets hold equal numbers of packets whatever the addresses look like, so
// heavy sources and links cost nothing extra.  A segment too long for one
// split is first split into about as many buckets as each of them will have,
// which then are the segments of the steps above.
//
// Against eight least-significant-digit passes (each bound by its chain of
// tiles and by 150 instructions per key; 53 us for 64 windows of 2^17 keys,
// 930 us for 2^27 keys with 16-bit window ids) this reads and writes the keys
// four times instead of nine: 64 windows in 242 us against 491, one window
// of 2^17 in 60-67 us against 82, 2^27 keys as one segment in 4.5 ms.  On one
// GB300, 2^27 keys in windows of 2^17: sample 0.17, count 0.38 (bound by issue
// slots, 72%), scatter 0.62 (by the latency of its loads: 0.93 with one 4-byte
// load per address instead of 16-byte vectors), local 1.7 ms (by
// shared-memory wavefronts, 75% of peak, 340 instructions per key; buckets of
// 2731 keys and 256 threads: 1.93 ms).
#include "ans_internal.cuh"

namespace ans {

namespace {

constexpr uint32_t kSsBucket = (kTile + kSsPerTile - 1) / kSsPerTile;  // keys per bucket aimed at
constexpr uint32_t kSsLocal = 2048;         // keys one CTA sorts on chip
constexpr uint32_t kSsMaxBuckets = 1024;    // buckets of one split
constexpr uint32_t kSsSampleMax = 16384;    // sampled keys of one segment
constexpr uint32_t kSsOversample = 16;      // sampled keys per bucket
constexpr uint32_t kSsRawBit = 0x80000000u; // level-2 parent: the segment itself, still unsplit input
constexpr uint32_t kSsDone = 0xFFFFFFFFu;   // level-2 parent: nothing to sort

// Buckets of an n-key split.  Level 1, the first of two splits: as many as
// the second split will make of each of its buckets.  An empty segment has
// none: it owns no tile, and behind the last tile there is no place for their
// counts.
__host__ __device__ __forceinline__ uint32_t ss_buckets(uint64_t n, bool level1, uint64_t one_level) {
  if (level1) {
    if (n <= one_level) return 0u;
    // (sqrtf is correctly rounded on both sides)
    const uint32_t r = (uint32_t)sqrtf((float)((n + kSsBucket - 1) / kSsBucket)) + 1;
    return r < kSsMaxBuckets ? r : kSsMaxBuckets;
  }
  if (n == 0) return 0u;
  return n <= kSsLocal ? 1u : (uint32_t)umin64((n + kSsBucket - 1) / kSsBucket, kSsMaxBuckets);
}
__device__ __forceinline__ uint32_t ss_levels(uint32_t nb) { return nb <= 1 ? 0u : 32u - __clz(nb - 1); }

// Where the keys of segment s come from.
struct SsIn {
  const uint32_t* src = nullptr;
  const uint32_t* dst = nullptr;
  const uint64_t* keys = nullptr;
  __device__ __forceinline__ uint64_t get(uint64_t i) const {
    return keys ? keys[i] : ((uint64_t)src[i] << 32) | dst[i];
  }
  // Raw packets from `at` on can be read four at a time (get4).
  __device__ __forceinline__ bool vectors(uint64_t at) const {
    return !keys && (((uintptr_t)(src + at) | (uintptr_t)(dst + at)) & 15u) == 0;
  }
  __device__ __forceinline__ void get4(uint64_t at, uint32_t v, uint64_t* k) const {
    const uint4 x = reinterpret_cast<const uint4*>(src + at)[v], y = reinterpret_cast<const uint4*>(dst + at)[v];
    k[0] = (uint64_t)x.x << 32 | y.x;
    k[1] = (uint64_t)x.y << 32 | y.y;
    k[2] = (uint64_t)x.z << 32 | y.z;
    k[3] = (uint64_t)x.w << 32 | y.w;
  }
};
constexpr uint32_t kSsNone = 0xFFFFFFFFu;

// One split's segments: the plan's own (raw packets), or, after a first
// split, the list seg2 (keys of the first split's buckets, or a raw segment
// that was small enough).
__device__ __forceinline__ SsIn ss_input(const SsArgs& a, uint32_t s, uint64_t start) {
  SsIn in;
  uint32_t raw = s;
  if (a.parent) {
    const uint32_t p = a.parent[s];
    if (!(p & kSsRawBit)) {
      in.keys = a.keys_in + start;
      return in;
    }
    raw = p & ~kSsRawBit;
  }
  window_inputs(a.plan, raw, a.src, a.dst, &in.src, &in.dst);
  return in;
}

struct SsSeg {
  uint32_t s, b0, nb, ft;
  uint64_t start, n;
};
__device__ __forceinline__ SsSeg ss_seg(const SsArgs& a, uint32_t s) {
  SsSeg g;
  g.s = s;
  g.ft = a.first_tile[s];
  g.b0 = g.ft * kSsPerTile;
  g.n = a.len[s];
  g.start = a.start[s];
  g.nb = ss_buckets(g.n, a.level1, a.one_level);
  if (a.parent && a.parent[s] == kSsDone) g.nb = 0;
  return g;
}
__device__ __forceinline__ uint32_t ss_find(const SsArgs& a, uint32_t t) {
  if (a.tile_seg) return a.tile_seg[t];
  uint32_t lo = 0, hi = a.nseg_d ? *a.nseg_d : a.nseg;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (a.first_tile[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

constexpr int kSsSampleThreads = 1024;

// Bitonic sort of sm[0 .. R * 1024) by 1024 threads, R keys per thread in
// registers (key r of thread t is element r * 1024 + t): strides below a warp
// by shuffles, above the CTA's width in registers, the rest through sm.
template <int R>
__device__ __forceinline__ void ss_bitonic_r(uint64_t* sm) {
  const uint32_t t = threadIdx.x;
  uint64_t v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = sm[r * 1024 + t];
  for (uint32_t k = 2; k <= R * 1024u; k <<= 1) {
#pragma unroll
    for (int lr = 4; lr >= 0; --lr) {  // strides of whole register rows
      const int jr = 1 << lr;
      if (jr < R && (uint32_t)jr * 1024u < k) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if ((r & jr) == 0 && r + jr < R) {
            const bool up = (((uint32_t)r * 1024u + t) & k) == 0;
            const uint64_t x = v[r], y = v[(r + jr) % R];
            const bool sw = (x > y) == up;
            v[r] = sw ? y : x;
            v[(r + jr) % R] = sw ? x : y;
          }
        }
      }
    }
    for (uint32_t j = min(k >> 1, 512u); j > 0; j >>= 1) {
      if (j >= 32) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) sm[r * 1024 + t] = v[r];
        __syncthreads();
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const uint64_t o = j >= 32 ? sm[(r * 1024 + t) ^ j] : __shfl_xor_sync(0xffffffffu, v[r], j);
        const bool up = (((uint32_t)r * 1024u + t) & k) == 0, low = (t & j) == 0;
        v[r] = (v[r] > o) == (up == low) ? o : v[r];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < R; ++r) sm[r * 1024 + t] = v[r];
  __syncthreads();
}
__device__ __forceinline__ void ss_bitonic(uint64_t* sm, uint32_t S) {
  if (S == 1024) ss_bitonic_r<1>(sm);
  else if (S == 2048) ss_bitonic_r<2>(sm);
  else if (S == 4096) ss_bitonic_r<4>(sm);
  else if (S == 8192) ss_bitonic_r<8>(sm);
  else ss_bitonic_r<16>(sm);
}


// The segment's splitters as a search tree: tree[1 .. 2^lv) in breadth-first
// order over the sorted splitters (padded with all-ones).  Bucket b holds the
// keys k with exactly b splitters <= k.  A splitter value drawn twice or more
// is one that fills at least a bucket: it is kept together with its
// successor, so that the bucket between the two holds copies of it alone.
__global__ void __launch_bounds__(kSsSampleThreads) k_ss_sample(SsArgs a) {
  extern __shared__ __align__(16) uint64_t sm[];
  __shared__ uint32_t s_w[kSsSampleThreads / 32], s_tot;
  const uint32_t nseg = a.nseg_d ? *a.nseg_d : a.nseg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t s = blockIdx.x; s < nseg; s += gridDim.x) {
    const SsSeg g = ss_seg(a, s);
    for (uint32_t i = tid; i < g.nb; i += kSsSampleThreads) a.cnt[g.b0 + i] = a.cur[g.b0 + i] = 0;
    if (g.nb <= 1) continue;
    const SsIn in = ss_input(a, s, g.start);
    const uint32_t lv = ss_levels(g.nb);
    uint32_t S = 1024;
    while (S < g.nb * kSsOversample && S < a.sample_max) S <<= 1;
    // one key from each of S equal stretches of the segment
    for (uint32_t i = tid; i < S; i += kSsSampleThreads) {
      const uint64_t at = (((uint64_t)i << 16 | (fmix32(i + 1) & 0xFFFFu)) * g.n) >> (16 + (31 - __clz(S)));
      sm[i] = in.get(at);
    }
    __syncthreads();
    ss_bitonic(sm, S);
    // splitter candidates 1 .. nb - 1 (at most 1023: one per thread)
    auto cand = [&](uint32_t i) { return sm[(uint32_t)(((uint64_t)i * S) / g.nb)]; };
    const uint32_t c = tid + 1;
    const bool in_range = c < g.nb;
    const uint64_t v = in_range ? cand(c) : 0ull;
    const bool first = in_range && (c == 1 || cand(c - 1) != v);
    const bool twice = first && c + 1 < g.nb && cand(c + 1) == v && v != ~0ull;
    // the successor is dropped if it is itself the next splitter
    bool succ = twice;
    if (twice) {
      uint32_t lo = c + 1, hi = g.nb;  // the next different candidate
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (cand(mid) > v) hi = mid; else lo = mid + 1;
      }
      if (lo < g.nb && cand(lo) == v + 1) succ = false;
    }
    const uint32_t mine = (first ? 1u : 0u) + (succ ? 1u : 0u);
    uint32_t x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    uint32_t off = 0;
    for (int w = 0; w < warp; ++w) off += s_w[w];
    if (tid == kSsSampleThreads - 1) s_tot = off + x;
    __syncthreads();  // every candidate has been read: sm is rewritten below
    const uint32_t at = off + x - mine, m = s_tot;
    if (first) sm[at] = v;
    if (succ) sm[at + 1] = v + 1;
    __syncthreads();
    const uint32_t full = 1u << lv;
    uint64_t* tree = a.tree + (uint64_t)g.b0 * 2;
    for (uint32_t i = 1 + tid; i < full; i += kSsSampleThreads) {
      const uint32_t l = 31u - __clz(i), j = i - (1u << l);
      const uint32_t at2 = (2 * j + 1) * (full >> (l + 1)) - 1;
      tree[i] = at2 < m ? sm[at2] : ~0ull;
    }
    // buckets that hold one value: between neighbours that differ by one
    for (uint32_t b = tid; b < g.nb; b += kSsSampleThreads)
      a.eq[g.b0 + b] = b >= 1 && (b < m ? sm[b] == sm[b - 1] + 1 : b == m && sm[b - 1] == ~0ull) ? 1 : 0;
    if (tid == 0) tree[0] = m;  // splitters: buckets 0 .. m
    __syncthreads();
  }
}

// kT threads take kP keys each.
template <int kT, int kP>
__global__ void __launch_bounds__(kT, 1536 / kT) k_ss_count(SsArgs a) {
  constexpr uint32_t kTT = kT * kP, kSub = kTile / kTT;
  __shared__ uint64_t s_tree[kSsMaxBuckets];
  __shared__ uint32_t s_h[kSsMaxBuckets];
  const uint32_t t = blockIdx.x / kSub;
  if (a.ntiles_d && t >= *a.ntiles_d) return;
  const SsSeg g = ss_seg(a, ss_find(a, t));
  const uint64_t off = (uint64_t)(t - g.ft) * kTile + (uint64_t)(blockIdx.x % kSub) * kTT;
  if (g.nb <= 1 || off >= g.n) return;
  const uint32_t count = (uint32_t)umin64(kTT, g.n - off);
  const uint32_t lv = ss_levels(g.nb);
  const uint64_t* tree = a.tree + (uint64_t)g.b0 * 2;
  for (uint32_t i = threadIdx.x; i < (1u << lv); i += kT) {
    s_tree[i] = tree[i];
    s_h[i] = 0;
  }
  const SsIn in = ss_input(a, g.s, g.start);
  uint64_t k[kP];
  const bool vec = count == kTT && in.vectors(off);
  if (vec) {
#pragma unroll
    for (int i = 0; i < kP; i += 4) in.get4(off, (i / 4) * kT + threadIdx.x, &k[i]);
  } else if (count == kTT && in.keys) {
    const uint64_t* kk = in.keys + off;
#pragma unroll
    for (int i = 0; i < kP; ++i) k[i] = kk[i * kT + threadIdx.x];
  } else {
#pragma unroll
    for (int i = 0; i < kP; ++i) {
      const uint32_t x = i * kT + threadIdx.x;
      k[i] = x < count ? in.get(off + x) : 0ull;
    }
  }
  __syncthreads();
  const uint32_t last = (uint32_t)s_tree[0];
  uint32_t node[kP];
#pragma unroll
  for (int i = 0; i < kP; ++i) node[i] = 1;
  for (uint32_t l = 0; l < lv; ++l) {
#pragma unroll
    for (int i = 0; i < kP; ++i) node[i] = 2 * node[i] + (k[i] >= s_tree[node[i]] ? 1u : 0u);
  }
  uint16_t* ids = a.ids + g.start + off;
  // (a key of all ones passes the padding too)
#pragma unroll
  for (int i = 0; i < kP; ++i) node[i] = min(node[i] - (1u << lv), last);
  if (vec) {
#pragma unroll
    for (int i = 0; i < kP; i += 4)
      reinterpret_cast<ushort4*>(ids)[(i / 4) * kT + threadIdx.x] =
          make_ushort4((uint16_t)node[i], (uint16_t)node[i + 1], (uint16_t)node[i + 2], (uint16_t)node[i + 3]);
  }
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const uint32_t x = i * kT + threadIdx.x;
    if (vec || x < count) {
      if (!vec) ids[x] = (uint16_t)node[i];
      atomicAdd(&s_h[node[i]], 1u);
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < g.nb; i += kT) {
    const uint32_t c = s_h[i];
    if (c) atomicAdd(&a.cnt[g.b0 + i], c);
  }
}

template <int kT, int kP>
constexpr size_t ss_scatter_smem() {
  return (size_t)kT * kP * 10;
}

template <int kT, int kP, int kMinB>
__global__ void __launch_bounds__(kT, kMinB) k_ss_scatter(SsArgs a) {
  constexpr uint32_t kTT = kT * kP, kSub = kTile / kTT;
  constexpr int kPer = kSsMaxBuckets / kT;  // buckets per thread
  static_assert(kPer * kT == kSsMaxBuckets, "");
  extern __shared__ __align__(16) uint8_t smem[];
  uint64_t* s_keys = reinterpret_cast<uint64_t*>(smem);
  uint16_t* s_ids = reinterpret_cast<uint16_t*>(smem + (size_t)kTT * 8);
  __shared__ uint32_t s_h[kSsMaxBuckets];    // count, then the bucket's first slot in the tile
  __shared__ uint32_t s_rel[kSsMaxBuckets];  // tile slot -> segment position
  __shared__ uint64_t s_w[kT / 32];
  const uint32_t t = blockIdx.x / kSub;
  if (a.ntiles_d && t >= *a.ntiles_d) return;
  const SsSeg g = ss_seg(a, ss_find(a, t));
  const uint64_t off = (uint64_t)(t - g.ft) * kTile + (uint64_t)(blockIdx.x % kSub) * kTT;
  if (g.nb <= 1 || off >= g.n) return;
  const uint32_t count = (uint32_t)umin64(kTT, g.n - off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t i = threadIdx.x; i < kSsMaxBuckets; i += kT) s_h[i] = 0;
  const SsIn in = ss_input(a, g.s, g.start);
  const uint16_t* ids = a.ids + g.start + off;
  uint64_t k[kP];
  uint32_t r[kP];  // bucket << 16 | rank; kSsNone: past the end
  if (count == kTT && in.vectors(off)) {
#pragma unroll
    for (int i = 0; i < kP; i += 4) {
      const uint32_t v = (i / 4) * kT + threadIdx.x;
      const ushort4 b = reinterpret_cast<const ushort4*>(ids)[v];
      in.get4(off, v, &k[i]);
      r[i] = (uint32_t)b.x << 16;
      r[i + 1] = (uint32_t)b.y << 16;
      r[i + 2] = (uint32_t)b.z << 16;
      r[i + 3] = (uint32_t)b.w << 16;
    }
  } else if (count == kTT && in.keys) {
    const uint64_t* kk = in.keys + off;
#pragma unroll
    for (int i = 0; i < kP; ++i) k[i] = kk[i * kT + threadIdx.x];
#pragma unroll
    for (int i = 0; i < kP; ++i) r[i] = (uint32_t)ids[i * kT + threadIdx.x] << 16;
  } else {
#pragma unroll
    for (int i = 0; i < kP; ++i) {
      const uint32_t x = i * kT + threadIdx.x;
      r[i] = x < count ? (uint32_t)ids[x] << 16 : kSsNone;
      k[i] = x < count ? in.get(off + x) : 0ull;
    }
  }
  uint32_t all[kPer];  // the segment's bucket sizes (a first split's cursors are places already)
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t b = threadIdx.x * kPer + j;
    all[j] = !a.level1 && b < g.nb ? a.cnt[g.b0 + b] : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kP; ++i)
    if (r[i] != kSsNone) r[i] |= atomicAdd(&s_h[r[i] >> 16], 1u);
  __syncthreads();
  // exclusive prefixes of the tile's counts (low) and the segment's (high)
  uint32_t got[kPer];
  uint64_t run = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t b = threadIdx.x * kPer + j;
    const uint32_t c = s_h[b];
    // space in the bucket; the answer is not needed before the write-out
    got[j] = c ? atomicAdd(&a.cur[g.b0 + b], c) : 0u;
    run += (uint64_t)all[j] << 32 | c;
  }
  uint64_t x = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  uint64_t before = x - run;
#pragma unroll
  for (int w = 0; w < kT / 32; ++w) before += w < warp ? s_w[w] : 0ull;
  const bool lead = !a.level1 && off == 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t b = threadIdx.x * kPer + j, c = s_h[b];
    s_h[b] = (uint32_t)before;
    s_rel[b] = (uint32_t)(before >> 32) - (uint32_t)before;
    if (lead && b < g.nb) a.bstart[g.b0 + b] = (uint32_t)(before >> 32);
    before += (uint64_t)all[j] << 32 | c;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    if (r[i] != kSsNone) {
      const uint32_t b = r[i] >> 16, pos = s_h[b] + (r[i] & 0xFFFFu);
      s_keys[pos] = k[i];
      s_ids[pos] = (uint16_t)b;
    }
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) s_rel[threadIdx.x * kPer + j] += got[j];
  __syncthreads();
  uint64_t* out = a.keys_split + g.start;
#pragma unroll 4
  for (uint32_t i = threadIdx.x; i < count; i += kT) out[s_rel[s_ids[i]] + i] = s_keys[i];
}

// ---- local sort --------------------------------------------------------------
constexpr int kSsLT = 128;  // threads
constexpr int kSsLP = 16;   // keys per thread
constexpr uint32_t kSsWarpKeys = 32 * kSsLP;
static_assert(kSsLT * kSsLP == kSsLocal, "one CTA sorts kSsLocal keys");
// one word of padding per run of a thread keeps threads that walk their runs
// off each other's banks
__device__ __forceinline__ uint32_t ss_pad(uint32_t i) { return i + i / kSsLP; }

template <typename K>
__device__ __forceinline__ void ss_cx(K& x, K& y) {
  const bool sw = x > y;
  const K lo = sw ? y : x, hi = sw ? x : y;
  x = lo;
  y = hi;
}

// Batcher's odd-even merge sort of a thread's keys (Batcher 1968).
template <typename K>
__device__ __forceinline__ void ss_sort_run(K (&k)[kSsLP]) {
#pragma unroll
  for (int lp = 0; (1 << lp) < kSsLP; ++lp) {
#pragma unroll
    for (int lq = lp; lq >= 0; --lq) {
      const int q = 1 << lq, j0 = lq == lp ? 0 : q;
#pragma unroll
      for (int i = 0; i < kSsLP; ++i) {  // i: the lower index of a comparator, if it is one
        const int x = i - j0;
        if (x >= 0 && (x & q) == 0 && i + q < kSsLP && (i >> (lp + 1)) == ((i + q) >> (lp + 1))) ss_cx(k[i], k[i + q]);
      }
    }
  }
}

// The keys k of threads 0 .. T - 1, 16 each, sorted into sm[ss_pad(0 ..)].
template <typename K>
__device__ __forceinline__ void ss_sort_keys(K (&k)[kSsLP], uint32_t T, K* sm) {
  const uint32_t tid = threadIdx.x, m16 = T * kSsLP;
  if (tid < T) {
    ss_sort_run(k);
#pragma unroll
    for (int j = 0; j < kSsLP; ++j) sm[tid * (kSsLP + 1) + j] = k[j];
  }
  for (uint32_t R = kSsLP; R < m16; R <<= 1) {
    const bool wide = 2 * R > kSsWarpKeys;  // a pair of runs spans warps
    if (wide) __syncthreads(); else __syncwarp();
    const uint32_t o = tid * kSsLP, g0 = o & ~(2 * R - 1);
    const bool act = o < m16 && g0 + R < m16;
    if (act) {
      const uint32_t A = g0, B = g0 + R, na = R, nb = min(R, m16 - B), diag = o - g0;
      uint32_t lo = diag > nb ? diag - nb : 0u, hi = diag < na ? diag : na;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (sm[ss_pad(A + mid)] <= sm[ss_pad(B + diag - 1 - mid)]) lo = mid + 1; else hi = mid;
      }
      uint32_t ai = A + lo, bi = B + diag - lo;
      const uint32_t ae = A + na, be = B + nb;
      K ka = sm[ss_pad(min(ai, ae - 1))], kb = sm[ss_pad(min(bi, be - 1))];
#pragma unroll
      for (int j = 0; j < kSsLP; ++j) {
        const bool pa = bi >= be || (ai < ae && ka <= kb);
        k[j] = pa ? ka : kb;
        const uint32_t nx = (pa ? ai : bi) + 1;
        if (pa) ai = nx; else bi = nx;
        // (one past a run's end is inside the buffer and never used)
        const K kn = sm[ss_pad(nx)];
        if (pa) ka = kn; else kb = kn;
      }
    }
    if (wide) __syncthreads(); else __syncwarp();
    if (act) {
#pragma unroll
      for (int j = 0; j < kSsLP; ++j) sm[tid * (kSsLP + 1) + j] = k[j];
    }
  }
  __syncthreads();
}

// Sort in.get(at .. at + m), 0 < m <= kSsLocal, into out[0 .. m); every
// thread of the CTA calls it.  sm: ss_pad(kSsLocal) + 1 keys.  Keys that share
// their high word (one source: half of the buckets of 2^30 packets of Zipf
// traffic) are sorted by their low words: half the shared-memory traffic and a
// third of the instructions of a comparison.
__device__ __forceinline__ void ss_sort_block(const SsIn& in, uint64_t at, uint32_t m, uint64_t* out, uint64_t* sm) {
  const uint32_t tid = threadIdx.x;
  uint64_t k[kSsLP];
  // any assignment of keys to threads will do: coalesced loads.  Threads
  // 0 .. T - 1 hold a run each, missing keys all ones (sorted last).
  const uint32_t T = (m + kSsLP - 1) / kSsLP;
  uint32_t high = 0, differ = 0;
  if (tid < T) {
    high = (uint32_t)(in.get(at) >> 32);
#pragma unroll
    for (int j = 0; j < kSsLP; ++j) {
      const uint32_t i = j * T + tid;
      k[j] = i < m ? in.get(at + i) : ~0ull;
      differ |= i < m ? (uint32_t)(k[j] >> 32) ^ high : 0u;
    }
  }
  if (__syncthreads_or((int)differ)) {
    ss_sort_keys(k, T, sm);
    for (uint32_t i = tid; i < m; i += kSsLT) out[i] = sm[ss_pad(i)];
  } else {
    uint32_t* s32 = reinterpret_cast<uint32_t*>(sm);
    uint32_t l[kSsLP];
#pragma unroll
    for (int j = 0; j < kSsLP; ++j) l[j] = (uint32_t)k[j];
    ss_sort_keys(l, T, s32);
    high = (uint32_t)(in.get(at) >> 32);
    for (uint32_t i = tid; i < m; i += kSsLT) out[i] = (uint64_t)high << 32 | s32[ss_pad(i)];
  }
  __syncthreads();  // sm may be reused
}

// How many of the first `diag` keys of merge(A, B) come from A.
__device__ __forceinline__ uint32_t ss_merge_path(const uint64_t* A, uint32_t na, const uint64_t* B, uint32_t nb,
                                                  uint32_t diag) {
  uint32_t lo = diag > nb ? diag - nb : 0u, hi = diag < na ? diag : na;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (A[mid] <= B[diag - 1 - mid]) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(kSsLT, 8) k_ss_local(SsArgs a) {
  __shared__ uint64_t sm[kSsLocal + kSsLocal / kSsLP + 1];
  const uint32_t t = blockIdx.x / kSsPerTile;
  if (a.ntiles_d && t >= *a.ntiles_d) return;
  const SsSeg g = ss_seg(a, ss_find(a, t));
  const uint32_t b = blockIdx.x - g.b0;
  if (b >= g.nb) return;
  if (g.nb == 1) {  // never split: the whole segment
    ss_sort_block(ss_input(a, g.s, g.start), 0, (uint32_t)g.n, a.keys_out + g.start, sm);
    return;
  }
  const uint32_t m = a.cnt[g.b0 + b];
  if (m == 0) return;
  const uint64_t at = g.start + a.bstart[g.b0 + b];
  uint64_t* from = a.keys_split + at;
  uint64_t* to = a.keys_out + at;
  if (a.eq[g.b0 + b]) {  // copies of one key
    const uint64_t v = from[0];
    for (uint32_t i = threadIdx.x; i < m; i += kSsLT) to[i] = v;
    return;
  }
  SsIn in;
  in.keys = from;
  if (m <= kSsLocal) {
    ss_sort_block(in, 0, m, to, sm);
    return;
  }
  // A bucket the sample misjudged: kSsLocal keys at a time, then merge rounds
  // between the two buffers, ending in keys_out.
  int rounds = 0;
  for (uint64_t r = kSsLocal; r < m; r <<= 1) ++rounds;
  uint64_t* x = rounds % 2 ? from : to;
  for (uint32_t c = 0; c < m; c += kSsLocal) ss_sort_block(in, c, min(kSsLocal, m - c), x + c, sm);
  __syncthreads();
  for (uint64_t R = kSsLocal; R < m; R <<= 1) {
    uint64_t* y = x == from ? to : from;
    for (uint64_t o = (uint64_t)threadIdx.x * kSsLP; o < m; o += (uint64_t)kSsLT * kSsLP) {
      const uint64_t g0 = o / (2 * R) * (2 * R);
      const uint64_t na = umin64(R, m - g0), nb = umin64(R, m - g0 - na);
      const uint64_t *A = x + g0, *B = A + na;
      const uint32_t diag = (uint32_t)(o - g0), end = (uint32_t)umin64(kSsLP, m - o);
      uint32_t ai = ss_merge_path(A, (uint32_t)na, B, (uint32_t)nb, diag);
      uint32_t bi = diag - ai;
      for (uint32_t j = 0; j < end; ++j) {
        const bool pa = bi >= nb || (ai < na && A[ai] <= B[bi]);
        y[o + j] = pa ? A[ai++] : B[bi++];
      }
    }
    __syncthreads();
    x = y;
  }
}

// Between count and scatter of a first split (one CTA): the starts of its
// buckets (their cursors), and the second split's segments: every bucket of a
// segment that is split, every other segment as it is.  seg2 arrays hold their
// starts, lengths, parents and first tiles.
__global__ void __launch_bounds__(1024) k_ss_plan2(SsArgs a, SsSeg2 o) {
  __shared__ uint32_t s_w[32], s_carry;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto scan = [&](uint32_t v) -> uint32_t {  // exclusive, carried from call to call
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    uint32_t off = 0, tot = 0;
    for (int w = 0; w < 32; ++w) {
      off += w < warp ? s_w[w] : 0u;
      tot += s_w[w];
    }
    const uint32_t r = s_carry + off + x - v;
    __syncthreads();
    if (tid == 0) s_carry += tot;
    __syncthreads();
    return r;
  };
  __shared__ uint2 s_big[1024];  // (segment, its first bucket's place in the list)
  __shared__ uint32_t s_nbig;
  if (tid == 0) s_carry = 0;
  __syncthreads();
  for (uint32_t s0 = 0; s0 < a.nseg; s0 += 1024) {
    const uint32_t s = s0 + tid;
    const bool in = s < a.nseg;
    const SsSeg g = ss_seg(a, in ? s : 0);
    if (tid == 0) s_nbig = 0;
    const uint32_t at = scan(!in ? 0u : g.nb ? g.nb : 1u);
    if (in && !g.nb) {
      o.start[at] = g.start;
      o.len[at] = g.n;
      o.parent[at] = s | kSsRawBit;
    } else if (in) {
      s_big[atomicAdd(&s_nbig, 1u)] = make_uint2(s, at);
    }
    __syncthreads();
    const uint32_t carry = s_carry;
    for (uint32_t e = 0; e < s_nbig; ++e) {  // one thread per bucket
      const SsSeg h = ss_seg(a, s_big[e].x);
      const uint32_t sum = tid < h.nb ? a.cnt[h.b0 + tid] : 0u;
      if (tid == 0) s_carry = 0;
      __syncthreads();
      const uint32_t run = scan(sum);
      if (tid < h.nb) {
        const uint32_t i = s_big[e].y + tid;
        o.start[i] = h.start + run;
        o.len[i] = sum;
        o.parent[i] = sum && a.eq[h.b0 + tid] ? kSsDone : 0u;
        a.cur[h.b0 + tid] = run;
      }
      __syncthreads();
    }
    if (tid == 0) s_carry = carry;
    __syncthreads();
  }
  const uint32_t n2 = s_carry;
  __syncthreads();
  if (tid == 0) s_carry = 0;
  __syncthreads();
  for (uint32_t s0 = 0; s0 < n2; s0 += 1024) {
    const uint32_t s = s0 + tid;
    const uint32_t at = scan(s < n2 ? (uint32_t)((o.len[s] + kTile - 1) / kTile) : 0u);
    if (s < n2) o.first_tile[s] = at;
  }
  if (tid == 0) {
    o.first_tile[n2] = s_carry;
    o.count[0] = n2;
    o.count[1] = s_carry;
  }
}

__global__ void __launch_bounds__(256) k_ss_tile_seg(SsSeg2 o) {
  const uint32_t n2 = o.count[0];
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < o.count[1]; t += gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = n2;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (o.first_tile[mid] <= t) lo = mid; else hi = mid;
    }
    o.tile_seg[t] = lo;
  }
}

template <typename F>
cudaError_t set_smem_once(F* f, size_t bytes, unsigned long long* done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 64 && ((*done >> dev) & 1ull)) return cudaSuccess;
  e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && dev < 64) *done |= 1ull << dev;
  return e;
}

}  // namespace

// (about sqrt(n / kSsBucket) + 1 buckets of an n-key segment, which is longer
// than 2^18 keys: at most n / 2^13, and 1024)
uint64_t ss_level1_buckets(uint64_t total, uint64_t nseg) {
  const uint64_t by_len = total / (1u << 13) + 1, by_seg = nseg * kSsMaxBuckets;
  return by_len < by_seg ? by_len : by_seg;
}

cudaError_t launch_ss_sample(const SsArgs& a0, uint64_t max_len, cudaStream_t st) {
  if (a0.ntiles == 0 || a0.nseg == 0) return cudaSuccess;
  static unsigned long long done = 0;
  cudaError_t e = set_smem_once(k_ss_sample, kSsSampleMax * 8, &done);
  if (e != cudaSuccess) return e;
  SsArgs a = a0;
  a.sample_max = 1024;
  const uint64_t want = (uint64_t)umin64(kSsSampleMax, (uint64_t)umax64(1, ss_buckets(max_len, a.level1, a.one_level)) * kSsOversample);
  while (a.sample_max < want) a.sample_max <<= 1;
  // (the splitters are compacted in the same buffer, which is as long as a
  // split's most buckets at least)
  const uint32_t grid = a.nseg < 65536u ? a.nseg : 65536u;
  k_ss_sample<<<grid, kSsSampleThreads, (size_t)a.sample_max * 8, st>>>(a);
  return cudaGetLastError();
}

// Tiles below this many are cut into four: 2048 keys per CTA fill the 152
// SMs from 2^18 keys on.
constexpr uint32_t kSsSmallTiles = 608;
int ss_shape(uint32_t ntiles) { return ntiles <= kSsSmallTiles ? 0 : 1; }

cudaError_t launch_ss_count(const SsArgs& a, cudaStream_t st) {
  if (a.ntiles == 0) return cudaSuccess;
  k_ss_count<256, 8><<<a.ntiles * 4, 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_ss_scatter(const SsArgs& a, cudaStream_t st) {
  if (a.ntiles == 0) return cudaSuccess;
  if (ss_shape(a.ntiles) == 0) {
    k_ss_scatter<256, 8, 4><<<a.ntiles * 4, 256, ss_scatter_smem<256, 8>(), st>>>(a);
  } else {
    static unsigned long long done = 0;
    cudaError_t e = set_smem_once(k_ss_scatter<512, 16, 2>, ss_scatter_smem<512, 16>(), &done);
    if (e != cudaSuccess) return e;
    k_ss_scatter<512, 16, 2><<<a.ntiles, 512, ss_scatter_smem<512, 16>(), st>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t launch_ss_local(const SsArgs& a, cudaStream_t st) {
  if (a.ntiles == 0) return cudaSuccess;
  k_ss_local<<<a.ntiles * kSsPerTile, kSsLT, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_ss_plan2(const SsArgs& a, const SsSeg2& o, cudaStream_t st) {
  k_ss_plan2<<<1, 1024, 0, st>>>(a, o);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_ss_tile_seg<<<512, 256, 0, st>>>(o);
  return cudaGetLastError();
}

}  // namespace ans
