// Column statistics of stored links by hash partitions of their destinations
// (Table I: unique destinations, max fan-in; Sec. IV-C: max destination
// packets).
//
// The three quantities only need equal destinations together, in any order.
// h = fmix32(destination) is a bijection; a segment of n links is cut into
// about n / kColPart partitions by the high bits of h.  k_finish, which reads
// every link anyway, counts the partitions; then
//   scatter  moves (destination, count) to its partition, ranks by one
//            shared-memory atomic per link, space by one global atomic per
//            partition and tile -- no order to keep, no look-back;
//   count    one CTA per partition counts its destinations in a shared-memory
//            table and adds the table's three quantities to the segment's.
// A partition with more destinations than the table takes (a segment of more
// than 2048 tables' worth of them, or destinations crowded into one) is cut by
// its CTA into parts of about kColPart links, by another mix of the
// destination, in memory, and the parts are counted one by one: two readings
// and a writing of its links more.  A part with too many still, or the
// partition where there is no such memory, is read again in 2, 4, ... classes.
// So every input ends here and no sort stands behind.  (9 million links of as
// many destinations: count 174 us, 225 with 64-bit counts, against 464 and 495
// for the four passes of a column sort; 2^25: 584 and 763 against 1588 and 1682.
// Reading all of it in classes, after tables filled to the brim: 5.0 ms and 10.6.)
//
// A destination with a large share of the links would make one partition, and
// one table slot, a queue.  In segments of kColHeavyLinks links or more those
// with 8 or more of 2048 sampled links are listed first (k_col_heavy) and
// added up by k_finish (a sum of 4.6 million links of bursty traffic: 127
// against 381 us).  Shorter segments do without: listing costs 20 us a launch
// and every link of k_finish a probe, and adding equal destinations of a warp
// once (__match_any_sync) makes one window of 2^17 packets 47 instead of 24.5 us.
//
// The column sorts and the one-CTA-per-window hashes that this replaces took
// 174 us for that window (24.5 now), 448 us for 64 windows and their sum.
#include "ans_internal.cuh"

namespace ans {

namespace {

constexpr uint32_t kColSlots = 4096;               // table slots of one CTA
constexpr uint32_t kColFill = kColSlots / 4 * 3;   // give up above this
constexpr uint32_t kColEarly = 920;                // or above this after 1024 links
constexpr uint32_t kColSubs = 512;                 // most parts of a cut partition
constexpr uint32_t kColNone = 0xFFFFFFFFu;         // empty slot (that destination is counted apart)
constexpr int kColThreads = 256;

constexpr uint32_t kColSample = 2048;
constexpr int kColHeavyThreads = 512;
constexpr uint32_t kColHeavyMin = 8;    // sampled links of a heavy destination
constexpr uint32_t kColHeavyMost = 48;  // destinations listed

// One CTA per segment: its heavy destinations, as a table of 64 slots
// (kColNone: empty).
__global__ void __launch_bounds__(kColHeavyThreads) k_col_heavy(SegPlan p, ColParts c, const uint32_t* __restrict__ col_ids,
                                                           const uint64_t* __restrict__ hdr) {
  __shared__ uint32_t t_key[2 * kColSample], t_cnt[2 * kColSample];
  __shared__ uint32_t s_key[kColHeavySlots], s_n[16];
  const uint32_t s = blockIdx.x;
  if (s >= p.nseg) return;
  const uint64_t n = hdr[2 * (uint64_t)s + 1];
  if (n < kColHeavyLinks) return;
  const uint32_t* d0 = col_ids + p.base[s];
  for (uint32_t i = threadIdx.x; i < 2 * kColSample; i += kColHeavyThreads) {
    t_key[i] = kColNone;
    t_cnt[i] = 0;
  }
  if (threadIdx.x < kColHeavySlots) s_key[threadIdx.x] = kColNone;
  if (threadIdx.x < 16) s_n[threadIdx.x] = 0;
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < kColSample; j += kColHeavyThreads) {  // one link of each stretch
    const uint32_t d = d0[(((uint64_t)j << 16 | (fmix32(j + 1) & 0xFFFFu)) * n) / ((uint64_t)kColSample << 16)];
    if (d == kColNone) continue;  // (the count has a place of its own for it)
    uint32_t i = fmix32(d) & (2 * kColSample - 1);
    for (;;) {  // at most half of the slots are taken
      const uint32_t cur = atomicCAS(&t_key[i], kColNone, d);
      if (cur == kColNone || cur == d) break;
      i = (i + 1) & (2 * kColSample - 1);
    }
    atomicAdd(&t_cnt[i], 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < 2 * kColSample; i += kColHeavyThreads)
    if (t_cnt[i] >= kColHeavyMin) atomicAdd(&s_n[31 - __clz(t_cnt[i])], 1u);
  __syncthreads();
  uint32_t lg = 15, most = 0;  // the lowest power of two that lists at most kColHeavyMost
  while (lg > 3 && most + s_n[lg - 1] <= kColHeavyMost) most += s_n[--lg];
  for (uint32_t i = threadIdx.x; i < 2 * kColSample; i += kColHeavyThreads) {
    if (t_cnt[i] < (1u << lg)) continue;
    uint32_t j = fmix32(t_key[i]) & (kColHeavySlots - 1);
    while (atomicCAS(&s_key[j], kColNone, t_key[i]) != kColNone) j = (j + 1) & (kColHeavySlots - 1);
  }
  __syncthreads();
  if (threadIdx.x < kColHeavySlots) c.hkey[(uint64_t)p.first_tile[s] * kColHeavyPerTile + threadIdx.x] = s_key[threadIdx.x];
}
static_assert(1u << 3 == kColHeavyMin, "the lowest count listed");

// The part of destination d among `subs` of its partition (its class comes
// from another mix).
__device__ __forceinline__ uint32_t col_sub(uint32_t d, uint32_t subs) {
  return __umulhi(fmix32(fmix32(d) ^ 0x7F4A7C15u), subs);
}

struct ColSeg {
  uint32_t ft, parts;
  uint64_t n;
};
__device__ __forceinline__ ColSeg col_seg(const SegPlan& p, uint32_t s, uint32_t max_parts) {
  ColSeg g;
  g.ft = p.first_tile[s];
  g.n = p.len[s];
  g.parts = col_parts(g.n, max_parts);
  return g;
}

// One sub-tile of kT * kP links per CTA.  kWide: 64-bit counts.
template <bool kWide, int kT, int kP>
__global__ void __launch_bounds__(kT, kP == 16 ? (kWide ? 1 : 2) : kT == 512 ? 3 : 4) k_col_scatter(SegPlan p, ColParts c, const uint32_t* __restrict__ col_ids,
                                                    const uint32_t* __restrict__ vals32,
                                                    const uint64_t* __restrict__ vals64, uint32_t* __restrict__ odst,
                                                    void* __restrict__ oval) {
  using V = typename std::conditional<kWide, uint64_t, uint32_t>::type;
  constexpr uint32_t kTT = kT * kP, kSub = kTile / kTT;
  extern __shared__ __align__(16) uint8_t smem[];
  V* s_val = reinterpret_cast<V*>(smem);
  uint32_t* s_dst = reinterpret_cast<uint32_t*>(smem + (size_t)kTT * sizeof(V));
  uint32_t* s_h = s_dst + kTT;  // [parts] count, then the partition's first slot in the tile
  uint32_t* s_rel = s_h + c.max_parts;  // [parts] tile slot -> segment position
  __shared__ uint64_t s_w[kT / 32];
  __shared__ uint32_t s_hkey[kColHeavySlots];
  const uint32_t t = blockIdx.x / kSub;
  const uint32_t s = find_seg(p, t);
  const ColSeg g = col_seg(p, s, c.max_parts);
  const uint64_t off = (uint64_t)(t - g.ft) * kTile + (uint64_t)(blockIdx.x % kSub) * kTT;
  if (g.parts <= 1 || off >= g.n) return;
  const uint32_t count = (uint32_t)umin64(kTT, g.n - off);
  const uint64_t base = p.base[s];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const V* vin = kWide ? (const V*)vals64 : (const V*)vals32;
  uint32_t d[kP], r[kP];
  V v[kP];
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    const uint32_t x = i * kT + threadIdx.x;
    d[i] = x < count ? col_ids[base + off + x] : 0u;
    v[i] = x < count ? vin[base + off + x] : V(0);
  }
  for (uint32_t b = threadIdx.x; b < g.parts; b += kT) s_h[b] = 0;
  const bool heavy = g.n >= kColHeavyLinks;
  if (heavy && threadIdx.x < kColHeavySlots) s_hkey[threadIdx.x] = c.hkey[(size_t)g.ft * kColHeavyPerTile + threadIdx.x];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    r[i] = kColNone;  // past the end, or a heavy destination's: not moved
    if (i * kT + threadIdx.x < count && !(heavy && col_heavy(s_hkey, d[i]) >= 0)) {
      const uint32_t b = col_part(d[i], g.parts);
      r[i] = b << 16 | atomicAdd(&s_h[b], 1u);
    }
  }
  __syncthreads();
  // exclusive prefixes of the tile's counts (low) and the segment's (high);
  // consecutive partitions per thread
  const uint32_t* cnt = c.cnt + (size_t)g.ft * kColPerTile;
  uint32_t* cur = c.cur + (size_t)g.ft * kColPerTile;
  const uint32_t per = (g.parts + kT - 1) / kT;
  const uint32_t b0 = min(threadIdx.x * per, g.parts), b1 = min(b0 + per, g.parts);
  constexpr int kB = kP == 16 ? 4 : 1;  // partitions whose loads and atomics are in flight together
  uint64_t run = 0;
  for (uint32_t c0 = b0; c0 < b1; c0 += kB) {
    uint32_t all[kB];
#pragma unroll
    for (int j = 0; j < kB; ++j) all[j] = c0 + j < b1 ? cnt[c0 + j] : 0u;
#pragma unroll
    for (int j = 0; j < kB; ++j)
      if (c0 + j < b1) run += (uint64_t)all[j] << 32 | s_h[c0 + j];
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
  uint32_t moved = 0;
#pragma unroll
  for (int w = 0; w < kT / 32; ++w) {
    before += w < warp ? s_w[w] : 0ull;
    moved += (uint32_t)s_w[w];
  }
  const bool lead = off == 0;
  for (uint32_t c0 = b0; c0 < b1; c0 += kB) {
    uint32_t all[kB], k[kB], got[kB];
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      const bool in = c0 + j < b1;
      all[j] = in ? cnt[c0 + j] : 0u;
      k[j] = in ? s_h[c0 + j] : 0u;
      got[j] = k[j] ? atomicAdd(&cur[c0 + j], k[j]) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      if (c0 + j < b1) {
        const uint32_t slot = (uint32_t)before, start = (uint32_t)(before >> 32);
        s_h[c0 + j] = slot;
        s_rel[c0 + j] = start + got[j] - slot;
        if (lead) c.start[(size_t)g.ft * kColPerTile + c0 + j] = start;
        before += (uint64_t)all[j] << 32 | k[j];
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kP; ++i) {
    if (r[i] != kColNone) {
      const uint32_t pos = s_h[r[i] >> 16] + (r[i] & 0xFFFFu);
      s_dst[pos] = d[i];
      s_val[pos] = v[i];
    }
  }
  __syncthreads();
  V* ov = reinterpret_cast<V*>(oval) + base;
#pragma unroll 4
  for (uint32_t i = threadIdx.x; i < moved; i += kT) {
    const uint32_t k = s_dst[i], o = s_rel[col_part(k, g.parts)] + i;
    odst[base + o] = k;
    ov[o] = s_val[i];
  }
}

// The links kd, vd[0 .. m) of an overfull partition moved to sd, sv, grouped
// into `subs` parts; start[0 .. subs] gets the parts' places.  Every thread of
// the CTA calls it; cur: `subs` shared words.
template <typename V>
__device__ __forceinline__ void col_cut(const uint32_t* kd, const V* vd, uint32_t m, uint32_t subs, uint32_t* sd, V* sv,
                                        uint32_t* start, uint32_t* cur) {
  static_assert(kColSubs == 2 * kColThreads, "two parts per thread in the scan");
  __shared__ uint32_t s_w[kColThreads / 32];
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t i = tid; i < subs; i += kColThreads) cur[i] = 0;
  __syncthreads();
#pragma unroll 4
  for (uint32_t u = tid; u < m; u += kColThreads) atomicAdd(&cur[col_sub(kd[u], subs)], 1u);
  __syncthreads();
  const uint32_t a = 2 * tid < subs ? cur[2 * tid] : 0u, b = 2 * tid + 1 < subs ? cur[2 * tid + 1] : 0u;
  uint32_t x = a + b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  uint32_t off = x - a - b;
  for (uint32_t w = 0; w < warp; ++w) off += s_w[w];
  if (2 * tid < subs) start[2 * tid] = cur[2 * tid] = off;
  if (2 * tid + 1 < subs) start[2 * tid + 1] = cur[2 * tid + 1] = off + a;
  if (tid == 0) start[subs] = m;
  __syncthreads();
#pragma unroll 4
  for (uint32_t u = tid; u < m; u += kColThreads) {
    const uint32_t d = kd[u];
    const V v = vd[u];
    const uint32_t at = atomicAdd(&cur[col_sub(d, subs)], 1u);
    sd[at] = d;
    sv[at] = v;
  }
  __syncthreads();
}

// One partition per CTA (one that was never split is the whole segment).
template <bool kWide>
__global__ void __launch_bounds__(kColThreads, kWide ? 3 : 4) k_col_count(SegPlan p, ColParts c,
                                                                          const uint32_t* __restrict__ col_ids,
                                                                          const uint32_t* __restrict__ vals32,
                                                                          const uint64_t* __restrict__ vals64,
                                                                          const uint32_t* __restrict__ pdst,
                                                                          const void* __restrict__ pval,
                                                                          ans_quantities* __restrict__ q) {
  using V = typename std::conditional<kWide, uint64_t, uint32_t>::type;
  extern __shared__ __align__(16) uint32_t t_key[];
  uint32_t* t_cnt = t_key + kColSlots;
  uint32_t* t_lo = t_cnt + kColSlots;
  uint32_t* t_hi = t_lo + kColSlots;  // kWide only
  __shared__ uint32_t s_fill, s_over, s_spec_cnt, s_spec_lo, s_spec_hi;
  __shared__ uint32_t s_start[kColSubs + 1];
  __shared__ unsigned long long s_red[3][kColThreads / 32];
  const uint32_t t = blockIdx.x / kColPerTile;
  const uint32_t s = find_seg(p, t);
  const ColSeg g = col_seg(p, s, c.max_parts);
  const uint32_t b = blockIdx.x - g.ft * kColPerTile;
  if (b >= g.parts || g.n == 0) return;
  const uint64_t base = p.base[s];
  const uint32_t* kd = col_ids + base;
  const V* vd = (kWide ? (const V*)vals64 : (const V*)vals32) + base;
  uint64_t m = g.n;
  uint32_t at = 0;
  if (g.parts > 1) {
    at = c.start[blockIdx.x];
    m = c.cnt[blockIdx.x];
    kd = pdst + base + at;
    vd = reinterpret_cast<const V*>(pval) + base + at;
  }
  const bool heavy = b == 0 && g.n >= kColHeavyLinks;  // this CTA adds the heavy destinations
  if (m == 0 && !heavy) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto add = [&](uint32_t* lo, uint32_t* hi, V x) {
    if constexpr (kWide) add64_shared(lo, hi, x);
    else atomicAdd(lo, x);
  };
  auto sum_of = [&](uint32_t lo, const uint32_t* hi) -> uint64_t { return kWide ? (uint64_t)*hi << 32 | lo : lo; };
  unsigned long long uniq = 0, mfan = 0, mpk = 0;
  uint32_t subs = 0;  // parts of a cut partition, 0: whole
  for (uint32_t sub = 0; sub < (subs ? subs : 1u); ++sub) {
    unsigned long long found = 0;
    uint32_t slots = 256;
    while (slots < m + m / 2 && slots < kColSlots) slots <<= 1;
    const bool watch = m > kColFill;  // it may hold too many destinations
    // (a first round of links with hardly a destination twice is one of far more
    // of them: cut at once)
    const uint32_t early = !subs && g.parts > 1 && c.sdst && m > kColFill / 5 * 6 ? kColEarly : kColFill;
    for (uint32_t R = 1, cls = 0; cls < R;) {
      for (uint32_t i = threadIdx.x; i < slots; i += kColThreads) {
        t_key[i] = kColNone;
        t_cnt[i] = 0;
        t_lo[i] = 0;
        if (kWide) t_hi[i] = 0;
      }
      if (threadIdx.x == 0) s_fill = s_over = s_spec_cnt = s_spec_lo = s_spec_hi = 0;
      __syncthreads();
      constexpr int kU = 4;  // links per thread in flight
      for (uint64_t u0 = 0; u0 < m; u0 += (uint64_t)kU * kColThreads) {
        if (__any_sync(0xffffffffu, *(volatile uint32_t*)&s_over)) break;  // (the warp as one)
        uint32_t d[kU], claimed = 0;
        V v[kU];
#pragma unroll
        for (int k = 0; k < kU; ++k) {
          const uint64_t u = u0 + (uint64_t)k * kColThreads + threadIdx.x;
          d[k] = u < m ? kd[u] : 0u;
          v[k] = u < m ? vd[u] : V(0);
        }
#pragma unroll
        for (int k = 0; k < kU; ++k) {
          if (u0 + (uint64_t)k * kColThreads + threadIdx.x < m) {
            if (d[k] == kColNone) {
              if (cls == 0) {
                atomicAdd(&s_spec_cnt, 1u);
                add(&s_spec_lo, &s_spec_hi, v[k]);
              }
            } else {
              const uint32_t h = fmix32(d[k]);
              if (R == 1 || (fmix32(h ^ 0x9E3779B9u) & (R - 1)) == cls) {
                uint32_t i = h & (slots - 1);
                for (uint32_t probe = 0; probe < slots; ++probe) {
                  uint32_t cur = *(volatile uint32_t*)&t_key[i];
                  if (cur == kColNone) {
                    cur = atomicCAS(&t_key[i], kColNone, d[k]);
                    if (cur == kColNone) {
                      cur = d[k];
                      ++claimed;
                    }
                  }
                  if (cur == d[k]) {
                    atomicAdd(&t_cnt[i], 1u);
                    add(&t_lo[i], &t_hi[i], v[k]);
                    break;
                  }
                  i = (i + 1) & (slots - 1);
                }
              }
            }
          }
          // Given up before the table is nearly full: every second link the
          // warps add up their new destinations, so that searches stay short (an
          // addition for every new destination made the count of 6 million
          // different ones 169 instead of 143 us; looking once a round of links,
          // overfull partitions took 18 times as long; after every link, ones of
          // few destinations 5% longer).
          if (watch && k % 2 == 1 && __any_sync(0xffffffffu, claimed)) {
            const uint32_t claims = __reduce_add_sync(0xffffffffu, claimed);
            claimed = 0;
            uint32_t fill = 0;
            if (lane == 0) fill = atomicAdd(&s_fill, claims) + claims;
            if (__shfl_sync(0xffffffffu, fill, 0) > (u0 ? kColFill : early)) {
              s_over = 1;
              break;
            }
          }
        }
      }
      __syncthreads();
      if (s_over) {
        __syncthreads();
        if (!subs && g.parts > 1 && c.sdst) break;  // cut below
        R <<= 1;  // twice the classes, from the start
        cls = 0;
        found = 0;
        continue;
      }
      for (uint32_t i = threadIdx.x; i < slots; i += kColThreads) {
        if (t_key[i] != kColNone) {
          ++found;
          mfan = umax64(mfan, t_cnt[i]);
          mpk = umax64(mpk, sum_of(t_lo[i], &t_hi[i]));
        }
      }
      if (threadIdx.x == 0 && s_spec_cnt) {
        ++found;
        mfan = umax64(mfan, s_spec_cnt);
        mpk = umax64(mpk, sum_of(s_spec_lo, &s_spec_hi));
      }
      ++cls;
      __syncthreads();  // the table is cleared for the next class
    }
    uniq += found;
    if (!subs && s_over) {
      subs = (uint32_t)umin64(kColSubs, (m + kColPart - 1) / kColPart);
      uint32_t* sd = c.sdst + base + at;
      V* sv = reinterpret_cast<V*>(c.sval) + base + at;
      col_cut<V>(kd, vd, (uint32_t)m, subs, sd, sv, s_start, t_key);
      kd = sd;
      vd = sv;
      m = s_start[1];
      sub = ~0u;  // from part 0 on
    } else if (sub + 1 < subs) {
      kd += s_start[sub + 1] - s_start[sub];
      vd += s_start[sub + 1] - s_start[sub];
      m = s_start[sub + 2] - s_start[sub + 1];
    }
  }
  if (heavy && threadIdx.x < kColHeavySlots) {
    const size_t at = (size_t)g.ft * kColHeavyPerTile + threadIdx.x;
    const unsigned long long f = c.hsum[2 * at];
    if (f) {
      ++uniq;
      mfan = umax64(mfan, f);
      mpk = umax64(mpk, c.hsum[2 * at + 1]);
    }
  }
  uniq = warp_sum(uniq);
  mfan = warp_max(mfan);
  mpk = warp_max(mpk);
  if (lane == 0) {
    s_red[0][warp] = uniq;
    s_red[1][warp] = mfan;
    s_red[2][warp] = mpk;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kColThreads / 32; ++w) {
      uniq += s_red[0][w];
      mfan = umax64(mfan, s_red[1][w]);
      mpk = umax64(mpk, s_red[2][w]);
    }
    atomicAdd((unsigned long long*)&q[s].unique_destinations, uniq);
    atomicMax((unsigned long long*)&q[s].max_destination_fanin, mfan);
    atomicMax((unsigned long long*)&q[s].max_destination_packets, mpk);
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

template <bool kWide, int kT, int kP>
cudaError_t scatter(const SegPlan& p, const ColParts& c, const uint32_t* col_ids, const uint32_t* vals32,
                    const uint64_t* vals64, uint32_t* odst, void* oval, cudaStream_t st) {
  constexpr size_t kItems = (size_t)kT * kP * (kWide ? 12 : 8);
  static unsigned long long done = 0;
  const cudaError_t e = set_smem_once(k_col_scatter<kWide, kT, kP>, kItems + (size_t)kColMaxParts * 8, &done);
  if (e != cudaSuccess) return e;
  k_col_scatter<kWide, kT, kP><<<p.ntiles * (kTile / (kT * kP)), kT, kItems + (size_t)c.max_parts * 8, st>>>(
      p, c, col_ids, vals32, vals64, odst, oval);
  return cudaGetLastError();
}

template <bool kWide>
cudaError_t run_scatter(const SegPlan& p, const ColParts& c, const uint32_t* col_ids, const uint32_t* vals32,
                        const uint64_t* vals64, uint32_t* odst, void* oval, cudaStream_t st) {
  if (c.max_parts <= 1) return cudaSuccess;
  // (c.max_parts: of the longest segment, or, in batches planned on the device,
  // of one that holds the whole batch, whose shape every window then takes: 2^27
  // packets in windows of 2^17 0.62 against 0.58 ms.)
  // With many partitions a CTA pays an atomic for nearly every one of them, so
  // it takes a whole tile (3 million links, 1108 partitions, 64-bit counts: 48
  // us, 85 by 2048 links); else 4096 links per CTA are faster (2^28 packets in
  // windows of 2^17: 1.30 against 1.63 ms), and 2048 fill the SMs sooner for
  // small plans.
  if (c.max_parts > 512) return scatter<kWide, 512, 16>(p, c, col_ids, vals32, vals64, odst, oval, st);
  return p.ntiles <= 608 ? scatter<kWide, 256, 8>(p, c, col_ids, vals32, vals64, odst, oval, st)
                         : scatter<kWide, 512, 8>(p, c, col_ids, vals32, vals64, odst, oval, st);
}

template <bool kWide>
cudaError_t run_count(const SegPlan& p, const ColParts& c, const uint32_t* col_ids, const uint32_t* vals32,
                      const uint64_t* vals64, const uint32_t* odst, const void* oval, ans_quantities* q,
                      cudaStream_t st) {
  constexpr size_t kSmem = (size_t)kColSlots * (kWide ? 16 : 12);
  static unsigned long long done = 0;
  const cudaError_t e = set_smem_once(k_col_count<kWide>, kSmem, &done);
  if (e != cudaSuccess) return e;
  k_col_count<kWide><<<p.ntiles * kColPerTile, kColThreads, kSmem, st>>>(p, c, col_ids, vals32, vals64, odst, oval, q);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_col_heavy(const SegPlan& p, const ColParts& c, const uint32_t* col_ids, const uint64_t* hdr,
                             cudaStream_t st) {
  if (p.ntiles == 0 || p.nseg == 0) return cudaSuccess;
  k_col_heavy<<<p.nseg, kColHeavyThreads, 0, st>>>(p, c, col_ids, hdr);
  return cudaGetLastError();
}

cudaError_t launch_col_scatter(const SegPlan& p, const ColParts& c, const uint32_t* col_ids, const uint32_t* vals32,
                               const uint64_t* vals64, uint32_t* odst, void* oval, cudaStream_t st) {
  if (p.ntiles == 0) return cudaSuccess;
  return vals32 ? run_scatter<false>(p, c, col_ids, vals32, nullptr, odst, oval, st)
                : run_scatter<true>(p, c, col_ids, nullptr, vals64, odst, oval, st);
}

cudaError_t launch_col_count(const SegPlan& p, const ColParts& c, const uint32_t* col_ids, const uint32_t* vals32,
                             const uint64_t* vals64, const uint32_t* odst, const void* oval, ans_quantities* q,
                             cudaStream_t st) {
  if (p.ntiles == 0) return cudaSuccess;
  return vals32 ? run_count<false>(p, c, col_ids, vals32, nullptr, odst, oval, q, st)
                : run_count<true>(p, c, col_ids, nullptr, vals64, odst, oval, q, st);
}

}  // namespace ans
