// f2: two-tier local chaining inside the potential SD regions (Section 3.3).
//
// For every region (query [qa, qb), target [ta, tb), strand o from
// sedef_extend) the query is X = G[qa, qb) and the target Y = G[ta, tb),
// reverse-complemented when o = 1, both read from the 2-bit packed genome
// (case does not matter; a base flagged in the N bit-vector matches
// nothing).
//   Seeds: maximal exact matches (x, y, L) of at least k2 = 11 bases.
//   Initial chains: seed b may follow a when it starts later on both axes
//   and the gaps from a's end to b's start are at most g1 = ceil(1000 *
//   delta_G) on both axes (negative where an indel makes them overlap); the
//   link adds the bases new on both axes, min(L_b, end_b - end_a on x,
//   end_b - end_a on y), and must add at least one; f(b) = max(L_b, best
//   f(a) + gain), the later seed on ties.  Chains are taken greedily by
//   decreasing f (earlier seed on ties), each back along its predecessors
//   to the first seed a chain already holds.
//   Final chains: initial chains (sorted by start) chained with gaps of at
//   most g2 = 10,000 on both axes and an affine penalty 25 + g / 50 for the
//   larger gap g; F(d) = S(d) + max(0, best F(c) - pen), a link only when it
//   raises the score, the later chain on ties; the same greedy extraction.
//   A final chain spanning at least 1,000 bases on both axes is an SD.
//
// Regions run in batches (at most 2^26 target k-mers).  Per batch:
//   k_c2_keys     one thread per target position: (region, 11-mer, y) keys
//   radix sort    by (region, 11-mer); y stays ascending
//   k_c2_mems     one thread per query position: the matching target range
//                 by binary search, left-maximal matches extended to the
//                 right (count pass, then write pass at scanned offsets), so
//                 a region's seeds come out sorted by (x, y)
//   k_c2_dp       one CTA per region: the chaining DP, 32 items at a time,
//                 predecessors only as far back as an item can still reach
//                 (its start at least the current start minus the gap bound
//                 minus the region's longest item)
//   k_c2_take     one CTA per region: the greedy extraction, as a minimum
//                 over every item's descendants
// (once for the seeds and once for the initial chains), and k_c2_emit
// compacts the final chains.
#include <cstring>

#include "common.cuh"

namespace sedef {
namespace {

constexpr int kK2 = 11;                  // seed length (Section 3.3)
constexpr int64_t kG2 = 10000;           // largest gap between initial chains (Section 3.3)
constexpr int64_t kGapOpen = 25;         // affine gap penalty: open
constexpr int64_t kGapDiv = 50;          // one more per kGapDiv gap bases
constexpr int64_t kMinSD = 1000;         // SD length (Section 3)
constexpr int64_t kMaxRegion = int64_t(1) << 20;

// A region of the batch: query and target starts, lengths, strand.
struct Reg {
  int64_t qa, ta, tb;
  int32_t nx, ny, o, pad;
};

__device__ __forceinline__ uint32_t base2(const uint32_t* packed, int64_t p) {
  return (packed[p >> 4] >> (2 * (p & 15))) & 3u;
}
__device__ __forceinline__ bool isn(const uint32_t* nbits, int64_t p) {
  return (nbits[p >> 5] >> (p & 31)) & 1u;
}

// Base of X (q) or Y (t) at offset u: 0-3, or 4 for a base that matches
// nothing.
__device__ __forceinline__ uint32_t xbase(const uint32_t* packed, const uint32_t* nbits,
                                          const Reg& R, int64_t u) {
  const int64_t p = R.qa + u;
  return isn(nbits, p) ? 4u : base2(packed, p);
}
__device__ __forceinline__ uint32_t ybase(const uint32_t* packed, const uint32_t* nbits,
                                          const Reg& R, int64_t u) {
  if (R.o == 0) {
    const int64_t p = R.ta + u;
    return isn(nbits, p) ? 4u : base2(packed, p);
  }
  const int64_t p = R.tb - 1 - u;
  return isn(nbits, p) ? 4u : (3u - base2(packed, p));
}

__device__ __forceinline__ int region_of(const int64_t* base, int nreg, int64_t g) {
  int lo = 0, hi = nreg;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (base[mid] <= g) lo = mid; else hi = mid;
  }
  return lo;
}

// Keys (region << 42 | code << 20 | y) of every target 11-mer of A, C, G, T.
__global__ void k_c2_keys(const uint32_t* packed, const uint32_t* nbits, const Reg* regs,
                          const int64_t* ybase_of, int nreg, int64_t total, uint64_t* keys) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= total) return;
  const int r = region_of(ybase_of, nreg, g);
  const Reg R = regs[r];
  const int64_t y = g - ybase_of[r];
  uint64_t key = ~0ull;
  if (y + kK2 <= R.ny) {
    uint64_t code = 0;
    bool ok = true;
    for (int u = 0; u < kK2; ++u) {
      const uint32_t b = ybase(packed, nbits, R, y + u);
      ok = ok && b < 4u;
      code = (code << 2) | (b & 3u);
    }
    if (ok) key = ((uint64_t)r << 42) | (code << 20) | (uint64_t)y;
  }
  keys[g] = key;
}

// Maximal exact matches per query position: counts (write = false) or
// seeds written at out[off[g] ..] (write = true) as x << 40 | y << 20 | L.
template <bool kWrite>
__global__ void k_c2_mems(const uint32_t* packed, const uint32_t* nbits, const Reg* regs,
                          const int64_t* xbase_of, int nreg, int64_t total, const uint64_t* skeys,
                          int64_t nkeys, uint32_t* count, const uint32_t* off, uint64_t* out) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= total) return;
  const int r = region_of(xbase_of, nreg, g);
  const Reg R = regs[r];
  const int64_t x = g - xbase_of[r];
  uint32_t n = 0;
  if (x + kK2 <= R.nx) {
    uint64_t code = 0;
    bool ok = true;
    for (int u = 0; u < kK2; ++u) {
      const uint32_t b = xbase(packed, nbits, R, x + u);
      ok = ok && b < 4u;
      code = (code << 2) | (b & 3u);
    }
    if (ok) {
      const uint64_t want = ((uint64_t)r << 42) | (code << 20);
      int64_t lo = 0, hi = nkeys;  // first key >= want
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (skeys[mid] < want) lo = mid + 1; else hi = mid;
      }
      const uint32_t xprev = x > 0 ? xbase(packed, nbits, R, x - 1) : 4u;
      uint64_t at = kWrite ? off[g] : 0;
      for (int64_t k = lo; k < nkeys && (skeys[k] >> 20) == (want >> 20); ++k) {
        const int64_t y = (int64_t)(skeys[k] & 0xFFFFFull);
        if (x > 0 && y > 0 && xprev < 4u && xprev == ybase(packed, nbits, R, y - 1)) continue;
        int64_t L = kK2;
        while (x + L < R.nx && y + L < R.ny) {
          const uint32_t b = xbase(packed, nbits, R, x + L);
          if (b >= 4u || b != ybase(packed, nbits, R, y + L)) break;
          ++L;
        }
        if (kWrite) out[at++] = ((uint64_t)x << 40) | ((uint64_t)y << 20) | (uint64_t)L;
        ++n;
      }
    }
  }
  if (!kWrite) count[g] = n;
}

// An item of a chaining tier: its box and its own score.
struct Item {
  int32_t x0, x1, y0, y1, score, seeds;
};

__device__ __forceinline__ Item seed_item(uint64_t s) {
  Item it;
  it.x0 = (int32_t)(s >> 40);
  it.y0 = (int32_t)((s >> 20) & 0xFFFFF);
  const int32_t L = (int32_t)(s & 0xFFFFF);
  it.x1 = it.x0 + L;
  it.y1 = it.y0 + L;
  it.score = L;
  it.seeds = 1;
  return it;
}

// Score a link c -> d adds, or INT_MIN when d cannot follow c.
__device__ __forceinline__ int32_t link_gain(const Item& c, const Item& d, int tier, int32_t g1) {
  if (tier == 1) {
    if (c.x0 >= d.x0 || c.y0 >= d.y0) return INT32_MIN;
    if (d.x0 - c.x1 > g1 || d.y0 - c.y1 > g1) return INT32_MIN;
    const int32_t g = min(d.score, min(d.x1 - c.x1, d.y1 - c.y1));
    return g > 0 ? g : INT32_MIN;
  }
  const int32_t gq = d.x0 - c.x1, gt = d.y0 - c.y1;
  if (gq < 0 || gt < 0 || gq > (int32_t)kG2 || gt > (int32_t)kG2) return INT32_MIN;
  return d.score - (int32_t)(kGapOpen + max(gq, gt) / kGapDiv);
}

constexpr int kC2Threads = 256;
constexpr int kC2Warps = kC2Threads / 32;

// The chaining DP of one tier: one CTA per region, items of region r at
// [ib[r], ib[r] + n[r]) in start order.  best[] and pred[] (region-local
// index, -1 for none) per item.
//
// 32 items at a time, one per lane of every warp: the warps share out the
// earlier items (each read once for all 32), one warp then settles the 32
// among themselves.  What bounds it is the chain of dependent steps: one
// item at a time by one warp paid a round trip to L2 per 32 predecessors of
// every item (a region of 100 kbp has thousands of initial chains, all of
// them within reach of tier 2): 34.3 -> 2.6 ms for the regions of a 4 Mbp
// genome.
__global__ void __launch_bounds__(kC2Threads) k_c2_dp(const Item* items, const int64_t* ib,
                                                      const uint32_t* n_of, int tier, int32_t g1,
                                                      int32_t* best, int32_t* pred) {
  __shared__ int32_t s_v[kC2Warps][32], s_a[kC2Warps][32];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const int r = blockIdx.x;
  const Item* it = items + ib[r];
  int32_t* f_of = best + ib[r];
  int32_t* p_of = pred + ib[r];
  const int32_t n = (int32_t)n_of[r];
  // the longest item bounds how far back a predecessor can start
  int32_t span = 0;
  for (int32_t u = threadIdx.x; u < n; u += kC2Threads) span = max(span, it[u].x1 - it[u].x0);
  span = (int32_t)__reduce_max_sync(0xffffffffu, (uint32_t)span);
  if (lane == 0) s_v[warp][0] = span;
  __syncthreads();
  for (int w = 0; w < kC2Warps; ++w) span = max(span, s_v[w][0]);
  const int32_t reach = (tier == 1 ? g1 : (int32_t)kG2) + span;
  int32_t from = 0;  // items before it are out of every later item's reach
  for (int32_t t0 = 0; t0 < n; t0 += 32) {
    const bool ok = t0 + lane < n;
    const Item d = it[ok ? t0 + lane : n - 1];
    const int32_t x_lo = __shfl_sync(0xffffffffu, d.x0, 0) - reach;
    while (from < t0) {
      const int32_t u = from + lane;
      const unsigned in = __ballot_sync(0xffffffffu, u >= t0 || it[u].x0 >= x_lo);
      if (in) {
        from += __ffs(in) - 1;
        break;
      }
      from += 32;
    }
    int32_t bv = INT32_MIN, ba = -1;  // best value through a predecessor, its index
#pragma unroll 4
    for (int32_t u = from + warp; u < t0; u += kC2Warps) {
      const int32_t g = link_gain(it[u], d, tier, g1);
      if (g != INT32_MIN) {
        const int32_t v = f_of[u] + g;
        if (v >= bv) {  // the later of equals
          bv = v;
          ba = u;
        }
      }
    }
    __syncthreads();  // s_v was last read for the items before
    s_v[warp][lane] = bv;
    s_a[warp][lane] = ba;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int w = 1; w < kC2Warps; ++w) {
        const int32_t v = s_v[w][lane], u = s_a[w][lane];
        if (v > bv || (v == bv && u > ba)) {
          bv = v;
          ba = u;
        }
      }
      const int last = min(32, n - t0);
      for (int t = 0; t < last; ++t) {
        // tier 1: f = max(L, best link); tier 2: F = S + max(0, best link - S)
        const int32_t f = __shfl_sync(0xffffffffu, max(bv, d.score), t);
        Item c;
        c.x0 = __shfl_sync(0xffffffffu, d.x0, t);
        c.x1 = __shfl_sync(0xffffffffu, d.x1, t);
        c.y0 = __shfl_sync(0xffffffffu, d.y0, t);
        c.y1 = __shfl_sync(0xffffffffu, d.y1, t);
        if (lane > t) {
          const int32_t g = link_gain(c, d, tier, g1);
          if (g != INT32_MIN && f + g >= bv) {
            bv = f + g;
            ba = t0 + t;
          }
        }
      }
      if (ok) {
        const bool linked = bv > d.score;
        f_of[t0 + lane] = linked ? bv : d.score;
        p_of[t0 + lane] = linked ? ba : -1;
      }
    }
    __syncthreads();
  }
}

// What the greedy extraction keeps per item: the item's best descendant and
// two buffers of ancestors, and per chain (at its last item) its furthest
// ends, seeds and number of items.
struct Take {
  unsigned long long* owner;
  int32_t *jump, *jump2;
  int32_t *x1, *y1, *seeds, *parts;
};

// Greedy extraction (one CTA per region): chains in order of decreasing best
// score (the earlier item on ties), each back along pred to the first item
// already taken.  An item goes to the first chain in that order whose walk
// reaches it, which is the least of (-score, index) over the item and all
// items whose walks pass it: a minimum over descendants, found by doubling
// the walks' stride (the walks themselves, one thread per region, took 27 ms
// where this takes 0.26).  A chain's score is its first item's plus every
// link's gain, the difference of the DP's values at its two ends; its box
// starts at its first item and ends at the furthest item end (tier 1) or at
// its last item's end (tier 2).  Writes the chains in the order of their
// first items, which is start order, to out[ib[r] ..] with their item counts
// in parts_out, and their number.
__global__ void __launch_bounds__(kC2Threads) k_c2_take(const Item* items, const int32_t* best,
                                                        const int32_t* pred, const int64_t* ib,
                                                        const uint32_t* n_of, int tier, Take T,
                                                        Item* out, int32_t* parts_out,
                                                        uint32_t* nout) {
  __shared__ int s_tmp[33];
  const int r = blockIdx.x;
  const int64_t b0 = ib[r];
  const int32_t n = (int32_t)n_of[r];
  const Item* it = items + b0;
  const int32_t* bst = best + b0;
  const int32_t* prd = pred + b0;
  unsigned long long* own = T.owner + b0;
  int32_t *x1 = T.x1 + b0, *y1 = T.y1 + b0, *seeds = T.seeds + b0, *parts = T.parts + b0;
  bool more = false;
  for (int32_t u = threadIdx.x; u < n; u += kC2Threads) {
    own[u] = ((unsigned long long)(0x7FFFFFFF - bst[u]) << 32) | (uint32_t)u;
    T.jump[b0 + u] = prd[u];
    more |= prd[u] >= 0;
    x1[u] = y1[u] = INT32_MIN;
    seeds[u] = parts[u] = 0;
  }
  // after round k an item knows its descendants up to 2^(k+1) - 1 links away
  int32_t *src = T.jump + b0, *dst = T.jump2 + b0;
  while (__syncthreads_or(more)) {
    more = false;
    for (int32_t u = threadIdx.x; u < n; u += kC2Threads) {
      const int32_t j = src[u];
      int32_t to = -1;
      if (j >= 0) {
        atomicMin(own + j, *(volatile unsigned long long*)(own + u));
        to = src[j];
      }
      dst[u] = to;
      more |= to >= 0;
    }
    int32_t* t = src;
    src = dst;
    dst = t;
  }
  for (int32_t u = threadIdx.x; u < n; u += kC2Threads) {
    const uint32_t h = (uint32_t)__ldcg(own + u);
    const Item c = it[u];
    if (tier == 1) {
      atomicMax(x1 + h, c.x1);
      atomicMax(y1 + h, c.y1);
    }
    atomicAdd(seeds + h, c.seeds);
    atomicAdd(parts + h, 1);
  }
  __syncthreads();
  int m = 0;
  for (int32_t base = 0; base < n; base += kC2Threads) {
    const int32_t u = base + threadIdx.x;
    bool first = false;
    uint32_t h = 0;
    if (u < n) {
      const unsigned long long o = __ldcg(own + u);
      h = (uint32_t)o;
      first = prd[u] < 0 || __ldcg(own + prd[u]) != o;
    }
    int tot;
    const int at = m + block_exclusive_sum(first ? 1 : 0, s_tmp, &tot);
    if (first) {
      Item c = it[u];
      c.score += bst[h] - bst[u];
      c.seeds = __ldcg(seeds + h);
      c.x1 = tier == 1 ? __ldcg(x1 + h) : it[h].x1;
      c.y1 = tier == 1 ? __ldcg(y1 + h) : it[h].y1;
      out[b0 + at] = c;
      parts_out[b0 + at] = __ldcg(parts + h);
    }
    m += tot;
  }
  if (threadIdx.x == 0) nout[r] = (uint32_t)m;
}

// Seeds (x << 40 | y << 20 | L) as chaining items.
__global__ void k_c2_items(const uint64_t* seeds, int64_t n, Item* items) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g < n) items[g] = seed_item(seeds[g]);
}

// Sum of n counts in 64 bits.
__global__ void k_c2_sum(const uint32_t* v, int64_t n, unsigned long long* total) {
  unsigned long long s = 0;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x)
    s += v[x];
  s = warp_sum(s);
  if (lane_id() == 0 && s) atomicAdd(total, s);
}

// Seed ranges of the regions from the seeds' offsets: ib[0..nreg], n[0..nreg).
__global__ void k_c2_ranges(const uint32_t* off, const int64_t* xbase_of, int nreg, int64_t* ib,
                            uint32_t* n) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r > nreg) return;
  ib[r] = off[xbase_of[r]];
  if (r < nreg) n[r] = off[xbase_of[r + 1]] - off[xbase_of[r]];
}

// Final chains of at least kMinSD bases on both axes, per region, sorted by
// (q0, q1, t0, t1, score) in genome coordinates, written at out[ob[r] ..]
// (one warp per region; few chains are that long, and they come by q0).
__global__ void k_c2_emit(const Item* fin, const int32_t* parts, const int64_t* ib,
                          const uint32_t* n_of, const Reg* regs, const int64_t* reg_index,
                          int nreg, const int64_t* ob, sedef_sd_t* out, uint32_t* nkept,
                          int count_only) {
  const int r = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (r >= nreg) return;
  const int lane = lane_id();
  const Reg R = regs[r];
  const int64_t b0 = ib[r];
  const uint32_t n = n_of[r];
  sedef_sd_t* row = out + (count_only ? 0 : ob[r]);
  uint32_t m = 0;
  for (uint32_t base = 0; base < n; base += 32) {
    const uint32_t u = base + lane;
    Item c;
    bool keep = false;
    if (u < n) {
      c = fin[b0 + u];
      keep = c.x1 - c.x0 >= kMinSD && c.y1 - c.y0 >= kMinSD;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (keep && !count_only) {
      sedef_sd_t s;
      s.region = (uint32_t)reg_index[r];
      s.o = (uint32_t)R.o;
      s.q0 = (uint32_t)(R.qa + c.x0);
      s.q1 = (uint32_t)(R.qa + c.x1);
      s.t0 = (uint32_t)(R.o ? R.tb - c.y1 : R.ta + c.y0);
      s.t1 = (uint32_t)(R.o ? R.tb - c.y0 : R.ta + c.y1);
      s.score = (uint32_t)c.score;
      s.seeds = (uint32_t)c.seeds;
      s.parts = (uint32_t)parts[b0 + u];
      s.reserved = 0;
      row[m + __popc(bal & lanemask_lt())] = s;
    }
    m += __popc(bal);
  }
  if (lane == 0) nkept[r] = m;
  __syncwarp();
  if (count_only || lane != 0) return;
  auto less = [](const sedef_sd_t& a, const sedef_sd_t& b) {
    if (a.q0 != b.q0) return a.q0 < b.q0;
    if (a.q1 != b.q1) return a.q1 < b.q1;
    if (a.t0 != b.t0) return a.t0 < b.t0;
    if (a.t1 != b.t1) return a.t1 < b.t1;
    if (a.score != b.score) return a.score < b.score;
    if (a.seeds != b.seeds) return a.seeds < b.seeds;
    return a.parts < b.parts;
  };
  for (uint32_t u = 1; u < m; ++u) {
    const sedef_sd_t s = row[u];
    uint32_t at = u;
    while (at > 0 && less(s, row[at - 1])) {
      row[at] = row[at - 1];
      --at;
    }
    if (at != u) row[at] = s;
  }
}

}  // namespace

int run_chain2(sedef_ctx* ctx, const uint32_t* packed, const uint32_t* nbits, int64_t nbases,
               const sedef_region_t* d_regions, int64_t nregions, const Derived& D,
               sedef_sd_t* out, int64_t cap, int64_t* nout) {
  cudaStream_t st = ctx_stream(ctx);
  *nout = 0;
  if (nregions == 0) return SEDEF_OK;
  std::vector<sedef_region_t> hr((size_t)nregions);
  SEDEF_CUDA(cudaMemcpyAsync(hr.data(), d_regions, (size_t)nregions * sizeof(sedef_region_t),
                             cudaMemcpyDeviceToHost, st));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  for (auto& R : hr) {
    if (R.qb < R.qa || R.tb < R.ta || (int64_t)R.qb > nbases || (int64_t)R.tb > nbases)
      return fail(SEDEF_ERR_INVALID, "sedef_chain2: region outside the sequence");
    if ((int64_t)(R.qb - R.qa) >= kMaxRegion || (int64_t)(R.tb - R.ta) >= kMaxRegion)
      return fail(SEDEF_ERR_UNSUPPORTED, "sedef_chain2: a region of 2^20 bases or more");
  }
  const int32_t g1 = (int32_t)std::ceil(1000.0 * D.delta_g - 1e-9);
  std::vector<sedef_sd_t> all;
  int64_t r0 = 0;
  const int64_t kBatchBases = int64_t(1) << 26;
  while (r0 < nregions) {
    // a batch: regions while their target bases fit the key budget
    int64_t r1 = r0, ysum = 0, xsum = 0;
    while (r1 < nregions && (r1 == r0 || ysum + (hr[r1].tb - hr[r1].ta) <= kBatchBases) &&
           r1 - r0 < (int64_t(1) << 21)) {
      ysum += hr[r1].tb - hr[r1].ta;
      xsum += hr[r1].qb - hr[r1].qa;
      ++r1;
    }
    const int nb = (int)(r1 - r0);
    const std::vector<char> used_before = ctx_pool_snapshot(ctx);
    // uploads: regions, y bases, x bases, region indices
    std::vector<Reg> regs(nb);
    std::vector<int64_t> yb(nb + 1, 0), xb(nb + 1, 0), rid(nb);
    for (int k = 0; k < nb; ++k) {
      const sedef_region_t& R = hr[r0 + k];
      regs[k] = {R.qa, R.ta, R.tb, (int32_t)(R.qb - R.qa), (int32_t)(R.tb - R.ta), (int32_t)R.o, 0};
      yb[k + 1] = yb[k] + regs[k].ny;
      xb[k + 1] = xb[k] + regs[k].nx;
      rid[k] = r0 + k;
    }
    const size_t up = sizeof(Reg) * nb + 8 * (size_t)(nb + 1) * 2 + 8 * (size_t)nb;
    char* d_up = (char*)ctx_alloc(ctx, up);
    if (!d_up) return SEDEF_ERR_OOM;
    Reg* d_regs = (Reg*)d_up;
    int64_t* d_yb = (int64_t*)(d_up + sizeof(Reg) * nb);
    int64_t* d_xb = d_yb + (nb + 1);
    int64_t* d_rid = d_xb + (nb + 1);
    SEDEF_CUDA(cudaMemcpyAsync(d_regs, regs.data(), sizeof(Reg) * nb, cudaMemcpyHostToDevice, st));
    SEDEF_CUDA(cudaMemcpyAsync(d_yb, yb.data(), 8 * (size_t)(nb + 1), cudaMemcpyHostToDevice, st));
    SEDEF_CUDA(cudaMemcpyAsync(d_xb, xb.data(), 8 * (size_t)(nb + 1), cudaMemcpyHostToDevice, st));
    SEDEF_CUDA(cudaMemcpyAsync(d_rid, rid.data(), 8 * (size_t)nb, cudaMemcpyHostToDevice, st));
    // target k-mer keys, sorted (a key that holds no k-mer sorts last)
    const int64_t ny = ysum > 0 ? ysum : 1;
    uint64_t* keys = (uint64_t*)ctx_alloc(ctx, (size_t)ny * 8);
    uint64_t* skeys = (uint64_t*)ctx_alloc(ctx, (size_t)ny * 8);
    if (!keys || !skeys) return SEDEF_ERR_OOM;
    int rbits = 1;
    while ((int64_t(1) << rbits) <= nb) ++rbits;
    if (ysum > 0) {
      SEDEF_KERNEL(ctx, "k_c2_keys", k_c2_keys<<<(int)((ysum + 255) / 256), 256, 0, st>>>(
                                         packed, nbits, d_regs, d_yb, nb, ysum, keys));
      SEDEF_TRY(radix_sort_u64(ctx, keys, nullptr, skeys, nullptr, ysum, 20, 42 + rbits));
    }
    // seeds: count, scan, write
    const int64_t nx = xsum > 0 ? xsum : 1;
    uint32_t* cnt = (uint32_t*)ctx_alloc(ctx, (size_t)(nx + 1) * 4);
    uint32_t* off = (uint32_t*)ctx_alloc(ctx, (size_t)(nx + 1) * 4);
    char* d_meta = (char*)ctx_alloc(ctx, 8 + (size_t)(nb + 1) * 8 * 2 + (size_t)nb * 4 * 4);
    if (!cnt || !off || !d_meta) return SEDEF_ERR_OOM;
    unsigned long long* d_total = (unsigned long long*)d_meta;
    int64_t* d_ib = (int64_t*)(d_meta + 8);
    int64_t* d_kb = d_ib + (nb + 1);
    uint32_t* d_n1 = (uint32_t*)(d_kb + (nb + 1));
    uint32_t* d_n2 = d_n1 + nb;
    uint32_t* d_n3 = d_n2 + nb;
    uint32_t* d_keep = d_n3 + nb;
    int64_t na = 0;
    if (xsum > 0 && ysum > 0) {
      SEDEF_KERNEL(ctx, "k_c2_mems", (k_c2_mems<false><<<(int)((xsum + 255) / 256), 256, 0, st>>>(
                                         packed, nbits, d_regs, d_xb, nb, xsum, skeys, ysum, cnt,
                                         nullptr, nullptr)));
      SEDEF_CUDA(cudaMemsetAsync(d_total, 0, 8, st));
      int64_t sg = (xsum + 255) / 256;
      if (sg > (int64_t)ctx_sm_count(ctx) * 8) sg = (int64_t)ctx_sm_count(ctx) * 8;
      SEDEF_KERNEL(ctx, "k_c2_sum", k_c2_sum<<<(int)sg, 256, 0, st>>>(cnt, xsum, d_total));
      SEDEF_TRY(scan_exclusive_u32(ctx, cnt, off, xsum, off + xsum));
      SEDEF_KERNEL(ctx, "k_c2_ranges",
                   k_c2_ranges<<<(nb + 256) / 256, 256, 0, st>>>(off, d_xb, nb, d_ib, d_n1));
      unsigned long long total = 0;
      std::vector<uint32_t> ncount(nb, 0);
      SEDEF_CUDA(cudaMemcpyAsync(&total, d_total, 8, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaMemcpyAsync(ncount.data(), d_n1, (size_t)nb * 4, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaStreamSynchronize(st));
      // the offsets are 32-bit; a batch with more seeds than that would need
      // more than 300 GB of items
      if (total >= (1ull << 32))
        return fail(SEDEF_ERR_OOM, "sedef_chain2: more than 2^32 seeds in a batch of regions");
      na = (int64_t)total;
      for (int k = 0; k < nb; ++k)
        if ((int64_t)ncount[k] >= (int64_t(1) << 22))
          return fail(SEDEF_ERR_UNSUPPORTED, "sedef_chain2: more than 2^22 seeds in a region");
    }
    std::vector<sedef_sd_t> rows;
    if (na > 0) {
      uint64_t* seeds = (uint64_t*)ctx_alloc(ctx, (size_t)na * 8);
      Item* items = (Item*)ctx_alloc(ctx, (size_t)na * sizeof(Item));
      Item* init = (Item*)ctx_alloc(ctx, (size_t)na * sizeof(Item));
      Item* fin = (Item*)ctx_alloc(ctx, (size_t)na * sizeof(Item));
      int32_t* best = (int32_t*)ctx_alloc(ctx, (size_t)na * 4);
      int32_t* pred = (int32_t*)ctx_alloc(ctx, (size_t)na * 4);
      int32_t* parts = (int32_t*)ctx_alloc(ctx, (size_t)na * 4);
      Take T;
      T.owner = (unsigned long long*)ctx_alloc(ctx, (size_t)na * 8);
      int32_t* words = (int32_t*)ctx_alloc(ctx, (size_t)na * 4 * 6);
      if (!seeds || !items || !init || !fin || !best || !pred || !parts || !T.owner || !words)
        return SEDEF_ERR_OOM;
      T.jump = words;
      T.jump2 = words + na;
      T.x1 = words + 2 * na;
      T.y1 = words + 3 * na;
      T.seeds = words + 4 * na;
      T.parts = words + 5 * na;
      SEDEF_KERNEL(ctx, "k_c2_mems", (k_c2_mems<true><<<(int)((xsum + 255) / 256), 256, 0, st>>>(
                                         packed, nbits, d_regs, d_xb, nb, xsum, skeys, ysum,
                                         nullptr, off, seeds)));
      SEDEF_KERNEL(ctx, "k_c2_items",
                   k_c2_items<<<(int)((na + 255) / 256), 256, 0, st>>>(seeds, na, items));
      // tier 1: DP, greedy extraction into initial chains (in start order)
      SEDEF_KERNEL(ctx, "k_c2_dp",
                   k_c2_dp<<<nb, kC2Threads, 0, st>>>(items, d_ib, d_n1, 1, g1, best, pred));
      SEDEF_KERNEL(ctx, "k_c2_take", k_c2_take<<<nb, kC2Threads, 0, st>>>(
                                         items, best, pred, d_ib, d_n1, 1, T, init, parts, d_n2));
      // tier 2 over the initial chains (region r at [ib[r], ib[r] + n2[r]))
      SEDEF_KERNEL(ctx, "k_c2_dp",
                   k_c2_dp<<<nb, kC2Threads, 0, st>>>(init, d_ib, d_n2, 2, g1, best, pred));
      SEDEF_KERNEL(ctx, "k_c2_take", k_c2_take<<<nb, kC2Threads, 0, st>>>(
                                         init, best, pred, d_ib, d_n2, 2, T, fin, parts, d_n3));
      // final chains of SD size: count, then rows per region
      const int rb = (int)(((int64_t)nb * 32 + 127) / 128);
      SEDEF_KERNEL(ctx, "k_c2_emit", k_c2_emit<<<rb, 128, 0, st>>>(fin, parts, d_ib, d_n3, d_regs,
                                                                  d_rid, nb, nullptr, nullptr, d_keep, 1));
      std::vector<uint32_t> keep(nb);
      SEDEF_CUDA(cudaMemcpyAsync(keep.data(), d_keep, (size_t)nb * 4, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaStreamSynchronize(st));
      std::vector<int64_t> kb(nb + 1, 0);
      for (int k = 0; k < nb; ++k) kb[k + 1] = kb[k] + keep[k];
      if (kb[nb] > 0) {
        sedef_sd_t* d_rows = (sedef_sd_t*)ctx_alloc(ctx, (size_t)kb[nb] * sizeof(sedef_sd_t));
        if (!d_rows) return SEDEF_ERR_OOM;
        SEDEF_CUDA(cudaMemcpyAsync(d_kb, kb.data(), (size_t)(nb + 1) * 8, cudaMemcpyHostToDevice, st));
        SEDEF_KERNEL(ctx, "k_c2_emit", k_c2_emit<<<rb, 128, 0, st>>>(fin, parts, d_ib, d_n3, d_regs,
                                                                    d_rid, nb, d_kb, d_rows, d_keep,
                                                                    0));
        rows.resize((size_t)kb[nb]);
        SEDEF_CUDA(cudaMemcpyAsync(rows.data(), d_rows, (size_t)kb[nb] * sizeof(sedef_sd_t),
                                   cudaMemcpyDeviceToHost, st));
        SEDEF_CUDA(cudaStreamSynchronize(st));
      }
    }
    all.insert(all.end(), rows.begin(), rows.end());
    ctx_pool_restore(ctx, used_before);
    r0 = r1;
  }
  *nout = (int64_t)all.size();
  if ((int64_t)all.size() > cap) return fail(SEDEF_ERR_CAPACITY, "sedef_chain2: output buffer too small");
  if (!all.empty())
    SEDEF_CUDA(cudaMemcpyAsync(out, all.data(), all.size() * sizeof(sedef_sd_t), cudaMemcpyHostToDevice,
                               st));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  return SEDEF_OK;
}

}  // namespace sedef
