// a7: chaining of each kept seed's minimizer anchors (Section 3.3) and the
// merge of chains into SD candidates.
//
// Chain: one warp per kept run finds its anchors, runs the DP over them in
// shared memory and writes the chain (k_chain_seeds).  In a self-search whose
// target records are the query records (a caller's index is compared with them
// first) the anchors are a join
// of two contiguous stretches: the window's records go into a hash table and
// the target span's records probe it.  Otherwise each query minimizer searches
// its posting list for the target span (an interpolated search, then a short
// gallop).  The anchors' order is (p, t') (t' = t for o = 0; for o = 1 the
// target axis is reversed).  The DP settles 32 anchors at a time, one per
// lane, from every earlier anchor within gap_max: the predecessor with the
// larger count, then the later one.  Seeds past the shared-memory sizes take
// three kernels instead (k_anchor_count, k_anchor_fill, k_chain_dp: anchors
// in device memory, the DP an anchor at a time).
//
// Merge: chains sorted by (o, q0); every chain links to the following chains
// whose query interval starts before its own ends; links are united with a
// lock-free union-find that always hooks the larger root under the smaller,
// so every component's root is its smallest member.
#include <cstring>
#include <string>

#include "common.cuh"

namespace sedef {

namespace {

struct ChainArgs {
  const sedef_run_t* runs;
  int64_t nruns;
  const uint64_t* qrec;
  int64_t nq;
  const uint64_t* tidx;     // hash-sorted target records (index)
  int64_t nt;
  const uint32_t* toff;
  const int64_t* qseq;
  int nqseq;
  const int64_t* tseq;
  int ntseq;
  const int32_t* mtab;
  int k, span, max_occ, self_mode, gap_max, diag_max;
  // live counts of a planned pass, the anchor capacity and its overflow flags
  const uint32_t* dnruns = nullptr;
  const uint32_t* dnq = nullptr;
  const uint32_t* dnt = nullptr;
  int64_t acap = 0;
  uint32_t* flags = nullptr;
  unsigned long long* atotal = nullptr;  // exact anchor total
  // seeds past k_chain_seeds' sizes: run indices and their number (big
  // nullptr: every run)
  uint32_t* big = nullptr;
  uint32_t* nbig = nullptr;
  // query records less target records, summed (k_same_records): zero when they
  // are the same; nullptr: known to be
  const unsigned long long* differ = nullptr;
};

// The chain DP is quadratic in a seed's anchors; a seed inside an unmasked
// low-complexity run can have millions.  Such seeds are refused.
constexpr int kMaxChainAnchors = 1 << 16;

__device__ __forceinline__ void resolve(ChainArgs& a) {
  a.nruns = live_n(a.nruns, a.dnruns);
  a.nq = live_n(a.nq, a.dnq);
  a.nt = live_n(a.nt, a.dnt);
}

// Postings of query record q's hash inside run `run`'s target span
// [j_a, j_b + n - k]: [*b0, *b1) of the index (empty when the list passes
// max_occ).  The start comes from an interpolated search of the posting
// list, the end from a gallop forward from it (the span is short).
__device__ __forceinline__ void record_postings(const ChainArgs& a, const sedef_run_t& run,
                                                uint64_t q, uint32_t* b0, uint32_t* b1) {
  const uint32_t h = rec_hash(q);
  const uint32_t st = a.toff[h], en = a.toff[h + 1];
  if (a.max_occ > 0 && (int)(en - st) > a.max_occ) {
    *b0 = *b1 = st;
    return;
  }
  const uint32_t tlo = run.j_a, thi = run.j_b + (uint32_t)a.span;
  *b0 = pos_lower_bound(a.tidx, st, en, (int64_t)tlo);
  *b1 = pos_gallop_forward(a.tidx, *b0, en, (int64_t)thi + 1);
}

// Visits the anchors of run `run` contributed by query record q among the
// postings [b0, b1): calls f(rank, p, t) for each, rank counting this
// record's anchors in (p, t') order.  Returns the number of anchors.
template <typename F>
__device__ int record_anchors(const ChainArgs& a, const sedef_run_t& run, uint64_t q, uint32_t b0,
                              uint32_t b1, F f) {
  const uint32_t p = rec_pos(q), sq = rec_strand(q);
  int cnt = 0;
  const int64_t i = run.i;
  auto visit = [&](int64_t y) {
    const uint64_t r = a.tidx[y];
    const uint32_t t = rec_pos(r);
    if ((sq ^ rec_strand(r)) != run.o) return;
    if (a.self_mode && (int64_t)t >= i && (int64_t)t <= i + a.span) return;
    f(cnt, p, t);
    ++cnt;
  };
  if (run.o == 0)
    for (int64_t y = b0; y < b1; ++y) visit(y);
  else
    for (int64_t y = (int64_t)b1 - 1; y >= (int64_t)b0; --y) visit(y);
  return cnt;
}

__device__ __forceinline__ void window_range(const ChainArgs& a, int64_t i, int64_t* qa, int64_t* qb) {
  auto pos_of = [](uint64_t r) { return (uint64_t)((r >> 1) & 0xFFFFFFFFull); };
  *qa = lower_bound_by(a.qrec, 0, a.nq, (uint64_t)i, pos_of);
  *qb = lower_bound_by(a.qrec, *qa, a.nq, (uint64_t)(i + a.span + 1), pos_of);
}

// The finalizer of SplitMix64 (Steele, Lea, Flood: Fast Splittable
// Pseudorandom Number Generators, 2014).
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Adds to differ[0..2) two mixes of every query record and takes those of the
// index's away.  Both sums are zero when the arrays hold the same records in
// any order, and otherwise with a chance of 2^-128: the join may take the
// target's records by position from the query's.  Bound by reading both
// arrays once (16 bytes a record).
__global__ void __launch_bounds__(256) k_same_records(const uint64_t* __restrict__ q,
                                                      const uint64_t* __restrict__ t, int64_t n,
                                                      unsigned long long* differ) {
  unsigned long long a = 0, b = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll 4
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
    const unsigned long long u = q[x], v = t[x];
    a += mix64(u) - mix64(v);
    b += mix64(~u) - mix64(~v);
  }
  a = warp_sum(a);
  b = warp_sum(b);
  if (lane_id() == 0 && (a | b)) {
    atomicAdd(differ, a);
    atomicAdd(differ + 1, b);
  }
}

// What k_chain_seeds keeps of a seed in shared memory.
constexpr int kSeedWarps = 8;
constexpr int kSeedQ = 256;            // query records
constexpr int kSeedTab = 2 * kSeedQ;   // hash-table slots
constexpr int kSeedA = 256;            // anchors
constexpr int kSeedTBits = 22;         // target span below 2^22 bases
struct alignas(16) SeedSmem {
  uint32_t tab[kSeedTab];    // hash + 1 of a query record (equal ones each have a slot)
  uint16_t info[kSeedTab];   // its offset in the window << 1 | strand
  uint32_t anchor[kSeedA];   // (p - i) << kSeedTBits | t' - lowest t', sorted
  uint16_t f[kSeedA];        // anchors of the best chain that ends here
  uint16_t first[kSeedA];    // its first anchor
  int n;
};

// Bound by the latency of its two record searches and, per seed, a thousand
// or so instructions.  Count, fill and DP as kernels of their own searched
// the records with one lane, the postings of every query record twice (in
// memory the size of the index) and kept the DP's state in device memory:
// 626 k seeds of a 200-genome batch 8.3 -> 2.6 ms, a 240 Mbp assembly's 3.5 ->
// 1.2 ms.
template <bool kJoin>
__global__ void __launch_bounds__(32 * kSeedWarps) k_chain_seeds(ChainArgs a, sedef_chain_t* out) {
  if (kJoin && a.differ && (a.differ[0] | a.differ[1]) != 0ull) return;  // other records
  resolve(a);
  __shared__ SeedSmem smem[kSeedWarps];
  SeedSmem& S = smem[threadIdx.x >> 5];
  const int lane = lane_id();
  const unsigned lt = lanemask_lt();
  unsigned long long anchors = 0;
  const int64_t nw = (int64_t)gridDim.x * kSeedWarps;
  for (int64_t r = (int64_t)blockIdx.x * kSeedWarps + (threadIdx.x >> 5); r < a.nruns; r += nw) {
    const sedef_run_t run = a.runs[r];
    if (!run.keep) {
      if (lane == 0) out[r].score = 0;
      continue;
    }
    const uint32_t i = run.i, tlo = run.j_a, thi = run.j_b + (uint32_t)a.span;
    const uint32_t o = run.o;
    const int64_t qa = warp_lower_pos(a.qrec, a.nq, i);
    bool big = thi - tlo >= (1u << kSeedTBits);
    int A = 0;
    __syncwarp();
    if (kJoin) {
      // ---- the window's records into the table
      for (int x = lane; x < kSeedTab / 4; x += 32)
        reinterpret_cast<uint4*>(S.tab)[x] = make_uint4(0, 0, 0, 0);
      if (lane == 0) S.n = 0;
      const int64_t ta = warp_lower_pos(a.qrec, a.nq, tlo);
      __syncwarp();
      int c = 0;
      for (int64_t x = qa; !big; x += 32) {
        const uint64_t q = x + lane < a.nq ? a.qrec[x + lane] : 0ull;
        const bool in = x + lane < a.nq && rec_pos(q) - i <= (uint32_t)a.span;
        c += __popc(__ballot_sync(0xffffffffu, in));
        if (c > kSeedQ) {
          big = true;
          break;
        }
        if (in) {
          const uint32_t h = rec_hash(q);
          if (!(a.max_occ > 0 && (int)(a.toff[h + 1] - a.toff[h]) > a.max_occ)) {
            uint32_t slot = (h * 0x9E3779B1u) >> 23;
            while (atomicCAS(&S.tab[slot], 0u, h + 1u) != 0u) slot = (slot + 1u) & (kSeedTab - 1);
            S.info[slot] = (uint16_t)(((rec_pos(q) - i) << 1) | rec_strand(q));
          }
        }
        if (!__all_sync(0xffffffffu, in)) break;
      }
      __syncwarp();
      // ---- the target span's records probe it
      for (int64_t x = ta; !big; x += 32) {
        const uint64_t t = x + lane < a.nq ? a.qrec[x + lane] : 0ull;
        const uint32_t p = rec_pos(t);
        const bool in = x + lane < a.nq && p - tlo <= thi - tlo;
        if (in && p - i > (uint32_t)a.span) {  // not in the window's own span
          const uint32_t h = rec_hash(t);
          for (uint32_t slot = (h * 0x9E3779B1u) >> 23; S.tab[slot] != 0u;
               slot = (slot + 1u) & (kSeedTab - 1)) {
            if (S.tab[slot] != h + 1u) continue;
            const uint32_t q = S.info[slot];
            if (((q ^ rec_strand(t)) & 1u) != o) continue;
            const int at = atomicAdd(&S.n, 1);
            if (at < kSeedA) S.anchor[at] = ((q >> 1) << kSeedTBits) | (o ? thi - p : p - tlo);
          }
        }
        __syncwarp();
        const int n = __shfl_sync(0xffffffffu, S.n, 0);  // the same answer for every lane
        if (n > kSeedA || !__all_sync(0xffffffffu, in)) break;
      }
      __syncwarp();
      A = S.n;
      big |= A > kSeedA;
      if (!big && A > 1) {
        // order by (p, t')
        int np = 2;
        while (np < A) np <<= 1;
        if (np <= 32) {
          uint32_t v = lane < A ? S.anchor[lane] : 0xFFFFFFFFu;
          for (int size = 2; size <= np; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
              const uint32_t w = __shfl_xor_sync(0xffffffffu, v, stride);
              v = ((lane & size) == 0) == ((lane & stride) == 0) ? min(v, w) : max(v, w);
            }
          if (lane < A) S.anchor[lane] = v;
        } else {
          for (int x = A + lane; x < np; x += 32) S.anchor[x] = 0xFFFFFFFFu;
          __syncwarp();
          for (int size = 2; size <= np; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
              for (int t = lane; t < (np >> 1); t += 32) {
                const int lo = ((t & ~(stride - 1)) << 1) | (t & (stride - 1)), hi = lo + stride;
                const uint32_t v = S.anchor[lo], w = S.anchor[hi];
                if ((v > w) == ((lo & size) == 0)) {
                  S.anchor[lo] = w;
                  S.anchor[hi] = v;
                }
              }
              __syncwarp();
            }
        }
        __syncwarp();
      }
    } else {
      // ---- postings of the window's records inside the target span, in order
      for (int64_t x = qa; !big; x += 32) {
        const uint64_t q = x + lane < a.nq ? a.qrec[x + lane] : 0ull;
        const bool in = x + lane < a.nq && rec_pos(q) - i <= (uint32_t)a.span;
        uint32_t b0 = 0, b1 = 0;
        int c = 0;
        if (in) {
          record_postings(a, run, q, &b0, &b1);
          c = record_anchors(a, run, q, b0, b1, [](int, uint32_t, uint32_t) {});
        }
        const int inc = warp_inclusive_sum(min(c, kSeedA + 1));
        const int to = A + inc - c;
        A += __shfl_sync(0xffffffffu, inc, 31);
        if (A > kSeedA) {
          big = true;
        } else if (c > 0) {
          record_anchors(a, run, q, b0, b1, [&](int rank, uint32_t p, uint32_t t) {
            S.anchor[to + rank] = ((p - i) << kSeedTBits) | (o ? thi - t : t - tlo);
          });
        }
        if (!__all_sync(0xffffffffu, in)) break;
      }
      __syncwarp();
    }
    if (big) {
      if (lane == 0) {
        out[r].score = 0;
        a.big[atomicAdd(a.nbig, 1u)] = (uint32_t)r;
      }
      continue;
    }
    anchors += A;
    // ---- the DP, 32 anchors at a time
    unsigned long long be = 0;  // best end: larger f, then the earlier anchor; f << 32 | ~index
    for (int t0 = 0; t0 < A; t0 += 32) {
      const int x = t0 + lane;
      const uint32_t ax = x < A ? S.anchor[x] : 0u;
      const int p = (int)(ax >> kSeedTBits), t = (int)(ax & ((1u << kSeedTBits) - 1u));
      int bf = 0, bb = -1;  // best predecessor's count and index
      auto look = [&](int pb, int tb, int f, int b) {
        const int dp = p - pb, dt = t - tb, dd = dp - dt;
        if (dp > 0 && dt > 0 && dp <= a.gap_max && dt <= a.gap_max && dd <= a.diag_max &&
            -dd <= a.diag_max && f >= bf) {  // the later of equals
          bf = f;
          bb = b;
        }
      };
      for (int b = 0; b < t0; ++b) {
        const uint32_t v = S.anchor[b];
        look((int)(v >> kSeedTBits), (int)(v & ((1u << kSeedTBits) - 1u)), S.f[b], b);
      }
      const int m = min(32, A - t0);
      int my_first = bb >= 0 ? S.first[bb] : x;
      for (int y = 0; y < m; ++y) {
        const int fy = __shfl_sync(0xffffffffu, bf + 1, y), py = __shfl_sync(0xffffffffu, p, y);
        const int ty = __shfl_sync(0xffffffffu, t, y), sy = __shfl_sync(0xffffffffu, my_first, y);
        if (lane > y) {
          const int before = bb;
          look(py, ty, fy, t0 + y);
          if (bb != before) my_first = sy;
        }
      }
      if (x < A) {
        S.f[x] = (uint16_t)(bf + 1);
        S.first[x] = (uint16_t)my_first;
        const unsigned long long v = ((unsigned long long)(bf + 1) << 32) | (0xFFFFFFFFu - (uint32_t)x);
        if (v > be) be = v;
      }
      __syncwarp();
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, be, d);
      if (v > be) be = v;
    }
    if (lane == 0) {
      sedef_chain_t c;
      c.i = i;
      c.qseq = c.q0 = c.q1 = c.tseq = c.t0 = c.t1 = 0;
      c.score = 0;
      c.s = run.s;
      c.o = o;
      c.reserved = 0;
      const int score = (int)(be >> 32);
      if (A > 0 && score >= a.mtab[run.s]) {
        // a chain advances on both axes: its ends are its box
        const uint32_t end = 0xFFFFFFFFu - (uint32_t)be;
        const uint32_t e1 = S.anchor[end], e0 = S.anchor[S.first[end]];
        const uint32_t tm = (1u << kSeedTBits) - 1u;
        c.q0 = i + (e0 >> kSeedTBits);
        c.q1 = i + (e1 >> kSeedTBits) + (uint32_t)a.k;
        c.t0 = o ? thi - (e1 & tm) : tlo + (e0 & tm);
        c.t1 = (o ? thi - (e0 & tm) : tlo + (e1 & tm)) + (uint32_t)a.k;
        c.qseq = (uint32_t)seq_of(a.qseq, a.nqseq, i);
        c.tseq = (uint32_t)seq_of(a.tseq, a.ntseq, tlo);
        c.score = (uint16_t)score;
      }
      out[r] = c;
    }
  }
  if (lane == 0 && anchors) atomicAdd(a.atotal, anchors);
}

// The seeds of the device-memory path: those k_chain_seeds left, or every run.
__device__ __forceinline__ int64_t seed_count(const ChainArgs& a) {
  return a.big ? (int64_t)*a.nbig : a.nruns;
}
__device__ __forceinline__ int64_t seed_run(const ChainArgs& a, int64_t r) {
  return a.big ? (int64_t)a.big[r] : r;
}

// Their anchors.
__global__ void k_anchor_count(ChainArgs a, uint32_t* count) {
  resolve(a);
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < seed_count(a);
       r += nw) {
    const sedef_run_t run = a.runs[seed_run(a, r)];
    if (!run.keep) {
      if (lane == 0) count[r] = 0;
      continue;
    }
    int total = 0;
    int64_t qa = 0, qb = 0;
    if (lane == 0) window_range(a, run.i, &qa, &qb);
    qa = __shfl_sync(0xffffffffu, qa, 0);
    qb = __shfl_sync(0xffffffffu, qb, 0);
    for (int64_t x = qa + lane; x < qb; x += 32) {
      const uint64_t q = a.qrec[x];
      uint32_t b0, b1;
      record_postings(a, run, q, &b0, &b1);
      total += record_anchors(a, run, q, b0, b1, [](int, uint32_t, uint32_t) {});
    }
    total = warp_sum(total);
    if (lane == 0) {
      count[r] = (uint32_t)total;
      if (total) atomicAdd(a.atotal, (unsigned long long)total);
    }
  }
}

// Writes anchors as (p << 32 | t') at the seed's offset, in (p, t') order.
__global__ void k_anchor_fill(ChainArgs a, const uint32_t* aoff, uint64_t* anchors) {
  resolve(a);
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < seed_count(a);
       r += nw) {
    const sedef_run_t run = a.runs[seed_run(a, r)];
    // 32-bit offsets: a range that wraps or ends past the capacity is skipped
    if (aoff[r + 1] == aoff[r] || aoff[r + 1] < aoff[r] || (int64_t)aoff[r + 1] > a.acap ||
        aoff[r + 1] - aoff[r] > (uint32_t)kMaxChainAnchors)
      continue;
    int64_t qa = 0, qb = 0;
    if (lane == 0) window_range(a, run.i, &qa, &qb);
    qa = __shfl_sync(0xffffffffu, qa, 0);
    qb = __shfl_sync(0xffffffffu, qb, 0);
    const uint32_t tref = run.j_b + (uint32_t)a.span;
    uint32_t base = aoff[r];
    for (int64_t x0 = qa; x0 < qb; x0 += 32) {
      const int64_t x = x0 + lane;
      int c = 0;
      uint64_t q = 0;
      uint32_t b0 = 0, b1 = 0;
      if (x < qb) {
        q = a.qrec[x];
        record_postings(a, run, q, &b0, &b1);
        c = record_anchors(a, run, q, b0, b1, [](int, uint32_t, uint32_t) {});
      }
      const int inc = warp_inclusive_sum(c);
      const uint32_t my = base + (uint32_t)(inc - c);
      if (x < qb && c > 0)
        record_anchors(a, run, q, b0, b1, [&](int rank, uint32_t p, uint32_t t) {
          const uint32_t tp = run.o ? tref - t : t;
          anchors[my + rank] = ((uint64_t)p << 32) | tp;
        });
      base += (uint32_t)__shfl_sync(0xffffffffu, inc, 31);
    }
  }
}

// DP over each of these seeds' anchors; writes the run's chain (score 0 =
// none).
__device__ void chain_one(const ChainArgs& a, int64_t r, const uint32_t* aoff, const uint64_t* anchors,
                          int32_t* f, int32_t* pred, sedef_chain_t* out) {
  const int lane = lane_id();
  const sedef_run_t run = a.runs[seed_run(a, r)];
  sedef_chain_t c;
  c.i = run.i;
  c.o = run.o;
  c.s = run.s;
  c.score = 0;
  c.reserved = 0;
  const uint32_t A0 = aoff[r], A = aoff[r + 1] - A0;
  const bool wrapped = aoff[r + 1] < A0;
  const bool over = wrapped || (int64_t)aoff[r + 1] > a.acap;
  const bool big = !wrapped && A > (uint32_t)kMaxChainAnchors;
  if ((over || big) && a.flags && lane == 0)
    atomicOr(a.flags, (over ? (uint32_t)kOverAnchors : 0u) | (big ? (uint32_t)kAnchorLimit : 0u));
  if (A == 0 || over || big) {
    if (lane == 0) {
      c.qseq = c.q0 = c.q1 = c.tseq = c.t0 = c.t1 = 0;
      out[seed_run(a, r)] = c;
    }
    return;
  }
  const uint64_t* an = anchors + A0;
  int32_t* F = f + A0;
  int32_t* P = pred + A0;
  uint32_t blo = 0;  // first predecessor with p >= p_a - gap_max
  for (uint32_t x = 0; x < A; ++x) {
    const uint64_t ax = an[x];
    const int64_t pa = (int64_t)(ax >> 32), ta = (int64_t)(uint32_t)ax;
    while (blo < x && (int64_t)(an[blo] >> 32) < pa - a.gap_max) ++blo;
    unsigned long long best = 0;  // (f + 1) << 32 | b
    for (uint32_t b = blo + lane; b < x; b += 32) {
      const uint64_t bx = an[b];
      const int64_t dp = pa - (int64_t)(bx >> 32), dt = ta - (int64_t)(uint32_t)bx;
      if (dp <= 0 || dt <= 0 || dp > a.gap_max || dt > a.gap_max) continue;
      const int64_t dd = dp - dt;
      if (dd > a.diag_max || -dd > a.diag_max) continue;
      const unsigned long long cand = ((unsigned long long)(F[b] + 1) << 32) | b;
      if (cand > best) best = cand;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, d);
      if (o > best) best = o;
    }
    if (lane == 0) {
      if (best) {
        F[x] = (int32_t)(best >> 32);
        P[x] = (int32_t)(uint32_t)best;
      } else {
        F[x] = 1;
        P[x] = -1;
      }
    }
    __syncwarp();
  }
  // best end: largest f, then smallest index
  unsigned long long be = 0;  // f << 32 | (~index)
  for (uint32_t x = lane; x < A; x += 32) {
    const unsigned long long v = ((unsigned long long)F[x] << 32) | (0xFFFFFFFFu - x);
    if (v > be) be = v;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, be, d);
    if (o > be) be = o;
  }
  if (lane != 0) return;
  const int score = (int)(be >> 32);
  const int end = (int)(0xFFFFFFFFu - (uint32_t)be);
  const uint32_t tref = run.j_b + (uint32_t)a.span;
  uint32_t q0 = 0xFFFFFFFFu, q1 = 0, t0 = 0xFFFFFFFFu, t1 = 0;
  for (int x = end; x >= 0; x = P[x]) {
    const uint64_t ax = an[x];
    const uint32_t p = (uint32_t)(ax >> 32), tp = (uint32_t)ax;
    const uint32_t t = run.o ? tref - tp : tp;
    q0 = min(q0, p);
    q1 = max(q1, p + (uint32_t)a.k);
    t0 = min(t0, t);
    t1 = max(t1, t + (uint32_t)a.k);
  }
  c.qseq = (uint32_t)seq_of(a.qseq, a.nqseq, run.i);
  c.tseq = (uint32_t)seq_of(a.tseq, a.ntseq, run.j_a);
  c.q0 = q0;
  c.q1 = q1;
  c.t0 = t0;
  c.t1 = t1;
  c.score = (score >= a.mtab[run.s]) ? (uint16_t)score : 0;
  out[seed_run(a, r)] = c;
}

__global__ void k_chain_dp(ChainArgs a, const uint32_t* aoff, const uint64_t* anchors, int32_t* f,
                           int32_t* pred, sedef_chain_t* out) {
  resolve(a);
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < seed_count(a); r += nw)
    chain_one(a, r, aoff, anchors, f, pred, out);
}

__global__ void k_max_u32(const uint32_t* v, int64_t n, uint32_t* out) {
  uint32_t m = 0;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x)
    m = max(m, v[x]);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, d));
  if (lane_id() == 0) atomicMax(out, m);
}

// Flags over all n slots (zero past the live count, so that a scan over n
// counts the live chains only).
__global__ void k_chain_flags(const sedef_chain_t* c, int64_t n, uint32_t* flag,
                              const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < n) flag[x] = (x < live_n(n, dn) && c[x].score > 0) ? 1u : 0u;
}

__global__ void k_chain_compact(const sedef_chain_t* c, int64_t n, const uint32_t* pos,
                                sedef_chain_t* out, int64_t cap, const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < live_n(n, dn) && c[x].score > 0 && (int64_t)pos[x] < cap) out[pos[x]] = c[x];
}

// ----------------------------------------------------------------- merge --

// What the links compare, in sorted order: [0] q0, q1, t0, t1; [1] o, query
// sequence, target sequence.
struct LinkBox {
  uint4 box, of;
};

struct MergeArgs {
  const sedef_chain_t* ch;
  int64_t n;
  const uint32_t* perm;  // sorted position -> chain index
  LinkBox* boxes;        // by sorted position
  int32_t* parent;       // over sorted positions
  int diag_max;
  double delta_g;
  const uint32_t* dn = nullptr;  // live chain count of a planned pass
};

__device__ __forceinline__ int uf_find(int32_t* parent, int x) {
  while (true) {
    const int p = parent[x];
    if (p == x) return x;
    const int g = parent[p];
    if (g != p) parent[x] = g;
    x = p;
  }
}

__device__ __forceinline__ void uf_union(int32_t* parent, int x, int y) {
  while (true) {
    x = uf_find(parent, x);
    y = uf_find(parent, y);
    if (x == y) return;
    if (x < y) {
      const int t = x;
      x = y;
      y = t;
    }
    if (atomicCAS(&parent[x], x, y) == x) return;  // hook the larger root under the smaller
  }
}

__device__ __forceinline__ int64_t diag_of(const LinkBox& c) {
  return c.of.x == 0 ? (int64_t)c.box.z - (int64_t)c.box.x : (int64_t)c.box.w + (int64_t)c.box.x;
}

__device__ __forceinline__ bool linked(const MergeArgs& a, const LinkBox& A, const LinkBox& B) {
  if (A.of.x != B.of.x || A.of.y != B.of.y || A.of.z != B.of.z) return false;
  if (B.box.x > A.box.y || A.box.x > B.box.y) return false;
  if (B.box.z > A.box.w || A.box.z > B.box.w) return false;
  const int64_t len = max((int64_t)A.box.y - A.box.x, (int64_t)B.box.y - B.box.x);
  const int64_t slack = a.diag_max + (int64_t)ceil(a.delta_g * (double)len);
  const int64_t dd = diag_of(A) - diag_of(B);
  return dd <= slack && -dd <= slack;
}

__global__ void k_merge_init(MergeArgs a) {
  const int64_t n = live_n(a.n, a.dn);
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < a.n) a.parent[x] = (int32_t)x;
  if (x >= n) return;
  const sedef_chain_t c = a.ch[a.perm[x]];
  a.boxes[x] = LinkBox{make_uint4(c.q0, c.q1, c.t0, c.t1), make_uint4(c.o, c.qseq, c.tseq, 0u)};
}

// A warp per chain looks at the following ones, 32 at a time, until they
// start past its end.  Where many copies chain against one stretch a chain
// has hundreds to look at: one thread per chain, through the permutation,
// took 1.77 ms for the chains of a 240 Mbp assembly, 0.58 ms this way.
__global__ void k_merge_link(MergeArgs a) {
  a.n = live_n(a.n, a.dn);
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < a.n; x += nw) {
    const LinkBox A = a.boxes[x];
    for (int64_t y0 = x + 1; y0 < a.n; y0 += 32) {
      const int64_t y = y0 + lane;
      bool in = false;
      if (y < a.n) {
        const LinkBox B = a.boxes[y];
        in = B.of.x == A.of.x && B.box.x <= A.box.y;
        if (in && linked(a, A, B)) uf_union(a.parent, (int)x, (int)y);
      }
      if (!__all_sync(0xffffffffu, in)) break;
    }
  }
}

struct Agg {
  uint32_t q0, q1, t0, t1, score, count;
};

__global__ void k_merge_agg(MergeArgs a, Agg* agg) {
  a.n = live_n(a.n, a.dn);
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= a.n) return;
  const int root = uf_find(a.parent, (int)x);
  const sedef_chain_t c = a.ch[a.perm[x]];
  atomicMin(&agg[root].q0, c.q0);
  atomicMax(&agg[root].q1, c.q1);
  atomicMin(&agg[root].t0, c.t0);
  atomicMax(&agg[root].t1, c.t1);
  atomicAdd(&agg[root].score, (uint32_t)c.score);
  atomicAdd(&agg[root].count, 1u);
}

__global__ void k_agg_init(Agg* agg, int64_t n) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < n) {
    agg[x].q0 = 0xFFFFFFFFu;
    agg[x].q1 = 0;
    agg[x].t0 = 0xFFFFFFFFu;
    agg[x].t1 = 0;
    agg[x].score = 0;
    agg[x].count = 0;
  }
}

__global__ void k_root_flags(const int32_t* parent, int64_t n, uint32_t* flag, const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < n) flag[x] = (x < live_n(n, dn) && parent[x] == (int32_t)x) ? 1u : 0u;
}

// Candidate keys: primary (q0, t0), tbits hold every target position; the tie
// order (o, q1, t1) is applied by k_cand_final after the primary sort.
__global__ void k_cand_emit(MergeArgs a, const Agg* agg, const uint32_t* pos, int tbits,
                            sedef_cand_t* tmp, uint64_t* key, int64_t ccap) {
  a.n = live_n(a.n, a.dn);
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= a.n || a.parent[x] != (int32_t)x || (int64_t)pos[x] >= ccap) return;
  const sedef_chain_t c = a.ch[a.perm[x]];
  const Agg g = agg[x];
  sedef_cand_t d;
  d.qseq = c.qseq;
  d.q0 = g.q0;
  d.q1 = g.q1;
  d.tseq = c.tseq;
  d.t0 = g.t0;
  d.t1 = g.t1;
  d.o = c.o;
  d.score = g.score;
  d.nchains = g.count;
  d.reserved = 0;
  tmp[pos[x]] = d;
  key[pos[x]] = ((uint64_t)g.q0 << tbits) | g.t0;
}

__device__ __forceinline__ bool cand_less(const sedef_cand_t& x, const sedef_cand_t& y) {
  if (x.q0 != y.q0) return x.q0 < y.q0;
  if (x.t0 != y.t0) return x.t0 < y.t0;
  if (x.o != y.o) return x.o < y.o;
  if (x.q1 != y.q1) return x.q1 < y.q1;
  if (x.t1 != y.t1) return x.t1 < y.t1;
  if (x.qseq != y.qseq) return x.qseq < y.qseq;
  if (x.tseq != y.tseq) return x.tseq < y.tseq;
  if (x.score != y.score) return x.score < y.score;
  return x.nchains < y.nchains;
}

// Gathers candidates in primary-key order, orders equal-key groups by the
// full comparator (groups are tiny) and converts to per-sequence coordinates.
__global__ void k_cand_final(const sedef_cand_t* tmp, const uint32_t* perm, const uint64_t* skey,
                             int64_t n, const int64_t* qseq, const int64_t* tseq, sedef_cand_t* out,
                             const uint32_t* dn) {
  n = live_n(n, dn);
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= n) return;
  if (x > 0 && skey[x - 1] == skey[x]) return;  // group leader handles the group
  int64_t e = x + 1;
  while (e < n && skey[e] == skey[x]) ++e;
  for (int64_t y = x; y < e; ++y) {
    // selection of the y-th smallest in the group (groups are tiny)
    sedef_cand_t best = tmp[perm[x]];
    bool set = false;
    for (int64_t z = x; z < e; ++z) {
      const sedef_cand_t c = tmp[perm[z]];
      int64_t rank = 0;
      for (int64_t u = x; u < e; ++u) {
        const sedef_cand_t d = tmp[perm[u]];
        if (cand_less(d, c) || (!cand_less(c, d) && u < z)) ++rank;
      }
      if (rank == y - x) {
        best = c;
        set = true;
        break;
      }
    }
    if (!set) best = tmp[perm[y]];
    sedef_cand_t o = best;
    o.q0 -= (uint32_t)qseq[best.qseq];
    o.q1 -= (uint32_t)qseq[best.qseq];
    o.t0 -= (uint32_t)tseq[best.tseq];
    o.t1 -= (uint32_t)tseq[best.tseq];
    out[y] = o;
  }
}

// (o, q0); qbits hold every query position.
__global__ void k_chain_keys(const sedef_chain_t* c, int64_t n, int qbits, uint64_t* key,
                             const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < live_n(n, dn)) key[x] = ((uint64_t)c[x].o << qbits) | c[x].q0;
}

int grid_of(int64_t n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

int scan_exclusive_u32(sedef_ctx* ctx, const uint32_t* in, uint32_t* out, int64_t n,
                       uint32_t* d_total);

static int upload_offsets(sedef_ctx* ctx, Planned* pl, const int64_t* h_q, int nq,
                          const int64_t* h_t, int nt, int64_t** d_q, int64_t** d_t) {
  cudaStream_t st = ctx_stream(ctx);
  const size_t bytes = (size_t)(nq + 1 + nt + 1) * 8;
  int64_t* h = (int64_t*)host_buf(ctx, pl, bytes);
  int64_t* d = (int64_t*)ctx_alloc(ctx, bytes);
  if (!h || !d) return SEDEF_ERR_OOM;
  std::memcpy(h, h_q, (size_t)(nq + 1) * 8);
  std::memcpy(h + nq + 1, h_t, (size_t)(nt + 1) * 8);
  SEDEF_CUDA(cudaMemcpyAsync(d, h, bytes, cudaMemcpyHostToDevice, st));
  *d_q = d;
  *d_t = d + nq + 1;
  return SEDEF_OK;
}

int run_chain(sedef_ctx* ctx, const sedef_run_t* runs, int64_t nruns, const uint64_t* qrec, int64_t nq,
              const int64_t* h_qoff, int nqseq, const uint64_t* tsorted, int64_t nt,
              const uint32_t* toff, const int64_t* h_toff, int ntseq, const Derived& D,
              const int32_t* h_mtab, sedef_chain_t* chains, int64_t cap, int64_t* nchains,
              Planned* pl, bool one_sketch) {
  cudaStream_t st = ctx_stream(ctx);
  int64_t *dq = nullptr, *dt = nullptr;
  SEDEF_TRY(upload_offsets(ctx, pl, h_qoff, nqseq, h_toff, ntseq, &dq, &dt));
  int32_t* dm = (int32_t*)ctx_alloc(ctx, (size_t)(kMaxWindowRecs + 1) * 4);
  if (!dm) return SEDEF_ERR_OOM;
  if (pl) {
    int32_t* hm = (int32_t*)host_buf(ctx, pl, (size_t)(kMaxWindowRecs + 1) * 4);
    if (!hm) return SEDEF_ERR_OOM;
    std::memcpy(hm, h_mtab, (size_t)(kMaxWindowRecs + 1) * 4);
    SEDEF_CUDA(cudaMemcpyAsync(dm, hm, (size_t)(kMaxWindowRecs + 1) * 4, cudaMemcpyHostToDevice, st));
  } else {
    SEDEF_CUDA(cudaMemcpyAsync(dm, h_mtab, (size_t)(kMaxWindowRecs + 1) * 4, cudaMemcpyHostToDevice, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));  // the mtab upload reads caller memory
  }

  ChainArgs a;
  a.runs = runs;
  a.nruns = nruns;
  a.qrec = qrec;
  a.nq = nq;
  a.tidx = tsorted;
  a.nt = nt;
  a.toff = toff;
  a.qseq = dq;
  a.nqseq = nqseq;
  a.tseq = dt;
  a.ntseq = ntseq;
  a.mtab = dm;
  a.k = D.k;
  a.span = D.span;
  a.max_occ = D.max_occ;
  a.self_mode = D.self_mode;
  a.gap_max = D.gap_max;
  a.diag_max = D.diag_max;
  if (pl) {
    a.dnruns = pl->n_runs;
    a.dnq = pl->n_rec;
    a.dnt = pl->n_rec;
    a.flags = pl->flags;
  }
  // a self-search's query records are its target records by position: where
  // the caller gave an index that may be another's, the join returns at once
  // when it is, and the search is launched after the counts are read
  const bool join = one_sketch || (D.self_mode != 0 && nq == nt && nqseq == ntseq &&
                    std::memcmp(h_qoff, h_toff, (size_t)(ntseq + 1) * sizeof(int64_t)) == 0);
  // Windows of more records than k_chain_seeds keeps, on average (the join
  // takes kSeedQ records, the search kSeedA anchors): its try came on top of
  // what the device-memory path costs.  Chains of 10 Mbp, before there were
  // two paths, with every seed tried, and now: joined w = 5 0.38, 0.47, 0.38 ms
  // (w = 6 0.34 -> 0.20 tried), searched w = 4 4.9, 6.2, 5.0 (w = 5 3.8 -> 1.9
  // tried).
  const bool dense = 2 * (D.span + 1) > (join ? kSeedQ * 9 / 10 : kSeedA) * (D.w + 1);
  // [0] anchors of every seed, [1] seeds for the device-memory path, [2] the
  // most anchors one of them has, [3] and [4] k_same_records' sums
  unsigned long long* sums = (unsigned long long*)ctx_alloc(ctx, 40);
  uint32_t* cnt = (uint32_t*)ctx_alloc(ctx, (size_t)(nruns + 1) * 4);
  a.big = dense ? nullptr : (uint32_t*)ctx_alloc(ctx, (size_t)nruns * 4);
  sedef_chain_t* tmp = (sedef_chain_t*)ctx_alloc(ctx, (size_t)nruns * sizeof(sedef_chain_t));
  // the big seeds' anchor offsets, then the chains' places
  uint32_t* pos = (uint32_t*)ctx_alloc(ctx, (size_t)(nruns + 1) * 4);
  if (!sums || !cnt || (!dense && !a.big) || !tmp || !pos) return SEDEF_ERR_OOM;
  SEDEF_CUDA(cudaMemsetAsync(sums, 0, 40, st));
  a.atotal = sums;
  a.nbig = (uint32_t*)(sums + 1);
  uint32_t* amax = (uint32_t*)(sums + 2);
  const int64_t most = (int64_t)ctx_sm_count(ctx) * 5;
  const int sg = (int)((nruns + kSeedWarps - 1) / kSeedWarps < most ? (nruns + kSeedWarps - 1) / kSeedWarps : most);
  if (join && !one_sketch && !dense) {
    a.differ = sums + 3;
    const int64_t cg = (nq + 1023) / 1024;
    SEDEF_KERNEL(ctx, "k_same_records",
                 k_same_records<<<(int)(cg < most ? (cg > 0 ? cg : 1) : most), 256, 0, st>>>(
                     qrec, tsorted, nq, sums + 3));
  }
  if (join && !dense)
    SEDEF_KERNEL(ctx, "k_chain_seeds", k_chain_seeds<true><<<sg, 32 * kSeedWarps, 0, st>>>(a, tmp));
  if (!join && !dense)
    SEDEF_KERNEL(ctx, "k_chain_seeds", k_chain_seeds<false><<<sg, 32 * kSeedWarps, 0, st>>>(a, tmp));
  int64_t nbig = nruns, A = 0;
  unsigned long long* h_sums = nullptr;
  if (!pl) {
    h_sums = (unsigned long long*)ctx_host(ctx, 40);
    if (!h_sums) return SEDEF_ERR_OOM;
  }
  if (!pl && !dense) {
    SEDEF_CUDA(cudaMemcpyAsync(h_sums, sums, 40, cudaMemcpyDeviceToHost, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));
    if (a.differ && (h_sums[3] | h_sums[4]) != 0ull) {
      SEDEF_KERNEL(ctx, "k_chain_seeds", k_chain_seeds<false><<<sg, 32 * kSeedWarps, 0, st>>>(a, tmp));
      SEDEF_CUDA(cudaMemcpyAsync(h_sums, sums, 24, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaStreamSynchronize(st));
    }
    nbig = (int64_t)(h_sums[1] & 0xFFFFFFFFull);
    ctx_set_anchor_total(ctx, (int64_t)h_sums[0]);
  }
  if (nbig > 0) {
    // the seeds past the shared-memory sizes (a planned pass does not know
    // whether there are any)
    uint32_t* aoff = pos;
    // a warp per seed; a pass that mostly has none of them starts fewer
    const int wb = grid_of(!pl || dense || nbig * 32 < most * 256 ? nbig * 32 : most * 256, 256);
    if (pl) SEDEF_CUDA(cudaMemsetAsync(cnt, 0, (size_t)(nbig + 1) * 4, st));
    SEDEF_KERNEL(ctx, "k_anchor_count", k_anchor_count<<<wb, 256, 0, st>>>(a, cnt));
    SEDEF_KERNEL(ctx, "k_max_u32",
                 k_max_u32<<<grid_of(nbig < 65536 ? nbig : 65536, 256), 256, 0, st>>>(cnt, nbig, amax));
    SEDEF_TRY(scan_exclusive_u32(ctx, cnt, aoff, nbig, aoff + nbig));
    if (pl) {
      // anchors: planned capacity; seeds past it or over the limit are
      // skipped and flagged by the DP
      A = pl->anchors;
      SEDEF_TRY(plan_check64(ctx, pl, a.atotal, A, 3));
    } else {
      uint32_t* h_tot = (uint32_t*)h_sums;
      SEDEF_CUDA(cudaMemcpyAsync(h_tot, aoff + nbig, 4, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaMemcpyAsync(h_tot + 1, amax, 4, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaMemcpyAsync(h_tot + 2, sums, 8, cudaMemcpyDeviceToHost, st));
      SEDEF_CUDA(cudaStreamSynchronize(st));
      A = h_tot[0];
      ctx_set_anchor_total(ctx, (int64_t)(((uint64_t)h_tot[3] << 32) | h_tot[2]));
      // refuse instead of running for hours
      if (h_tot[1] > (uint32_t)kMaxChainAnchors)
        return fail(SEDEF_ERR_UNSUPPORTED,
                    "sedef_chain: a seed has " + std::to_string(h_tot[1]) +
                        " anchors (limit 65536); soft-mask low-complexity repeats or set max_occ");
    }
    a.acap = A;
    uint64_t* anchors = (uint64_t*)ctx_alloc(ctx, (size_t)(A ? A : 1) * 8);
    int32_t* f = (int32_t*)ctx_alloc(ctx, (size_t)(A ? A : 1) * 4);
    int32_t* pred = (int32_t*)ctx_alloc(ctx, (size_t)(A ? A : 1) * 4);
    if (!anchors || !f || !pred) return SEDEF_ERR_OOM;
    SEDEF_KERNEL(ctx, "k_anchor_fill", k_anchor_fill<<<wb, 256, 0, st>>>(a, aoff, anchors));
    SEDEF_KERNEL(ctx, "k_chain_dp", k_chain_dp<<<wb, 256, 0, st>>>(a, aoff, anchors, f, pred, tmp));
  }
  uint32_t* flag = cnt;  // reuse
  const uint32_t* dn = pl ? pl->n_runs : nullptr;
  SEDEF_KERNEL(ctx, "k_chain_flags",
               k_chain_flags<<<grid_of(nruns, 256), 256, 0, st>>>(tmp, nruns, flag, dn));
  SEDEF_TRY(scan_exclusive_u32(ctx, flag, pos, nruns, pos + nruns));
  if (pl) {
    pl->n_chains = pos + nruns;
    SEDEF_TRY(plan_check(ctx, pl, pos + nruns, cap, 4));
    *nchains = cap;
    SEDEF_KERNEL(ctx, "k_chain_compact",
                 k_chain_compact<<<grid_of(nruns, 256), 256, 0, st>>>(tmp, nruns, pos, chains, cap, dn));
    return SEDEF_OK;
  }
  uint32_t* h_tot = (uint32_t*)ctx_host(ctx, 8);
  if (!h_tot) return SEDEF_ERR_OOM;
  SEDEF_CUDA(cudaMemcpyAsync(h_tot, pos + nruns, 4, cudaMemcpyDeviceToHost, st));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  *nchains = *h_tot;
  if (*nchains > cap) return fail(SEDEF_ERR_CAPACITY, "sedef_chain: chain buffer too small");
  SEDEF_KERNEL(ctx, "k_chain_compact",
               k_chain_compact<<<grid_of(nruns, 256), 256, 0, st>>>(tmp, nruns, pos, chains, cap,
                                                                    nullptr));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  return SEDEF_OK;
}

int run_merge(sedef_ctx* ctx, const sedef_chain_t* chains, int64_t n, const int64_t* h_qoff,
              int nqseq, const int64_t* h_toff, int ntseq, const Derived& D, sedef_cand_t* cands,
              int64_t cap, int64_t* ncands, Planned* pl) {
  cudaStream_t st = ctx_stream(ctx);
  if (n >= (int64_t(1) << 31)) return fail(SEDEF_ERR_UNSUPPORTED, "too many chains");
  const uint32_t* dn = pl ? pl->n_chains : nullptr;
  int64_t *dq = nullptr, *dt = nullptr;
  SEDEF_TRY(upload_offsets(ctx, pl, h_qoff, nqseq, h_toff, ntseq, &dq, &dt));
  // 56 bytes a chain: the flags and their sums take the sort keys' place, the
  // components' boxes that of the chains'
  uint64_t* key = (uint64_t*)ctx_alloc(ctx, (size_t)(n + 1) * 8);
  uint64_t* skey = (uint64_t*)ctx_alloc(ctx, (size_t)n * 8);
  uint32_t* perm = (uint32_t*)ctx_alloc(ctx, (size_t)n * 4);
  int32_t* parent = (int32_t*)ctx_alloc(ctx, (size_t)n * 4);
  LinkBox* boxes = (LinkBox*)ctx_alloc(ctx, (size_t)n * sizeof(LinkBox));
  if (!key || !skey || !perm || !parent || !boxes) return SEDEF_ERR_OOM;
  uint32_t* flag = (uint32_t*)key;
  uint32_t* pos = flag + (n + 1);
  static_assert(sizeof(Agg) <= sizeof(LinkBox), "a component's box fits in a chain's place");
  Agg* agg = (Agg*)boxes;
  const int g = grid_of(n, 256);
  // sort keys of only as many bits as the positions have
  const int qbits = bits_below(h_qoff[nqseq] + 1), tbits = bits_below(h_toff[ntseq] + 1);
  SEDEF_KERNEL(ctx, "k_chain_keys", k_chain_keys<<<g, 256, 0, st>>>(chains, n, qbits, key, dn));
  SEDEF_TRY(radix_sort_u64(ctx, key, nullptr, skey, perm, n, 0, qbits + 1, dn));
  MergeArgs a;
  a.ch = chains;
  a.n = n;
  a.perm = perm;
  a.boxes = boxes;
  a.parent = parent;
  a.diag_max = D.diag_max;
  a.delta_g = D.delta_g;
  a.dn = dn;
  SEDEF_KERNEL(ctx, "k_merge_init", k_merge_init<<<g, 256, 0, st>>>(a));
  const int64_t most = (int64_t)ctx_sm_count(ctx) * 8;
  SEDEF_KERNEL(ctx, "k_merge_link",
               k_merge_link<<<(int)((n + 7) / 8 < most ? (n + 7) / 8 : most), 256, 0, st>>>(a));
  SEDEF_KERNEL(ctx, "k_agg_init", k_agg_init<<<g, 256, 0, st>>>(agg, n));
  SEDEF_KERNEL(ctx, "k_merge_agg", k_merge_agg<<<g, 256, 0, st>>>(a, agg));
  SEDEF_KERNEL(ctx, "k_root_flags", k_root_flags<<<g, 256, 0, st>>>(parent, n, flag, dn));
  SEDEF_TRY(scan_exclusive_u32(ctx, flag, pos, n, pos + n));
  int64_t nc;
  const uint32_t* dnc = nullptr;
  if (pl) {
    nc = cap;
    dnc = pos + n;
    pl->n_cands = dnc;
    SEDEF_TRY(plan_check(ctx, pl, dnc, cap, 5));
    *ncands = cap;
  } else {
    uint32_t* h_tot = (uint32_t*)ctx_host(ctx, 8);
    if (!h_tot) return SEDEF_ERR_OOM;
    SEDEF_CUDA(cudaMemcpyAsync(h_tot, pos + n, 4, cudaMemcpyDeviceToHost, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));
    nc = *h_tot;
    *ncands = nc;
    if (nc > cap) return fail(SEDEF_ERR_CAPACITY, "sedef_merge: candidate buffer too small");
  }
  if (nc == 0) return SEDEF_OK;
  sedef_cand_t* tmp = (sedef_cand_t*)ctx_alloc(ctx, (size_t)nc * sizeof(sedef_cand_t));
  uint64_t* ckey = nc <= n ? skey : (uint64_t*)ctx_alloc(ctx, (size_t)nc * 8);
  uint64_t* cskey = (uint64_t*)ctx_alloc(ctx, (size_t)nc * 8);
  uint32_t* cperm = (uint32_t*)ctx_alloc(ctx, (size_t)nc * 4);
  if (!tmp || !ckey || !cskey || !cperm) return SEDEF_ERR_OOM;
  SEDEF_KERNEL(ctx, "k_cand_emit", k_cand_emit<<<g, 256, 0, st>>>(a, agg, pos, tbits, tmp, ckey, nc));
  SEDEF_TRY(radix_sort_u64(ctx, ckey, nullptr, cskey, cperm, nc, 0, qbits + tbits, dnc));
  SEDEF_KERNEL(ctx, "k_cand_final",
               k_cand_final<<<grid_of(nc, 256), 256, 0, st>>>(tmp, cperm, cskey, nc, dq, dt, cands,
                                                              dnc));
  if (pl) return SEDEF_OK;
  SEDEF_CUDA(cudaStreamSynchronize(st));
  return SEDEF_OK;
}

}  // namespace sedef
