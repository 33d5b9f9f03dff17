// a4-a6: candidate lookup, sliding count of shared minimizers against m(s),
// and the winnowed MinHash refine (Sections 2.2 and 3.1).
//
// Every tier takes the same steps for a query window:
//   1. every posting of the window's query minimizers is a hit (t, hash, o).
//      Hits are counted into direct-mapped counters keyed by (t >> 10, o): a
//      target window [j, j+n-k] lies inside bins j>>10 and (j>>10)+1, so a j
//      can only pass when those two counters sum to m or more (aliasing and
//      hits counted twice only add false candidates).  The table has the
//      smallest power of two >= 4 H slots (H = the window's posting entries)
//      up to the tier's size, so the prefilter stays selective when posting
//      lists are long (a large target);
//   2. W_Q: the distinct hashes (s of them, each with its strand set) and m;
//   3. hits whose bin pair can pass are collected and sorted by (o, t), and
//      the runs found exactly from them.  Any j whose true count reaches m
//      has all of its hits collected, and a count computed from a subset
//      never exceeds the true one, so the runs are exact.
// Tiers, by what a window needs: the warp tier (a warp per window), the
// narrow, the broad and the deep CTA tier (k_filter_cta: 2,048, 4,096 and
// 12,288 collected hits), the second wide tier (16,384, counters of 16 bits).  Windows none of them can hold go to a global path
// that writes their hits to global memory, radix-sorts them by (window, o, t)
// and sweeps their dense groups.  The autotuner may leave the warp tier out
// for tiers 1 and 2, CTAs of chosen shapes over windows of up to 2,048
// entries (launch_fast; the second wide tier is one of these): W_Q sorted in
// shared memory, 16-bit counters, and one thread that sweeps each dense group
// (m consecutive hits within n-k bases) with per-hash counters.
//
// Refine (k_refine_batch): each run's span records become events (position,
// rank among W_Q), set up by a warp; then one lane per run rolls the target
// window over the run's breakpoints, keeping a count per rank, the shared
// hashes and the threshold that says which of them lie among the s smallest
// of W_Q u W_T, so the estimate |S(W_Q u W_T) n W_Q n W_T| is exact at every
// breakpoint.  Runs past the batched kernel's limits go to k_refine (one
// warp per run, bitsets over the sorted domain).
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <mutex>
#include <thread>

#include "common.cuh"

namespace sedef {

namespace {

constexpr int kQCap = 256;        // query records per window (fast path)
constexpr int kBinShift = 10;     // 1024-base bins (>= n - k + 1)
constexpr int kSlots = 2048;      // (bin, o) counters (16-bit)
constexpr int kHMax = 65535;      // hits per window (fast path; 16-bit counters)
constexpr uint32_t kNone = 0xFFFFFFFFu;

struct FArgs {
  const uint64_t* qrec;
  const uint64_t* trec;
  const uint64_t* tsorted;
  const uint32_t* toff;
  const int64_t* tseq;   // target sequence offsets (ntseq + 1)
  const int64_t* qseq;   // query sequence offsets (nqseq + 1)
  const int32_t* mtab;
  const uint32_t* win_i;   // window start (global)
  const uint32_t* win_qa;  // first query record of the window
  const uint32_t* win_qb;  // one past the last
  const int32_t* win_seq;  // query sequence of the window
  // per query record of a self-search: its hash's posting range from after
  // its own entry on (after_own), narrowed to the record's own genome in a
  // batch, or (kNone, 0) when the list passes max_occ; nullptr when the tiers
  // look postings up themselves
  const uint2* qpost;
  const uint32_t* tsamp;  // positions of every kSampleStride-th index entry, or nullptr
  int64_t nwin;
  int ntseq, nqseq;
  int64_t ttotal;  // target total length
  int k, n, span, max_occ, self_mode, overlap;
  int after_own;   // qpost holds only the entries after a record's own one
  sedef_run_t* runs;
  unsigned long long* nruns;
  int64_t run_cap;
  uint32_t* ov_list;
  unsigned int* nov;
  unsigned long long* stats;  // [0] hits enumerated, [1] hits collected (fast path)
};

// A self-search has no use for a hit at t when no valid target start is at or
// before it (starts lie at i + n - overlap or later), or when t lies in the
// query window's own span.  Half of all hits, the mates before the window,
// go this way.
__device__ __forceinline__ uint32_t first_useful(const FArgs& a, int64_t i) {
  const int64_t lo = a.self_mode ? i + a.n - a.overlap : 0;
  return lo < 0 ? 0u : (uint32_t)min(lo, (int64_t)0xFFFFFFFF);
}
__device__ __forceinline__ bool useless_hit(const FArgs& a, uint32_t t, uint32_t i, uint32_t lo) {
  return a.self_mode && (t < lo || t - i <= (uint32_t)a.span);
}

// ----------------------------------------------------------- run emission --

struct RunState {
  bool open;
  int64_t ja, jb, jmx;
  int mx;
  // the target sequence that held the last position looked up
  int64_t seq_lo = 0, seq_hi = -1;
  int seq = 0;
};

struct WinInfo {
  int64_t i;
  int qseq;
  int s, m, o;
};

__device__ __forceinline__ void emit_run(const FArgs& a, const WinInfo& w, RunState& r) {
  if (!r.open) return;
  r.open = false;
  const unsigned long long slot = atomicAdd(a.nruns, 1ull);
  if ((int64_t)slot < a.run_cap) {
    sedef_run_t out;
    out.i = (uint32_t)w.i;
    out.j_a = (uint32_t)r.ja;
    out.j_b = (uint32_t)r.jb;
    out.j_at_max = (uint32_t)r.jmx;
    out.j_star = 0;
    out.s = (uint16_t)w.s;
    out.m = (uint16_t)w.m;
    out.max_shared = (uint16_t)r.mx;
    out.est = 0;
    out.den = 0;
    out.o = (uint8_t)w.o;
    out.keep = 0;
    a.runs[slot] = out;
  }
}

// The shared count is `shared` on every j of [j0, j1]; split by target
// sequence and the validity rules, and extend / open / close runs.
__device__ void segment(const FArgs& a, const WinInfo& w, RunState& r, int64_t j0, int64_t j1,
                        int shared) {
  if (shared < w.m) {
    emit_run(a, w, r);
    return;
  }
  int64_t x = j0 < 0 ? 0 : j0;
  while (x <= j1 && x < a.ttotal) {
    if (x < r.seq_lo || x >= r.seq_hi) {
      r.seq = seq_of(a.tseq, a.ntseq, x);
      r.seq_lo = a.tseq[r.seq];
      r.seq_hi = a.tseq[r.seq + 1];
    }
    const int u = r.seq;
    const int64_t st = r.seq_lo, en = r.seq_hi;
    int64_t lo = st, hi = en - a.n;
    bool ok = true;
    if (a.self_mode) {
      if (u < w.qseq) ok = false;
      else if (u == w.qseq) lo = max(lo, w.i + a.n - a.overlap);
      else if (a.self_mode == 2) ok = false;  // independent genomes
    }
    const int64_t pend = min(j1, en - 1);
    const int64_t vlo = max(x, lo), vhi = min(pend, hi);
    if (ok && vlo <= vhi) {
      if (r.open && vlo == r.jb + 1) {
        r.jb = vhi;
      } else {
        emit_run(a, w, r);
        r.open = true;
        r.ja = vlo;
        r.jb = vhi;
        r.mx = -1;
      }
      if (shared > r.mx) {
        r.mx = shared;
        r.jmx = vlo;
      }
    }
    x = pend + 1;
  }
}

// Exact sweep of one dense group [Jlo, Jhi] over one strand's hits (sorted
// by t; get(x) returns (t, hid)).  cnt[] holds one zeroed counter per hash
// id and is zero again on return.  A group never shares a run with another
// (they are separated by target starts that cannot pass), so the run state
// starts empty and every run is emitted before returning.  Single thread.
template <typename Get>
__device__ void sweep_group(const FArgs& a, const WinInfo& w, Get get, int64_t L, uint16_t* cnt,
                            int64_t Jlo, int64_t Jhi) {
  const int span = a.span;
  RunState r;
  r.open = false;
  int64_t lo = 0, hi = L;  // first hit with t >= Jlo
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)get(mid).x < Jlo) lo = mid + 1; else hi = mid;
  }
  int64_t e = lo, l = lo;
  int shared = 0;
  int64_t j = Jlo;
  while (e < L && (int64_t)get(e).x <= j + span) {
    if (cnt[get(e).y]++ == 0) ++shared;
    ++e;
  }
  while (true) {
    const int64_t ne = e < L ? (int64_t)get(e).x - span : INT64_MAX;
    const int64_t nl = l < e ? (int64_t)get(l).x + 1 : INT64_MAX;
    int64_t nx = min(ne, nl);
    if (nx > Jhi + 1) nx = Jhi + 1;
    segment(a, w, r, j, nx - 1, shared);
    if (nx > Jhi) break;
    j = nx;
    while (l < e && (int64_t)get(l).x + 1 <= j) {
      if (--cnt[get(l).y] == 0) --shared;
      ++l;
    }
    while (e < L && (int64_t)get(e).x - span <= j) {
      if (cnt[get(e).y]++ == 0) ++shared;
      ++e;
    }
  }
  for (int64_t x = l; x < e; ++x) cnt[get(x).y] = 0;
  emit_run(a, w, r);
}

// Dense groups of one strand's t-sorted hits (warp-cooperative; every lane
// calls).  Hit x is dense when the m hits from x on fit in n-k bases; every
// j whose count reaches m lies in [t(x+m-1) - (n-k), t(x)] for some dense x.
// Overlapping or touching such ranges form a group.  emit(mine, Jlo, Jhi) is
// called by every lane, for the groups of the lanes with `mine`, in
// increasing order (a lane that starts a group closes the one before it, so
// up to 32 groups go out at once: one after another, a window whose every hit
// is a group took 0.5 us for each of its thousands, 1.46 -> 0.12 ms for the
// global path of a 950 kbp region against a 3.1 Gbp index).
template <typename Get, typename Emit>
__device__ void find_groups(Get get, int64_t L, int m, int span, Emit emit) {
  m = max(m, 1);  // a threshold of 0 (a tiny tau) asks no more of the hits than 1
  const int lane = lane_id();
  const unsigned lt = lanemask_lt();
  int64_t carry_hi = INT64_MIN;  // largest jhi of the dense hits seen so far
  int64_t cur_lo = 0;
  bool open = false;
  for (int64_t base = 0; base + m - 1 < L; base += 32) {
    const int64_t x = base + lane;
    bool dense = false;
    int64_t jlo = 0, jhi = INT64_MIN;
    if (x + m - 1 < L) {
      const int64_t ta = get(x).x, tb = get(x + m - 1).x;
      if (tb - ta <= span) {
        dense = true;
        jlo = tb - span;
        jhi = ta;
      }
    }
    const unsigned dm = __ballot_sync(0xffffffffu, dense);
    // the hits are sorted, so the nearest dense one before has the largest jhi
    const int64_t near = __shfl_sync(0xffffffffu, jhi, dm & lt ? 31 - __clz(dm & lt) : lane);
    const int64_t before = dm & lt ? near : carry_hi;
    const bool start = dense && (before == INT64_MIN || jlo > before + 1);
    const unsigned starts = __ballot_sync(0xffffffffu, start);
    const int64_t lo_near = __shfl_sync(0xffffffffu, jlo, starts & lt ? 31 - __clz(starts & lt) : lane);
    emit(start && (open || (starts & lt)), starts & lt ? lo_near : cur_lo, before);
    if (starts) {
      cur_lo = __shfl_sync(0xffffffffu, jlo, 31 - __clz(starts));
      open = true;
    }
    if (dm) carry_hi = __shfl_sync(0xffffffffu, jhi, 31 - __clz(dm));
  }
  emit(open && lane == 0, cur_lo, carry_hi);
}

// ------------------------------------------------------ block bitonic sort --

template <typename T>
__device__ void block_sort(T* v, int n) {  // n a power of two
  for (int size = 2; size <= n; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < (n >> 1); t += blockDim.x) {
        // pair t of this stage: stride is a power of two
        const int lo = ((t & ~(stride - 1)) << 1) | (t & (stride - 1));
        const int hi = lo + stride;
        const bool asc = (lo & size) == 0;
        const T x = v[lo], y = v[hi];
        if ((x > y) == asc) {
          v[lo] = y;
          v[hi] = x;
        }
      }
      __syncthreads();
    }
}

__device__ __forceinline__ int next_pow2(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Builds W_Q for a window from its query records (already in qkey[0..c) as
// hash<<1|strand), sorted in place.  Writes dh (hash), dm (strand mask),
// pst/plen (posting range) for the kept hashes; returns s.  Uses the whole
// block.  `flag` needs c ints of scratch.
struct QBuild {
  uint32_t* qkey;
  uint32_t* dh;
  uint8_t* dm;
  uint32_t* pst;
  uint32_t* plen;
  int* tmp;
};

// Record positions of every kSampleStride-th entry of the sorted index
// (samp[k] = pos(idx[k * kSampleStride])): a search first brackets its
// answer between two samples, an array small enough to stay in L2, and then
// reads one stretch of kSampleStride index entries (one 128-byte line).
constexpr int kSampleShift = 4, kSampleStride = 1 << kSampleShift;

// pos_lower_bound over the samples, then over the bracketed stretch.
__host__ __device__ __forceinline__ uint32_t pos_lower_bound_sampled(const uint64_t* idx,
                                                                     const uint32_t* samp,
                                                                     uint32_t a0, uint32_t a1,
                                                                     int64_t key) {
  uint32_t lo = a0, hi = a1;  // pos(x) < key below lo; pos(x) >= key from hi (or hi = a1)
  if (a0 < a1) {
    const uint32_t k0 = (a0 + kSampleStride - 1) >> kSampleShift, k1 = (a1 - 1) >> kSampleShift;
    if (k0 <= k1) {  // samples inside the list: the first one at or past key
      uint32_t l = k0, h = k1 + 1;
      while (l < h) {
        const uint32_t m = l + ((h - l) >> 1);
        if ((int64_t)samp[m] >= key) h = m; else l = m + 1;
      }
      if (l <= k1) hi = l << kSampleShift;
      if (l > k0) lo = ((l - 1) << kSampleShift) + 1;
    }
  }
  while (lo < hi) {
    const uint32_t m = lo + ((hi - lo) >> 1);
    if ((int64_t)rec_pos(idx[m]) >= key) hi = m; else lo = m + 1;
  }
  return lo;
}

// Narrows a posting list [*st, *st + *len) to the positions in [lo, hi)
// (one genome of a batch).
__host__ __device__ __forceinline__ void posting_window(const uint64_t* idx, const uint32_t* samp,
                                                        uint32_t* st, uint32_t* len, int64_t lo,
                                                        int64_t hi) {
  const uint32_t a0 = *st, a1 = *st + *len;
  const uint32_t l =
      samp ? pos_lower_bound_sampled(idx, samp, a0, a1, lo) : pos_lower_bound(idx, a0, a1, lo);
  const uint32_t l2 = pos_gallop_forward(idx, l, a1, hi);
  *st = l;
  *len = l2 - l;
}

__global__ void k_sample_pos(const uint64_t* __restrict__ idx, int64_t nt, const uint32_t* dnt,
                             uint32_t* __restrict__ samp) {
  const int64_t n = live_n(nt, dnt);
  const int64_t ns = (n + kSampleStride - 1) >> kSampleShift;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < ns;
       k += (int64_t)gridDim.x * blockDim.x)
    samp[k] = rec_pos(idx[k << kSampleShift]);
}

// Posting range of every query record of a self-search, resolved once per
// record rather than once per window that holds it (a record lies in n / step
// windows), by threads that each follow one record's chain of dependent
// loads.  Records are sorted by position, so neighbouring threads share a
// genome and often a hash.
__global__ void k_qpost(FArgs a, int64_t nq, const uint32_t* dnq, uint2* out) {
  const int64_t n = live_n(nq, dnq);
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t r = a.qrec[x];
    const uint32_t h = rec_hash(r);
    uint32_t st = a.toff[h], len = a.toff[h + 1] - st;
    if (a.max_occ > 0 && (int)len > a.max_occ) {
      out[x] = make_uint2(kNone, 0u);
      continue;
    }
    int64_t lo = a.after_own ? (int64_t)rec_pos(r) + 1 : 0, hi = INT64_MAX;
    if (a.self_mode == 2) {
      const int sq = seq_of(a.qseq, a.nqseq, (int64_t)rec_pos(r));
      lo = max(lo, a.tseq[sq]);
      hi = a.tseq[sq + 1];
    }
    posting_window(a.tsorted, a.tsamp, &st, &len, lo, hi);
    out[x] = make_uint2(st, len);
  }
}

__device__ int build_wq(const FArgs& a, QBuild q, int c, int64_t seq_lo = 0, int64_t seq_hi = 0) {
  const int np = next_pow2(c < 2 ? 2 : c);
  for (int x = threadIdx.x; x < np; x += blockDim.x)
    if (x >= c) q.qkey[x] = kNone;
  __syncthreads();
  block_sort(q.qkey, np);
  // distinct hashes: first occurrence flags, block-wide compaction
  __shared__ int s_count;
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  for (int base = 0; base < c; base += blockDim.x) {
    const int x = base + threadIdx.x;
    int keep = 0;
    uint32_t h = 0, st = 0, len = 0, mask = 0;
    if (x < c) {
      h = q.qkey[x] >> 1;
      if (x == 0 || (q.qkey[x - 1] >> 1) != h) {
        for (int y = x; y < c && (q.qkey[y] >> 1) == h; ++y) mask |= 1u << (q.qkey[y] & 1u);
        st = a.toff[h];
        len = a.toff[h + 1] - st;
        keep = (a.max_occ > 0 && (int)len > a.max_occ) ? 0 : 1;
        // independent genomes: only the query's own sequence can hold targets
        if (keep && a.self_mode == 2)
          posting_window(a.tsorted, a.tsamp, &st, &len, seq_lo, seq_hi);
      }
    }
    int tot;
    const int ex = block_exclusive_sum(keep, q.tmp, &tot);
    if (keep) {
      const int d = s_count + ex;
      q.dh[d] = h;
      q.dm[d] = (uint8_t)mask;
      q.pst[d] = st;
      q.plen[d] = len;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_count += tot;
    __syncthreads();
  }
  return s_count;
}

// Posting ranges in index order (eager self-search).  The query records of a
// self-search are the index's own records, and the entries of the index with
// one hash (in a batch: one hash in one genome) form a run whose entries
// after e are the posting range of e's record.  So the ranges come from one
// walk over the index: a warp reads 32 consecutive entries, splits them into
// runs, and in a batch searches only for the ends of the run that leaves its
// 32 entries.  Each range goes to its record, found by the rank of the
// record's position among all record positions: a bitmap of the positions
// with the count of set bits before each 32-bit word.
struct RankWord {
  uint32_t before;  // record positions below this word's first position
  uint32_t bits;    // record positions inside it
};

// bits[p >> 5] |= 1 << (p & 31) for every record position p (rec sorted by
// position, so the lanes with one word are consecutive: each run of them is
// OR-ed into its first lane, which alone writes).
__global__ void k_pos_bits(const uint64_t* __restrict__ rec, int64_t n, uint32_t* __restrict__ bits) {
  const int lane = lane_id();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~(int64_t)31; base < n;
       base += stride) {
    const int64_t x = base + lane;
    const bool ok = x < n;
    const uint32_t p = ok ? rec_pos(rec[x]) : 0u;
    const uint32_t w = ok ? (p >> 5) : 0xFFFFFFFFu;
    uint32_t v = ok ? (1u << (p & 31)) : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t ov = __shfl_down_sync(0xffffffffu, v, d);
      const uint32_t ow = __shfl_down_sync(0xffffffffu, w, d);
      if (lane + d < 32 && ow == w) v |= ov;
    }
    const uint32_t pw = __shfl_up_sync(0xffffffffu, w, 1);
    if (ok && (lane == 0 || pw != w)) atomicOr(bits + w, v);
  }
}

__global__ void k_pos_popc(const uint32_t* __restrict__ bits, int64_t nw, uint32_t* __restrict__ cnt) {
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nw;
       w += (int64_t)gridDim.x * blockDim.x)
    cnt[w] = __popc(bits[w]);
}

__global__ void k_rank_words(const uint32_t* __restrict__ bits, const uint32_t* __restrict__ before,
                             int64_t nw, RankWord* __restrict__ rw) {
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nw;
       w += (int64_t)gridDim.x * blockDim.x)
    rw[w] = RankWord{before[w], bits[w]};
}

// Sequence of every 2^16 bases of the target, so that a position's sequence
// is a read and a short walk.
constexpr int kSeqShift = 16;
__global__ void k_seq_table(const int64_t* __restrict__ tseq, int ntseq, int64_t blocks,
                            int32_t* __restrict__ tab) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < blocks) tab[x] = seq_of(tseq, ntseq, x << kSeqShift);
}

// Four entries a lane keep four of each access in flight.  With keys, the
// ranges go there in index order (position << 32 | first entry, end) for
// k_qpost_place; else straight to their records.
__global__ void __launch_bounds__(256) k_qpost_index(FArgs a, int64_t n, const RankWord* __restrict__ rw,
                                                     const int32_t* __restrict__ seq_tab,
                                                     uint2* __restrict__ out,
                                                     uint64_t* __restrict__ keys,
                                                     uint32_t* __restrict__ vals) {
  constexpr int kAhead = 4;  // chunks of 32 entries; one more is read to see where the last run ends
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const bool batch = a.self_mode == 2;
  for (int64_t e0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * kAhead); e0 < n;
       e0 += nw * (32 * kAhead)) {
    uint32_t h[kAhead + 1], p[kAhead + 1], hi[kAhead];
    int g[kAhead + 1];
    RankWord q[kAhead];
#pragma unroll
    for (int c = 0; c <= kAhead; ++c) {
      const int64_t e = e0 + c * 32 + lane;
      const uint64_t r = e < n ? a.tsorted[e] : ~0ull;
      h[c] = e < n ? rec_hash(r) : 0xFFFFFFFFu;
      p[c] = rec_pos(r);
      g[c] = -1;
    }
#pragma unroll
    for (int c = 0; c < kAhead; ++c) {
      q[c] = RankWord{0u, 0u};
      hi[c] = 0;
      if (h[c] != 0xFFFFFFFFu) {
        if (!keys) q[c] = rw[p[c] >> 5];
        hi[c] = a.toff[h[c] + 1];
      }
    }
    unsigned ends[kAhead];  // lanes whose entry is the last of its run
    if (batch) {
#pragma unroll
      for (int c = 0; c <= kAhead; ++c) {
        if (h[c] != 0xFFFFFFFFu) {
          int x = seq_tab[p[c] >> kSeqShift];
          while (x + 1 < a.ntseq && a.tseq[x + 1] <= (int64_t)p[c]) ++x;
          g[c] = x;
        }
      }
#pragma unroll
      for (int c = 0; c < kAhead; ++c) {
        uint32_t nh = __shfl_down_sync(0xffffffffu, h[c], 1);
        int ng = __shfl_down_sync(0xffffffffu, g[c], 1);
        const uint32_t h0 = __shfl_sync(0xffffffffu, h[c + 1], 0);
        const int g0 = __shfl_sync(0xffffffffu, g[c + 1], 0);
        if (lane == 31) {
          nh = h0;
          ng = g0;
        }
        ends[c] = __ballot_sync(0xffffffffu, nh != h[c] || ng != g[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < kAhead; ++c) {
      const int64_t e = e0 + c * 32 + lane;
      if (h[c] == 0xFFFFFFFFu) continue;
      uint32_t re = hi[c];
      if (batch) {
        bool found = false;
#pragma unroll
        for (int d = c; d < kAhead; ++d) {
          const unsigned m = d == c ? ends[d] & ~((1u << lane) - 1u) : ends[d];
          if (!found && m) {
            re = (uint32_t)(e0 + d * 32 + __ffs(m));
            found = true;
          }
        }
        if (!found)  // the run goes on past these entries
          re = pos_gallop_forward(a.tsorted, (uint32_t)(e0 + kAhead * 32), hi[c], a.tseq[g[c] + 1]);
      }
      uint32_t rs = (uint32_t)e + 1;
      if (!a.after_own) {
        const uint32_t lo = a.toff[h[c]];
        rs = batch ? pos_lower_bound(a.tsorted, lo, (uint32_t)e, a.tseq[g[c]]) : lo;
      }
      if (a.max_occ > 0 && (int)(hi[c] - a.toff[h[c]]) > a.max_occ) rs = re = kNone;
      if (keys) {
        keys[e] = ((uint64_t)p[c] << 32) | rs;
        vals[e] = re;
      } else {
        out[q[c].before + __popc(q[c].bits & ((1u << (p[c] & 31)) - 1u))] = make_uint2(rs, re - rs);
      }
    }
  }
}

// The ranges of k_qpost_index, parted by position, to their records.
__global__ void k_qpost_place(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals,
                              int64_t n, const RankWord* __restrict__ rw, uint2* __restrict__ out) {
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = keys[x];
    const uint32_t p = (uint32_t)(k >> 32), rs = (uint32_t)k;
    const RankWord q = rw[p >> 5];
    out[q.before + __popc(q.bits & ((1u << (p & 31)) - 1u))] = make_uint2(rs, vals[x] - rs);
  }
}

// From this many records on the ranges (8 bytes each) and rank words are well
// past L2, and an entry's two random accesses go to device memory: parting
// the ranges by position first (one radix pass) makes them local: 119 M
// records 6.2 -> 2.7 ms, 24 M 0.77 -> 0.6 ms.
constexpr int64_t kPartRecords = int64_t(16) << 20;

// ------------------------------------------------------------- fast path --

template <int TPB, int LCAP, int GCAP, int SLOTS>
struct FastSmemT {
  uint32_t qkey[kQCap];
  uint32_t dh[kQCap];
  uint32_t pst[kQCap];
  uint32_t plen[kQCap];
  uint32_t pre[kQCap + 1];
  uint8_t dm[kQCap];
  uint32_t slots[SLOTS / 2];  // two 16-bit counters per word
  unsigned long long hits[LCAP];
  uint32_t glo[GCAP];     // dense groups: Jlo (clamped to >= 0), Jhi
  uint32_t ghi[GCAP];
  uint16_t cnt[TPB / 32][kQCap];  // one counter array per warp
  int tmp[33];
  int64_t win;
  int nhit, s, ovf, ng0, ng;
};

// Where a tier of the shared-memory path takes its windows from (all
// windows, or a list) and where it sends the windows it cannot hold.
struct TierIO {
  const uint32_t* in_list;        // nullptr: windows 0..nwin-1
  const unsigned int* in_count;
  uint32_t* out_list;
  unsigned int* out_count;
  unsigned int* next;             // work counter of this tier
  int stats;                      // count hits in the filter statistics
  // windows with more than hlim hits are handed over before their hits are
  // enumerated: to wide_list when set (the next larger shape), else to out_list
  uint32_t hlim = 0xFFFFFFFFu;
  uint32_t* wide_list = nullptr;
  unsigned int* wide_count = nullptr;
};

// (bin, o) counter slot of a hit in a direct-mapped table of mask+1 slots
__device__ __forceinline__ uint32_t slot_of(uint32_t t, uint32_t o, uint32_t mask) {
  return (((t >> kBinShift) << 1) | o) & mask;
}

__device__ __forceinline__ uint32_t slot_count(const uint32_t* slots, uint32_t s) {
  return (slots[s >> 1] >> ((s & 1) * 16)) & 0xFFFFu;
}

// Enumerates the window's hits: calls f(t, hid, o) for every posting of every
// kept hash with a compatible relative strand (self positions skipped).
template <typename Smem, typename F>
__device__ __forceinline__ void for_hits(const FArgs& a, const Smem& S, int64_t i, int H, F f) {
  const uint32_t tlo = first_useful(a, i);
  for (int e = threadIdx.x; e < H; e += blockDim.x) {
    int lo = 0, hi = S.s;  // list with pre[l] <= e < pre[l+1]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if ((int)S.pre[mid] <= e) lo = mid; else hi = mid;
    }
    const uint64_t r = __ldg(a.tsorted + S.pst[lo] + (uint32_t)(e - (int)S.pre[lo]));
    const uint32_t t = rec_pos(r), st = rec_strand(r);
    if (useless_hit(a, t, (uint32_t)i, tlo)) continue;
    const uint32_t qm = S.dm[lo];
    if ((qm >> st) & 1u) f(t, (uint32_t)lo, 0u);
    if ((qm >> (st ^ 1u)) & 1u) f(t, (uint32_t)lo, 1u);
  }
}

// One query window through a shared-memory tier: W_Q, the prefilter, the
// collected hits, dense groups and the exact sweep; a window the tier
// cannot hold goes to io.out_list (or io.wide_list).  Every thread of the
// block calls it.
template <int TPB, int LCAP, int GCAP, int SLOTS>
__device__ void fast_window(const FArgs& a, const TierIO& io,
                            FastSmemT<TPB, LCAP, GCAP, SLOTS>& S, int64_t wdx) {
  constexpr int kFThreads = TPB;
  constexpr int kLCap = LCAP;
  constexpr int kGCap = GCAP;
  const int64_t i = __ldcg(a.win_i + wdx);
  const uint32_t qa = __ldcg(a.win_qa + wdx), qb = __ldcg(a.win_qb + wdx);
  const int c = (int)(qb - qa);
  if (c == 0) return;
  if (c > kQCap) {
    if (threadIdx.x == 0) io.out_list[atomicAdd(io.out_count, 1u)] = (uint32_t)wdx;
    return;
  }
  for (int x = threadIdx.x; x < c; x += blockDim.x) {
    const uint64_t r = __ldcg(a.qrec + qa + x);
    S.qkey[x] = (rec_hash(r) << 1) | rec_strand(r);
  }
  __syncthreads();
  QBuild qb_;
  qb_.qkey = S.qkey;
  qb_.dh = S.dh;
  qb_.dm = S.dm;
  qb_.pst = S.pst;
  qb_.plen = S.plen;
  qb_.tmp = S.tmp;
  int64_t seq_lo = 0, seq_hi = 0;
  if (a.self_mode == 2) {
    const int sq = __ldcg(a.win_seq + wdx);
    seq_lo = a.tseq[sq];
    seq_hi = a.tseq[sq + 1];
  }
  const int s = build_wq(a, qb_, c, seq_lo, seq_hi);
  if (s == 0) return;
  // prefix of posting lengths (hit enumeration)
  if (threadIdx.x < 32) {
    uint32_t run = 0;
    for (int base = 0; base < s; base += 32) {
      const int x = base + threadIdx.x;
      const uint32_t v = x < s ? S.plen[x] : 0u;
      const uint32_t inc = warp_inclusive_sum(v);
      if (x < s) S.pre[x] = run + inc - v;
      run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (threadIdx.x == 0) S.pre[s] = run;
  }
  if (threadIdx.x == 0) {
    S.s = s;
    S.nhit = 0;
    S.ovf = 0;
  }
  __syncthreads();
  const uint32_t H = S.pre[s];
  if (H == 0) return;
  if (H > (uint32_t)kHMax || H > io.hlim) {
    if (threadIdx.x == 0) {
      if (H <= (uint32_t)kHMax && io.wide_list)
        io.wide_list[atomicAdd(io.wide_count, 1u)] = (uint32_t)wdx;
      else
        io.out_list[atomicAdd(io.out_count, 1u)] = (uint32_t)wdx;
    }
    return;
  }
  uint32_t nslots = kSlots;
  while (nslots < 4u * H && nslots < (uint32_t)SLOTS) nslots <<= 1;
  const uint32_t smask = nslots - 1;
  for (uint32_t x = threadIdx.x; x < nslots / 2; x += blockDim.x) S.slots[x] = 0;
  __syncthreads();
  const int m = a.mtab[s];
  // pass 1: (bin, o) counts
  for_hits(a, S, i, (int)H, [&](uint32_t t, uint32_t, uint32_t o) {
    const uint32_t sl = slot_of(t, o, smask);
    atomicAdd(&S.slots[sl >> 1], 1u << ((sl & 1) * 16));
  });
  __syncthreads();
  // pass 2: collect the hits of bins whose pair (b, b+1) or (b-1, b) may pass
  for_hits(a, S, i, (int)H, [&](uint32_t t, uint32_t hid, uint32_t o) {
    const uint32_t b = t >> kBinShift;
    const uint32_t c0 = slot_count(S.slots, slot_of(t, o, smask));
    const uint32_t cn = slot_count(S.slots, (((b + 1) << 1) | o) & smask);
    bool need = c0 + cn >= (uint32_t)m;
    if (!need && b > 0) {
      const uint32_t cp = slot_count(S.slots, (((b - 1) << 1) | o) & smask);
      need = cp + c0 >= (uint32_t)m;
    }
    if (need) {
      const int at = atomicAdd(&S.nhit, 1);
      if (at < kLCap)
        S.hits[at] = ((unsigned long long)o << 63) | ((unsigned long long)t << 20) | hid;
    }
  });
  __syncthreads();
  const int L = S.nhit;
  if (L > kLCap) {
    if (threadIdx.x == 0) io.out_list[atomicAdd(io.out_count, 1u)] = (uint32_t)wdx;
    return;
  }
  // statistics count the windows this tier finishes (each window once)
  if (L < m) {
    if (io.stats && threadIdx.x == 0) {
      atomicAdd(a.stats + 0, (unsigned long long)H);
      atomicAdd(a.stats + 1, (unsigned long long)L);
    }
    return;
  }
  const int np = next_pow2(L < 2 ? 2 : L);
  for (int x = L + threadIdx.x; x < np; x += blockDim.x) S.hits[x] = ~0ull;
  __syncthreads();
  block_sort(S.hits, np);
  // dense groups of both strands (warp 0), then one warp per group
  int split = 0;
  {
    // first hit with o = 1
    int lo2 = 0, hi2 = L;
    while (lo2 < hi2) {
      const int mid = (lo2 + hi2) >> 1;
      if ((S.hits[mid] >> 63) == 0) lo2 = mid + 1; else hi2 = mid;
    }
    split = lo2;
  }
  if (threadIdx.x < 32) {
    int ng = 0;
    for (int o = 0; o < 2; ++o) {
      const unsigned long long* base = S.hits + (o ? split : 0);
      const int64_t cnt = o ? L - split : split;
      find_groups(
          [&](int64_t x) {
            const unsigned long long h = base[x];
            return make_uint2((uint32_t)(h >> 20), (uint32_t)(h & 0xFFFFFu));
          },
          cnt, m, a.span, [&](bool mine, int64_t lo, int64_t hi) {
            const unsigned b = __ballot_sync(0xffffffffu, mine);
            const int g = ng + __popc(b & lanemask_lt());
            if (mine && g < kGCap) {
              S.glo[g] = (uint32_t)(lo < 0 ? 0 : lo);
              S.ghi[g] = (uint32_t)hi;
            }
            ng += __popc(b);
          });
      if (o == 0 && threadIdx.x == 0) S.ng0 = ng;
    }
    if (threadIdx.x == 0) S.ng = ng;
  }
  __syncthreads();
  const int ng = S.ng, ng0 = S.ng0;
  if (ng > kGCap) {
    if (threadIdx.x == 0) io.out_list[atomicAdd(io.out_count, 1u)] = (uint32_t)wdx;
    return;
  }
  if (io.stats && threadIdx.x == 0) {
    atomicAdd(a.stats + 0, (unsigned long long)H);
    atomicAdd(a.stats + 1, (unsigned long long)L);
  }
  {
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      WinInfo w;
      w.i = i;
      w.qseq = __ldcg(a.win_seq + wdx);
      w.s = s;
      w.m = m;
      for (int g = warp; g < ng; g += kFThreads / 32) {
        w.o = g < ng0 ? 0 : 1;
        const unsigned long long* base = S.hits + (w.o ? split : 0);
        const int64_t cnt = w.o ? L - split : split;
        sweep_group(a, w,
                    [&](int64_t x) {
                      const unsigned long long h = base[x];
                      return make_uint2((uint32_t)(h >> 20), (uint32_t)(h & 0xFFFFFu));
                    },
                    cnt, S.cnt[warp], (int64_t)S.glo[g], (int64_t)S.ghi[g]);
      }
    }
  }
}

// SLOTS is the largest (bin, o) table; a window uses the smallest power of
// two >= 4 H (at least 2,048 slots), so that aliasing stays rare however
// many hits the window has.
template <int TPB, int LCAP, int GCAP, int SLOTS>
__global__ void __launch_bounds__(TPB) k_filter_fast(FArgs a, TierIO io) {
  using FastSmem = FastSmemT<TPB, LCAP, GCAP, SLOTS>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FastSmem& S = *reinterpret_cast<FastSmem*>(smem_raw);
  for (int x = threadIdx.x; x < kQCap * (TPB / 32); x += blockDim.x) (&S.cnt[0][0])[x] = 0;
  const int64_t count = io.in_list ? (int64_t)*io.in_count : a.nwin;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const int64_t k = atomicAdd(io.next, 1u);
      S.win = k < count ? (io.in_list ? (int64_t)io.in_list[k] : k) : -1;
    }
    __syncthreads();
    const int64_t wdx = S.win;
    if (wdx < 0) break;
    fast_window<TPB, LCAP, GCAP, SLOTS>(a, io, S, wdx);
  }
}

// ------------------------------------------------------------- warp tier --
//
// Small windows (at most 2,048 posting entries and 128 collected hits, or 256
// in the form for many records) by one warp each, no block barriers:
//   1. every posting of every query record is counted into 8-bit (bin, o)
//      counters, without building W_Q first: a hash that occurs twice in the
//      window only counts too much.  The number of distinct hashes is bounded
//      from below by the bits they set in a 2,048-bit map, and with it m.
//      When no two adjacent bins reach that m the window is done: most
//      windows end here;
//   2. the others build W_Q in a hash table (exact s and m; the table's slot
//      is a hash's id) and collect the hits of the bins whose pair can pass;
//   3. the collected hits are sorted by (o, t) in registers, and the runs of
//      each strand come from its events: the hits of one hash at most span + 1
//      apart keep it in the target window over one stretch of starts, so only
//      a stretch's first hit enters and only its last one leaves.  The shared
//      count after an event is the number of enters up to it less the number
//      of leaves, found by rank (a binary search) for all events at once;
//      a run starts where it first reaches m and ends where it falls below.
// Windows past a limit go to the next tier.
//
// Bound by instruction issue and, as a window's path is long and the warps
// of an SM are all at different places of it, by the instruction cache: sorts
// unrolled in place, or four chunks of postings in flight, made it slower
// (13.5 -> 18.8 ms on the batch below; one to three in flight in a loop of one
// copy 8.2 -> 8.4 to 8.9), and a separate small kernel for step 1 gained 5%
// there and lost 16% on an assembly.  The form that built W_Q for
// every window, looked at the hits before the window too, searched the
// posting lists per hit and swept groups with one lane took about 4,600
// instructions a window: 4.7 M windows of a 200-genome batch 21.7 -> 7.0 ms
// (tier 1 over the windows handed on 3.9 -> 0.2 ms), a 240 Mbp assembly 10.8
// -> 3.0 ms.  Of that the sort by the number of hits (32, 64, 128) gave 0.5 ms
// on the batch, and room for 128 collected hits instead of 256, which makes
// 32 warps per SM of 28, 0.7 more; 2,048 counters and 36 warps gave 0.4 more
// there and cost 0.5 on the assembly (more windows look as if they passed).

constexpr int kWWarps = 4;

// QC: query records, SLOTS: 8-bit (bin, o) counters, WL: collected hits, WH:
// posting entries, MINB: CTAs per SM.
template <int QC_, int SLOTS_, int WL_, int WH_, int MINB_>
struct WindowShape {
  static constexpr int QC = QC_, SLOTS = SLOTS_, WL = WL_, WH = WH_, MINB = MINB_;
  static constexpr int TS = 2 * QC;  // W_Q table slots
  static_assert(WH / 32 >= 64, "the map of hashes lies over the list starts");
  static_assert(TS * 4 <= WL * 8, "W_Q's table lies over the hits");
  static_assert(WL * 16 <= SLOTS, "the strands' events lie over the counters");
};
using WarpSparse = WindowShape<128, 4096, 128, 2048, 8>;
using WarpDense = WindowShape<256, 4096, 256, 2048, 5>;

template <typename W>
struct WindowSmemT {
  uint32_t table[W::SLOTS / 4];       // counters; then the strands' events
  uint2 lists[W::QC];                 // posting lists; then per-hash places
  unsigned long long hits[W::WL];     // W_Q's hash table; then the collected hits
  uint32_t starts[W::WH / 32];        // map of hashes; then bit e: a list starts at hit e
  uint32_t strands[W::TS / 16];       // W_Q's strands, two bits per table slot
};

// Sorts n 64-bit keys in shared memory (n <= 32 * NR) through registers.
// The stages are loops and not unrolled: the kernel around it is bound by its
// instruction cache when they are.
template <int NR>
__device__ __noinline__ void warp_sort_hits(unsigned long long* v, int n) {
  const int lane = lane_id();
  unsigned long long r[NR];
#pragma unroll
  for (int x = 0; x < NR; ++x) {
    const int at = x * 32 + lane;
    r[x] = at < n ? v[at] : ~0ull;
  }
#pragma unroll 1
  for (int size = 2; size <= 32 * NR; size <<= 1) {
#pragma unroll 1
    for (int stride = size >> 1; stride >= NR; stride >>= 1) {
      const bool keep_min = (((lane * NR) & size) == 0) == ((lane & (stride / NR)) == 0);
#pragma unroll
      for (int x = 0; x < NR; ++x) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, r[x], stride / NR);
        if ((o < r[x]) == keep_min) r[x] = o;
      }
    }
#pragma unroll
    for (int stride = NR / 2; stride > 0; stride >>= 1) {
      if (stride >= size) continue;
#pragma unroll
      for (int x = 0; x < NR; ++x) {
        if (x & stride) continue;
        const bool asc = ((lane * NR + x) & size) == 0;
        const unsigned long long p = r[x], q = r[x | stride];
        if ((p > q) == asc) {
          r[x] = q;
          r[x | stride] = p;
        }
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int x = 0; x < NR; ++x) v[lane * NR + x] = r[x];
  __syncwarp();
}

// First place in v[0..n) whose value is >= x.
__device__ __forceinline__ int lb_u32(const uint32_t* v, int n, uint32_t x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (v[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// hits: o << 63 | t << 20 | hid, with these flags once a strand's stretches are known
constexpr unsigned long long kHitNoEnter = 1ull << 52, kHitNoLeave = 1ull << 53;
__device__ __forceinline__ uint32_t hit_pos(unsigned long long h) { return (uint32_t)(h >> 20); }

// Where a strand's events go (shared memory of one warp).
struct EventMem {
  uint32_t* enter;   // sorted target positions; a window [j, j + span] holds them from j + span on
  uint32_t* leave;   // first j + span past the stretch
  uint16_t* val;     // shared count at each enter
  uint32_t* end;     // per run: its last j + span
  uint16_t* first;   // per run: the enter that starts it
  uint16_t* last;    // per hash id: its last hit
  int nlast;         // hash ids
};

// The places for a strand of n hits: 16 n bytes at `words`, nlast entries at `last`.
__device__ __forceinline__ EventMem event_mem(uint32_t* words, int n, uint16_t* last, int nlast) {
  EventMem M;
  M.enter = words;
  M.leave = words + n;
  M.end = words + 2 * n;
  M.val = reinterpret_cast<uint16_t*>(words + 3 * n);
  M.first = M.val + n;
  M.last = last;
  M.nlast = nlast;
  return M;
}

// Whether two adjacent bins that begin in word x of the counter table reach m
// on a strand: the word holds bins 2x and 2x + 1, both strands; the bins wrap
// around after nw words.
__device__ __forceinline__ bool word_passes(const uint32_t* table, int x, int nw, uint32_t m) {
  const uint32_t c0 = table[x], c1 = table[(x + 1) & (nw - 1)];
  const uint32_t s0 = c0 & 0x00FF00FFu, s1 = (c0 >> 8) & 0x00FF00FFu;  // strands 0 and 1
  const uint32_t n0 = c1 & 0x00FF00FFu, n1 = (c1 >> 8) & 0x00FF00FFu;
  return (s0 & 0xFFFFu) + (s0 >> 16) >= m || (s1 & 0xFFFFu) + (s1 >> 16) >= m ||
         (s0 >> 16) + (n0 & 0xFFFFu) >= m || (s1 >> 16) + (n1 & 0xFFFFu) >= m;
}

// Emits the run of starts whose j + span are first..last of one strand (ne
// enters with their counts, nl leaves), split by target sequence and the
// validity rules.  by_lane: each lane has a run of its own; else the warp has
// one run and shares its enters out.
__device__ __forceinline__ void emit_valid(const FArgs& a, const WinInfo& w, const uint32_t* enter,
                                           const uint16_t* val, int ne, const uint32_t* leave, int nl,
                                           uint32_t first, uint32_t last, bool by_lane) {
  const int lane = lane_id();
  const uint32_t span = (uint32_t)a.span;
  const int64_t lo = (int64_t)first - span, hi = (int64_t)last - span;
  int64_t x = lo < 0 ? 0 : lo;
  for (int u = seq_of(a.tseq, a.ntseq, x); u < a.ntseq && x <= hi; ++u) {
    const int64_t st = a.tseq[u], en = a.tseq[u + 1];
    bool ok = true;
    int64_t from = st;
    if (a.self_mode) {
      if (u < w.qseq) ok = false;
      else if (u == w.qseq) from = max(from, w.i + a.n - a.overlap);
      else if (a.self_mode == 2) ok = false;  // independent genomes
    }
    const int64_t vlo = max(x, from), vhi = min(hi, en - a.n);
    x = en;
    if (!ok || vlo > vhi) continue;
    // the largest count on [vlo, vhi]: at vlo, or at an enter after it
    const uint32_t j0 = (uint32_t)(vlo + span), j1 = (uint32_t)(vhi + span);
    int e = lb_u32(enter, ne, j0);
    e += e < ne && enter[e] == j0 ? 1 : 0;
    int l = lb_u32(leave, nl, j0);
    l += l < nl && leave[l] == j0 ? 1 : 0;
    uint32_t best = 0;  // count, then the earliest
    for (int y = by_lane ? e : e + lane; y < ne && enter[y] <= j1; y += by_lane ? 1 : 32)
      best = max(best, ((uint32_t)val[y] << 16) | (uint32_t)(0xFFFF - y));
    if (!by_lane) best = __reduce_max_sync(0xffffffffu, best);
    RunState run;
    run.open = true;
    run.ja = vlo;
    run.jb = vhi;
    run.mx = e - l;
    run.jmx = vlo;
    if ((int)(best >> 16) > run.mx) {
      run.mx = (int)(best >> 16);
      run.jmx = (int64_t)enter[0xFFFF - (best & 0xFFFFu)] - span;
    }
    if (by_lane || lane == 0) emit_run(a, w, run);
  }
}

// The runs of one strand from its n collected hits, sorted by t.
// The whole warp calls.
__device__ __noinline__ void strand_runs(const FArgs& a, const WinInfo& w, unsigned long long* hits, int n,
                            const EventMem& M) {
  const int lane = lane_id();
  const uint32_t span = (uint32_t)a.span;
  for (int x = lane; x < M.nlast / 2; x += 32) reinterpret_cast<uint32_t*>(M.last)[x] = 0xFFFFFFFFu;
  __syncwarp();
  // stretches: a hit joined to the previous one of its hash does not enter,
  // and that one does not leave
  for (int base = 0; base < n; base += 32) {
    const int x = base + lane;
    const bool ok = x < n;
    const unsigned long long h = ok ? hits[x] : 0ull;
    const uint32_t t = hit_pos(h), id = (uint32_t)h & 0xFFFFFu;
    const unsigned peers = __match_any_sync(0xffffffffu, ok ? id : (0x80000000u | (uint32_t)lane));
    const unsigned lower = peers & lanemask_lt();
    int p = -1;
    if (ok) {
      if (lower) p = base + 31 - __clz(lower);
      else if (M.last[id] != 0xFFFFu) p = M.last[id];
    }
    const bool joined = p >= 0 && t - hit_pos(hits[p]) <= span + 1u;
    __syncwarp();
    if (joined) {
      atomicOr(reinterpret_cast<unsigned int*>(hits + x) + 1, (unsigned int)(kHitNoEnter >> 32));
      atomicOr(reinterpret_cast<unsigned int*>(hits + p) + 1, (unsigned int)(kHitNoLeave >> 32));
    }
    if (ok && (peers >> lane) == 1u) M.last[id] = (uint16_t)x;
    __syncwarp();
  }
  int ne = 0, nl = 0;
  for (int base = 0; base < n; base += 32) {
    const int x = base + lane;
    const unsigned long long h = x < n ? hits[x] : (kHitNoEnter | kHitNoLeave);
    const uint32_t t = hit_pos(h);
    const unsigned be = __ballot_sync(0xffffffffu, !(h & kHitNoEnter));
    const unsigned bl = __ballot_sync(0xffffffffu, !(h & kHitNoLeave));
    if (!(h & kHitNoEnter)) M.enter[ne + __popc(be & lanemask_lt())] = t;
    // t + 1 + span, short of wrapping (no window starts that far)
    if (!(h & kHitNoLeave))
      M.leave[nl + __popc(bl & lanemask_lt())] = t < 0xFFFFFFFFu - span - 1u ? t + span + 1u : 0xFFFFFFFFu;
    ne += __popc(be);
    nl += __popc(bl);
  }
  __syncwarp();
  const int m = w.m;
  int nr = 0, nend = 0;
  for (int base = 0; base < ne; base += 32) {
    const int x = base + lane;
    bool start = false;
    if (x < ne) {
      const uint32_t j = M.enter[x];
      const int before = lb_u32(M.leave, nl, j);             // leaves before j
      const int upto = before + (before < nl && M.leave[before] == j ? 1 : 0);
      const int v = x + 1 - upto;
      M.val[x] = (uint16_t)v;
      start = v >= m && x - before < m;
    }
    const unsigned b = __ballot_sync(0xffffffffu, start);
    if (start) M.first[nr + __popc(b & lanemask_lt())] = (uint16_t)x;
    nr += __popc(b);
  }
  if (nr == 0) return;
  for (int base = 0; base < nl; base += 32) {
    const int x = base + lane;
    bool stop = false;
    uint32_t j = 0;
    if (x < nl) {
      j = M.leave[x];
      const int before = lb_u32(M.enter, ne, j);
      const int upto = before + (before < ne && M.enter[before] == j ? 1 : 0);
      stop = upto - (x + 1) < m && before - x >= m;
    }
    const unsigned b = __ballot_sync(0xffffffffu, stop);
    if (stop) M.end[nend + __popc(b & lanemask_lt())] = j - 1u;
    nend += __popc(b);
  }
  __syncwarp();
  // every run starts and ends once, in order.  Many runs: one per lane; few:
  // the warp takes them in turn and shares their enters out.
  const bool by_lane = nr >= 8;
  for (int r = by_lane ? lane : 0; r < nr; r += by_lane ? 32 : 1)
    emit_valid(a, w, M.enter, M.val, ne, M.leave, nl, M.enter[M.first[r]], M.end[r], by_lane);
}

// posting_window by value (out of line, see warp_sort_hits).
__device__ __noinline__ uint2 posting_window_of(const uint64_t* idx, const uint32_t* samp, uint32_t st,
                                                uint32_t len, int64_t lo, int64_t hi) {
  posting_window(idx, samp, &st, &len, lo, hi);
  return make_uint2(st, len);
}

template <typename W>
__global__ void __launch_bounds__(32 * kWWarps, W::MINB) k_filter_warp(FArgs a, TierIO io,
                                                                     int per_grab) {
  constexpr int QC = W::QC, TS = W::TS, kWL = W::WL, kWH = W::WH, kWSlots = W::SLOTS;
  constexpr int NC = QC / 32;    // records per lane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  WindowSmemT<W>& S = reinterpret_cast<WindowSmemT<W>*>(smem_raw)[warp];
  const uint32_t lt = lanemask_lt();
  const int64_t count = io.in_list ? (int64_t)*io.in_count : a.nwin;
  unsigned long long n_hits = 0, n_collected = 0;
  while (true) {
    // several windows at a time: they share query records, and the work
    // counter is one word for the whole grid
    int64_t k0 = 0;
    if (lane == 0) k0 = (int64_t)atomicAdd(io.next, (unsigned int)per_grab);
    k0 = __shfl_sync(0xffffffffu, k0, 0);
    if (k0 >= count) break;
    const int nk = (int)min((int64_t)per_grab, count - k0);
    uint32_t l_w = 0, l_i = 0, l_qa = 0, l_qb = 0;
    if (lane < nk) {
      l_w = io.in_list ? io.in_list[k0 + lane] : (uint32_t)(k0 + lane);
      l_i = a.win_i[l_w];
      l_qa = a.win_qa[l_w];
      l_qb = a.win_qb[l_w];
    }
    {
      // windows of too many records go on together: side by side in the list
      // they share records and postings in the tiers after this one
      const bool over = l_qb - l_qa > (uint32_t)QC;
      const unsigned bo = __ballot_sync(0xffffffffu, over);
      if (bo) {
        unsigned int to = 0;
        if (lane == 0) to = atomicAdd(io.out_count, (unsigned int)__popc(bo));
        to = __shfl_sync(0xffffffffu, to, 0);
        if (over) io.out_list[to + __popc(bo & lt)] = l_w;
      }
    }
    for (int kk = 0; kk < nk; ++kk) {
      const uint32_t wdx = __shfl_sync(0xffffffffu, l_w, kk), i = __shfl_sync(0xffffffffu, l_i, kk);
      const uint32_t qa = __shfl_sync(0xffffffffu, l_qa, kk);
      const int c = (int)(__shfl_sync(0xffffffffu, l_qb, kk) - qa);
      if (c == 0 || c > QC) continue;
      auto hand_over = [&](bool wide) {
        if (lane != 0) return;
        if (wide && io.wide_list) io.wide_list[atomicAdd(io.wide_count, 1u)] = wdx;
        else io.out_list[atomicAdd(io.out_count, 1u)] = wdx;
      };
      __syncwarp();  // the previous window's shared memory is free
      S.starts[lane] = 0u;
      S.starts[lane + 32] = 0u;
      __syncwarp();
      // ---- the records: hash and strand, posting range
      uint32_t key[NC], st[NC], len[NC];
      unsigned kept = 0;
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) {
        const int x = ch * 32 + lane;
        key[ch] = st[ch] = len[ch] = 0;
        if (x < c) {
          const uint64_t r = __ldg(a.qrec + qa + x);
          const uint32_t h = rec_hash(r);
          key[ch] = (h << 1) | rec_strand(r);
          if (a.qpost) {
            const uint2 pp = __ldg(a.qpost + qa + x);
            st[ch] = pp.x;
            len[ch] = pp.y;
            if (pp.x != kNone) kept |= 1u << ch;
          } else {
            st[ch] = a.toff[h];
            len[ch] = a.toff[h + 1] - st[ch];
            if (!(a.max_occ > 0 && (int)len[ch] > a.max_occ)) {
              kept |= 1u << ch;
              if (a.self_mode == 2) {
                const int sq = a.win_seq[wdx];
                const uint2 pw = posting_window_of(a.tsorted, a.tsamp, st[ch], len[ch], a.tseq[sq], a.tseq[sq + 1]);
                st[ch] = pw.x;
                len[ch] = pw.y;
              }
            }
          }
          if ((kept >> ch) & 1u) {
            const uint32_t g = (h * 0x9E3779B1u) >> 21;
            atomicOr(&S.starts[g >> 5], 1u << (g & 31));
          } else {
            len[ch] = 0;
          }
        }
      }
      __syncwarp();
      const int s_least = (int)__reduce_add_sync(0xffffffffu, __popc(S.starts[lane]) + __popc(S.starts[lane + 32]));
      if (s_least == 0) continue;  // every hash passes max_occ
      // ---- posting lists with an entry, one after another
      uint32_t H = 0;
      uint32_t at[NC];
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) {
        at[ch] = 0;
        if (ch * 32 >= c) break;
        const uint32_t v = min(len[ch], 1u << 20);  // no sum can wrap
        const uint32_t inc = warp_inclusive_sum(v);
        at[ch] = H + inc - v;
        H += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (H == 0) continue;
      if (H > io.hlim || H > (uint32_t)kWH) {
        hand_over(true);
        continue;
      }
      __syncwarp();
      S.starts[lane] = 0u;
      S.starts[lane + 32] = 0u;
      uint32_t nslots = 512;
      while (nslots < 4u * H && nslots < (uint32_t)kWSlots) nslots <<= 1;
      const uint32_t smask = nslots - 1;
      for (int x = lane; x < (int)nslots / 16; x += 32)
        reinterpret_cast<uint4*>(S.table)[x] = make_uint4(0, 0, 0, 0);
      __syncwarp();
      int nlist = 0;
      uint32_t lid[NC];
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) {
        lid[ch] = 0;
        if (ch * 32 >= c) break;
        const unsigned some = __ballot_sync(0xffffffffu, len[ch] > 0);
        if (len[ch] > 0) {
          lid[ch] = nlist + __popc(some & lt);
          S.lists[lid[ch]] = make_uint2(st[ch] - at[ch], key[ch] & 1u);
          atomicOr(&S.starts[at[ch] >> 5], 1u << (at[ch] & 31));
        }
        nlist += __popc(some);
      }
      __syncwarp();
      // hit e lies in the last list that starts at or before it; f is called
      // by every lane (on: the lane has a hit that a target window can use)
      const uint32_t tlo = first_useful(a, i);
      auto each_hit = [&](auto f) {
        int lists_before = -1;
        for (uint32_t base = 0; base < H; base += 32) {
          const unsigned sb = S.starts[base >> 5];
          const int li = lists_before + __popc(sb & (lt | (1u << lane)));
          lists_before += __popc(sb);
          bool on = base + lane < H;
          uint32_t t = 0, o = 0, y = 0;
          if (on) {
            const uint2 list = S.lists[li];
            const uint64_t r = __ldg(a.tsorted + (list.x + base + lane));
            t = rec_pos(r);
            y = list.y;
            o = (y ^ rec_strand(r)) & 1u;
            on = !useless_hit(a, t, i, tlo);
          }
          f(on, t, o, y);
        }
      };
      uint32_t most = 0;  // the largest counter
      each_hit([&](bool on, uint32_t t, uint32_t o, uint32_t) {
        if (!on) return;
        const uint32_t sl = slot_of(t, o, smask), sh = (sl & 3u) * 8u;
        const uint32_t was = (atomicAdd(&S.table[sl >> 2], 1u << sh) >> sh) & 0xFFu;
        most = max(most, was + 1u);
      });
      most = __reduce_max_sync(0xffffffffu, most);
      if (most > 255u) {  // a counter ran into its neighbour
        hand_over(false);
        continue;
      }
      __syncwarp();
      {
        const uint32_t m = (uint32_t)a.mtab[s_least];
        bool pass = 2u * most >= m;
        if (pass) {
          pass = false;
          const int nw = (int)nslots / 4;
          for (int x = lane; x < nw; x += 32) pass |= word_passes(S.table, x, nw, m);
        }
        if (!__any_sync(0xffffffffu, pass)) {
          n_hits += H;
          continue;
        }
      }
      // ---- W_Q: a hash's id is its slot; a record whose hash and strand are
      // in already adds nothing
      uint32_t* tab = reinterpret_cast<uint32_t*>(S.hits);
      for (int x = lane; x < TS / 4; x += 32) reinterpret_cast<uint4*>(tab)[x] = make_uint4(0, 0, 0, 0);
      if (lane < TS / 16) S.strands[lane] = 0u;
      __syncwarp();
      int fresh = 0;
#pragma unroll
      for (int ch = 0; ch < NC; ++ch) {
        if ((kept >> ch) & 1u) {
          const uint32_t h = key[ch] >> 1;
          uint32_t slot = (h * 0x9E3779B1u) >> (QC == 128 ? 24 : 23);
          while (true) {  // at most QC keys in TS slots: a free slot is always found
            const uint32_t old = atomicCAS(&tab[slot], 0u, h + 1u);
            if (old == 0u) ++fresh;
            if (old == 0u || old == h + 1u) break;
            slot = (slot + 1u) & (uint32_t)(TS - 1);
          }
          const uint32_t bit = 1u << ((slot & 15) * 2 + (key[ch] & 1u));
          const bool twice = (atomicOr(&S.strands[slot >> 4], bit) & bit) != 0u;
          if (len[ch] > 0) S.lists[lid[ch]].y = (key[ch] & 1u) | (twice ? 2u : 0u) | (slot << 2);
        }
      }
      const int s = (int)__reduce_add_sync(0xffffffffu, fresh);
      const int m = a.mtab[s];
      __syncwarp();
      int L = 0;
      each_hit([&](bool on, uint32_t t, uint32_t o, uint32_t y) {
        bool need = false;
        if (on && !(y & 2u)) {
          const uint32_t b = t >> kBinShift;
          auto cnt = [&](uint32_t bin) {
            const uint32_t sl = ((bin << 1) | o) & smask;
            return (S.table[sl >> 2] >> ((sl & 3u) * 8u)) & 0xFFu;
          };
          const uint32_t c0 = cnt(b);
          need = c0 + cnt(b + 1) >= (uint32_t)m || (b > 0 && c0 + cnt(b - 1) >= (uint32_t)m);
        }
        const unsigned bn = __ballot_sync(0xffffffffu, need);
        const int to = L + __popc(bn & lt);
        if (need && to < kWL)
          S.hits[to] = ((unsigned long long)o << 63) | ((unsigned long long)t << 20) | (y >> 2);
        L += __popc(bn);
      });
      __syncwarp();
      if (L > kWL) {
        hand_over(false);
        continue;
      }
      n_hits += H;
      n_collected += L;
      if (L < m) continue;
      if (L <= 32) warp_sort_hits<1>(S.hits, L);
      else if (L <= 64) warp_sort_hits<2>(S.hits, L);
      else if (kWL <= 128 || L <= 128) warp_sort_hits<4>(S.hits, L);
      else warp_sort_hits<8>(S.hits, L);
      int split = 0;  // first hit with o = 1
      for (int base = 0; base < L; base += 32)
        split += __popc(__ballot_sync(0xffffffffu, base + lane < L && (S.hits[base + lane] >> 63) == 0));
      const EventMem M = event_mem(S.table, L, reinterpret_cast<uint16_t*>(S.lists), TS);
      WinInfo w;
      w.i = i;
      w.qseq = a.win_seq[wdx];
      w.s = s;
      w.m = m;
#pragma unroll 1
      for (int o = 0; o < 2; ++o) {
        const int n = o ? L - split : split;
        if (n < m) continue;
        w.o = o;
        strand_runs(a, w, S.hits + (o ? split : 0), n, M);
        __syncwarp();
      }
    }
  }
  if (io.stats && lane == 0) {
    if (n_hits) atomicAdd(a.stats + 0, n_hits);
    if (n_collected) atomicAdd(a.stats + 1, n_collected);
  }
}

template <typename W>
int launch_warp_tier_as(sedef_ctx* ctx, const FArgs& a, const TierIO& io, int64_t max_windows,
                        const char* name) {
  const size_t sm = sizeof(WindowSmemT<W>) * kWWarps;
  SEDEF_TRY(ensure_smem_attr((const void*)k_filter_warp<W>, sm));
  int per_sm = 0;
  SEDEF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_warp<W>, 32 * kWWarps, sm));
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)ctx_sm_count(ctx) * per_sm;
  // a few windows: one per warp; many: eight at a time
  int64_t grab = max_windows / (grid * kWWarps * 4);
  grab = grab < 1 ? 1 : (grab > 8 ? 8 : grab);
  const int64_t need = (max_windows + kWWarps - 1) / kWWarps;
  if (grid > need) grid = need;
  if (grid < 1) grid = 1;
  SEDEF_KERNEL(ctx, name,
               k_filter_warp<W><<<(int)grid, 32 * kWWarps, sm, ctx_stream(ctx)>>>(a, io, (int)grab));
  return SEDEF_OK;
}

// w: winnowing window.  A query window holds 2 / (w + 1) of its starts as
// records on average; the shape for 256 records has five CTAs per SM where
// the one for 128 has eight, so it is taken only where 128 would not do.
int launch_warp_tier(sedef_ctx* ctx, const FArgs& a, const TierIO& io, int64_t max_windows, int w,
                     const char* name) {
  if (1.35 * 2.0 * (a.span + 1) / (w + 1) <= 128.0)
    return launch_warp_tier_as<WarpSparse>(ctx, a, io, max_windows, name);
  return launch_warp_tier_as<WarpDense>(ctx, a, io, max_windows, name);
}

// -------------------------------------------------------------- CTA tier --
//
// A CTA per window, for windows with more records, posting entries or
// collected hits than a warp keeps:
//   1. W_Q in a hash table, a record per thread (a hash's id is its slot);
//   2. the posting chunks, a contiguous stretch for each warp and four chunks
//      in flight, counted into 8-bit (bin, o) counters; each hit's counter is
//      kept (16 bits);
//   3. the counters become a bit each: reaches m with a neighbour.  The sum of
//      all counters tells whether one ran over;
//   4. the kept counters are looked up in those bits and the records of the
//      few that are set are read again;
//   5. those hits are sorted by chunks in registers, merged by rank;
//   6. the runs come from the strands' events as in the warp tier, with every
//      step shared out to all warps.
//
// Bound by instruction issue (two thirds of the slots) and by latency: some
// 4,000 cycles until a window's posting ranges are known, then steps that a
// barrier ends.  A window of 10 k entries and 800 collected hits against a
// 3.1 Gbp index takes 86 k cycles with four CTAs on an SM: postings 25 k,
// second look 18 k, sort 14 k, runs 20 k.  46 k windows against that index
// took 8.3 ms in a form that sorted the records (28 barriers), searched the
// lists for each hit and swept groups one by one; 3.1 with this one's first
// form, which read every posting twice (without keeping the counters: the
// narrow shape 2.5 ms instead of 2.3), sorted with a barrier per stage and
// left the runs of a strand to one warp; 2.3 now.  A 240 Mbp assembly's 79 k:
// 3.5 -> 2.4 ms, and the windows that go on to the broad and the deep shape,
// with twice the room for hits in the same memory, 2.0 -> 0.45 ms.  Six or
// eight chunks in flight gave the same.

// SLOTS: 8-bit (bin, o) counters, WL: collected hits, WH: posting entries,
// WC: posting entries whose counter is kept for the second look, TPB:
// threads, MINB: CTAs per SM.
template <int SLOTS_, int WL_, int WH_, int WC_, int TPB_, int MINB_>
struct CtaShape {
  static constexpr int QC = 256;      // query records
  static constexpr int TS = 2 * QC;   // W_Q table slots
  static constexpr int SLOTS = SLOTS_, WL = WL_, WH = WH_, WC = WC_, TPB = TPB_, MINB = MINB_;
  static constexpr int WARPS = TPB / 32;
  static constexpr int BUF = SLOTS > 8 * WL ? SLOTS : 8 * WL;  // bytes of the counters' array
  static constexpr int KEEP = 2 * WC > 8 * WL ? 2 * WC : 8 * WL;  // bytes of the kept counters' array
  static_assert(TPB >= QC && WL % 256 == 0 && WL < 0xFFFF, "a record per thread; 16-bit hit numbers");
  static_assert((SLOTS <= 32768 || WC == 0) && WH <= 65536 && WC % 32 == 0,
                "16 bits for a counter, with one value to spare, and for an entry");
  static_assert(TS * 4 <= WL * 8, "W_Q's table lies over the hits");
  static_assert(SLOTS / 8 + 4 * WL <= BUF, "the needed entries lie behind the counters' bits");
  static_assert(WARPS * TS * 4 <= 8 * WL, "the warps' last hits per hash lie over the events");
  static_assert(WH / 32 >= 2 * (WL / 32), "the event bits lie over the list starts");
};
using CtaNarrow = CtaShape<16384, 2048, 16384, 16384, 256, 4>;
using CtaBroad = CtaShape<32768, 4096, 65536, 16384, 256, 3>;
// One CTA per SM, the smaller one beside the serving kernel: 64 registers per
// thread, so that both kernels' registers fit.
using CtaDeep = CtaShape<65536, 12288, 65536, 0, 512, 2>;
using CtaMid = CtaShape<65536, 8192, 65536, 0, 512, 2>;

template <typename W>
struct CtaSmemT {
  uint32_t table[W::BUF / 4];         // counters; a bit per counter and the needed entries; hits or events
  // W_Q's hash table; the kept counters; then hits or events
  unsigned long long hits[W::KEEP / 8];
  uint2 lists[W::QC];                 // posting lists
  uint32_t starts[W::WH / 32];        // bit e: a list starts at hit e; later event bits
  uint32_t strands[W::TS / 16];       // W_Q's strands, two bits per table slot
  uint32_t sum[4][W::WARPS];
  uint32_t uncounted;                 // hits less counters
  int nhit;
  int64_t win;
};

// Sorts the n distinct keys v[0..n) by the whole CTA: a chunk per warp in
// registers, then merged in pairs by rank, between v and w; returns where
// they end up.  Both hold n rounded up to 256.
template <typename W>
__device__ unsigned long long* cta_sort_hits(unsigned long long* v, unsigned long long* w, int n) {
  const int warp = threadIdx.x >> 5;
  int chunk = 32;
  while (chunk < 256 && chunk * W::WARPS < n) chunk <<= 1;
  for (int from = warp * chunk; from < n; from += W::WARPS * chunk) {
    const int len = min(chunk, n - from);
    if (chunk == 32) warp_sort_hits<1>(v + from, len);
    else if (chunk == 64) warp_sort_hits<2>(v + from, len);
    else if (chunk == 128) warp_sort_hits<4>(v + from, len);
    else warp_sort_hits<8>(v + from, len);
  }
  __syncthreads();
  for (int width = chunk; width < n; width <<= 1) {
    for (int x = threadIdx.x; x < n; x += W::TPB) {
      const unsigned long long key = v[x];
      const int other = (x & ~(width - 1)) ^ width;  // the chunk this one merges with
      int lo = 0, hi = min(width, n - other);
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (v[other + mid] < key) lo = mid + 1; else hi = mid;
      }
      w[(x & ~(2 * width - 1)) + (x & (width - 1)) + lo] = key;
    }
    __syncthreads();
    unsigned long long* const t = v;
    v = w;
    w = t;
  }
  return v;
}

// strand_runs for both strands of a window by the whole CTA: each warp takes
// an equal stretch of the hits (then of the events), whose places come from
// the counts of the stretches before.  hits: n sorted hits; events: 8 n
// bytes for enters and leaves; what follows lies over the hits.
template <typename W>
__device__ void cta_runs(const FArgs& a, WinInfo w, unsigned long long* hits, uint32_t* events, int n,
                         CtaSmemT<W>& S) {
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  const uint32_t lt = lanemask_lt();
  const uint32_t span = (uint32_t)a.span;
  uint32_t* bits0 = S.starts;                // per word of 32 hits or events
  uint32_t* bits1 = S.starts + W::WL / 32;
  auto mine = [&](int count, int* from, int* to) {
    const int words = (count + 31) >> 5, per = (words + W::WARPS - 1) / W::WARPS;
    *from = min(warp * per, words);
    *to = min(*from + per, words);
  };
  // sum of row r before this warp, and in all
  auto places = [&](int r, int* before, int* total) {
    const uint32_t v = lane < W::WARPS ? S.sum[r][lane] : 0u;
    *before = (int)__reduce_add_sync(0xffffffffu, lane < warp ? v : 0u);
    *total = (int)__reduce_add_sync(0xffffffffu, v);
  };
  int w0, w1;
  // ---- stretches: a hit joined to the previous one of its hash does not
  // enter, and that one does not leave; first within this warp's hits
  mine(n, &w0, &w1);
  uint16_t* last = reinterpret_cast<uint16_t*>(events) + warp * (2 * W::TS);
  for (int x = lane; x < W::TS; x += 32) reinterpret_cast<uint32_t*>(last)[x] = 0xFFFFFFFFu;
  __syncwarp();
  auto join = [&](int p, int x, uint32_t t) {
    if (t - hit_pos(hits[p]) > span + 1u) return;
    atomicOr(reinterpret_cast<unsigned int*>(hits + x) + 1, (unsigned int)(kHitNoEnter >> 32));
    atomicOr(reinterpret_cast<unsigned int*>(hits + p) + 1, (unsigned int)(kHitNoLeave >> 32));
  };
  // strand and hash of a hit
  auto key_of = [](unsigned long long h) { return ((uint32_t)h & 0xFFFFFu) | ((uint32_t)(h >> 63) * W::TS); };
  for (int wd = w0; wd < w1; ++wd) {
    const int x = wd * 32 + lane;
    const bool ok = x < n;
    const unsigned long long h = ok ? hits[x] : 0ull;
    const uint32_t key = key_of(h);
    const unsigned peers = __match_any_sync(0xffffffffu, ok ? key : (0x80000000u | (uint32_t)lane));
    const unsigned lower = peers & lt;
    int p = -1;
    if (ok) {
      if (lower) p = wd * 32 + 31 - __clz(lower);
      else if (last[key] != 0xFFFFu) p = last[key];
    }
    const unsigned alone = __ballot_sync(0xffffffffu, ok && p < 0);
    if (lane == 0) bits0[wd] = alone;
    __syncwarp();
    if (p >= 0) join(p, x, hit_pos(h));
    if (ok && (peers >> lane) == 1u) last[key] = (uint16_t)x;
    __syncwarp();
  }
  __syncthreads();
  // then with the hits of the warps before
  if (warp > 0) {
    for (int wd = w0; wd < w1; ++wd) {
      if (!((bits0[wd] >> lane) & 1u)) continue;
      const int x = wd * 32 + lane;
      const unsigned long long h = hits[x];
      const uint16_t* l = last + key_of(h);
      for (int q = warp - 1; q >= 0; --q) {
        l -= 2 * W::TS;
        if (*l == 0xFFFFu) continue;
        join(*l, x, hit_pos(h));
        break;
      }
    }
  }
  __syncthreads();
  // ---- enters and leaves, strand 0's and then strand 1's
  {
    int ne = 0, nl = 0, ne0 = 0, nl0 = 0;
    for (int wd = w0; wd < w1; ++wd) {
      const int x = wd * 32 + lane;
      const unsigned long long h = x < n ? hits[x] : (kHitNoEnter | kHitNoLeave);
      const unsigned be = __ballot_sync(0xffffffffu, !(h & kHitNoEnter));
      const unsigned bl = __ballot_sync(0xffffffffu, !(h & kHitNoLeave));
      const unsigned b0 = __ballot_sync(0xffffffffu, !(h >> 63));
      ne += __popc(be);
      nl += __popc(bl);
      ne0 += __popc(be & b0);
      nl0 += __popc(bl & b0);
    }
    if (lane == 0) {
      S.sum[0][warp] = ne;
      S.sum[1][warp] = nl;
      S.sum[2][warp] = ne0;
      S.sum[3][warp] = nl0;
    }
  }
  __syncthreads();
  uint32_t* enter = events;
  uint32_t* leave = events + n;
  int ne, nl, ne0, nl0;
  {
    int e, l, skip;
    places(0, &e, &ne);
    places(1, &l, &nl);
    places(2, &skip, &ne0);
    places(3, &skip, &nl0);
    for (int wd = w0; wd < w1; ++wd) {
      const int x = wd * 32 + lane;
      const unsigned long long h = x < n ? hits[x] : (kHitNoEnter | kHitNoLeave);
      const uint32_t t = hit_pos(h);
      const unsigned be = __ballot_sync(0xffffffffu, !(h & kHitNoEnter));
      const unsigned bl = __ballot_sync(0xffffffffu, !(h & kHitNoLeave));
      if (!(h & kHitNoEnter)) enter[e + __popc(be & lt)] = t;
      // t + 1 + span, short of wrapping (no window starts that far)
      if (!(h & kHitNoLeave))
        leave[l + __popc(bl & lt)] = t < 0xFFFFFFFFu - span - 1u ? t + span + 1u : 0xFFFFFFFFu;
      e += __popc(be);
      l += __popc(bl);
    }
  }
  __syncthreads();
  // ---- shared counts: where runs start and end
  uint16_t* val = reinterpret_cast<uint16_t*>(hits);  // shared count at each enter
  uint16_t* first = val + n;                          // per run: the enter that starts it
  uint32_t* end = reinterpret_cast<uint32_t*>(hits) + n;  // per run: its last j + span
  const int m = w.m;
  int e0, e1, l0, l1;
  mine(ne, &e0, &e1);
  mine(nl, &l0, &l1);
  {
    int c = 0;
    for (int wd = e0; wd < e1; ++wd) {
      const int x = wd * 32 + lane;
      bool start = false;
      if (x < ne) {
        const int o = x >= ne0;
        const int xe = x - (o ? ne0 : 0), lb = o ? nl0 : 0, ln = o ? nl - nl0 : nl0;
        const uint32_t j = enter[x];
        const int before = lb_u32(leave + lb, ln, j);  // leaves before j
        const int upto = before + (before < ln && leave[lb + before] == j ? 1 : 0);
        const int v = xe + 1 - upto;
        val[x] = (uint16_t)v;
        start = v >= m && xe - before < m;
      }
      const unsigned b = __ballot_sync(0xffffffffu, start);
      if (lane == 0) bits0[wd] = b;
      c += __popc(b);
    }
    int d = 0;
    for (int wd = l0; wd < l1; ++wd) {
      const int x = wd * 32 + lane;
      bool stop = false;
      if (x < nl) {
        const int o = x >= nl0;
        const int xl = x - (o ? nl0 : 0), eb = o ? ne0 : 0, en = o ? ne - ne0 : ne0;
        const uint32_t j = leave[x];
        const int before = lb_u32(enter + eb, en, j);
        const int upto = before + (before < en && enter[eb + before] == j ? 1 : 0);
        stop = upto - (xl + 1) < m && before - xl >= m;
      }
      const unsigned b = __ballot_sync(0xffffffffu, stop);
      if (lane == 0) bits1[wd] = b;
      d += __popc(b);
    }
    if (lane == 0) {
      S.sum[0][warp] = c;
      S.sum[1][warp] = d;
    }
  }
  __syncthreads();
  int nr, at, to, skip;
  places(0, &at, &nr);
  places(1, &to, &skip);
  if (nr == 0) return;
  for (int wd = e0; wd < e1; ++wd) {
    const unsigned b = bits0[wd];
    if ((b >> lane) & 1u) first[at + __popc(b & lt)] = (uint16_t)(wd * 32 + lane);
    at += __popc(b);
  }
  for (int wd = l0; wd < l1; ++wd) {
    const unsigned b = bits1[wd];
    if ((b >> lane) & 1u) end[to + __popc(b & lt)] = leave[wd * 32 + lane] - 1u;
    to += __popc(b);
  }
  __syncthreads();
  // ---- every run starts and ends once, in order; many runs: one per lane;
  // few: a warp each, which shares their enters out
  const bool by_lane = nr >= 4 * W::WARPS;
  for (int r = by_lane ? lane * W::WARPS + warp : warp; r < nr; r += by_lane ? W::TPB : W::WARPS) {
    const int o = first[r] >= ne0;
    w.o = o;
    emit_valid(a, w, enter + (o ? ne0 : 0), val + (o ? ne0 : 0), o ? ne - ne0 : ne0,
               leave + (o ? nl0 : 0), o ? nl - nl0 : nl0, enter[first[r]], end[r], by_lane);
  }
}

// For the 16 counters of four words of the table (one word: two bins, both
// strands): whether a counter and that of the same strand in the bin before
// or after reach m.  before, after: the words on either side.
__device__ __forceinline__ uint32_t pass_bits(uint32_t before, uint4 c, uint32_t after, uint32_t m) {
  const uint32_t word[6] = {before, c.x, c.y, c.z, c.w, after};
  const uint32_t reach = (0x8000u - m) * 0x10001u;  // a 16-bit field plus this: top bit set from m on
  uint32_t out = 0;
#pragma unroll
  for (int x = 1; x <= 4; ++x) {
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      // 16-bit fields: the word's two bins; the bin before and the bin after
      const uint32_t own = __byte_perm(word[x], 0u, o ? 0x4341 : 0x4240);
      const uint32_t side = __byte_perm(word[x - 1], word[x + 1], o ? 0x0503 : 0x0402) & 0x00FF00FFu;
      const uint32_t pair = own + __byte_perm(own, 0u, 0x1032);
      const uint32_t hit = ((pair + reach) | (own + side + reach)) & 0x80008000u;
      // bits 15 and 31 to counters o and 2 + o
      out |= ((hit >> 15) & 1u) << (4 * (x - 1) + o) | (hit >> 31) << (4 * (x - 1) + 2 + o);
    }
  }
  return out;
}

// One query window by the whole CTA; a window the shape cannot hold goes to
// io.out_list, or for its posting entries to io.wide_list.  The caller
// synchronizes the CTA before and after.  Query-side data is read past L1: a
// serving slot's buffers are refilled while the kernel runs.
template <typename W>
__device__ void cta_window(const FArgs& a, const TierIO& io, CtaSmemT<W>& S, int64_t wdx) {
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  const uint32_t lt = lanemask_lt(), le = lt | (1u << lane);
  const uint32_t i = __ldcg(a.win_i + wdx), qa = __ldcg(a.win_qa + wdx);
  const int c = (int)(__ldcg(a.win_qb + wdx) - qa);
  if (c == 0) return;
  auto hand_over = [&](bool wide) {
    if (tid != 0) return;
    if (wide && io.wide_list) io.wide_list[atomicAdd(io.wide_count, 1u)] = (uint32_t)wdx;
    else io.out_list[atomicAdd(io.out_count, 1u)] = (uint32_t)wdx;
  };
  if (c > W::QC) return hand_over(false);
  uint32_t* tab = reinterpret_cast<uint32_t*>(S.hits);  // W_Q
  if (tid < W::TS / 4) reinterpret_cast<uint4*>(tab)[tid] = make_uint4(0, 0, 0, 0);
  if (tid < W::TS / 16) S.strands[tid] = 0u;
  if (tid == 0) {
    S.uncounted = 0;
    S.nhit = 0;
  }
  // ---- this thread's record: hash and strand, posting range
  uint32_t key = 0, st = 0, len = 0;
  bool kept = false;
  if (tid < c) {
    const uint64_t r = __ldcg(a.qrec + qa + tid);
    const uint32_t h = rec_hash(r);
    key = (h << 1) | rec_strand(r);
    if (a.qpost) {
      const uint2 pp = __ldcg(a.qpost + qa + tid);
      st = pp.x;
      len = pp.y;
      kept = pp.x != kNone;
    } else {
      st = a.toff[h];
      len = a.toff[h + 1] - st;
      kept = !(a.max_occ > 0 && (int)len > a.max_occ);
      if (kept && a.self_mode == 2) {
        const int sq = __ldcg(a.win_seq + wdx);
        posting_window(a.tsorted, a.tsamp, &st, &len, a.tseq[sq], a.tseq[sq + 1]);
      }
    }
    if (!kept) len = 0;
  }
  // ---- posting lists with an entry, one after another
  const uint32_t v = min(len, 1u << 20);  // no sum can wrap
  const uint32_t inc = warp_inclusive_sum(v);
  const unsigned some = __ballot_sync(0xffffffffu, len > 0);
  if (lane == 31) S.sum[0][warp] = inc;
  if (lane == 0) S.sum[1][warp] = __popc(some);
  __syncthreads();
  uint32_t at = inc - v, lid = __popc(some & lt), H = 0;
#pragma unroll
  for (int x = 0; x < W::QC / 32; ++x) {
    const uint32_t y = S.sum[0][x];
    if (x < warp) {
      at += y;
      lid += S.sum[1][x];
    }
    H += y;
  }
  if (H == 0) return;
  if (H > io.hlim || H > (uint32_t)W::WH) return hand_over(true);
  const int nchunk = (int)(H + 31) >> 5;
  uint32_t nslots = 1024;
  while (nslots < 4u * H && nslots < (uint32_t)W::SLOTS) nslots <<= 1;
  const uint32_t smask = nslots - 1;
  for (int x = tid; x < nchunk; x += W::TPB) S.starts[x] = 0u;
  for (int x = tid; x < (int)nslots / 16; x += W::TPB)
    reinterpret_cast<uint4*>(S.table)[x] = make_uint4(0, 0, 0, 0);
  // ---- W_Q: a hash's id is its slot; a record whose hash and strand are in
  // already adds nothing
  bool fresh = false;
  uint32_t how = 0;
  if (kept) {
    const uint32_t h = key >> 1;
    static_assert(W::TS == 512, "nine bits of the hash pick a slot");
    uint32_t slot = (h * 0x9E3779B1u) >> 23;
    while (true) {  // at most QC keys in TS slots: a free slot is always found
      const uint32_t old = atomicCAS(&tab[slot], 0u, h + 1u);
      fresh = old == 0u;
      if (fresh || old == h + 1u) break;
      slot = (slot + 1u) & (uint32_t)(W::TS - 1);
    }
    const uint32_t bit = 1u << ((slot & 15) * 2 + (key & 1u));
    const bool twice = (atomicOr(&S.strands[slot >> 4], bit) & bit) != 0u;
    how = (key & 1u) | (twice ? 2u : 0u) | (slot << 2);
  }
  const int s = __syncthreads_count(fresh);
  const int m = a.mtab[s];
  if (len > 0) {
    S.lists[lid] = make_uint2(st - at, how);
    atomicOr(&S.starts[at >> 5], 1u << (at & 31));
  }
  __syncthreads();
  // this warp's chunks of 32 hits, and the lists that start before them
  const int per = (nchunk + W::WARPS - 1) / W::WARPS;
  const int c0 = min(warp * per, nchunk), c1 = min(c0 + per, nchunk);
  int first_list = 0;
  for (int x = lane; x < c0; x += 32) first_list += __popc(S.starts[x]);
  first_list = (int)__reduce_add_sync(0xffffffffu, first_list) - 1;
  const uint32_t tlo = first_useful(a, i);
  constexpr int kAhead = 4;  // chunks in flight
  // calls f(ch, sl) for kAhead chunks from ch on, from chunk c on: each hit's
  // counter, kNoSlot for none
  constexpr uint32_t kNoSlot = 0xFFFFFFFFu;  // its low 16 bits are no counter either
  auto each_hits = [&](int c, int lists_before, auto f) {
    for (int ch = c; ch < c1; ch += kAhead) {
      uint64_t r[kAhead];
      uint32_t y[kAhead], sl[kAhead];
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        const uint32_t e = (uint32_t)(ch + q) * 32 + lane;
        r[q] = 0;
        y[q] = 2u;
        if (ch + q < c1) {
          const unsigned sb = S.starts[ch + q];
          const int li = lists_before + __popc(sb & le);
          lists_before += __popc(sb);
          if (e < H) {
            const uint2 list = S.lists[li];
            y[q] = list.y;
            r[q] = __ldg(a.tsorted + (list.x + e));
          }
        }
      }
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        const uint32_t t = rec_pos(r[q]);
        const bool on = !(y[q] & 2u) && !useless_hit(a, t, i, tlo);
        sl[q] = on ? slot_of(t, (y[q] ^ rec_strand(r[q])) & 1u, smask) : kNoSlot;
      }
      f(ch, sl);
    }
  };
  uint16_t* kept_sl = reinterpret_cast<uint16_t*>(S.hits);
  {
    uint32_t n_on = 0;
    each_hits(c0, first_list, [&](int ch, const auto& sl) {
#pragma unroll
      for (int q = 0; q < kAhead; ++q) {
        if (ch + q < c1 && ch + q < W::WC / 32) kept_sl[(ch + q) * 32 + lane] = (uint16_t)sl[q];
        if (sl[q] == kNoSlot) continue;
        atomicAdd(&S.table[sl[q] >> 2], 1u << ((sl[q] & 3u) * 8u));
        ++n_on;
      }
    });
    n_on = __reduce_add_sync(0xffffffffu, n_on);
    if (lane == 0) atomicAdd(&S.uncounted, n_on);
  }
  __syncthreads();
  // ---- a bit per counter: its bin and the one before or after reach m.  A
  // counter that ran into its neighbour makes the bytes' sum less than the
  // hits counted.
  {
    constexpr int kPer = (W::SLOTS / 16 + W::TPB - 1) / W::TPB;  // four words at a time
    const int nw = (int)nslots / 4;
    uint32_t bits[(kPer + 1) / 2] = {};
    uint32_t counted = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int x = (q * W::TPB + tid) * 4;
      if (x >= nw) break;
      const uint4 c4 = *reinterpret_cast<const uint4*>(S.table + x);
      bits[q / 2] |= pass_bits(S.table[(x - 1) & (nw - 1)], c4, S.table[(x + 4) & (nw - 1)],
                               (uint32_t)m) << (16 * (q & 1));
      counted = __dp4a(c4.x, 0x01010101u, __dp4a(c4.y, 0x01010101u,
                __dp4a(c4.z, 0x01010101u, __dp4a(c4.w, 0x01010101u, counted))));
    }
    uint32_t any = 0;
#pragma unroll
    for (int q = 0; q < (kPer + 1) / 2; ++q) any |= bits[q];
    counted = __reduce_add_sync(0xffffffffu, counted);
    if (lane == 0) atomicSub(&S.uncounted, counted);
    any = __syncthreads_or(any != 0u);
    if (S.uncounted != 0u) return hand_over(false);
    if (!any) {
      if (io.stats && tid == 0) atomicAdd(a.stats + 0, (unsigned long long)H);
      return;
    }
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int x = q * W::TPB + tid;
      if (x * 4 >= nw) break;
      reinterpret_cast<uint16_t*>(S.table)[x] = (uint16_t)(bits[q / 2] >> (16 * (q & 1)));
    }
  }
  __syncthreads();
  // ---- the entries whose counter's bit is set, with their lists; then their
  // records again
  uint32_t* needed = S.table + W::SLOTS / 32;  // list << 16 | entry
  auto bit_of = [&](uint32_t sl) {
    return sl != kNoSlot && ((S.table[(sl >> 5) & (W::SLOTS / 32 - 1)] >> (sl & 31u)) & 1u) != 0u;
  };
  // N chunks from ch on
  int lists_before = first_list;
  auto take = [&](int ch, const auto& sl) {
    constexpr int N = sizeof(sl) / 4;
    unsigned b[N];
    int n = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      b[q] = __ballot_sync(0xffffffffu, bit_of(sl[q]));
      n += __popc(b[q]);
    }
    int to = 0;
    if (n && lane == 0) to = atomicAdd(&S.nhit, n);
    to = __shfl_sync(0xffffffffu, to, 0);
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const unsigned sb = ch + q < c1 ? S.starts[ch + q] : 0u;
      const int k = to + __popc(b[q] & lt);
      if (((b[q] >> lane) & 1u) && k < W::WL)
        needed[k] = (uint32_t)(lists_before + __popc(sb & le)) << 16 | (uint32_t)((ch + q) * 32 + lane);
      to += __popc(b[q]);
      lists_before += __popc(sb);
    }
  };
  int ch = c0;
  constexpr int kKept = 4;
  for (; ch < c1 && (W::WC >= W::WH || ch + kKept <= W::WC / 32); ch += kKept) {
    uint32_t sl[kKept];
#pragma unroll
    for (int q = 0; q < kKept; ++q) {
      const uint32_t v = ch + q < c1 ? kept_sl[(ch + q) * 32 + lane] : 0xFFFFu;
      sl[q] = v == 0xFFFFu ? kNoSlot : v;
    }
    take(ch, sl);
  }
  if (W::WC < W::WH) each_hits(ch, lists_before, take);
  __syncthreads();
  const int L = S.nhit;
  if (L > W::WL) return hand_over(false);
  for (int x = tid; x < L; x += kAhead * W::TPB) {
    uint64_t r[kAhead];
    uint32_t y[kAhead];
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      if (x + q * W::TPB >= L) break;
      const uint32_t z = needed[x + q * W::TPB];
      const uint2 list = S.lists[z >> 16];
      y[q] = list.y;
      r[q] = __ldg(a.tsorted + (list.x + (z & 0xFFFFu)));
    }
#pragma unroll
    for (int q = 0; q < kAhead; ++q) {
      if (x + q * W::TPB >= L) break;
      S.hits[x + q * W::TPB] = ((unsigned long long)((y[q] ^ rec_strand(r[q])) & 1u) << 63) |
                               ((unsigned long long)rec_pos(r[q]) << 20) | (y[q] >> 2);
    }
  }
  __syncthreads();
  if (io.stats && tid == 0) {
    atomicAdd(a.stats + 0, (unsigned long long)H);
    atomicAdd(a.stats + 1, (unsigned long long)L);
  }
  if (L < m) return;
  unsigned long long* const other = reinterpret_cast<unsigned long long*>(S.table);
  unsigned long long* const sorted = cta_sort_hits<W>(S.hits, other, L);
  WinInfo w;
  w.i = i;
  w.qseq = __ldcg(a.win_seq + wdx);
  w.s = s;
  w.m = m;
  w.o = 0;
  cta_runs<W>(a, w, sorted, reinterpret_cast<uint32_t*>(sorted == other ? S.hits : other), L, S);
}

template <typename W>
__global__ void __launch_bounds__(W::TPB, W::MINB) k_filter_cta(FArgs a, TierIO io) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CtaSmemT<W>& S = *reinterpret_cast<CtaSmemT<W>*>(smem_raw);
  const int64_t count = (int64_t)*io.in_count;
  unsigned int next = 0;
  if (threadIdx.x == 0) next = atomicAdd(io.next, 1u);
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) {
      S.win = (int64_t)next < count ? (int64_t)io.in_list[next] : -1;
      if (S.win >= 0) next = atomicAdd(io.next, 1u);  // waited for after this window
    }
    __syncthreads();
    if (S.win < 0) break;
    cta_window(a, io, S, S.win);
  }
}

template <typename W>
int launch_cta_tier(sedef_ctx* ctx, const FArgs& a, const TierIO& io, int64_t max_windows,
                    const char* name) {
  const size_t sm = sizeof(CtaSmemT<W>);
  SEDEF_TRY(ensure_smem_attr((const void*)k_filter_cta<W>, sm));
  int per_sm = 0;
  SEDEF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_cta<W>, W::TPB, sm));
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)ctx_sm_count(ctx) * per_sm;
  if (grid > max_windows) grid = max_windows;
  if (grid < 1) grid = 1;
  SEDEF_KERNEL(ctx, name, k_filter_cta<W><<<(int)grid, W::TPB, sm, ctx_stream(ctx)>>>(a, io));
  return SEDEF_OK;
}

// ------------------------------------------------------------- slow path --

constexpr int kSThreads = 256;

struct SlowSmem {
  uint32_t qkey[kMaxWindowRecs];
  uint32_t dh[kMaxWindowRecs];
  uint32_t pst[kMaxWindowRecs];
  uint32_t plen[kMaxWindowRecs];
  uint8_t dm[kMaxWindowRecs];
  uint16_t cnt[kMaxWindowRecs];
  int tmp[33];
  unsigned long long acc;
};

__device__ int slow_wq(const FArgs& a, SlowSmem& S, int64_t wdx) {
  const uint32_t qa = a.win_qa[wdx], qb = a.win_qb[wdx];
  const int c = (int)(qb - qa);
  for (int x = threadIdx.x; x < c; x += blockDim.x) {
    const uint64_t r = a.qrec[qa + x];
    S.qkey[x] = (rec_hash(r) << 1) | rec_strand(r);
  }
  __syncthreads();
  QBuild q;
  q.qkey = S.qkey;
  q.dh = S.dh;
  q.dm = S.dm;
  q.pst = S.pst;
  q.plen = S.plen;
  q.tmp = S.tmp;
  int64_t seq_lo = 0, seq_hi = 0;
  if (a.self_mode == 2) {
    const int sq = a.win_seq[wdx];
    seq_lo = a.tseq[sq];
    seq_hi = a.tseq[sq + 1];
  }
  return build_wq(a, q, c, seq_lo, seq_hi);
}

// Hits of overflow window v: visits (t, hid, o) for every compatible posting.
template <typename F>
__device__ void slow_hits(const FArgs& a, const SlowSmem& S, int s, int64_t i, F f) {
  const uint32_t tlo = first_useful(a, i);
  for (int l = 0; l < s; ++l) {
    const uint32_t st0 = S.pst[l], len = S.plen[l];
    const uint32_t qm = S.dm[l];
    for (uint32_t x = threadIdx.x; x < len; x += blockDim.x) {
      const uint64_t r = a.tsorted[st0 + x];
      const uint32_t t = rec_pos(r), st = rec_strand(r);
      if (useless_hit(a, t, (uint32_t)i, tlo)) continue;
      if ((qm >> st) & 1u) f(t, (uint32_t)l, 0u);
      if ((qm >> (st ^ 1u)) & 1u) f(t, (uint32_t)l, 1u);
    }
  }
}

template <typename C>
__global__ void __launch_bounds__(kSThreads) k_slow_count(FArgs a, int64_t nov, C* counts,
                                                          int32_t* s_out, const uint32_t* dnov,
                                                          unsigned long long* total) {
  __shared__ SlowSmem S;
  nov = live_n(nov, dnov);
  for (int64_t v = blockIdx.x; v < nov; v += gridDim.x) {
    __syncthreads();
    const int64_t wdx = a.ov_list[v];
    const int s = slow_wq(a, S, wdx);
    if (threadIdx.x == 0) S.acc = 0;
    __syncthreads();
    unsigned long long mine = 0;
    slow_hits(a, S, s, a.win_i[wdx], [&](uint32_t, uint32_t, uint32_t) { ++mine; });
    atomicAdd(&S.acc, mine);
    __syncthreads();
    if (threadIdx.x == 0) {
      counts[v] = (C)S.acc;
      s_out[v] = s;
      if (total) atomicAdd(total, S.acc);
    }
  }
}

// Writes keys (local window << 33 | o << 32 | t) and hash ids for windows
// [v0, v1) of the overflow list at offsets base[v] - base[v0].
// Windows whose hits would end past `hcap` are skipped (a planned pass
// reports them as an overflow).
__global__ void __launch_bounds__(kSThreads) k_slow_emit(FArgs a, int64_t v0, int64_t v1,
                                                         const unsigned long long* base,
                                                         uint64_t* keys, uint32_t* vals,
                                                         const uint32_t* dnov, int64_t hcap) {
  __shared__ SlowSmem S;
  __shared__ unsigned long long cursor;
  v1 = live_n(v1, dnov);
  for (int64_t v = v0 + blockIdx.x; v < v1; v += gridDim.x) {
    if (base[v + 1] < base[v] || (int64_t)(base[v + 1] - base[v0]) > hcap) continue;
    __syncthreads();
    const int64_t wdx = a.ov_list[v];
    const int s = slow_wq(a, S, wdx);
    if (threadIdx.x == 0) cursor = base[v] - base[v0];
    __syncthreads();
    const uint64_t lw = (uint64_t)(v - v0);
    slow_hits(a, S, s, a.win_i[wdx], [&](uint32_t t, uint32_t hid, uint32_t o) {
      const unsigned long long at = atomicAdd(&cursor, 1ull);
      keys[at] = (lw << 33) | ((uint64_t)o << 32) | t;
      vals[at] = hid;
    });
  }
}

// A dense group of an overflow window: one task of the sweep.
struct SlowTask {
  uint32_t v;   // overflow-list index
  uint32_t o;
  int64_t jlo, jhi;
};

__device__ __forceinline__ void slow_segment(const uint64_t* keys, int64_t lo, int64_t hi,
                                             int64_t* split) {
  int64_t l = lo, h = hi;  // first key with o = 1
  while (l < h) {
    const int64_t mid = (l + h) >> 1;
    if (((keys[mid] >> 32) & 1u) == 0) l = mid + 1; else h = mid;
  }
  *split = l;
}

// Writes a task for each lane that has one.  The whole warp calls.
__device__ __forceinline__ void slow_task(SlowTask* tasks, unsigned long long* ntask, int64_t task_cap,
                                          bool has, uint32_t v, uint32_t o, int64_t jlo, int64_t jhi) {
  const unsigned b = __ballot_sync(0xffffffffu, has);
  if (b == 0) return;
  unsigned long long at = 0;
  if (lane_id() == 0) at = atomicAdd(ntask, (unsigned long long)__popc(b));
  at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & lanemask_lt());
  if (has && (int64_t)at < task_cap) {
    SlowTask t;
    t.v = v;
    t.o = o;
    t.jlo = jlo < 0 ? 0 : jlo;
    t.jhi = jhi;
    tasks[at] = t;
  }
}

// A window's hits are shared out to `parts` warps, kGroupHits of a strand at a
// time: a warp takes the groups that start among them, to their ends.  Whether
// a dense hit starts a group depends on the nearest dense hit before it alone,
// at most span + 1 back.  As many parts as the grid has warps to spare for the
// windows at hand; one part takes a strand in one go.  (One warp for a window
// of 22 k hits, through both strands: 0.48 ms, 0.05 in 32 parts; 32 parts for
// each of 40 k windows of 500 or 1,800 hits: 1.56 and 4.9 ms, 0.18 and 0.48 with
// a warp each.)
constexpr int kGroupHits = 512;
constexpr int kGroupParts = 32;

__global__ void k_slow_groups(FArgs a, int64_t v0, int64_t v1, const unsigned long long* base,
                              const int32_t* s_of, const uint64_t* keys, SlowTask* tasks,
                              unsigned long long* ntask, int64_t task_cap, const uint32_t* dnov,
                              int64_t hcap) {
  const int lane = lane_id();
  const unsigned lt = lanemask_lt();
  v1 = live_n(v1, dnov);
  if (v1 <= v0) return;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  int parts = 1;  // a power of two: the grid's warps are a multiple of kGroupParts
  while (parts < kGroupParts && 2 * parts * (v1 - v0) <= warps) parts <<= 1;
  const int64_t chunk = parts > 1 ? kGroupHits : INT64_MAX / 2;
  const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t part = w & (parts - 1);
  for (int64_t v = v0 + w / parts; v < v1; v += warps / parts) {
    const int s = s_of[v];
    if (s == 0 || base[v + 1] < base[v] || (int64_t)(base[v + 1] - base[v0]) > hcap) continue;
    const int m = max(a.mtab[s], 1);
    const int64_t lo = (int64_t)(base[v] - base[v0]), hi = (int64_t)(base[v + 1] - base[v0]);
    if (part > 0 && lo + part * chunk >= hi) continue;
    int64_t split;
    slow_segment(keys, lo, hi, &split);
    for (int o = 0; o < 2; ++o) {
      const uint64_t* k = keys + (o ? split : lo);
      const int64_t n = o ? hi - split : split - lo;  // hits of the strand
      const int64_t nd = n - m + 1;                   // the first of m hits lies before this one
      auto dense = [&](int64_t x, int64_t* jlo, int64_t* jhi) {
        if (x < 0 || x >= nd) return false;
        const int64_t ta = (uint32_t)k[x], tb = (uint32_t)k[x + m - 1];
        *jlo = tb - a.span;
        *jhi = ta;
        return tb - ta <= a.span;
      };
      for (int64_t x0 = part ? part * chunk : 0; x0 < nd; x0 += parts * chunk) {
        const int64_t x1 = min(x0 + chunk, nd);
        int64_t carry_hi = INT64_MIN, cur_lo = 0;  // jhi of the nearest dense hit before; the open group
        bool open = false;
        const int64_t reach = (int64_t)(uint32_t)k[x0] - a.span - 1;
        for (int64_t y = x0 - 32; y > -32; y -= 32) {
          int64_t jlo, jhi = 0;
          const unsigned dm = __ballot_sync(0xffffffffu, dense(y + lane, &jlo, &jhi));
          if (dm) {
            carry_hi = __shfl_sync(0xffffffffu, jhi, 31 - __clz(dm));
            break;
          }
          if (y <= 0 || (int64_t)(uint32_t)k[y] < reach) break;
        }
        for (int64_t y = x0; y < x1 || (open && y < nd); y += 32) {
          const int64_t x = y + lane;
          int64_t jlo = 0, jhi = INT64_MIN;
          const bool is = dense(x, &jlo, &jhi);
          const unsigned dm = __ballot_sync(0xffffffffu, is);
          const int64_t near = __shfl_sync(0xffffffffu, jhi, dm & lt ? 31 - __clz(dm & lt) : lane);
          const int64_t before = dm & lt ? near : carry_hi;
          const bool start = is && (before == INT64_MIN || jlo > before + 1);
          const unsigned starts = __ballot_sync(0xffffffffu, start);
          const int64_t lo_near = __shfl_sync(0xffffffffu, jlo, starts & lt ? 31 - __clz(starts & lt) : lane);
          // a start closes the group before it, when that one is this warp's
          const int own = (int)min(max(x1 - y, (int64_t)0), (int64_t)32);
          const unsigned mine = own >= 32 ? 0xffffffffu : (1u << own) - 1u;
          const bool closes = start && (starts & lt ? (((starts & lt & mine) >> (31 - __clz(starts & lt))) & 1u) != 0u : open);
          slow_task(tasks, ntask, task_cap, closes, (uint32_t)v, (uint32_t)o,
                    starts & lt ? lo_near : cur_lo, before);
          if (starts) {
            const int l = 31 - __clz(starts);
            cur_lo = __shfl_sync(0xffffffffu, jlo, l);
            open = ((mine >> l) & 1u) != 0u;
          }
          if (dm) carry_hi = __shfl_sync(0xffffffffu, jhi, 31 - __clz(dm));
        }
        slow_task(tasks, ntask, task_cap, open && lane == 0, (uint32_t)v, (uint32_t)o, cur_lo, carry_hi);
      }
    }
  }
}

// One warp per task; lane 0 sweeps the group with the warp's counters.
constexpr int kTaskWarps = 8;

__global__ void __launch_bounds__(32 * kTaskWarps) k_slow_tasks(
    FArgs a, int64_t v0, const unsigned long long* base, const int32_t* s_of,
    const uint64_t* keys, const uint32_t* vals, const SlowTask* tasks,
    const unsigned long long* ntask, int64_t task_cap) {
  __shared__ uint16_t cnt[kTaskWarps][kMaxWindowRecs];
  const int warp = threadIdx.x >> 5;
  for (int x = threadIdx.x & 31; x < kMaxWindowRecs; x += 32) cnt[warp][x] = 0;
  __syncwarp();
  if ((threadIdx.x & 31) != 0) return;
  const int64_t nt = min((int64_t)*ntask, task_cap);
  for (int64_t t = (int64_t)blockIdx.x * kTaskWarps + warp; t < nt;
       t += (int64_t)gridDim.x * kTaskWarps) {
    const SlowTask task = tasks[t];
    const int64_t v = task.v;
    const int64_t wdx = a.ov_list[v];
    const int s = s_of[v];
    WinInfo w;
    w.i = a.win_i[wdx];
    w.qseq = a.win_seq[wdx];
    w.s = s;
    w.m = a.mtab[s];
    w.o = (int)task.o;
    const int64_t lo = (int64_t)(base[v] - base[v0]), hi = (int64_t)(base[v + 1] - base[v0]);
    int64_t split;
    slow_segment(keys, lo, hi, &split);
    const int64_t b = task.o ? split : lo, e = task.o ? hi : split;
    sweep_group(a, w, [&](int64_t x) { return make_uint2((uint32_t)keys[b + x], vals[b + x]); },
                e - b, cnt[warp], task.jlo, task.jhi);
  }
}

// ---------------------------------------------------------- window table --

__global__ void k_windows(const uint64_t* __restrict__ qrec, int64_t nq,
                          const int64_t* __restrict__ qseq, int nqseq,
                          const int64_t* __restrict__ wbase, int64_t nwin, int step, int span,
                          uint32_t* wi, uint32_t* wqa, uint32_t* wqb, int32_t* wseq,
                          const uint32_t* dnq) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= nwin) return;
  nq = live_n(nq, dnq);
  int lo = 0, hi = nqseq;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (wbase[mid] <= w) lo = mid; else hi = mid;
  }
  const int64_t i = qseq[lo] + (w - wbase[lo]) * step;
  auto pos = [](uint64_t r) { return (uint64_t)((r >> 1) & 0xFFFFFFFFull); };
  const int64_t a = lower_bound_by(qrec, 0, nq, (uint64_t)i, pos);
  const int64_t b = lower_bound_by(qrec, a, nq, (uint64_t)(i + span + 1), pos);
  wi[w] = (uint32_t)i;
  wqa[w] = (uint32_t)a;
  wqb[w] = (uint32_t)b;
  wseq[w] = lo;
}

// Sort keys of the runs: (window index, o, j_a), tbits hold every j_a.  part
// 0: the whole key when it fits 64 bits; part 1: j_a alone and part 2:
// (window, o), for a two-pass stable sort otherwise.
__global__ void k_run_keys(const sedef_run_t* runs, int64_t n, const int64_t* qseq, int nqseq,
                           const int64_t* wbase, int step, int part, int tbits, uint64_t* keys,
                           const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= live_n(n, dn)) return;
  const sedef_run_t r = runs[x];
  const int sq = seq_of(qseq, nqseq, r.i);
  const uint64_t widx = (uint64_t)(wbase[sq] + ((int64_t)r.i - qseq[sq]) / step);
  if (part == 0) keys[x] = (((widx << 1) | r.o) << tbits) | r.j_a;
  else if (part == 1) keys[x] = r.j_a;
  else keys[x] = (widx << 1) | r.o;
}

__global__ void k_permute_u64(const uint64_t* in, const uint32_t* perm, int64_t n, uint64_t* out,
                              const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < live_n(n, dn)) out[x] = in[perm[x]];
}

__global__ void k_compose_perm(const uint32_t* first, const uint32_t* second, int64_t n,
                               uint32_t* out, const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < live_n(n, dn)) out[x] = first[second[x]];
}

__global__ void k_widen_u32(const uint32_t* in, int64_t n, unsigned long long* out) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < n) out[x] = in[x];
}

__global__ void k_gather_runs(const sedef_run_t* in, const uint32_t* perm, int64_t n, sedef_run_t* out,
                              const uint32_t* dn) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < live_n(n, dn)) out[x] = in[perm[x]];
}

// ----------------------------------------------------------------- refine --
//
// Two kernels: k_refine_batch (at most 256 query records and 512 span records
// per run) and k_refine (any run, in pieces of at most 1024 span records) for
// the runs that k_refine_batch hands over.
//
// The estimate at j never exceeds the number of W_Q hashes shared with the
// window (the filter's shared_o(j)), so it is evaluated only where that
// count exceeds the best estimate so far, and the run is finished as soon
// as the best estimate reaches the run's max_shared.

constexpr int kRWarpsBig = 4;  // large kernel

template <int QC, int RC>
struct RefineWarpT {
  static constexpr int DC = QC + RC;  // domain: W_Q u span hashes
  static_assert((DC & (DC - 1)) == 0, "the sort pads the domain to a power of two");
  uint32_t dom[DC];      // sorted distinct hashes
  uint16_t cntT[DC];     // records of this hash in the target window
  uint16_t cntS[DC];     // shared-compatible records of this hash in the window
  uint8_t qm[DC];        // strand mask for W_Q members (0 = not in W_Q)
  uint32_t pb[DC / 32];  // present: in W_Q or cntT > 0
  uint32_t sb[DC / 32];  // shared: cntS > 0
  uint32_t tpos[RC];     // span record positions (sorted)
  uint16_t tdx[RC];      // domain index of each span record
  uint8_t tsh[RC];       // record is shared-compatible
  uint32_t wq_h[QC];     // W_Q hashes (sorted)
  uint8_t wq_m[QC];      // W_Q strand masks
};

__device__ __forceinline__ void warp_sort_u32(uint32_t* v, int n) {  // n power of two
  for (int size = 2; size <= n; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = lane_id(); t < (n >> 1); t += 32) {
        const int lo = ((t & ~(stride - 1)) << 1) | (t & (stride - 1));
        const int hi = lo + stride;
        const bool asc = (lo & size) == 0;
        const uint32_t x = v[lo], y = v[hi];
        if ((x > y) == asc) {
          v[lo] = y;
          v[hi] = x;
        }
      }
      __syncwarp();
    }
}

__device__ __forceinline__ int dom_find(const uint32_t* dom, int D, uint32_t h) {
  int lo = 0, hi = D;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (dom[mid] < h) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// theta = domain index of the s-th present bit, est = shared bits at or
// below it (warp-wide; same word layout as estimate()).
__device__ __forceinline__ void theta_est(const uint32_t* pb, const uint32_t* sb, int nwords,
                                          int s, int* theta, int* est) {
  const int lane = lane_id();
  const uint32_t p0 = (2 * lane < nwords) ? pb[2 * lane] : 0u;
  const uint32_t p1 = (2 * lane + 1 < nwords) ? pb[2 * lane + 1] : 0u;
  const uint32_t s0 = (2 * lane < nwords) ? sb[2 * lane] : 0u;
  const uint32_t s1 = (2 * lane + 1 < nwords) ? sb[2 * lane + 1] : 0u;
  const int pc = __popc(p0) + __popc(p1);
  const int inc = warp_inclusive_sum(pc);
  const int before = inc - pc;
  const unsigned owner = __ballot_sync(0xffffffffu, before < s && inc >= s);
  const int ol = __ffs(owner) - 1;
  int cnt = (inc < s) ? (__popc(s0) + __popc(s1)) : 0;  // lanes wholly below theta
  int th = 0;
  if (lane == ol) {
    int need = s - before;
    const uint32_t wp[2] = {p0, p1}, ws[2] = {s0, s1};
    cnt = 0;
    for (int x = 0; x < 2; ++x) {
      const int c = __popc(wp[x]);
      if (c < need) {
        cnt += __popc(ws[x]);
        need -= c;
        continue;
      }
      uint32_t v = wp[x];
      for (int y = 1; y < need; ++y) v &= v - 1u;
      const int b = __ffs(v) - 1;
      const uint32_t below = (b >= 31) ? 0xFFFFFFFFu : ((2u << b) - 1u);
      cnt += __popc(ws[x] & below);
      th = (2 * lane + x) * 32 + b;
      break;
    }
  }
  *est = warp_sum(cnt);
  *theta = __shfl_sync(0xffffffffu, th, ol);
}

struct RefineArgs {
  sedef_run_t* runs;
  int64_t nruns;
  const uint64_t* qrec;
  int64_t nq;
  const uint64_t* trec;
  int64_t nt;
  const uint32_t* dnruns = nullptr;  // live counts of a planned pass
  const uint32_t* dnt = nullptr;
  const uint32_t* toff;
  const int32_t* mtab;
  int span, max_occ, self_mode;
  uint32_t* big;        // runs handed to the large kernel
  unsigned int* nbig;
  const uint4* ranges;  // per run: query records [x, y), span records [z, w)
  unsigned long long* next;  // chunk counters of the two kernels
  // k_refine_batch: event words (ev_words + kEvPad per warp), W_Q hashes per roll
  uint32_t* events = nullptr;
  int ev_words = 0;
  int scap = 0;
};

template <int QC, int RC>
__global__ void __launch_bounds__(32 * kRWarpsBig) k_refine(RefineArgs a) {
  a.nruns = live_n(a.nruns, a.dnruns);
  a.nt = live_n(a.nt, a.dnt);
  using RW = RefineWarpT<QC, RC>;
  constexpr int DC = RW::DC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  RW& R = reinterpret_cast<RW*>(smem_raw)[warp];
  auto pos_of = [](uint64_t r) { return (uint64_t)((r >> 1) & 0xFFFFFFFFull); };
  const int64_t count = (int64_t)*a.nbig;
  // contiguous chunks of runs per warp (runs of one window are adjacent, so
  // W_Q is built once per window and chunk), handed out dynamically
  constexpr int kChunk = 16;
  int64_t prev_qa = -1, prev_qb = -1;
  int s = 0;
  while (true) {
    int64_t c0 = 0;
    if (lane == 0) c0 = (int64_t)atomicAdd(a.next + 1, (unsigned long long)kChunk);
    c0 = __shfl_sync(0xffffffffu, c0, 0);
    if (c0 >= count) break;
    const int64_t c1 = min(count, c0 + kChunk);
  for (int64_t t = c0; t < c1; ++t) {
    const int64_t ri = (int64_t)a.big[t];
    const sedef_run_t run = a.runs[ri];
    const int64_t i = run.i, ja = run.j_a, jb = run.j_b;
    const int o = run.o;
    const uint4 rg = a.ranges[ri];  // query records [qa, qb), span records from rlo on
    const int64_t qa = rg.x, qb = rg.y;
    int64_t rlo = rg.z;
    const int c = (int)(qb - qa);
    if (qa != prev_qa || qb != prev_qb) {
    prev_qa = qa;
    prev_qb = qb;
    // ---- W_Q: sorted hashes with strand masks (capped hashes dropped)
    const int npq = next_pow2(c < 2 ? 2 : c);
    for (int x = lane; x < npq; x += 32) {
      uint32_t key = kNone;
      if (x < c) {
        const uint64_t r = a.qrec[qa + x];
        key = (rec_hash(r) << 1) | rec_strand(r);
      }
      R.dom[x] = key;  // the domain array doubles as the sort buffer
    }
    __syncwarp();
    warp_sort_u32(R.dom, npq);
    s = 0;
    for (int base = 0; base < c; base += 32) {
      const int x = base + lane;
      uint32_t h = 0, mask = 0;
      bool first = false;
      if (x < c) {
        h = R.dom[x] >> 1;
        first = (x == 0) || ((R.dom[x - 1] >> 1) != h);
        if (first) {
          for (int y = x; y < c && (R.dom[y] >> 1) == h; ++y) mask |= 1u << (R.dom[y] & 1u);
          if (a.max_occ > 0 && (int)(a.toff[h + 1] - a.toff[h]) > a.max_occ) first = false;
        }
      }
      const unsigned bal = __ballot_sync(0xffffffffu, first);
      if (first) {
        const int d = s + __popc(bal & lanemask_lt());
        R.wq_h[d] = h;
        R.wq_m[d] = (uint8_t)mask;
      }
      s += __popc(bal);
    }
    __syncwarp();
    }
    const int mx = run.max_shared;
    int best = -1;
    int64_t jstar = ja;
    int64_t plo = ja;
    bool finished = false;
    while (plo <= jb && !finished) {
      // ---- the piece [plo, phi]: span records [rlo, rhi), at most RC
      int64_t phi = jb, rhi = 0;
      if (lane == 0) {
        const int64_t rcap_end = rlo + RC < a.nt ? rlo + RC : a.nt;
        rhi = lower_bound_by(a.trec, rlo, a.nt, (uint64_t)(jb + a.span + 1), pos_of);
        if (rhi > rcap_end) {
          const int64_t lim = (int64_t)pos_of(a.trec[rcap_end]);  // first record that does not fit
          phi = lim - a.span - 1;
          rhi = rcap_end;
        }
      }
      phi = __shfl_sync(0xffffffffu, phi, 0);
      rhi = __shfl_sync(0xffffffffu, rhi, 0);
      const int nr = (int)(rhi - rlo);
      // ---- relevant span records.  Only W_Q hashes with a compatible,
      // non-self occurrence in the span (the candidates C) can ever count,
      // and a candidate's rank among W_Q u W_T depends only on the hashes
      // below it.  So the roll needs the candidates' compatible occurrences
      // and the non-W_Q records whose hash is below max(C); every other
      // record leaves the estimate unchanged.  W_Q itself stays in the
      // domain, so at least s hashes are always present.  cntT/cntS double
      // as a scratch array of the kept records' hashes until the domain is
      // built.
      uint32_t* tmp_h = reinterpret_cast<uint32_t*>(R.cntT);  // DC u32 (cntT then cntS)
      auto wq_find = [&](uint32_t h) {  // index in W_Q or -1
        int lo2 = 0, hi2 = s;
        while (lo2 < hi2) {
          const int mid = (lo2 + hi2) >> 1;
          if (R.wq_h[mid] < h) lo2 = mid + 1; else hi2 = mid;
        }
        return (lo2 < s && R.wq_h[lo2] == h) ? lo2 : -1;
      };
      uint32_t cmax = 0;
      bool have_c = false;
      for (int base = 0; base < nr; base += 32) {
        const int x = base + lane;
        bool cand = false;
        uint32_t h = 0;
        if (x < nr) {
          const uint64_t r = a.trec[rlo + x];
          h = rec_hash(r);
          const uint32_t t = rec_pos(r), st = rec_strand(r);
          const int q = wq_find(h);
          const bool self = a.self_mode && (int64_t)t >= i && (int64_t)t <= i + a.span;
          cand = q >= 0 && !self && ((R.wq_m[q] >> (st ^ (uint32_t)o)) & 1u);
        }
        uint32_t hm = cand ? h : 0u;
        const bool any = __any_sync(0xffffffffu, cand);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) hm = max(hm, __shfl_xor_sync(0xffffffffu, hm, d));
        if (any) {
          cmax = have_c ? max(cmax, hm) : hm;
          have_c = true;
        }
      }
      int nrel = 0;
      for (int base = 0; base < nr && have_c; base += 32) {
        const int x = base + lane;
        bool keep = false;
        uint32_t h = 0, t = 0, st = 0;
        if (x < nr) {
          const uint64_t r = a.trec[rlo + x];
          h = rec_hash(r);
          t = rec_pos(r);
          st = rec_strand(r);
          const int q = wq_find(h);
          if (q >= 0) {
            const bool self = a.self_mode && (int64_t)t >= i && (int64_t)t <= i + a.span;
            keep = !self && ((R.wq_m[q] >> (st ^ (uint32_t)o)) & 1u);
          } else {
            keep = h < cmax;
          }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (keep) {
          const int y = nrel + __popc(bal & lanemask_lt());
          R.tpos[y] = t;
          tmp_h[y] = h;
          R.tsh[y] = (uint8_t)st;  // strand for now
        }
        nrel += __popc(bal);
      }
      __syncwarp();
      // ---- domain: sorted distinct hashes of W_Q u kept records
      const int nd0 = s + nrel;
      const int npd = next_pow2(nd0 < 2 ? 2 : nd0);
      for (int x = lane; x < npd; x += 32) {
        uint32_t v = kNone;
        if (x < s) v = R.wq_h[x];
        else if (x < nd0) v = tmp_h[x - s];
        R.dom[x] = v;
      }
      __syncwarp();
      warp_sort_u32(R.dom, npd);
      int D = 0;
      for (int base = 0; base < nd0; base += 32) {
        const int x = base + lane;
        const uint32_t v = x < nd0 ? R.dom[x] : kNone;
        const bool first = x < nd0 && (x == 0 || R.dom[x - 1] != v);
        const unsigned bal = __ballot_sync(0xffffffffu, first);
        __syncwarp();
        if (first) R.dom[D + __popc(bal & lanemask_lt())] = v;
        __syncwarp();
        D += __popc(bal);
      }
      for (int x = lane; x < nrel; x += 32) R.tdx[x] = (uint16_t)dom_find(R.dom, D, tmp_h[x]);
      __syncwarp();
      const int nwords = (D + 31) >> 5;
      for (int x = lane; x < D; x += 32) {
        R.cntT[x] = 0;
        R.cntS[x] = 0;
        R.qm[x] = 0;
      }
      for (int x = lane; x < DC / 32; x += 32) {
        R.pb[x] = 0;
        R.sb[x] = 0;
      }
      __syncwarp();
      for (int x = lane; x < s; x += 32) {
        const int d = dom_find(R.dom, D, R.wq_h[x]);
        R.qm[d] = R.wq_m[x];
        atomicOr(&R.pb[d >> 5], 1u << (d & 31));
      }
      __syncwarp();
      for (int x = lane; x < nrel; x += 32) {
        const uint32_t t = R.tpos[x], st = R.tsh[x];
        const int d = R.tdx[x];
        const bool self = a.self_mode && (int64_t)t >= i && (int64_t)t <= i + a.span;
        R.tsh[x] = (!self && ((R.qm[d] >> (st ^ (uint32_t)o)) & 1u)) ? 1 : 0;
      }
      __syncwarp();
      // ---- roll the target window over [plo, phi].  theta is the domain
      // index of the s-th present hash (the largest member of U) and est the
      // number of shared hashes at or below it.  After the first breakpoint
      // lane 0 keeps both exact through every enter and leave, one record at
      // a time: a hash joining below theta pushes theta down to its
      // predecessor, one leaving at or below theta pulls theta up to its
      // successor, and a W_Q hash at or below theta changes est when it
      // becomes or stops being shared.
      int e = 0, l = 0;
      int64_t j = plo;
      if (lane == 0) {
        while (e < nrel && (int64_t)R.tpos[e] <= j + a.span) {
          const int d = R.tdx[e];
          if (R.cntT[d]++ == 0) R.pb[d >> 5] |= 1u << (d & 31);
          if (R.tsh[e] && R.cntS[d]++ == 0) R.sb[d >> 5] |= 1u << (d & 31);
          ++e;
        }
      }
      __syncwarp();
      int theta = 0, est = 0;
      theta_est(R.pb, R.sb, nwords, s, &theta, &est);
      int fin = 0;
      if (lane == 0) {
        auto bit = [&](const uint32_t* bs, int d) { return (int)((bs[d >> 5] >> (d & 31)) & 1u); };
        auto pred = [&](int d) {  // largest present index below d
          int w = d >> 5;
          uint32_t bits = R.pb[w] & ((1u << (d & 31)) - 1u);
          while (bits == 0 && w > 0) bits = R.pb[--w];
          return bits ? w * 32 + 31 - __clz(bits) : 0;
        };
        auto succ = [&](int d) {  // smallest present index above d
          int w = d >> 5;
          uint32_t bits = ((d & 31) == 31) ? 0u : (R.pb[w] & ~((2u << (d & 31)) - 1u));
          while (bits == 0 && w + 1 < nwords) bits = R.pb[++w];
          return bits ? w * 32 + __ffs(bits) - 1 : d;
        };
        auto enter = [&](int x) {
          const int d = R.tdx[x];
          if (R.cntT[d]++ == 0 && R.qm[d] == 0) {
            R.pb[d >> 5] |= 1u << (d & 31);
            if (d < theta) {
              const int old = theta;
              theta = pred(theta);
              est -= bit(R.sb, old);
            }
          }
          if (R.tsh[x] && R.cntS[d]++ == 0) {
            R.sb[d >> 5] |= 1u << (d & 31);
            if (d <= theta) ++est;
          }
        };
        auto leave = [&](int x) {
          const int d = R.tdx[x];
          if (--R.cntT[d] == 0 && R.qm[d] == 0) {
            R.pb[d >> 5] &= ~(1u << (d & 31));
            if (d <= theta) {
              theta = succ(theta);
              est += bit(R.sb, theta);
            }
          }
          if (R.tsh[x] && --R.cntS[d] == 0) {
            R.sb[d >> 5] &= ~(1u << (d & 31));
            if (d <= theta) --est;
          }
        };
        while (true) {
          if (est > best) {
            best = est;
            jstar = j;
            if (best >= mx) {
              fin = 1;
              break;
            }
          }
          const int64_t ne = e < nrel ? (int64_t)R.tpos[e] - a.span : INT64_MAX;
          const int64_t nl = l < e ? (int64_t)R.tpos[l] + 1 : INT64_MAX;
          const int64_t nx = min(ne, nl);
          if (nx > phi) break;
          j = nx;
          while (l < e && (int64_t)R.tpos[l] + 1 <= j) leave(l++);
          while (e < nrel && (int64_t)R.tpos[e] - a.span <= j) enter(e++);
        }
      }
      jstar = __shfl_sync(0xffffffffu, jstar, 0);
      finished = __shfl_sync(0xffffffffu, fin, 0) != 0;
      best = __shfl_sync(0xffffffffu, best, 0);
      plo = phi + 1;
      if (plo <= jb && !finished) {
        if (lane == 0) rlo = lower_bound_by(a.trec, rlo, a.nt, (uint64_t)plo, pos_of);
        rlo = __shfl_sync(0xffffffffu, rlo, 0);
      }
      __syncwarp();
    }
    if (lane == 0) {
      sedef_run_t& out = a.runs[ri];
      out.est = (uint16_t)(best < 0 ? 0 : best);
      out.den = (uint16_t)s;
      out.j_star = (uint32_t)jstar;
      out.keep = (best >= a.mtab[s]) ? 1 : 0;
    }
    __syncwarp();
  }
  }
}

// ------------------------------------------------- batched refine ----
//
// A warp sets up runs one at a time (cooperatively), writing each run's
// events to its own stretch of device memory, then every lane rolls one run,
// so up to 32 rolls proceed side by side.
//
// The estimate needs no merged domain.  W_Q's hashes h_0 < ... < h_{s-1} are
// all in the union, so h_r is among the union's s smallest exactly when
// r + 1 + #{distinct non-W_Q hashes of the window below h_r} <= s.  The left
// side grows with r: a threshold R (how many h_r pass) decides, and est is
// the number of shared h_r with r < R.  A non-W_Q record acts only through
// its rank q among W_Q (it lies below h_q, ..., h_{s-1}); one whose rank is s
// never does.  So the state of a roll is a count per rank c[q], the shared
// bits, R, and B = the sum of c[q] below R; one hash entering or leaving
// moves R by at most one.
//
// A hash is in the window while any of its records is: records of one hash
// at most span + 1 apart cover one stretch of target starts, so only a
// stretch's first record enters and only its last one leaves, and nothing
// counts occurrences.  The setup finds a record's previous occurrence with
// an open-addressing table of the span's hashes (no sort).
//
// What bounds it: instruction issue (setup) and the latency of the dependent
// shared-memory accesses (roll).  Events live in device memory (L2) so that
// shared memory holds 32 rolls per warp instead of the six or so whose
// events fit there; a lane reads its two event streams 16 bytes at a time,
// one load ahead.  Measured against the form that sorted a merged domain per
// run into shared-memory slots and took 32 runs per warp whatever their
// number: 1.26 M runs of a 200-genome batch 17.4 -> 4.1 ms, 2.5 M runs of a
// 240 Mbp assembly 19.7 -> 5.0 ms, 299 runs of a 2 Mbp genome 1.75 -> 0.08 ms.
// Runs beyond its limits (more than 256 query records,
// 512 span records, a span of 65,536 bases, more W_Q hashes than the launch's
// counters or a count past 255) go to the large kernel.

constexpr int kBWarps = 4;
constexpr int kBQC = 256, kBRC = 512;
constexpr int kEvWords = 8192;  // event words of a warp's stretch
constexpr int kEvPad = 16;      // read ahead past the last event
// event: position - j_a (bits 0-15), rank among W_Q (16-23), flags
constexpr uint32_t kEvW = 1u << 24;        // a W_Q hash
constexpr uint32_t kEvNoEnter = 1u << 25;  // its hash is already in the window
constexpr uint32_t kEvNoLeave = 1u << 26;  // its hash stays in the window
// hash table of a run's kept records: keys, then their last event index
constexpr int kBTabMax = 1024;
constexpr int kBTabWords = kBTabMax + kBTabMax / 2;

// Shared words of a warp for rolls with at most scap W_Q hashes: 8-bit
// counts and shared bits for 32 lanes, each lane in its own bank (the setup's
// hash table lies over them).  A count past 255 sends its run to the large
// kernel.  32 warps fit on an SM at w = 16; with counts of 16 bits and room
// for 256 W_Q hashes there were 20, and 2.5 M runs of a 240 Mbp assembly took
// 6.6 ms instead of 5.0, 1.26 M of a 200-genome batch 5.4 instead of 4.1.
__host__ __device__ constexpr int roll_words(int scap) {
  return (scap / 4 + scap / 32) * 32 > kBTabWords ? (scap / 4 + scap / 32) * 32 : kBTabWords;
}
__host__ __device__ constexpr size_t refine_warp_bytes(int scap) {
  return (size_t)scap * 5 + (size_t)roll_words(scap) * 4;
}

// Rolls one run (single lane) over target starts j_a + [0, jend].  cnt and sb
// are the lane's zeroed counters and shared bits (one 32-bit word per 32).
// False: a count ran over.
__device__ bool roll_run(const uint32_t* __restrict__ ev, int nrel, int s, int mx, int jend, int span,
                         uint32_t* cnt, uint32_t* sb, int* best_out, int* jstar_out) {
  const uint4* ev4 = reinterpret_cast<const uint4*>(ev);
  auto count = [&](int q) -> uint8_t& {
    return reinterpret_cast<uint8_t*>(cnt + ((q >> 2) << 5))[q & 3];
  };
  auto shared_bit = [&](int r) { return (int)((sb[(r >> 5) << 5] >> (r & 31)) & 1u); };
  uint4 eb = ev4[0], en = ev4[1], lb = eb, ln = en;  // next events of either stream
  int e = 0, l = 0, j = 0;
  int best = -1, jstar = 0;
  int R = s, B = 0, est = 0;
  while (true) {
    const int ne = e < nrel ? max((int)(eb.x & 0xFFFFu) - span, 0) : INT_MAX;
    const int nl = l < nrel ? (int)(lb.x & 0xFFFFu) + 1 : INT_MAX;
    const int nx = min(ne, nl);
    if (nx > j) {  // every event up to j is in
      if (est > best) {
        best = est;
        jstar = j;
        if (best >= mx) break;
      }
      if (nx > jend) break;
      j = nx;
    }
    if (ne <= nl) {
      const uint32_t v = eb.x;
      eb.x = eb.y;
      eb.y = eb.z;
      eb.z = eb.w;
      if ((++e & 3) == 0) {
        eb = en;
        en = ev4[(e >> 2) + 1];
      }
      if (v & kEvNoEnter) continue;
      const int q = (int)((v >> 16) & 0xFFu);
      if (v & kEvW) {
        sb[(q >> 5) << 5] |= 1u << (q & 31);
        if (q < R) ++est;
      } else {
        if (++count(q) == 0) return false;
        if (q < R && R + ++B > s) {
          --R;
          B -= count(R);
          est -= shared_bit(R);
        }
      }
    } else {
      const uint32_t v = lb.x;
      lb.x = lb.y;
      lb.y = lb.z;
      lb.z = lb.w;
      if ((++l & 3) == 0) {
        lb = ln;
        ln = ev4[(l >> 2) + 1];
      }
      if (v & kEvNoLeave) continue;
      const int q = (int)((v >> 16) & 0xFFu);
      if (v & kEvW) {
        sb[(q >> 5) << 5] &= ~(1u << (q & 31));
        if (q < R) --est;
      } else {
        --count(q);
        if (q < R) --B;
        if (q <= R && R < s) {
          const int c = count(R);
          if (R + 1 + B + c <= s) {
            B += c;
            est += shared_bit(R);
            ++R;
          }
        }
      }
    }
  }
  *best_out = best;
  *jstar_out = jstar;
  return true;
}

// Sorts 32 * NR keys held by a warp (key of index lane * NR + x in v[x]).
template <typename T, int NR>
__device__ __forceinline__ void warp_sort_regs(T (&v)[NR]) {
  const int lane = lane_id();
#pragma unroll
  for (int size = 2; size <= 32 * NR; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= NR) {
        const bool keep_min = (((lane * NR) & size) == 0) == ((lane & (stride / NR)) == 0);
#pragma unroll
        for (int x = 0; x < NR; ++x) {
          const T o = __shfl_xor_sync(0xffffffffu, v[x], stride / NR);
          v[x] = keep_min ? min(v[x], o) : max(v[x], o);
        }
      } else {
#pragma unroll
        for (int x = 0; x < NR; ++x) {
          if (x & stride) continue;
          const bool asc = ((lane * NR + x) & size) == 0;
          const T p = v[x], q = v[x | stride];
          v[x] = asc ? min(p, q) : max(p, q);
          v[x | stride] = asc ? max(p, q) : min(p, q);
        }
      }
    }
  }
}


// Query records [qa, qa + c) as sorted (hash << 1 | strand) keys in buf[0..32 * NR).
template <int NR>
__device__ __forceinline__ void sort_window(const uint64_t* __restrict__ qrec, int64_t qa, int c,
                                            uint32_t* buf) {
  const int lane = lane_id();
  uint32_t v[NR];
#pragma unroll
  for (int x = 0; x < NR; ++x) {
    const int at = x * 32 + lane;
    v[x] = kNone;
    if (at < c) {
      const uint64_t r = qrec[qa + at];
      v[x] = (rec_hash(r) << 1) | rec_strand(r);
    }
  }
  warp_sort_regs(v);
#pragma unroll
  for (int x = 0; x < NR; ++x) buf[lane * NR + x] = v[x];
}

__global__ void __launch_bounds__(32 * kBWarps) k_refine_batch(RefineArgs a) {
  a.nruns = live_n(a.nruns, a.dnruns);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  const int scap = a.scap;
  unsigned char* base_s = smem_raw + (size_t)warp * refine_warp_bytes(scap);
  uint32_t* scratch = reinterpret_cast<uint32_t*>(base_s);
  uint32_t* wq_h = scratch + roll_words(scap);
  uint8_t* wq_m = reinterpret_cast<uint8_t*>(wq_h + scap);
  const int64_t nwarps = (int64_t)gridDim.x * kBWarps;
  uint32_t* ev_base = a.events + ((int64_t)blockIdx.x * kBWarps + warp) * (a.ev_words + kEvPad);
  // few runs: spread them over the warps (one warp took 32 runs one after
  // another in 0.46 ms while the others had none); many: 32 neighbours at a
  // time, as runs of one window share W_Q
  int64_t chunk = (a.nruns + nwarps - 1) / nwarps;
  chunk = chunk < 1 ? 1 : (chunk > 32 ? 32 : chunk);
  int64_t prev_qa = -1, prev_qb = -1;
  int s = 0, smax = 0;
  int nslots = 0, used = 0;
  int64_t my_run = 0;  // this lane's run
  int my_off = 0, my_nrel = 0, my_s = 0;

  auto flush = [&]() {
    __syncwarp();
    const int nw = (scap / 4) * 32;  // counters, then shared bits
    uint4* z4 = reinterpret_cast<uint4*>(scratch);
    for (int x = lane; x < (smax + 3) / 4 * 8; x += 32) z4[x] = make_uint4(0, 0, 0, 0);
    for (int x = lane; x < (smax + 31) / 32 * 8; x += 32) z4[nw / 4 + x] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    if (lane < nslots) {
      const sedef_run_t run = a.runs[my_run];
      int best, jstar;
      if (roll_run(ev_base + my_off, my_nrel, my_s, run.max_shared, (int)(run.j_b - run.j_a), a.span,
                   scratch + lane, scratch + nw + lane, &best, &jstar)) {
        sedef_run_t& out = a.runs[my_run];
        out.est = (uint16_t)(best < 0 ? 0 : best);
        out.den = (uint16_t)my_s;
        out.j_star = run.j_a + (uint32_t)jstar;
        out.keep = (best >= a.mtab[my_s]) ? 1 : 0;
      } else {
        a.big[atomicAdd(a.nbig, 1u)] = (uint32_t)my_run;
      }
    }
    __syncwarp();
    nslots = 0;
    used = 0;
    smax = 0;
  };

  while (true) {
    int64_t c0 = 0;
    if (lane == 0) c0 = (int64_t)atomicAdd(a.next, (unsigned long long)chunk);
    c0 = __shfl_sync(0xffffffffu, c0, 0);
    if (c0 >= a.nruns) break;
    const int64_t c1 = min(a.nruns, c0 + chunk);
    for (int64_t ri = c0; ri < c1; ++ri) {
      const sedef_run_t run = a.runs[ri];
      const int64_t i = run.i;
      const int o = run.o;
      const uint4 rg = a.ranges[ri];
      const int64_t qa = rg.x, qb = rg.y, rlo = rg.z, rend = rg.w;
      const int c = (int)(qb - qa);
      const int nr = (int)(rend - rlo);
      bool big = c > kBQC || nr > kBRC || (int64_t)run.j_b + a.span - run.j_a >= 65536;
      // ---- W_Q (kept from the previous run of the same window)
      if (!big && (qa != prev_qa || qb != prev_qb)) {
        prev_qa = qa;
        prev_qb = qb;
        __syncwarp();
        uint32_t* buf = scratch;
        if (c <= 64) sort_window<2>(a.qrec, qa, c, buf);
        else if (c <= 128) sort_window<4>(a.qrec, qa, c, buf);
        else sort_window<8>(a.qrec, qa, c, buf);
        __syncwarp();
        s = 0;
        for (int base = 0; base < c; base += 32) {
          const int x = base + lane;
          uint32_t h = 0, mask = 0;
          bool first = false;
          if (x < c) {
            h = buf[x] >> 1;
            first = (x == 0) || ((buf[x - 1] >> 1) != h);
            if (first) {
              for (int y = x; y < c && (buf[y] >> 1) == h; ++y) mask |= 1u << (buf[y] & 1u);
              if (a.max_occ > 0 && (int)(a.toff[h + 1] - a.toff[h]) > a.max_occ) first = false;
            }
          }
          const unsigned bal = __ballot_sync(0xffffffffu, first);
          if (first) {
            const int d = s + __popc(bal & lanemask_lt());
            if (d < scap) {
              wq_h[d] = h;
              wq_m[d] = (uint8_t)mask;
            }
          }
          s += __popc(bal);
        }
        __syncwarp();
      }
      if (big || s > scap) {
        if (lane == 0) a.big[atomicAdd(a.nbig, 1u)] = (uint32_t)ri;
        continue;
      }
      if (nslots == 32 || used + nr + 8 > a.ev_words) flush();
      // ---- the span's hashes: a table with at most 5/8 of its slots taken
      const int tsz = nr <= 320 ? kBTabMax / 2 : kBTabMax;
      uint32_t* tab = scratch;
      uint16_t* tval = reinterpret_cast<uint16_t*>(scratch + tsz);
      __syncwarp();
      {
        uint4* z4 = reinterpret_cast<uint4*>(scratch);
        for (int x = lane; x < tsz / 4; x += 32) z4[x] = make_uint4(0, 0, 0, 0);
        for (int x = lane; x < tsz / 8; x += 32) z4[tsz / 4 + x] = make_uint4(kNone, kNone, kNone, kNone);
      }
      __syncwarp();
      // ---- one pass over the span records: rank among W_Q, whether the
      // record counts, its hash's previous occurrence, the event
      uint32_t* ev = ev_base + used;
      int nrel = 0;
      uint64_t ahead = lane < nr ? a.trec[rlo + lane] : 0;
      for (int base = 0; base < nr; base += 32) {
        const uint64_t r = ahead;
        const bool ok = base + lane < nr;
        if (base + 32 + lane < nr) ahead = a.trec[rlo + base + 32 + lane];
        const uint32_t h = rec_hash(r), t = rec_pos(r);
        const int q = lb_u32(wq_h, s, h);
        bool keep = ok && q < s;
        bool member = false;
        if (keep && wq_h[q] == h) {
          member = true;
          const bool self = a.self_mode && (int64_t)t >= i && (int64_t)t <= i + a.span;
          keep = !self && ((wq_m[q] >> (rec_strand(r) ^ (uint32_t)o)) & 1u);
        }
        const unsigned bk = __ballot_sync(0xffffffffu, keep);
        const int y = nrel + __popc(bk & lanemask_lt());
        uint32_t slot = 0;
        bool seen = false;
        if (keep) {
          slot = (h * 0x9E3779B1u) >> (nr <= 320 ? 23 : 22);
          while (true) {  // a free slot is always found
            const uint32_t old = atomicCAS(&tab[slot], 0u, h + 1u);
            if (old == 0u) break;
            if (old == h + 1u) {
              seen = true;
              break;
            }
            slot = (slot + 1u) & (uint32_t)(tsz - 1);
          }
        }
        uint32_t v = (t - run.j_a) | ((uint32_t)q << 16) | (member ? kEvW : 0u);
        bool last = true;  // the last record of its hash in these 32
        if (__any_sync(0xffffffffu, seen)) {
          // the previous occurrence: the nearest lower lane with the hash,
          // else the table's (written after an earlier 32)
          const unsigned peers = __match_any_sync(0xffffffffu, keep ? h : (0x80000000u | (uint32_t)lane));
          const unsigned lower = peers & lanemask_lt();
          const int pl = lower ? 31 - __clz(lower) : lane;
          const uint32_t pt = __shfl_sync(0xffffffffu, t, pl);
          last = (peers >> lane) == 1u;
          int py = -1;
          uint32_t gap = kNone;
          if (keep && lower) {
            py = nrel + __popc(bk & ((1u << pl) - 1u));
            gap = t - pt;
          } else if (seen && tval[slot] != 0xFFFFu) {
            py = tval[slot];
            gap = t - run.j_a - (ev[py] & 0xFFFFu);
          }
          const bool joined = py >= 0 && gap <= (uint32_t)a.span + 1u;
          if (joined) v |= kEvNoEnter;
          if (keep) ev[y] = v;
          __syncwarp();
          if (joined) ev[py] |= kEvNoLeave;  // one successor per record
        } else if (keep) {
          ev[y] = v;
        }
        if (keep && last) tval[slot] = (uint16_t)y;
        nrel += __popc(bk);
        __syncwarp();
      }
      if (lane == nslots) {
        my_run = ri;
        my_off = used;
        my_nrel = nrel;
        my_s = s;
      }
      ++nslots;
      used += (nrel + 3) & ~3;
      smax = max(smax, s);
    }
  }
  flush();
}

// Every run to the large kernel.
__global__ void k_refine_all(RefineArgs a) {
  const int64_t n = live_n(a.nruns, a.dnruns);
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x < n) a.big[x] = (uint32_t)x;
  if (x == 0) *a.nbig = (unsigned int)n;
}

// Per-run record ranges for the refine: query records of the run's window
// (from the window table) and target records of its span [j_a, j_b+n-k].
__global__ void k_run_ranges(const sedef_run_t* runs, int64_t n, const int64_t* qseq, int nqseq,
                             const int64_t* wbase, int step, const uint32_t* win_qa,
                             const uint32_t* win_qb, const uint64_t* trec, int64_t nt, int span,
                             uint4* ranges, const uint32_t* dn, const uint32_t* dnt) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= live_n(n, dn)) return;
  nt = live_n(nt, dnt);
  const sedef_run_t r = runs[x];
  const int sq = seq_of(qseq, nqseq, r.i);
  const int64_t w = wbase[sq] + ((int64_t)r.i - qseq[sq]) / step;
  auto pos_of = [](uint64_t v) { return (uint64_t)((v >> 1) & 0xFFFFFFFFull); };
  const int64_t lo = lower_bound_by(trec, 0, nt, (uint64_t)r.j_a, pos_of);
  // the span holds few records: gallop from lo
  const uint64_t end_pos = (uint64_t)r.j_b + (uint64_t)span + 1;
  int64_t stepg = 1, hi = lo;
  while (hi < nt && pos_of(trec[hi]) < end_pos) {
    hi = lo + stepg;
    stepg <<= 1;
  }
  if (hi > nt) hi = nt;
  const int64_t b = lower_bound_by(trec, lo + (stepg >> 2), hi, end_pos, pos_of);
  ranges[x] = make_uint4(win_qa[w], win_qb[w], (uint32_t)lo, (uint32_t)b);
}

// ------------------------------------------------------- tier launchers --

template <int TPB, int LCAP, int GCAP, int SLOTS = kSlots>
int launch_fast(sedef_ctx* ctx, const FArgs& a, const TierIO& io_in, int64_t max_windows,
                const char* name) {
  const size_t sm = sizeof(FastSmemT<TPB, LCAP, GCAP, SLOTS>);
  static_assert(sizeof(FastSmemT<TPB, LCAP, GCAP, SLOTS>) <= 227 * 1024,
                "a filter tier must fit one CTA's shared memory");
  SEDEF_TRY(ensure_smem_attr((const void*)k_filter_fast<TPB, LCAP, GCAP, SLOTS>, sm));
  // a table of 2,048 counters separates about as many hits: a window with
  // more passes nearly all of them on to its sort, and is better off in the
  // CTA tier (measured when these shapes came after the warp tier on every
  // pass: a 100 Mbp chromosome's tiers 17.6 ms with the line at twice as many
  // hits and 10.2 ms with it here; half as many: the next tier's fixed cost per
  // window, a 240 Mbp assembly's pass 57.0 -> 65.7 ms)
  TierIO io = io_in;
  io.hlim = (uint32_t)(SLOTS == kSlots ? SLOTS : 2 * SLOTS);
  int per_sm = 0;
  SEDEF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm,
                                                           k_filter_fast<TPB, LCAP, GCAP, SLOTS>,
                                                           TPB, sm));
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)ctx_sm_count(ctx) * per_sm;
  if (grid > max_windows) grid = max_windows;
  if (grid < 1) grid = 1;
  SEDEF_KERNEL(ctx, name,
               k_filter_fast<TPB, LCAP, GCAP, SLOTS><<<(int)grid, TPB, sm, ctx_stream(ctx)>>>(a, io));
  return SEDEF_OK;
}

using FastLaunch = int (*)(sedef_ctx*, const FArgs&, const TierIO&, int64_t, const char*);

// First-tier shapes the autotuner chooses from: threads per window, hits and
// dense groups the window may hold in shared memory.
const FastLaunch kTier1[] = {launch_fast<128, 2048, 512>, launch_fast<64, 1024, 256>,
                             launch_fast<256, 2048, 512>, launch_fast<128, 1024, 256>};
constexpr int kNumTier1 = 4;
// Second-tier shapes (windows the first tier could not hold).
const FastLaunch kTier2[] = {launch_fast<256, 8192, 2048>, launch_fast<256, 4096, 1024>,
                             launch_fast<512, 8192, 2048>};
constexpr int kNumTier2 = 3;
// Second wide tier: windows with more collected hits than the CTA tiers keep
// (regions with many homologous copies) or with a counter past 255, before
// the global path.  32,768
// (bin, o) slots and 16,384 collected hits.
constexpr int kWideSlots = 32768;
const FastLaunch kTierWide2 = launch_fast<512, 16384, 1024, kWideSlots>;
// The second wide tier in the form that fits beside the serving kernel
// (8,192 collected hits instead of 16,384), for a context whose tier cap
// leaves the full one out.
const FastLaunch kTierWideMid = launch_fast<512, 8192, 1024, kWideSlots>;
using WideMidSmem = FastSmemT<512, 8192, 1024, kWideSlots>;
static_assert(sizeof(FastSmemT<512, 8192, 2048, 2048>) <= kTierSmemFloor &&
                  sizeof(WindowSmemT<WarpDense>) * kWWarps <= kTierSmemFloor,
              "a tier that always runs needs more shared memory than a tier cap may be");
static_assert(sizeof(CtaSmemT<CtaNarrow>) <= kTierSmemFloor && sizeof(CtaSmemT<CtaBroad>) <= kTierSmemFloor &&
                  sizeof(CtaSmemT<CtaMid>) <= sizeof(WideMidSmem) &&
                  sizeof(CtaSmemT<CtaDeep>) <= sizeof(FastSmemT<512, 16384, 1024, kWideSlots>),
              "a CTA tier runs where its neighbour in the chain does");
// variant = (warp tier off) * 12 + t1 * kNumTier2 + t2
constexpr int kNumShapes = kNumTier1 * kNumTier2;
constexpr int kNumVariants = 2 * kNumShapes;

}  // namespace

int filter_variant_count() { return kNumVariants; }

int scan_exclusive_u32(sedef_ctx* ctx, const uint32_t* in, uint32_t* out, int64_t n,
                       uint32_t* d_total);

namespace {

// The global path (eager) over the windows a.ov_list[0..nov): hits counted
// per window, then batches of at most 2^27 hits emitted, radix-sorted by
// (window, o, t) and swept by dense group.  Adds the hits to
// *slow_hits_total.
int global_path_eager(sedef_ctx* ctx, const FArgs& a, int64_t nov, unsigned long long* counters,
                      int64_t* slow_hits_total) {
  cudaStream_t st = ctx_stream(ctx);
  // slow path: count, then batches of emit -> sort -> sweep
  unsigned long long* ocnt = (unsigned long long*)ctx_alloc(ctx, (size_t)(nov + 1) * 8);
  int32_t* os = (int32_t*)ctx_alloc(ctx, (size_t)(nov + 1) * 4);
  if (!ocnt || !os) return SEDEF_ERR_OOM;
  int64_t sgrid = nov < (int64_t)ctx_sm_count(ctx) * 4 ? nov : (int64_t)ctx_sm_count(ctx) * 4;
  SEDEF_KERNEL(ctx, "k_slow_count",
               k_slow_count<unsigned long long><<<(int)sgrid, kSThreads, 0, st>>>(a, nov, ocnt, os,
                                                                                  nullptr, nullptr));
  std::vector<unsigned long long> hc(nov + 1, 0);
  SEDEF_CUDA(cudaMemcpyAsync(hc.data(), ocnt, (size_t)nov * 8, cudaMemcpyDeviceToHost, st));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  std::vector<unsigned long long> base(nov + 1, 0);
  for (int64_t v = 0; v < nov; ++v) base[v + 1] = base[v] + hc[v];
  unsigned long long* d_base = (unsigned long long*)ctx_alloc(ctx, (size_t)(nov + 1) * 8);
  if (!d_base) return SEDEF_ERR_OOM;
  SEDEF_CUDA(cudaMemcpyAsync(d_base, base.data(), (size_t)(nov + 1) * 8, cudaMemcpyHostToDevice, st));
  *slow_hits_total += (int64_t)base[nov];
  const unsigned long long budget = 1ull << 27;  // hits per batch
  int64_t v0 = 0;
  while (v0 < nov) {
    int64_t v1 = v0 + 1;
    while (v1 < nov && base[v1 + 1] - base[v0] <= budget && v1 - v0 < (1 << 20)) ++v1;
    const unsigned long long nh = base[v1] - base[v0];
    // a batch's scratch goes back to the pool once the batch has run
    const std::vector<char> used_before = ctx_pool_snapshot(ctx);
    if (nh > 0) {
      uint64_t* keys = (uint64_t*)ctx_alloc(ctx, (size_t)nh * 8);
      uint32_t* vals = (uint32_t*)ctx_alloc(ctx, (size_t)nh * 4);
      uint64_t* skeys = (uint64_t*)ctx_alloc(ctx, (size_t)nh * 8);
      uint32_t* svals = (uint32_t*)ctx_alloc(ctx, (size_t)nh * 4);
      if (!keys || !vals || !skeys || !svals) return SEDEF_ERR_OOM;
      const int64_t nb = v1 - v0;
      int g = (int)(nb < (int64_t)ctx_sm_count(ctx) * 4 ? nb : (int64_t)ctx_sm_count(ctx) * 4);
      SEDEF_KERNEL(ctx, "k_slow_emit",
                   k_slow_emit<<<g, kSThreads, 0, st>>>(a, v0, v1, d_base, keys, vals, nullptr,
                                                        (int64_t)nh));
      int wbits = 0;
      while ((int64_t(1) << wbits) < nb) ++wbits;
      SEDEF_TRY(radix_sort_u64(ctx, keys, vals, skeys, svals, (int64_t)nh, 0, 33 + wbits));
      SlowTask* tasks = (SlowTask*)ctx_alloc(ctx, (size_t)nh * sizeof(SlowTask));
      if (!tasks) return SEDEF_ERR_OOM;
      SEDEF_CUDA(cudaMemsetAsync(counters + 6, 0, 8, st));
      // a warp per part of a window, up to eight CTAs per SM
      const int64_t gw = (nb * kGroupParts + 7) / 8, g8 = (int64_t)ctx_sm_count(ctx) * 8;
      const int g2 = (int)(gw < g8 ? gw : g8);
      SEDEF_KERNEL(ctx, "k_slow_groups",
                   k_slow_groups<<<g2, 256, 0, st>>>(a, v0, v1, d_base, os, skeys, tasks,
                                                     counters + 6, (int64_t)nh, nullptr,
                                                     (int64_t)nh));
      SEDEF_KERNEL(ctx, "k_slow_tasks",
                   k_slow_tasks<<<ctx_sm_count(ctx) * 8, 32 * kTaskWarps, 0, st>>>(
                       a, v0, d_base, os, skeys, svals, tasks, counters + 6, (int64_t)nh));
      SEDEF_CUDA(cudaStreamSynchronize(st));
    }
    ctx_pool_restore(ctx, used_before);
    v0 = v1;
  }
  return SEDEF_OK;
}

// Whether the ranges pay.  They cost a walk over all records whatever the
// windows; they save a window's records a look into the offset table, the hits
// before the window (half of the mean posting list) and, in a batch, the search
// for the genome's part of the list.  Measured with and without them (w = 16,
// n = 750: 87 records a window), the walk takes 36 ps a record and seven
// launches, the search of a planned pass 52; a window gains 0.75 ns at 10 Mbp,
// 2 to 3 at 100 Mbp, 11 at 1 Gbp, 6 to 13 in batches of 100 and 200 Mbp.
// Filter of 1 Gbp with windows every 250 bases 80.9 ms with, 123 without;
// every 3,000 equal; every 1 Mbp 3.8 and 0.23; of 10 Mbp 0.37 and 0.35; of 200
// genomes of 1 Mbp 1.7 and 7.0, every 5,000 bases 1.0 and 0.59.  Windows past
// the tiers' 256 records do not read them.
bool ranges_pay(const Derived& D, int64_t nwin, int64_t nt, bool planned) {
  const double records = 2.0 * (D.span + 1) / (D.w + 1);
  if (records > kQCap) return false;
  const double list = (double)nt / (double)(int64_t(1) << (2 * D.k));
  const double gain_ns = (double)nwin * records * ((D.self_mode == 2 ? 0.057 : 0.023) + 0.015 * list);
  const double cost_ns = planned ? 5e3 + 0.052 * (double)nt : 60e3 + 0.036 * (double)nt;
  return gain_ns > cost_ns;
}

// Every query record's useful posting range of a self-search, once (the tiers
// read them by record offset).  An eager pass walks the index when the query
// records are its records, with the same sequence offsets (walk); a planned
// pass, whose counts live on the device, searches per record.  With target
// starts at i + n - overlap or later and overlap <= n, only the entries after
// the record's own one can be hits.  SEDEF_ERR_OOM: no room for them (kernels
// that are queued by then only touch this function's own blocks).
int posting_ranges(sedef_ctx* ctx, const FArgs& a, int64_t nq, int64_t nt, const uint32_t* dnq, bool walk,
                   uint2** out) {
  cudaStream_t st = ctx_stream(ctx);
  uint2* qp = (uint2*)ctx_alloc(ctx, (size_t)nq * sizeof(uint2));
  if (!qp) return SEDEF_ERR_OOM;
  *out = qp;
  int64_t g = (nq + 255) / 256;
  if (g > (int64_t)ctx_sm_count(ctx) * 16) g = (int64_t)ctx_sm_count(ctx) * 16;
  if (g < 1) g = 1;
  if (!walk) {
    SEDEF_KERNEL(ctx, "k_qpost", k_qpost<<<(int)g, 256, 0, st>>>(a, nq, dnq, qp));
    return SEDEF_OK;
  }
  const int64_t nw = (a.ttotal + 31) >> 5;
  uint32_t* pbits = (uint32_t*)ctx_alloc(ctx, (size_t)(nw + 1) * 4);
  uint32_t* pcnt = (uint32_t*)ctx_alloc(ctx, (size_t)(nw + 1) * 4);
  uint32_t* pbef = (uint32_t*)ctx_alloc(ctx, (size_t)(nw + 1) * 4);
  RankWord* rw = (RankWord*)ctx_alloc(ctx, (size_t)(nw + 1) * sizeof(RankWord));
  const int64_t sblocks = ((a.ttotal - 1) >> kSeqShift) + 1;
  int32_t* stab = (int32_t*)ctx_alloc(ctx, (size_t)sblocks * 4);
  if (!pbits || !pcnt || !pbef || !rw || !stab) return SEDEF_ERR_OOM;
  int64_t gw = (nw + 255) / 256;
  if (gw > (int64_t)ctx_sm_count(ctx) * 16) gw = (int64_t)ctx_sm_count(ctx) * 16;
  if (gw < 1) gw = 1;
  SEDEF_CUDA(cudaMemsetAsync(pbits, 0, (size_t)(nw + 1) * 4, st));
  SEDEF_KERNEL(ctx, "k_pos_bits", k_pos_bits<<<(int)g, 256, 0, st>>>(a.qrec, nq, pbits));
  SEDEF_KERNEL(ctx, "k_pos_popc", k_pos_popc<<<(int)gw, 256, 0, st>>>(pbits, nw, pcnt));
  SEDEF_TRY(scan_exclusive_u32(ctx, pcnt, pbef, nw, pbef + nw));
  SEDEF_KERNEL(ctx, "k_rank_words", k_rank_words<<<(int)gw, 256, 0, st>>>(pbits, pbef, nw, rw));
  SEDEF_KERNEL(ctx, "k_seq_table",
               k_seq_table<<<(int)((sblocks + 255) / 256), 256, 0, st>>>(a.tseq, a.ntseq, sblocks, stab));
  int64_t gq = (nt + 1023) / 1024;
  if (gq > (int64_t)ctx_sm_count(ctx) * 8) gq = (int64_t)ctx_sm_count(ctx) * 8;
  uint64_t *pk = nullptr, *pks = nullptr;
  uint32_t *pv = nullptr, *pvs = nullptr;
  const std::vector<char> no_parts = ctx_pool_snapshot(ctx);
  if (nt >= kPartRecords) {
    pk = (uint64_t*)ctx_alloc(ctx, (size_t)nt * 8);
    pks = pk ? (uint64_t*)ctx_alloc(ctx, (size_t)nt * 8) : nullptr;
    pv = pks ? (uint32_t*)ctx_alloc(ctx, (size_t)nt * 4) : nullptr;
    pvs = pv ? (uint32_t*)ctx_alloc(ctx, (size_t)nt * 4) : nullptr;
    if (!pvs) pk = nullptr;  // no room under the context's cap
  }
  SEDEF_KERNEL(ctx, "k_qpost", k_qpost_index<<<(int)gq, 256, 0, st>>>(a, nt, rw, stab, qp, pk, pv));
  if (pk) {
    const int pb = bits_below(a.ttotal);
    // two CTAs per SM: the CTAs drift apart, and with more of them the
    // stretch of records being written no longer stays in L2 (119 M
    // records: 0.9 ms; four CTAs per SM 1.7, eight 4.4)
    const int64_t gp = (int64_t)ctx_sm_count(ctx) * 2;
    const int sorted = radix_sort_u64(ctx, pk, pv, pks, pvs, nt, 32 + (pb > 8 ? pb - 8 : 0), 32 + pb);
    if (sorted == SEDEF_ERR_OOM) {
      // no room for the sort's own scratch: straight to their records after all
      SEDEF_KERNEL(ctx, "k_qpost",
                   k_qpost_index<<<(int)gq, 256, 0, st>>>(a, nt, rw, stab, qp, nullptr, nullptr));
    } else {
      SEDEF_TRY(sorted);
      SEDEF_KERNEL(ctx, "k_qpost_place", k_qpost_place<<<(int)gp, 256, 0, st>>>(pks, pvs, nt, rw, qp));
    }
  }
  ctx_pool_restore(ctx, no_parts);
  return SEDEF_OK;
}

// Orders the `total` raw runs by (window, o, j_a) into `runs` and refines
// them (the winnowed MinHash estimate at every breakpoint of each run).
// druns / dnt: live counts of a planned pass (nullptr when eager).
int order_and_refine(sedef_ctx* ctx, const FArgs& a, const Derived& D, int nqseq,
                     const int64_t* d_wbase, int64_t nwin, const uint32_t* wqa, const uint32_t* wqb,
                     const uint64_t* qrec, int64_t nq, const uint64_t* trec, int64_t nt,
                     const uint32_t* toff, unsigned long long* counters, sedef_run_t* raw,
                     int64_t total, sedef_run_t* runs, const uint32_t* druns, const uint32_t* dnt) {
  cudaStream_t st = ctx_stream(ctx);
  // counters for a third more W_Q hashes than a window holds on average
  // (2 / (w + 1) of its starts): the sizes between runs differ by a few
  int scap = ((int)(1.35 * 2.0 * (D.span + 1) / (D.w + 1)) + 31) / 32 * 32;
  scap = scap < 64 ? 64 : (scap > kBQC ? kBQC : scap);
  const size_t batch_sm = refine_warp_bytes(scap) * kBWarps;
  SEDEF_TRY(ensure_smem_attr((const void*)k_refine_batch, batch_sm));
  SEDEF_TRY(ensure_smem_attr((const void*)k_refine<kMaxWindowRecs, 1024>,
                             sizeof(RefineWarpT<kMaxWindowRecs, 1024>) * kRWarpsBig));
  // order runs by (i, o); the sweep emits each window's runs in j order
  ctx_set_stage(ctx, "runsort");
  uint64_t* keys = (uint64_t*)ctx_alloc(ctx, (size_t)total * 8);
  uint64_t* skeys = (uint64_t*)ctx_alloc(ctx, (size_t)total * 8);
  uint32_t* perm = (uint32_t*)ctx_alloc(ctx, (size_t)total * 4);
  if (!keys || !skeys || !perm) return SEDEF_ERR_OOM;
  const int tb = (int)((total + 255) / 256);
  int wb = 1;
  while ((int64_t(1) << wb) < nwin) ++wb;
  const int tbits = bits_below(a.ttotal + 1);
  if (tbits + 1 + wb <= 64) {
    SEDEF_KERNEL(ctx, "k_run_keys",
                 k_run_keys<<<tb, 256, 0, st>>>(raw, total, a.qseq, nqseq, d_wbase, D.step, 0, tbits,
                                                keys, druns));
    SEDEF_TRY(radix_sort_u64(ctx, keys, nullptr, skeys, perm, total, 0, tbits + 1 + wb, druns));
  } else {
    // stable two-pass order: by j_a, then by (window, o)
    uint32_t* perm1 = (uint32_t*)ctx_alloc(ctx, (size_t)total * 4);
    uint32_t* perm2 = (uint32_t*)ctx_alloc(ctx, (size_t)total * 4);
    uint64_t* k2 = (uint64_t*)ctx_alloc(ctx, (size_t)total * 8);
    if (!perm1 || !perm2 || !k2) return SEDEF_ERR_OOM;
    SEDEF_KERNEL(ctx, "k_run_keys",
                 k_run_keys<<<tb, 256, 0, st>>>(raw, total, a.qseq, nqseq, d_wbase, D.step, 1, tbits,
                                                keys, druns));
    SEDEF_TRY(radix_sort_u64(ctx, keys, nullptr, skeys, perm1, total, 0, tbits, druns));
    SEDEF_KERNEL(ctx, "k_run_keys",
                 k_run_keys<<<tb, 256, 0, st>>>(raw, total, a.qseq, nqseq, d_wbase, D.step, 2, tbits,
                                                keys, druns));
    SEDEF_KERNEL(ctx, "k_permute_u64",
                 k_permute_u64<<<tb, 256, 0, st>>>(keys, perm1, total, k2, druns));
    SEDEF_TRY(radix_sort_u64(ctx, k2, nullptr, skeys, perm2, total, 0, wb + 1, druns));
    SEDEF_KERNEL(ctx, "k_compose_perm",
                 k_compose_perm<<<tb, 256, 0, st>>>(perm1, perm2, total, perm, druns));
  }
  SEDEF_KERNEL(ctx, "k_gather_runs",
               k_gather_runs<<<tb, 256, 0, st>>>(raw, perm, total, runs, druns));
  // refine: k_refine_batch over all runs, then the large kernel over the runs
  // it handed over (their count stays on the device)
  ctx_set_stage(ctx, "refine");
  uint32_t* big = (uint32_t*)ctx_alloc(ctx, (size_t)total * 4);
  if (!big) return SEDEF_ERR_OOM;
  RefineArgs ra;
  ra.runs = runs;
  ra.nruns = total;
  ra.qrec = qrec;
  ra.nq = nq;
  ra.trec = trec;
  ra.nt = nt;
  ra.dnruns = druns;
  ra.dnt = dnt;
  ra.toff = toff;
  ra.mtab = a.mtab;
  ra.span = D.span;
  ra.max_occ = D.max_occ;
  ra.self_mode = D.self_mode;
  ra.big = big;
  ra.nbig = (unsigned int*)(counters + 3);
  uint4* ranges = (uint4*)ctx_alloc(ctx, (size_t)total * sizeof(uint4));
  if (!ranges) return SEDEF_ERR_OOM;
  SEDEF_KERNEL(ctx, "k_run_ranges",
               k_run_ranges<<<tb, 256, 0, st>>>(runs, total, a.qseq, nqseq, d_wbase, D.step, wqa, wqb,
                                                trec, nt, D.span, ranges, druns, dnt));
  ra.ranges = ranges;
  ra.next = counters + 6;
  SEDEF_CUDA(cudaMemsetAsync(counters + 6, 0, 16, st));
  using Big = RefineWarpT<kMaxWindowRecs, 1024>;
  const size_t big_sm = sizeof(Big) * kRWarpsBig;
  int rper = 0;
  SEDEF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&rper, k_refine_batch, 32 * kBWarps,
                                                           batch_sm));
  if (rper < 1) rper = 1;
  int64_t rgrid = (total + kBWarps - 1) / kBWarps;
  if (rgrid > (int64_t)ctx_sm_count(ctx) * rper) rgrid = (int64_t)ctx_sm_count(ctx) * rper;
  if (rgrid < 1) rgrid = 1;
  // a warp's events: room for the runs it takes at a time; under a cap on the
  // context's scratch fewer warps, and where not even one CTA's fit the large
  // kernel takes every run
  ra.scap = scap;
  const std::vector<char> used_before = ctx_pool_snapshot(ctx);
  while (ctx_extras(ctx)) {
    const int64_t per_warp = (total + rgrid * kBWarps - 1) / (rgrid * kBWarps);
    ra.ev_words = per_warp * (kBRC + 8) < kEvWords ? (int)per_warp * (kBRC + 8) : kEvWords;
    ra.events = (uint32_t*)ctx_alloc(ctx, (size_t)(rgrid * kBWarps) * (ra.ev_words + kEvPad) * 4);
    if (ra.events || rgrid == 1) break;
    rgrid /= 2;
  }
  if (ra.events) {
    SEDEF_KERNEL(ctx, "k_refine",
                 k_refine_batch<<<(int)rgrid, 32 * kBWarps, batch_sm, st>>>(ra));
  } else {
    SEDEF_KERNEL(ctx, "k_refine_all", k_refine_all<<<tb, 256, 0, st>>>(ra));
  }
  SEDEF_KERNEL(ctx, "k_refine_big",
               k_refine<kMaxWindowRecs, 1024><<<ctx_sm_count(ctx), 32 * kRWarpsBig, big_sm,
                                                       st>>>(ra));
  ctx_pool_restore(ctx, used_before);  // the events
  return SEDEF_OK;
}

}  // namespace

int run_filter(sedef_ctx* ctx, const uint64_t* qrec, int64_t nq, const int64_t* h_qoff, int nqseq,
               const uint64_t* trec, const uint64_t* tsorted, const uint32_t* toff, int64_t nt,
               const int64_t* h_toff, int ntseq, const Derived& D, const int32_t* h_mtab,
               sedef_run_t* runs, int64_t cap, int64_t* nruns, int tune, Planned* pl) {
  cudaStream_t st = ctx_stream(ctx);
  StageScope stage(ctx, "filter");  // the caller's label comes back on return
  if (pl && tune) return fail(SEDEF_ERR_INVALID, "sedef_filter: no autotuning inside a planned pass");
  // live record counts of a planned pass (query and target are one sketch)
  const uint32_t* dnq = pl ? pl->n_rec : nullptr;
  const uint32_t* dnt = pl ? pl->n_rec : nullptr;
  // windows per query sequence
  std::vector<int64_t> wbase(nqseq + 1, 0);
  for (int s = 0; s < nqseq; ++s) {
    const int64_t len = h_qoff[s + 1] - h_qoff[s];
    const int64_t cnt = len >= D.n ? (len - D.n) / D.step + 1 : 0;
    wbase[s + 1] = wbase[s] + cnt;
  }
  const int64_t nwin = wbase[nqseq];
  *nruns = 0;
  if (nwin == 0 || nq == 0 || nt == 0) return SEDEF_OK;
  // uploads: query offsets, target offsets, window bases, m table
  const size_t up_bytes = (size_t)(nqseq + 1) * 8 * 2 + (size_t)(ntseq + 1) * 8 +
                          (size_t)(kMaxWindowRecs + 1) * 4;
  char* h_up = (char*)host_buf(ctx, pl, up_bytes + 64);
  char* d_up = (char*)ctx_alloc(ctx, up_bytes + 64);
  if (!h_up || !d_up) return SEDEF_ERR_OOM;
  size_t o = 0;
  int64_t* h_q = (int64_t*)(h_up + o);
  const size_t oq = o;
  std::memcpy(h_q, h_qoff, (size_t)(nqseq + 1) * 8);
  o += (size_t)(nqseq + 1) * 8;
  const size_t ot = o;
  std::memcpy(h_up + o, h_toff, (size_t)(ntseq + 1) * 8);
  o += (size_t)(ntseq + 1) * 8;
  const size_t ow = o;
  std::memcpy(h_up + o, wbase.data(), (size_t)(nqseq + 1) * 8);
  o += (size_t)(nqseq + 1) * 8;
  const size_t om = o;
  std::memcpy(h_up + o, h_mtab, (size_t)(kMaxWindowRecs + 1) * 4);
  SEDEF_CUDA(cudaMemcpyAsync(d_up, h_up, up_bytes, cudaMemcpyHostToDevice, st));

  uint32_t* wi = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* wqa = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* wqb = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  int32_t* wseq = (int32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* ovl = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* ovl1 = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* ovlw = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* ovlw2 = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  uint32_t* ovlx = (uint32_t*)ctx_alloc(ctx, (size_t)nwin * 4);
  if (!ovlw || !ovlw2 || !ovlx) return SEDEF_ERR_OOM;
  // [0] runs, [1] windows for the global path, [2] tier-1 work, [3] large
  // refine runs, [4] hits, [5] collected hits, [6]/[7] task and refine work,
  // [8] tier-2 work, [9] windows tier 1 handed to tier 2, [10] sample size,
  // [11] global-path hits (planned pass), [12]/[13] warp-tier hand-overs and
  // work, [14] windows for the broad CTA tier, [15] its work, [16]/[17] the
  // same for the deep CTA tier, [20] its work counter, [21] what it handed to
  // the second wide tier, [18]/[19] for the narrow CTA tier
  unsigned long long* counters = (unsigned long long*)ctx_alloc(ctx, 256);
  sedef_run_t* raw = (sedef_run_t*)ctx_alloc(ctx, (size_t)(cap > 0 ? cap : 1) * sizeof(sedef_run_t));
  if (!wi || !wqa || !wqb || !wseq || !ovl || !ovl1 || !counters || !raw) return SEDEF_ERR_OOM;

  SEDEF_CUDA(cudaMemsetAsync(counters, 0, 256, st));

  FArgs a;
  a.qrec = qrec;
  a.trec = trec;
  a.tsorted = tsorted;
  a.toff = toff;
  a.qseq = (const int64_t*)(d_up + oq);
  a.tseq = (const int64_t*)(d_up + ot);
  a.mtab = (const int32_t*)(d_up + om);
  a.win_i = wi;
  a.win_qa = wqa;
  a.win_qb = wqb;
  a.win_seq = wseq;
  a.nwin = nwin;
  a.ntseq = ntseq;
  a.nqseq = nqseq;
  a.ttotal = h_toff[ntseq];
  a.k = D.k;
  a.n = D.n;
  a.span = D.span;
  a.max_occ = D.max_occ;
  a.self_mode = D.self_mode;
  a.overlap = D.overlap;
  a.runs = raw;
  a.nruns = counters;
  a.run_cap = cap;
  a.ov_list = ovl;
  a.nov = (unsigned int*)(counters + 1);
  a.stats = counters + 4;

  a.qpost = nullptr;
  a.tsamp = nullptr;
  if (D.self_mode == 2) {
    // every posting search of a batch self-search starts from the samples
    const int64_t ns = (nt + kSampleStride - 1) >> kSampleShift;
    uint32_t* samp = (uint32_t*)ctx_alloc(ctx, (size_t)ns * 4);
    if (!samp) return SEDEF_ERR_OOM;
    int64_t g = (ns + 255) / 256;
    if (g > (int64_t)ctx_sm_count(ctx) * 16) g = (int64_t)ctx_sm_count(ctx) * 16;
    SEDEF_KERNEL(ctx, "k_sample_pos", k_sample_pos<<<(int)g, 256, 0, st>>>(tsorted, nt, dnt, samp));
    a.tsamp = samp;
  }
  a.after_own = D.overlap <= D.n ? 1 : 0;
  const std::vector<char> used_before = ctx_pool_snapshot(ctx);
  if (ctx_extras(ctx) && (D.self_mode == 2 || (D.self_mode == 1 && a.after_own)) &&
      ranges_pay(D, nwin, nt, pl != nullptr)) {
    // The walk ranks target positions among the query's, so both have to be
    // one array (the autotuner may be given others).
    const bool walk = !pl && qrec == trec && nq == nt && nqseq == ntseq &&
                      std::memcmp(h_qoff, h_toff, (size_t)(ntseq + 1) * sizeof(int64_t)) == 0;
    uint2* qp = nullptr;
    const int got = posting_ranges(ctx, a, nq, nt, dnq, walk, &qp);
    if (got == SEDEF_ERR_OOM) {
      // no room under the context's cap: the tiers look postings up themselves
      ctx_pool_restore(ctx, used_before);
      qp = nullptr;
    } else {
      SEDEF_TRY(got);
    }
    a.qpost = qp;
  }
  SEDEF_KERNEL(ctx, "k_windows",
               k_windows<<<(int)((nwin + 255) / 256), 256, 0, st>>>(
                   qrec, nq, a.qseq, nqseq, (const int64_t*)(d_up + ow), nwin, D.step, D.span, wi,
                   wqa, wqb, wseq, dnq));
  if (tune) {
    // time the warp tier (the variants with it launch the same kernels: it
    // stands for them as variant 0) and every shape that takes its place, on a
    // uniform sample of windows (at least 65,536 or a sixteenth of them, so
    // that a run lasts long enough to time); keep the fastest
    const int64_t want = nwin / 16 > 65536 ? nwin / 16 : 65536;
    const int64_t stride = nwin > want ? nwin / want : 1;
    std::vector<uint32_t> sample;
    for (int64_t w = 0; w < nwin; w += stride) sample.push_back((uint32_t)w);
    const unsigned int ns = (unsigned int)sample.size();
    uint32_t* d_sample = (uint32_t*)ctx_alloc(ctx, (size_t)ns * 4 + 8);
    if (!d_sample) return SEDEF_ERR_OOM;
    SEDEF_CUDA(cudaMemcpyAsync(d_sample, sample.data(), (size_t)ns * 4, cudaMemcpyHostToDevice, st));
    SEDEF_CUDA(cudaMemcpyAsync(counters + 10, &ns, 4, cudaMemcpyHostToDevice, st));
    cudaEvent_t e0, e1;
    SEDEF_CUDA(cudaEventCreate(&e0));
    SEDEF_CUDA(cudaEventCreate(&e1));
    int best_v = 0;
    float best_ms = 1e30f;
    for (int v = 0; v < kNumVariants; v = v == 0 ? kNumShapes : v + 1) {
      float ms = 0.f;
      const int sh = v % kNumShapes;
      const bool warp_tier = v < kNumShapes;
      float best_rep = 1e30f;
      for (int rep = 0; rep < 3; ++rep) {  // the first repetition warms up
        SEDEF_CUDA(cudaMemsetAsync(counters, 0, 80, st));
        SEDEF_CUDA(cudaMemsetAsync(counters + 12, 0, 80, st));
        TierIO io0{d_sample, (const unsigned int*)(counters + 10), ovlx,
                   (unsigned int*)(counters + 18), (unsigned int*)(counters + 13), 0};
        TierIO io{d_sample, (const unsigned int*)(counters + 10), ovl1,
                  (unsigned int*)(counters + 9), (unsigned int*)(counters + 2), 0};
        io.wide_list = ovlx;
        io.wide_count = (unsigned int*)(counters + 18);
        TierIO io2{ovl1, (const unsigned int*)(counters + 9), ovlx, (unsigned int*)(counters + 18),
                   (unsigned int*)(counters + 8), 0};
        TierIO iox{ovlx, (const unsigned int*)(counters + 18), ovlw, (unsigned int*)(counters + 14),
                   (unsigned int*)(counters + 19), 0};
        TierIO iow{ovlw, (const unsigned int*)(counters + 14), ovlw2,
                   (unsigned int*)(counters + 16), (unsigned int*)(counters + 15), 0};
        TierIO iod{ovlw2, (const unsigned int*)(counters + 16), ovl1,
                   (unsigned int*)(counters + 21), (unsigned int*)(counters + 20), 0};
        TierIO iow2{ovl1, (const unsigned int*)(counters + 21), ovl,
                    (unsigned int*)(counters + 1), (unsigned int*)(counters + 17), 0};
        SEDEF_CUDA(cudaEventRecord(e0, st));
        if (warp_tier) {
          SEDEF_TRY(launch_warp_tier(ctx, a, io0, ns, D.w, "k_filter_tune"));
        } else {
          SEDEF_TRY(kTier1[sh / kNumTier2](ctx, a, io, ns, "k_filter_tune"));
          SEDEF_TRY(kTier2[sh % kNumTier2](ctx, a, io2, ns, "k_filter_tune"));
        }
        SEDEF_TRY(launch_cta_tier<CtaNarrow>(ctx, a, iox, ns, "k_filter_tune"));
        SEDEF_TRY(launch_cta_tier<CtaBroad>(ctx, a, iow, ns, "k_filter_tune"));
        SEDEF_TRY(launch_cta_tier<CtaDeep>(ctx, a, iod, ns, "k_filter_tune"));
        SEDEF_TRY(kTierWide2(ctx, a, iow2, ns, "k_filter_tune"));
        SEDEF_CUDA(cudaEventRecord(e1, st));
        SEDEF_CUDA(cudaEventSynchronize(e1));
        SEDEF_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        if (rep > 0 && ms < best_rep) best_rep = ms;
      }
      ms = best_rep;
      if (ms < best_ms) {
        best_ms = ms;
        best_v = v;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    ctx_set_filter_variant(ctx, best_v);
    *nruns = best_v;
    return SEDEF_OK;
  }
  {
    // the warp tier over all windows, or where the variant leaves it out tier
    // 1 (autotuned shape) over all windows and tier 2 (4,096-8,192 hits in
    // shared memory) over what it could not hold; the CTA tiers over the
    // windows those hand on, the second wide tier after that, the global path
    // last
    int v = ctx_filter_variant(ctx);
    if (v < 0 || v >= kNumVariants) v = 0;
    const int sh = v % kNumShapes;
    const bool warp_tier = v < kNumShapes;
    if (warp_tier) {
      TierIO io0{nullptr, nullptr, ovlx, (unsigned int*)(counters + 18),
                 (unsigned int*)(counters + 13), 1};
      SEDEF_TRY(launch_warp_tier(ctx, a, io0, nwin, D.w, "k_filter_warp"));
    } else {
      TierIO io1{nullptr, nullptr, ovl1, (unsigned int*)(counters + 9),
                 (unsigned int*)(counters + 2), 1};
      io1.wide_list = ovlx;
      io1.wide_count = (unsigned int*)(counters + 18);
      SEDEF_TRY(kTier1[sh / kNumTier2](ctx, a, io1, nwin, "k_filter_fast"));
      TierIO io2{ovl1, (const unsigned int*)(counters + 9), ovlx, (unsigned int*)(counters + 18),
                 (unsigned int*)(counters + 8), 1};
      SEDEF_TRY(kTier2[sh % kNumTier2](ctx, a, io2, nwin, "k_filter_mid"));
    }
    TierIO iox{ovlx, (const unsigned int*)(counters + 18), ovlw, (unsigned int*)(counters + 14),
               (unsigned int*)(counters + 19), 1};
    SEDEF_TRY(launch_cta_tier<CtaNarrow>(ctx, a, iox, nwin, "k_filter_cta"));
    // where the deep and the second wide tier's CTA would pass the context's
    // cap, their
    // 8,192-hit form takes its place, or, where that would pass it too, the
    // wide tier hands its leftovers straight to the global path
    const size_t scap = ctx_tier_smem_cap(ctx);
    const bool wide2 = sizeof(FastSmemT<512, 16384, 1024, kWideSlots>) <= scap;
    const bool mid = !wide2 && sizeof(WideMidSmem) <= scap;
    const bool second = wide2 || mid;
    TierIO iow{ovlw, (const unsigned int*)(counters + 14), second ? ovlw2 : ovl,
               (unsigned int*)(counters + (second ? 16 : 1)), (unsigned int*)(counters + 15), 1};
    SEDEF_TRY(launch_cta_tier<CtaBroad>(ctx, a, iow, nwin, "k_filter_wide"));
    TierIO iod{ovlw2, (const unsigned int*)(counters + 16), ovl1, (unsigned int*)(counters + 21),
               (unsigned int*)(counters + 20), 1};
    TierIO iow2{ovl1, (const unsigned int*)(counters + 21), ovl, (unsigned int*)(counters + 1),
                (unsigned int*)(counters + 17), 1};
    if (wide2) {
      SEDEF_TRY(launch_cta_tier<CtaDeep>(ctx, a, iod, nwin, "k_filter_deep"));
      SEDEF_TRY(kTierWide2(ctx, a, iow2, nwin, "k_filter_wide2"));
    } else if (mid) {
      SEDEF_TRY(launch_cta_tier<CtaMid>(ctx, a, iod, nwin, "k_filter_deep"));
      SEDEF_TRY(kTierWideMid(ctx, a, iow2, nwin, "k_filter_widemid"));
    }
  }
  // only the tiers read the posting ranges: what follows may use their memory
  ctx_pool_restore(ctx, used_before);
  a.qpost = nullptr;

  unsigned long long* h_cnt = nullptr;
  int64_t nov = 0, slow_hits_total = 0;
  if (pl) {
    // planned: the global path over the live overflow list in one batch of
    // at most pl->slow_hits hits
    const uint32_t* dnov = (const uint32_t*)(counters + 1);
    const int64_t H = pl->slow_hits > 0 ? pl->slow_hits : 1;
    uint32_t* cnt32 = (uint32_t*)ctx_alloc(ctx, (size_t)(nwin + 1) * 4);
    uint32_t* base32 = (uint32_t*)ctx_alloc(ctx, (size_t)(nwin + 1) * 4);
    unsigned long long* d_base = (unsigned long long*)ctx_alloc(ctx, (size_t)(nwin + 1) * 8);
    int32_t* os = (int32_t*)ctx_alloc(ctx, (size_t)(nwin + 1) * 4);
    uint64_t* keys = (uint64_t*)ctx_alloc(ctx, (size_t)H * 8);
    uint32_t* vals = (uint32_t*)ctx_alloc(ctx, (size_t)H * 4);
    uint64_t* skeys = (uint64_t*)ctx_alloc(ctx, (size_t)H * 8);
    uint32_t* svals = (uint32_t*)ctx_alloc(ctx, (size_t)H * 4);
    SlowTask* tasks = (SlowTask*)ctx_alloc(ctx, (size_t)H * sizeof(SlowTask));
    if (!cnt32 || !base32 || !d_base || !os || !keys || !vals || !skeys || !svals || !tasks)
      return SEDEF_ERR_OOM;
    SEDEF_CUDA(cudaMemsetAsync(cnt32, 0, (size_t)(nwin + 1) * 4, st));
    const int sgrid = (int)(nwin < (int64_t)ctx_sm_count(ctx) * 4 ? nwin : (int64_t)ctx_sm_count(ctx) * 4);
    SEDEF_KERNEL(ctx, "k_slow_count",
                 k_slow_count<uint32_t><<<sgrid, kSThreads, 0, st>>>(a, nwin, cnt32, os, dnov,
                                                                     counters + 11));
    // 32-bit offsets: a window whose range wraps is skipped; the exact
    // 64-bit total (counters[11]) decides the overflow
    SEDEF_TRY(scan_exclusive_u32(ctx, cnt32, base32, nwin, base32 + nwin));
    SEDEF_KERNEL(ctx, "k_widen_u32",
                 k_widen_u32<<<(int)((nwin + 256) / 256), 256, 0, st>>>(base32, nwin + 1, d_base));
    const uint32_t* dhits = base32 + nwin;
    SEDEF_TRY(plan_check64(ctx, pl, counters + 11, H, 1));
    SEDEF_KERNEL(ctx, "k_slow_emit",
                 k_slow_emit<<<sgrid, kSThreads, 0, st>>>(a, 0, nwin, d_base, keys, vals, dnov, H));
    int wbits = 0;
    while ((int64_t(1) << wbits) < nwin) ++wbits;
    SEDEF_TRY(radix_sort_u64(ctx, keys, vals, skeys, svals, H, 0, 33 + wbits, dhits));
    SEDEF_CUDA(cudaMemsetAsync(counters + 6, 0, 8, st));
    const int64_t gw = (nwin * kGroupParts + 7) / 8, g8 = (int64_t)ctx_sm_count(ctx) * 8;
    const int g2 = (int)(gw < g8 ? gw : g8);
    SEDEF_KERNEL(ctx, "k_slow_groups",
                 k_slow_groups<<<g2, 256, 0, st>>>(a, 0, nwin, d_base, os, skeys, tasks,
                                                   counters + 6, H, dnov, H));
    SEDEF_KERNEL(ctx, "k_slow_tasks",
                 k_slow_tasks<<<ctx_sm_count(ctx) * 8, 32 * kTaskWarps, 0, st>>>(
                     a, 0, d_base, os, skeys, svals, tasks, counters + 6, H));
  } else {
    h_cnt = (unsigned long long*)ctx_host(ctx, 64);
    if (!h_cnt) return SEDEF_ERR_OOM;
    SEDEF_CUDA(cudaMemcpyAsync(h_cnt, counters, 16, cudaMemcpyDeviceToHost, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));
    nov = (int64_t)(h_cnt[1] & 0xFFFFFFFFull);
  }

  if (nov > 0) {
    SEDEF_TRY(global_path_eager(ctx, a, nov, counters, &slow_hits_total));
    SEDEF_CUDA(cudaMemcpyAsync(h_cnt, counters, 8, cudaMemcpyDeviceToHost, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));
  }
  // runs: the exact count (eager) or the planned capacity with the live
  // count on the device (the low word of counters[0])
  const uint32_t* druns = nullptr;
  int64_t total;
  if (pl) {
    total = cap;
    druns = (const uint32_t*)counters;
    pl->n_runs = druns;
    SEDEF_TRY(plan_check(ctx, pl, druns, cap, 2));
    *nruns = cap;
    if (total == 0) return SEDEF_OK;
  } else {
    total = (int64_t)h_cnt[0];
    *nruns = total;
    if (total > cap) return fail(SEDEF_ERR_CAPACITY, "sedef_filter: run buffer too small");
    if (total == 0) return SEDEF_OK;
  }
  SEDEF_TRY(order_and_refine(ctx, a, D, nqseq, (const int64_t*)(d_up + ow), nwin, wqa, wqb, qrec,
                             nq, trec, nt, toff, counters, raw, total, runs, druns, dnt));
  if (pl) return SEDEF_OK;
  SEDEF_CUDA(cudaMemcpyAsync(h_cnt, counters, 64, cudaMemcpyDeviceToHost, st));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  {
    const int64_t stats[7] = {nwin, nov, (int64_t)h_cnt[4], (int64_t)h_cnt[5], total,
                              (int64_t)(h_cnt[3] & 0xFFFFFFFFull), slow_hits_total};
    ctx_set_stats(ctx, stats, 7);
  }
  return SEDEF_OK;
}

}  // namespace sedef

// ===================================================== continuous batching ==
//
// Serving against a resident target index.  A persistent kernel (one small
// CTA per SM, so that every SM keeps room for the kernels of other streams)
// drains a work queue of query windows: a
// ring of (slot, window) items in mapped host memory that the host
// publishes as requests are admitted into free slots.  A slot holds one
// request's query sketch, window table and outputs in device memory that
// the server allocated once.  A CTA claims an item only when the ring holds
// one (compare-and-swap on the device head below the published tail), runs
// the window through the shared-memory tier into its slot's runs (windows
// the tier cannot hold into the slot's overflow list), and the CTA that
// finishes a slot's last window writes the slot's epoch into a mapped
// completion word.  The host then runs the global path for the overflow
// windows, the run ordering, refine, chaining and merging of that slot on
// its own stream while the kernel keeps serving the other slots.  A CTA that
// finds the ring empty sleeps and polls; when nothing arrives for
// idle_timeout (or the host raises the stop word) it leaves, and a CTA that
// left on the idle limit records SEDEF_ERR_TIMEOUT in the control block.
// The host relaunches the kernel when work arrives and no CTA is running.
// Query-side data is read past L1 (a slot's buffers are refilled while the
// kernel runs).
namespace sedef {
namespace {

constexpr int kServeMaxSlots = 64;
// One CTA per SM of 256 threads (16 K registers) and ~53 KB of shared
// memory: the rest of every SM stays free for the admission and finishing
// kernels (a CTA of the deep and second wide tiers takes 32 K registers, a sort
// pass 16 to 20 K), which would otherwise wait for the persistent kernel to
// leave.
constexpr int kServeTPB = CtaNarrow::TPB;
using ServeSmem = CtaSmemT<CtaNarrow>;
// Windows with more posting entries than the shape keeps go to the slot's
// wide list before they are read; the finishing call runs the broad CTA tier
// over them as an ordinary launch beside k_serve, as the narrow one of a
// whole-genome pass hands them on.
// Finishing calls that may run at once (each on its own stream and context).
constexpr int kServeFinishers = 5;

struct ServeItem {
  uint32_t slot, window;
};

// Control block in mapped host memory (both sides read and write it).
struct ServeCtl {
  unsigned long long tail;                   // items published (host)
  int stop;                                  // host: leave now
  int status;                                // device: SEDEF_ERR_TIMEOUT after an idle exit
  long long nwin[kServeMaxSlots];            // host: windows of the slot's request
  unsigned int epoch[kServeMaxSlots];        // host: admission number of the slot
  unsigned int done_epoch[kServeMaxSlots];   // device: epoch whose last window finished
};

// Per-slot constants in device memory (written once, at creation).
struct SlotDev {
  FArgs a;              // the slot's query, windows and outputs
  unsigned int* done;   // windows finished (reset at admission)
  uint32_t* wide_list;  // windows with more hits than k_serve keeps (for the broad CTA tier)
  unsigned int* wide_count;
  uint32_t* mid_list;   // windows k_serve could not hold (for the 8,192-hit tier)
  unsigned int* mid_count;
};

struct ServeArgs {
  const SlotDev* slots;
  const ServeItem* ring;     // mapped host memory (device view)
  unsigned long long ring_cap;
  ServeCtl* ctl;             // mapped host memory (device view)
  unsigned long long* head;  // device memory
  unsigned long long idle_ns;
};

__device__ __forceinline__ unsigned long long ld_acquire_sys(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.sys.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__global__ void __launch_bounds__(kServeTPB) k_serve(ServeArgs sv) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ServeSmem& S = *reinterpret_cast<ServeSmem*>(smem_raw);
  __shared__ long long s_item;
  __shared__ unsigned int s_slot, s_window;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) {
      // claim the next published item; sleep while there is none, at most
      // idle_ns in a row
      long long got = -1;
      const unsigned long long idle_from = global_ns();
      unsigned int nap = 256;
      while (true) {
        const unsigned long long t = ld_acquire_sys(&sv.ctl->tail);
        const unsigned long long h = *(volatile unsigned long long*)sv.head;
        if (h < t) {
          if (atomicCAS(sv.head, h, h + 1) == h) {
            got = (long long)h;
            break;
          }
          continue;
        }
        if (*(volatile int*)&sv.ctl->stop) break;
        if (global_ns() - idle_from > sv.idle_ns) {
          *(volatile int*)&sv.ctl->status = SEDEF_ERR_TIMEOUT;
          __threadfence_system();
          break;
        }
        __nanosleep(nap);
        if (nap < 8192) nap <<= 1;
      }
      s_item = got;
      if (got >= 0) {
        const volatile ServeItem* it = sv.ring + (unsigned long long)got % sv.ring_cap;
        s_slot = it->slot;
        s_window = it->window;
      }
    }
    __syncthreads();
    if (s_item < 0) break;
    const unsigned int slot = s_slot;
    const SlotDev& sd = sv.slots[slot];
    TierIO io;
    io.in_list = nullptr;
    io.in_count = nullptr;
    io.out_list = sd.mid_list;
    io.out_count = sd.mid_count;
    io.next = nullptr;
    io.stats = 1;
    io.wide_list = sd.wide_list;
    io.wide_count = sd.wide_count;
    cta_window(sd.a, io, S, (int64_t)s_window);
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();  // this window's runs and hand-overs before its count
      const unsigned int d = atomicAdd(sd.done, 1u) + 1u;
      if ((long long)d == *(volatile long long*)&sv.ctl->nwin[slot]) {
        __threadfence_system();
        *(volatile unsigned int*)&sv.ctl->done_epoch[slot] =
            *(volatile unsigned int*)&sv.ctl->epoch[slot];
        __threadfence_system();
      }
    }
  }
}

}  // namespace

// Host side of one server.
struct Server {
  int device = 0;
  int nslots = 0;
  int64_t slot_bases = 0;
  Derived D;
  sedef_params P;
  std::vector<int32_t> mtab;
  // the resident target (owned by the caller)
  const uint64_t* trec = nullptr;
  const uint64_t* tsorted = nullptr;
  const uint32_t* toff = nullptr;
  int64_t nt = 0;
  std::vector<int64_t> h_toff;
  // streams and contexts: admission, the persistent kernel, finishing (one
  // stream and context per concurrent sedef_server_finish call)
  cudaStream_t s_prep = nullptr, s_kern = nullptr;
  sedef_ctx* c_prep = nullptr;
  struct Finisher {
    cudaStream_t stream = nullptr;
    sedef_ctx* ctx = nullptr;
    bool busy = false;
  };
  std::vector<Finisher> fins;
  std::condition_variable fin_cv;
  cudaEvent_t kern_done = nullptr;
  bool kern_launched = false;
  char* d_shared = nullptr;  // target offsets and the m table
  // mapped host memory: host views and device views
  ServeCtl* ctl = nullptr;
  ServeCtl* d_ctl = nullptr;
  ServeItem* ring = nullptr;
  ServeItem* d_ring = nullptr;
  unsigned long long ring_cap = 0;
  unsigned long long tail = 0;
  unsigned long long* d_head = nullptr;
  SlotDev* d_slots = nullptr;
  double idle_s = 1.0;
  struct Slot {
    uint8_t* seq = nullptr;
    uint32_t *packed = nullptr, *mask = nullptr, *nbits = nullptr;
    uint64_t* qrec = nullptr;
    int64_t rec_cap = 0;
    uint32_t *wi = nullptr, *wqa = nullptr, *wqb = nullptr, *ov = nullptr, *wl = nullptr,
             *ml = nullptr;
    int32_t* wseq = nullptr;
    int64_t win_cap = 0;
    sedef_run_t* raw = nullptr;
    int64_t run_cap = 0;
    unsigned long long* counters = nullptr;  // 32 words, as in the filter
    unsigned int* done = nullptr;
    char* d_up = nullptr;                    // query offsets (2) and window bases (2)
    int state = 0;                           // 0 free, 1 admitted, 2 queued, 3 filtered
    unsigned int epoch = 0;
    int64_t len = 0, nrec = 0, nwin = 0;
    FArgs a;
    // candidates of a finished slot kept until the caller's buffer holds them
    std::vector<sedef_cand_t> fin;
    bool fin_ready = false;
  };
  std::vector<Slot> slots;
  std::vector<void*> dev_allocs;
  std::mutex mu;
};

namespace {

// Shared memory per CTA that other kernels find on an SM beside one k_serve
// CTA: the largest split (228 KB) less k_serve's block and the 1 KB the SM
// reserves for each of the two CTAs.
int64_t server_smem_left() { return 228 * 1024 - (int64_t)sizeof(ServeSmem) - 2 * 1024; }
static_assert(228 * 1024 - sizeof(ServeSmem) - 2 * 1024 >= kTierSmemFloor &&
                  228 * 1024 - sizeof(ServeSmem) - 2 * 1024 >= sizeof(WideMidSmem),
              "the finishing tiers must fit beside k_serve");

int server_alloc(Server* s, void** p, size_t bytes) {
  if (cudaMalloc(p, bytes ? bytes : 256) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return fail(SEDEF_ERR_OOM, "server: device allocation failed");
  }
  s->dev_allocs.push_back(*p);
  return SEDEF_OK;
}

// Launches the persistent kernel unless a launch is still running.  Caller
// holds mu.
int server_kick(Server* s) {
  if (s->kern_launched) {
    const cudaError_t q = cudaEventQuery(s->kern_done);
    if (q == cudaErrorNotReady) return SEDEF_OK;
    if (q != cudaSuccess) return cuda_fail(q, "server: kernel event");
  }
  __atomic_store_n(&s->ctl->status, 0, __ATOMIC_RELEASE);
  ServeArgs sv;
  sv.slots = s->d_slots;
  sv.ring = s->d_ring;
  sv.ring_cap = s->ring_cap;
  sv.ctl = s->d_ctl;
  sv.head = s->d_head;
  sv.idle_ns = (unsigned long long)(s->idle_s * 1e9);
  k_serve<<<ctx_sm_count(s->c_prep), kServeTPB, sizeof(ServeSmem), s->s_kern>>>(sv);
  count_launch();
  SEDEF_LAUNCHED("k_serve");
  SEDEF_CUDA(cudaEventRecord(s->kern_done, s->s_kern));
  s->kern_launched = true;
  return SEDEF_OK;
}

// Admission work of one slot on the prep stream: query upload, pack,
// sketch, window table, counters; synchronizes.
int server_prepare(Server* s, Server::Slot& L, const uint8_t* h_query, int64_t len) {
  sedef_ctx* c = s->c_prep;
  cudaStream_t st = s->s_prep;
  ctx_pool_reset(c);
  if (len == 0) {
    L.len = L.nrec = L.nwin = 0;
    return SEDEF_OK;
  }
  SEDEF_CUDA(cudaMemcpyAsync(L.seq, h_query, (size_t)len, cudaMemcpyHostToDevice, st));
  SEDEF_TRY(launch_pack(c, L.seq, len, L.packed, L.mask, L.nbits));
  const int64_t qoff[2] = {0, len};
  int64_t nrec = 0;
  SEDEF_TRY(run_sketch(c, L.packed, L.mask, L.nbits, qoff, 1, s->D, L.qrec, L.rec_cap, &nrec));
  if (nrec > L.rec_cap) return fail(SEDEF_ERR_CAPACITY, "server: sketch exceeds the slot");
  const int64_t nwin = len >= s->D.n ? (len - s->D.n) / s->D.step + 1 : 0;
  const int64_t up[4] = {0, len, 0, nwin};  // query offsets, window bases
  int64_t* h_up = (int64_t*)ctx_host(c, 64);
  if (!h_up) return SEDEF_ERR_OOM;
  std::memcpy(h_up, up, sizeof(up));
  SEDEF_CUDA(cudaMemcpyAsync(L.d_up, h_up, sizeof(up), cudaMemcpyHostToDevice, st));
  SEDEF_CUDA(cudaMemsetAsync(L.counters, 0, 256 + 64, st));
  if (nwin > 0 && nrec > 0)
    SEDEF_KERNEL(c, "k_windows",
                 k_windows<<<(int)((nwin + 255) / 256), 256, 0, st>>>(
                     L.qrec, nrec, (const int64_t*)L.d_up, 1, (const int64_t*)L.d_up + 2, nwin,
                     s->D.step, s->D.span, L.wi, L.wqa, L.wqb, L.wseq, nullptr));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  L.len = len;
  L.nrec = nrec;
  L.nwin = (nrec > 0) ? nwin : 0;
  L.a.qrec = L.qrec;
  L.a.nwin = L.nwin;
  return SEDEF_OK;
}

}  // namespace
}  // namespace sedef

extern "C" {

using sedef::Server;

int sedef_server_destroy(sedef_server* srv) {
  using namespace sedef;
  Server* s = (Server*)srv;
  if (!s) return SEDEF_OK;
  cudaSetDevice(s->device);
  if (s->ctl) {
    __atomic_store_n(&s->ctl->stop, 1, __ATOMIC_RELEASE);
    if (s->kern_launched) cudaEventSynchronize(s->kern_done);
  }
  if (s->s_prep) cudaStreamSynchronize(s->s_prep);
  for (auto& F : s->fins)
    if (F.stream) cudaStreamSynchronize(F.stream);
  if (s->c_prep) sedef_destroy(s->c_prep);
  for (auto& F : s->fins)
    if (F.ctx) sedef_destroy(F.ctx);
  for (void* p : s->dev_allocs) cudaFree(p);
  if (s->ctl) cudaFreeHost(s->ctl);
  if (s->ring) cudaFreeHost(s->ring);
  if (s->kern_done) cudaEventDestroy(s->kern_done);
  if (s->s_prep) cudaStreamDestroy(s->s_prep);
  if (s->s_kern) cudaStreamDestroy(s->s_kern);
  for (auto& F : s->fins)
    if (F.stream) cudaStreamDestroy(F.stream);
  delete s;
  return SEDEF_OK;
}

int sedef_server_create(sedef_ctx* ctx, const uint64_t* d_trec, const uint64_t* d_tsorted,
                        const uint32_t* d_toff, int64_t nt, const int64_t* h_toff, int32_t ntseq,
                        const sedef_params* p, int32_t slots, int64_t slot_bases,
                        double idle_timeout_s, sedef_server** out) {
  using namespace sedef;
  if (!ctx || !out || !p) return fail(SEDEF_ERR_INVALID, "NULL argument");
  *out = nullptr;
  Derived D;
  SEDEF_TRY(derive(p, &D));
  if (D.self_mode != 0) return fail(SEDEF_ERR_INVALID, "sedef_server_create: self_mode must be 0");
  if (slots < 1 || slots > kServeMaxSlots)
    return fail(SEDEF_ERR_INVALID, "sedef_server_create: slots must be in [1, 64]");
  if (slot_bases < D.n || slot_bases >= (int64_t(1) << 31))
    return fail(SEDEF_ERR_INVALID, "sedef_server_create: slot_bases must be in [n, 2^31)");
  if (!(idle_timeout_s > 0 && idle_timeout_s < 3600))
    return fail(SEDEF_ERR_INVALID, "sedef_server_create: idle timeout must be in (0, 3600) s");
  if (ntseq < 1 || !h_toff || h_toff[0] != 0 || nt < 1 || !d_trec || !d_tsorted || !d_toff)
    return fail(SEDEF_ERR_INVALID, "sedef_server_create: bad target index");
  for (int u = 0; u < ntseq; ++u)
    if (h_toff[u + 1] < h_toff[u]) return fail(SEDEF_ERR_INVALID, "target offsets decrease");
  SEDEF_CUDA(cudaSetDevice(ctx_device(ctx)));
  Server* s = new Server();
  auto bail = [&](int st) {
    const std::string msg = sedef_last_error();
    sedef_server_destroy((sedef_server*)s);
    set_error(msg);
    return st;
  };
  s->device = ctx_device(ctx);
  s->nslots = slots;
  s->slot_bases = slot_bases;
  s->D = D;
  s->P = *p;
  s->idle_s = idle_timeout_s;
  s->trec = d_trec;
  s->tsorted = d_tsorted;
  s->toff = d_toff;
  s->nt = nt;
  s->h_toff.assign(h_toff, h_toff + ntseq + 1);
  s->mtab.resize(kMaxWindowRecs + 1);
  mtable(p, s->mtab.data(), kMaxWindowRecs, nullptr);
  s->fins.resize(kServeFinishers);
  bool made = cudaStreamCreateWithFlags(&s->s_prep, cudaStreamNonBlocking) == cudaSuccess &&
              cudaStreamCreateWithFlags(&s->s_kern, cudaStreamNonBlocking) == cudaSuccess &&
              cudaEventCreateWithFlags(&s->kern_done, cudaEventDisableTiming) == cudaSuccess;
  for (auto& F : s->fins)
    made = made && cudaStreamCreateWithFlags(&F.stream, cudaStreamNonBlocking) == cudaSuccess;
  if (!made) {
    cudaGetLastError();
    return bail(fail(SEDEF_ERR_CUDA, "sedef_server_create: stream or event creation failed"));
  }
  int st = sedef_create(s->device, s->s_prep, &s->c_prep);
  if (st == SEDEF_OK) st = sedef_set_scratch_limit(s->c_prep, ctx_scratch_limit(ctx));
  // admission and finishing run beside the persistent kernel: nothing they
  // allocate may wait for it
  if (st == SEDEF_OK) st = ctx_use_stream_ordered_alloc(s->c_prep);
  for (auto& F : s->fins) {
    if (st == SEDEF_OK) st = sedef_create(s->device, F.stream, &F.ctx);
    if (st == SEDEF_OK) st = sedef_set_scratch_limit(F.ctx, ctx_scratch_limit(ctx));
    if (st == SEDEF_OK) st = ctx_use_stream_ordered_alloc(F.ctx);
    if (st != SEDEF_OK) break;
    ctx_set_filter_variant(F.ctx, ctx_filter_variant(ctx));
    // the finishing tiers keep to the shared memory left beside k_serve
    ctx_set_tier_smem_cap(F.ctx, (size_t)server_smem_left());
  }
  if (st != SEDEF_OK) return bail(st);
  // An SM splits its unified L1 / shared memory when a CTA arrives on an
  // idle SM and keeps the split while any CTA stays.  The persistent kernel
  // stays, so it asks for the largest shared-memory split: the other
  // streams' kernels then find 228 - 53 KB per SM (the large refine kernel
  // takes 125 KB) instead of waiting for the persistent kernel to leave.
  if (cudaFuncSetAttribute(k_serve, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sizeof(ServeSmem)) != cudaSuccess ||
      cudaFuncSetAttribute(k_serve, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess) {
    cudaGetLastError();
    return bail(fail(SEDEF_ERR_CUDA, "sedef_server_create: kernel attributes refused"));
  }
  const size_t up = (size_t)(ntseq + 1) * 8 + (size_t)(kMaxWindowRecs + 1) * 4;
  if ((st = server_alloc(s, (void**)&s->d_shared, up)) != SEDEF_OK) return bail(st);
  if (cudaMemcpy(s->d_shared, h_toff, (size_t)(ntseq + 1) * 8, cudaMemcpyHostToDevice) !=
          cudaSuccess ||
      cudaMemcpy(s->d_shared + (ntseq + 1) * 8, s->mtab.data(), (size_t)(kMaxWindowRecs + 1) * 4,
                 cudaMemcpyHostToDevice) != cudaSuccess)
    return bail(fail(SEDEF_ERR_CUDA, "sedef_server_create: upload failed"));
  s->slots.resize(slots);
  const int64_t win_cap = (slot_bases - D.n) / D.step + 1;
  s->ring_cap = (unsigned long long)(win_cap * slots);
  if (cudaHostAlloc((void**)&s->ctl, sizeof(ServeCtl), cudaHostAllocMapped) != cudaSuccess ||
      cudaHostAlloc((void**)&s->ring, s->ring_cap * sizeof(ServeItem), cudaHostAllocMapped) !=
          cudaSuccess) {
    cudaGetLastError();
    return bail(fail(SEDEF_ERR_OOM, "sedef_server_create: mapped host allocation failed"));
  }
  std::memset(s->ctl, 0, sizeof(ServeCtl));
  if (cudaHostGetDevicePointer((void**)&s->d_ctl, s->ctl, 0) != cudaSuccess ||
      cudaHostGetDevicePointer((void**)&s->d_ring, s->ring, 0) != cudaSuccess) {
    cudaGetLastError();
    return bail(fail(SEDEF_ERR_CUDA, "sedef_server_create: no device view of mapped memory"));
  }
  if ((st = server_alloc(s, (void**)&s->d_head, 8)) != SEDEF_OK) return bail(st);
  if ((st = server_alloc(s, (void**)&s->d_slots, sizeof(SlotDev) * slots)) != SEDEF_OK)
    return bail(st);
  if (cudaMemset(s->d_head, 0, 8) != cudaSuccess)
    return bail(fail(SEDEF_ERR_CUDA, "sedef_server_create: memset failed"));
  std::vector<SlotDev> sdev(slots);
  for (int k = 0; k < slots; ++k) {
    Server::Slot& L = s->slots[k];
    L.rec_cap = slot_bases;
    L.win_cap = win_cap;
    L.run_cap = win_cap * 64 + 4096;
    void* v = nullptr;
#define SALLOC(field, type, bytes)                                   \
  do {                                                               \
    if ((st = server_alloc(s, &v, (size_t)(bytes))) != SEDEF_OK) return bail(st); \
    L.field = (type)v;                                               \
  } while (0)
    SALLOC(seq, uint8_t*, slot_bases);
    SALLOC(packed, uint32_t*, ((slot_bases + 15) / 16) * 4);
    SALLOC(mask, uint32_t*, ((slot_bases + 31) / 32) * 4);
    SALLOC(nbits, uint32_t*, ((slot_bases + 31) / 32) * 4);
    SALLOC(qrec, uint64_t*, L.rec_cap * 8);
    SALLOC(wi, uint32_t*, win_cap * 4 * 7);
    SALLOC(raw, sedef_run_t*, L.run_cap * (int64_t)sizeof(sedef_run_t));
    SALLOC(counters, unsigned long long*, 256 + 64 + 64);
#undef SALLOC
    L.wqa = L.wi + win_cap;
    L.wqb = L.wqa + win_cap;
    L.ov = L.wqb + win_cap;
    L.wl = L.ov + win_cap;
    L.ml = L.wl + win_cap;
    L.wseq = (int32_t*)(L.ml + win_cap);
    L.done = (unsigned int*)((char*)L.counters + 256);
    L.d_up = (char*)L.counters + 256 + 64;
    FArgs& a = L.a;
    std::memset(&a, 0, sizeof(a));
    a.qrec = L.qrec;
    a.trec = d_trec;
    a.tsorted = d_tsorted;
    a.toff = d_toff;
    a.tseq = (const int64_t*)s->d_shared;
    a.qseq = (const int64_t*)L.d_up;
    a.mtab = (const int32_t*)(s->d_shared + (ntseq + 1) * 8);
    a.win_i = L.wi;
    a.win_qa = L.wqa;
    a.win_qb = L.wqb;
    a.win_seq = L.wseq;
    a.ntseq = ntseq;
    a.nqseq = 1;
    a.ttotal = h_toff[ntseq];
    a.k = D.k;
    a.n = D.n;
    a.span = D.span;
    a.max_occ = D.max_occ;
    a.self_mode = 0;
    a.overlap = D.overlap;
    a.runs = L.raw;
    a.nruns = L.counters;
    a.run_cap = L.run_cap;
    a.ov_list = L.ov;
    a.nov = (unsigned int*)(L.counters + 1);
    a.stats = L.counters + 4;
    sdev[k].a = a;
    sdev[k].done = L.done;
    sdev[k].wide_list = L.wl;
    sdev[k].wide_count = (unsigned int*)(L.counters + 14);
    sdev[k].mid_list = L.ml;
    sdev[k].mid_count = (unsigned int*)(L.counters + 16);
  }
  if (cudaMemcpy(s->d_slots, sdev.data(), sizeof(SlotDev) * slots, cudaMemcpyHostToDevice) !=
      cudaSuccess)
    return bail(fail(SEDEF_ERR_CUDA, "sedef_server_create: slot table upload failed"));
  *out = (sedef_server*)s;
  return SEDEF_OK;
}

int sedef_server_submit(sedef_server* srv, const uint8_t* h_query, int64_t len, int32_t* slot_out) {
  using namespace sedef;
  Server* s = (Server*)srv;
  if (!s || !slot_out || (len > 0 && !h_query)) return fail(SEDEF_ERR_INVALID, "NULL argument");
  *slot_out = -1;
  if (len < 0 || len > s->slot_bases)
    return fail(SEDEF_ERR_UNSUPPORTED, "sedef_server_submit: query longer than a slot holds");
  SEDEF_CUDA(cudaSetDevice(s->device));
  int k = -1;
  {
    std::lock_guard<std::mutex> g(s->mu);
    for (int x = 0; x < s->nslots && k < 0; ++x)
      if (s->slots[x].state == 0) k = x;
    if (k < 0) return fail(SEDEF_ERR_CAPACITY, "sedef_server_submit: no free slot");
    s->slots[k].state = 1;
  }
  Server::Slot& L = s->slots[k];
  const int st = server_prepare(s, L, h_query, len);
  std::lock_guard<std::mutex> g(s->mu);
  if (st != SEDEF_OK) {
    L.state = 0;
    return st;
  }
  L.epoch += 1;
  *slot_out = k;
  if (L.nwin == 0) {  // nothing to filter: the slot is done at once
    L.state = 3;
    return SEDEF_OK;
  }
  __atomic_store_n(&s->ctl->nwin[k], (long long)L.nwin, __ATOMIC_RELAXED);
  __atomic_store_n(&s->ctl->epoch[k], L.epoch, __ATOMIC_RELAXED);
  for (int64_t w = 0; w < L.nwin; ++w) {
    ServeItem& it = s->ring[(s->tail + (unsigned long long)w) % s->ring_cap];
    it.slot = (uint32_t)k;
    it.window = (uint32_t)w;
  }
  s->tail += (unsigned long long)L.nwin;
  L.state = 2;
  __atomic_store_n(&s->ctl->tail, s->tail, __ATOMIC_RELEASE);  // items before the tail
  return server_kick(s);
}

int sedef_server_poll(sedef_server* srv, double wait_s, int32_t* slot_out) {
  using namespace sedef;
  Server* s = (Server*)srv;
  if (!s || !slot_out) return fail(SEDEF_ERR_INVALID, "NULL argument");
  *slot_out = -1;
  SEDEF_CUDA(cudaSetDevice(s->device));
  const auto t0 = std::chrono::steady_clock::now();
  while (true) {
    {
      std::lock_guard<std::mutex> g(s->mu);
      bool queued = false;
      for (int k = 0; k < s->nslots; ++k) {
        Server::Slot& L = s->slots[k];
        if (L.state == 2 &&
            __atomic_load_n(&s->ctl->done_epoch[k], __ATOMIC_ACQUIRE) == L.epoch)
          L.state = 3;
        if (L.state == 3) {
          L.state = 4;  // handed to the caller for sedef_server_finish
          *slot_out = k;
          return SEDEF_OK;
        }
        queued |= L.state == 2;
      }
      // items left behind by a kernel that went idle are served by a new one
      if (queued) SEDEF_TRY(server_kick(s));
    }
    const double el =
        std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (el >= wait_s) return SEDEF_OK;
    std::this_thread::sleep_for(std::chrono::microseconds(50));
  }
}

int sedef_server_finish(sedef_server* srv, int32_t slot, sedef_cand_t* h_cands, int64_t cap,
                        int64_t* h_ncands) {
  using namespace sedef;
  Server* s = (Server*)srv;
  if (!s || !h_ncands || slot < 0 || slot >= (s ? s->nslots : 0))
    return fail(SEDEF_ERR_INVALID, "bad argument");
  *h_ncands = 0;
  Server::Slot& L = s->slots[slot];
  {
    std::lock_guard<std::mutex> g(s->mu);
    if (L.state != 4) return fail(SEDEF_ERR_INVALID, "sedef_server_finish: slot not polled");
  }
  if (L.fin_ready) {  // a second call after SEDEF_ERR_CAPACITY
    *h_ncands = (int64_t)L.fin.size();
    if ((int64_t)L.fin.size() > cap)
      return fail(SEDEF_ERR_CAPACITY, "sedef_server_finish: candidate buffer too small");
    if (!L.fin.empty()) std::memcpy(h_cands, L.fin.data(), L.fin.size() * sizeof(sedef_cand_t));
    L.fin_ready = false;
    std::lock_guard<std::mutex> g(s->mu);
    L.state = 0;
    return SEDEF_OK;
  }
  SEDEF_CUDA(cudaSetDevice(s->device));
  // a free finishing stream and context, held for the whole call
  struct FinLease {
    Server* s;
    Server::Finisher* f = nullptr;
    explicit FinLease(Server* sv) : s(sv) {
      std::unique_lock<std::mutex> g(s->mu);
      s->fin_cv.wait(g, [&] {
        for (auto& F : s->fins)
          if (!F.busy) {
            F.busy = true;
            f = &F;
            return true;
          }
        return false;
      });
    }
    ~FinLease() {
      {
        std::lock_guard<std::mutex> g(s->mu);
        f->busy = false;
      }
      s->fin_cv.notify_one();
    }
  } lease(s);
  sedef_ctx* c = lease.f->ctx;
  cudaStream_t st = lease.f->stream;
  ctx_pool_reset(c);
  auto release = [&](int status) {
    std::lock_guard<std::mutex> g(s->mu);
    L.state = 0;
    return status;
  };
  const int64_t qoff[2] = {0, L.len};
  int64_t nc = 0;
  if (L.nwin > 0) {
    {
      // the windows k_serve handed on for their many hits: the broad tier,
      // as an ordinary launch beside k_serve; what it cannot hold, and what
      // k_serve could not hold, goes through the 8,192-hit deep and second
      // wide tiers, and what those cannot hold joins the slot's overflow list
      StageScope stage(c, "filter");
      TierIO iow{L.wl, (const unsigned int*)(L.counters + 14), L.ml,
                 (unsigned int*)(L.counters + 16), (unsigned int*)(L.counters + 15), 1};
      int wst = launch_cta_tier<CtaBroad>(c, L.a, iow, L.nwin, "k_filter_wide");
      // the broad tier is through with the slot's wide list
      TierIO iod{L.ml, (const unsigned int*)(L.counters + 16), L.wl,
                 (unsigned int*)(L.counters + 21), (unsigned int*)(L.counters + 20), 1};
      if (wst == SEDEF_OK) wst = launch_cta_tier<CtaMid>(c, L.a, iod, L.nwin, "k_filter_deep");
      TierIO iom{L.wl, (const unsigned int*)(L.counters + 21), L.ov,
                 (unsigned int*)(L.counters + 1), (unsigned int*)(L.counters + 17), 1};
      if (wst == SEDEF_OK) wst = kTierWideMid(c, L.a, iom, L.nwin, "k_filter_widemid");
      if (wst != SEDEF_OK) return release(wst);
    }
    unsigned long long* h_cnt = (unsigned long long*)ctx_host(c, 64);
    if (!h_cnt) return release(SEDEF_ERR_OOM);
    if (cudaMemcpyAsync(h_cnt, L.counters, 16, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return release(fail(SEDEF_ERR_CUDA, "sedef_server_finish: counter copy failed"));
    const int64_t nov = (int64_t)(h_cnt[1] & 0xFFFFFFFFull);
    int64_t slow = 0;
    int status = SEDEF_OK;
    if (nov > 0) status = global_path_eager(c, L.a, nov, L.counters, &slow);
    if (status == SEDEF_OK &&
        (cudaMemcpyAsync(h_cnt, L.counters, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
         cudaStreamSynchronize(st) != cudaSuccess))
      status = fail(SEDEF_ERR_CUDA, "sedef_server_finish: counter copy failed");
    if (status != SEDEF_OK) return release(status);
    const int64_t total = (int64_t)h_cnt[0];
    sedef_cand_t* cands = nullptr;
    auto candidates = [&]() -> int {  // of the raw runs, into cands and nc
      sedef_run_t* runs = (sedef_run_t*)ctx_alloc(c, (size_t)total * sizeof(sedef_run_t));
      if (!runs) return SEDEF_ERR_OOM;
      if (total > L.run_cap) {
        // more runs than the slot holds: the whole filter again, sized exactly
        int64_t got = 0;
        SEDEF_TRY(run_filter(c, L.qrec, L.nrec, qoff, 1, s->trec, s->tsorted, s->toff, s->nt,
                             s->h_toff.data(), (int)s->h_toff.size() - 1, s->D, s->mtab.data(), runs,
                             total, &got, 0));
      } else {
        StageScope stage(c, "runsort");
        SEDEF_TRY(order_and_refine(c, L.a, s->D, 1, (const int64_t*)L.d_up + 2, L.nwin, L.wqa, L.wqb,
                                   L.qrec, L.nrec, s->trec, s->nt, s->toff, L.counters, L.raw, total,
                                   runs, nullptr, nullptr));
      }
      sedef_chain_t* chains = (sedef_chain_t*)ctx_alloc(c, (size_t)total * sizeof(sedef_chain_t));
      if (!chains) return SEDEF_ERR_OOM;
      int64_t nch = 0;
      {
        StageScope stage(c, "chain");
        SEDEF_TRY(run_chain(c, runs, total, L.qrec, L.nrec, qoff, 1, s->tsorted, s->nt, s->toff,
                            s->h_toff.data(), (int)s->h_toff.size() - 1, s->D, s->mtab.data(),
                            chains, total, &nch));
      }
      if (nch == 0) return SEDEF_OK;
      cands = (sedef_cand_t*)ctx_alloc(c, (size_t)nch * sizeof(sedef_cand_t));
      if (!cands) return SEDEF_ERR_OOM;
      StageScope stage(c, "merge");
      return run_merge(c, chains, nch, qoff, 1, s->h_toff.data(), (int)s->h_toff.size() - 1, s->D, cands,
                       nch, &nc);
    };
    if (total > 0) {
      status = candidates();
      if (status == SEDEF_ERR_OOM) {
        // once more without the buffers a call can do without
        ctx_pool_release(c);
        ctx_set_extras(c, false);
        // the runs handed to the large refine kernel are counted anew
        if (cudaMemsetAsync(L.counters + 3, 0, 8, st) == cudaSuccess) status = candidates();
        ctx_set_extras(c, true);
      }
      if (status != SEDEF_OK) return release(status);
    }
    if (nc > cap) {  // keep them for the next call; the slot stays handed out
      L.fin.resize((size_t)nc);
      if (cudaMemcpyAsync(L.fin.data(), cands, (size_t)nc * sizeof(sedef_cand_t),
                          cudaMemcpyDeviceToHost, st) != cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess)
        return release(fail(SEDEF_ERR_CUDA, "sedef_server_finish: copy failed"));
      L.fin_ready = true;
      *h_ncands = nc;
      return fail(SEDEF_ERR_CAPACITY, "sedef_server_finish: candidate buffer too small");
    }
    if (nc > 0 &&
        cudaMemcpyAsync(h_cands, cands, (size_t)nc * sizeof(sedef_cand_t), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess)
      return release(fail(SEDEF_ERR_CUDA, "sedef_server_finish: copy failed"));
  }
  if (cudaStreamSynchronize(st) != cudaSuccess)
    return release(fail(SEDEF_ERR_CUDA, "sedef_server_finish: stream failed"));
  *h_ncands = nc;
  return release(SEDEF_OK);
}

int sedef_server_smem_left(sedef_server* srv, int64_t* bytes) {
  if (!srv || !bytes) return sedef::fail(SEDEF_ERR_INVALID, "NULL argument");
  *bytes = sedef::server_smem_left();
  return SEDEF_OK;
}

int sedef_server_status(sedef_server* srv, int32_t* running, int32_t* timed_out) {
  using namespace sedef;
  Server* s = (Server*)srv;
  if (!s) return fail(SEDEF_ERR_INVALID, "NULL argument");
  std::lock_guard<std::mutex> g(s->mu);
  int run = 0;
  if (s->kern_launched) {
    const cudaError_t q = cudaEventQuery(s->kern_done);
    if (q == cudaErrorNotReady) run = 1;
    else if (q != cudaSuccess) return cuda_fail(q, "server: kernel event");
  }
  const int tmo = __atomic_load_n(&s->ctl->status, __ATOMIC_ACQUIRE) == SEDEF_ERR_TIMEOUT;
  if (running) *running = run;
  if (timed_out) *timed_out = tmo;
  return (!run && tmo) ? SEDEF_ERR_TIMEOUT : SEDEF_OK;
}

}  // extern "C"
