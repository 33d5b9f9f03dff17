// a3 index: device-wide exclusive scan, stable LSD radix sort of uint64 keys
// (optionally with uint32 payloads) over a chosen bit range, and the offset
// table over all 4^k hashes.
//
// The sort takes 8-bit digits over only the significant bits (2k = 24 hash
// bits for the index: 3 passes).  One kernel counts the digits of every pass
// in one read of the keys; then each pass is one kernel: a CTA takes tiles of
// 4,096 keys in ticket order, every warp ranks its keys by votes, the CTA
// finds where each digit of its tile goes by a decoupled look-back over the
// tiles before it (or, should they not publish in time, by counting their keys
// itself), stages the tile in shared memory in digit order, and
// consecutive threads write consecutive output addresses (coalesced runs per
// digit).  Up to 4,096 keys are sorted by one CTA in one launch, all passes
// in shared memory.
#include "common.cuh"

namespace sedef {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t block_scan_tile(uint32_t (&v)[kScanItems], int* tmp,
                                                    uint32_t* total) {
  uint32_t s = 0;
#pragma unroll
  for (int x = 0; x < kScanItems; ++x) s += v[x];
  int tot;
  const int ex = block_exclusive_sum((int)s, tmp, &tot);
  uint32_t run = (uint32_t)ex;
#pragma unroll
  for (int x = 0; x < kScanItems; ++x) {
    const uint32_t t = v[x];
    v[x] = run;
    run += t;
  }
  *total = (uint32_t)tot;
  return (uint32_t)ex;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const uint32_t* __restrict__ in,
                                                              int64_t n, uint32_t* __restrict__ sums) {
  __shared__ int tmp[33];
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t s = 0;
#pragma unroll
  for (int x = 0; x < kScanItems; ++x)
    if (base + x < n) s += in[base + x];
  int tot;
  block_exclusive_sum((int)s, tmp, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = (uint32_t)tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(const uint32_t* __restrict__ in,
                                                             uint32_t* __restrict__ out, int64_t n,
                                                             const uint32_t* __restrict__ tile_off,
                                                             uint32_t* __restrict__ total) {
  __shared__ int tmp[33];
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
#pragma unroll
  for (int x = 0; x < kScanItems; ++x) v[x] = (base + x < n) ? in[base + x] : 0u;
  uint32_t tot;
  block_scan_tile(v, tmp, &tot);
  const uint32_t add = tile_off ? tile_off[blockIdx.x] : 0u;
#pragma unroll
  for (int x = 0; x < kScanItems; ++x)
    if (base + x < n) out[base + x] = v[x] + add;
  if (total && threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) *total = add + tot;
}

// ------------------------------------------------------------- radix sort --

constexpr int kRsThreads = 256;  // one per digit value
constexpr int kRsItems = 16;
constexpr int kRsTile = kRsThreads * kRsItems;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsPasses = 8;

__device__ __forceinline__ uint32_t digit_of(uint64_t key, int shift, uint32_t dmask) {
  return (uint32_t)(key >> shift) & dmask;
}

// Lanes with the caller's digit (9 bits, 256: no key).  Nine votes: the match
// instruction goes through a warp's distinct values one by one.
__device__ __forceinline__ unsigned digit_peers(uint32_t d) {
  unsigned peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const unsigned set = __ballot_sync(0xffffffffu, (d >> b) & 1u);
    peers &= (d >> b) & 1u ? set : ~set;
  }
  return peers;
}

// Bits of each pass: 8 from bit_lo + 8 p, fewer in the last.
struct RsBits {
  int lo, hi;
  __host__ __device__ int passes() const { return (hi - lo + 7) / 8; }
  __host__ __device__ int shift(int p) const { return lo + 8 * p; }
  __host__ __device__ uint32_t mask(int p) const {
    const int b = hi - shift(p);
    return (1u << (b < 8 ? b : 8)) - 1u;
  }
};

// Scratch of one sort: zeroed before it.  Status words hold a pass number and
// a flag over a count, so that the next pass needs no clearing.
struct RsScratch {
  unsigned int* ticket;        // per pass
  uint32_t* hist;              // [pass][256] keys of each digit
  unsigned long long* status;  // [tile][256]
  unsigned int polls;          // reads of one unpublished status before the wait ends
};

// Digit counts of every pass.
__global__ void __launch_bounds__(kRsThreads) k_rs_hist(const uint64_t* __restrict__ keys, int64_t n,
                                                        RsBits bits, uint32_t* __restrict__ hist,
                                                        const uint32_t* __restrict__ dn) {
  __shared__ uint32_t h[kRsPasses][256];
  n = live_n(n, dn);
  const int np = bits.passes();
  for (int p = 0; p < np; ++p) h[p][threadIdx.x] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * kRsThreads;
  for (int64_t base = (int64_t)blockIdx.x * kRsThreads; base < n; base += stride) {
    const int64_t x = base + threadIdx.x;
    const bool ok = x < n;
    const uint64_t k = ok ? keys[x] : 0ull;
    for (int p = 0; p < np; ++p) {
      const uint32_t d = digit_of(k, bits.shift(p), bits.mask(p));
      // one digit for the whole warp (the high bits of small numbers): one
      // atomic instead of 32 on one address
      const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
      if (__all_sync(0xffffffffu, ok && d == d0)) {
        if (lane_id() == 0) atomicAdd(&h[p][d], 32u);
      } else if (ok) {
        atomicAdd(&h[p][d], 1u);
      }
    }
  }
  __syncthreads();
  for (int p = 0; p < np; ++p) {
    const uint32_t c = h[p][threadIdx.x];
    if (c) atomicAdd(hist + p * 256 + threadIdx.x, c);
  }
}

template <bool kVals>
struct RsSmem {
  uint32_t wcnt[kRsWarps][256];  // keys of a digit per warp, then before it
  uint32_t dstart[256];          // where a digit starts in the tile
  uint32_t base[256];            // where a digit starts in the output
  uint32_t gofs[256];            // output place of the digit's first key of this tile, less dstart
  int tmp[33];
  long long tile;
  uint64_t keys[kRsTile];
  uint32_t vals[kVals ? kRsTile : 1];
};

// Ranks the warp's kRsItems rounds of 32 keys by digit: loc[r] = keys of the
// same digit before this one in the warp; wcnt = the warp's counts.
__device__ __forceinline__ void rank_round(uint32_t* wcnt, uint32_t d, uint32_t lt, uint32_t& loc) {
  const unsigned peers = digit_peers(d);
  const uint32_t rank = __popc(peers & lt);
  const uint32_t before = d < 256 ? wcnt[d] : 0u;
  __syncwarp();
  if (d < 256 && rank == 0) wcnt[d] = before + __popc(peers);
  __syncwarp();
  loc = before + rank;
}

// This thread's digit among the first `end` keys, counted by its warp: what a
// tile whose wait ran out would have read from the tiles before it, so every
// key goes to its place whatever the other CTAs do.  cnt: the warp's row, which
// only its own staging reads.  Out of line: the pass has no registers to spare.
__device__ __noinline__ uint32_t count_before(const uint64_t* kin, int64_t end, int shift, uint32_t dmask,
                                              uint32_t* cnt) {
  __syncwarp();
  cnt[threadIdx.x] = 0;
  __syncwarp();
  for (int64_t x = threadIdx.x & 31; x < end; x += 32) {
    const uint32_t d = digit_of(kin[x], shift, dmask);
    if ((d >> 5) == (threadIdx.x >> 5)) atomicAdd(cnt + d, 1u);
  }
  __syncwarp();
  return cnt[threadIdx.x];
}

// One pass.  Bound by the integer pipe: six to seven warp instructions a key,
// most of them the votes (73% of the pipe and 60% of the issue slots busy in a
// sort of 14.3 M records, waits for the keys' loads next).  Between CTAs a
// thread per digit reads eight tiles' status at once.  194 M records over 24
// bits: 8.0 -> 5.2 ms with the count, 2.1 TB/s or 31% of the copy rate (before:
// three kernels a pass, 147 registers and one CTA of 256 threads per SM).
template <bool kVals>
__global__ void __launch_bounds__(kRsThreads, kVals ? 3 : 4) k_rs_pass(
    const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint64_t* __restrict__ kout,
    uint32_t* __restrict__ vout, int64_t n, RsBits bits, int pass, RsScratch sc, int iota_vals,
    const uint32_t* __restrict__ dn) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RsSmem<kVals>& S = *reinterpret_cast<RsSmem<kVals>*>(smem_raw);
  n = live_n(n, dn);
  const int64_t ntiles = (n + kRsTile - 1) / kRsTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int shift = bits.shift(pass);
  const uint32_t dmask = bits.mask(pass);
  const uint32_t lt = lanemask_lt();
  const unsigned long long kAgg = (unsigned long long)(2 * pass + 1) << 32;
  const unsigned long long kPrefix = (unsigned long long)(2 * pass + 2) << 32;
  if (threadIdx.x == 0) S.tile = (long long)atomicAdd(sc.ticket + pass, 1u);
  {
    int tot;
    S.base[threadIdx.x] =
        (uint32_t)block_exclusive_sum((int)sc.hist[pass * 256 + threadIdx.x], S.tmp, &tot);
  }
  __syncthreads();
  while (true) {
    const int64_t tile = S.tile;
    if (tile >= ntiles) break;
    for (int x = threadIdx.x; x < kRsWarps * 256; x += kRsThreads) (&S.wcnt[0][0])[x] = 0;
    const int cnt = (int)min((int64_t)kRsTile, n - tile * kRsTile);
    const int base = warp * (32 * kRsItems) + lane;  // this thread's keys: every 32nd from here
    const uint64_t* kt = kin + tile * kRsTile + base;
    uint64_t key[kRsItems];
    uint32_t loc[kRsItems];
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) key[r] = base + r * 32 < cnt ? kt[r * 32] : 0ull;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsItems; ++r)
      rank_round(S.wcnt[warp], base + r * 32 < cnt ? digit_of(key[r], shift, dmask) : 256u, lt, loc[r]);
    __syncthreads();
    uint32_t count = 0;
    const int d = threadIdx.x;
    {
#pragma unroll
      for (int w = 0; w < kRsWarps; ++w) {
        const uint32_t c = S.wcnt[w][d];
        S.wcnt[w][d] = count;
        count += c;
      }
    }
    unsigned long long* mine = sc.status + tile * 256 + d;
    if (tile > 0) st_relaxed_gpu(mine, kAgg | count);
    int tot;
    const uint32_t start = (uint32_t)block_exclusive_sum((int)count, S.tmp, &tot);
    S.dstart[d] = start;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
      if (base + r * 32 < cnt) {
        const uint32_t x = digit_of(key[r], shift, dmask);
        loc[r] += S.dstart[x] + S.wcnt[warp][x];
        S.keys[loc[r]] = key[r];
      }
    }
    if (kVals) {
      const int64_t at = tile * kRsTile + base;
#pragma unroll
      for (int r = 0; r < kRsItems; ++r)
        if (base + r * 32 < cnt)
          S.vals[loc[r]] = iota_vals ? (uint32_t)(at + r * 32) : vin[at + r * 32];
    }
    // keys of this digit in the tiles before: a tile's predecessors were all
    // taken before it by CTAs that publish their counts before they wait
    uint32_t before = 0;
    bool ran_out = false;
    if (tile > 0) {
      int64_t j = tile - 1;
      unsigned int spins = 0;
      bool done = false;
      while (!done) {
        constexpr int kWide = 8;
        unsigned long long v[kWide];
#pragma unroll
        for (int x = 0; x < kWide; ++x)
          v[x] = j - x >= 0 ? ld_relaxed_gpu(sc.status + (j - x) * 256 + d) : kPrefix;
#pragma unroll
        for (int x = 0; x < kWide; ++x) {
          if (v[x] < kAgg) {  // not yet: read again from this tile
            if (++spins > sc.polls) ran_out = done = true;
            break;
          }
          spins = 0;
          before += (uint32_t)v[x];
          if (v[x] >= kPrefix) {
            done = true;
            break;
          }
          --j;
        }
      }
    }
    if (__any_sync(0xffffffffu, ran_out))
      before = count_before(kin, tile * kRsTile, shift, dmask, S.wcnt[warp]);
    st_relaxed_gpu(mine, kPrefix | (before + count));
    S.gofs[d] = S.base[d] + before - start;
    if (threadIdx.x == 0) S.tile = (long long)atomicAdd(sc.ticket + pass, 1u);
    __syncthreads();
#pragma unroll 4
    for (int x = threadIdx.x; x < cnt; x += kRsThreads) {
      const uint64_t kk = S.keys[x];
      const uint32_t o = S.gofs[digit_of(kk, shift, dmask)] + (uint32_t)x;
      kout[o] = kk;
      if (kVals) vout[o] = S.vals[x];
    }
    __syncthreads();
  }
}

// Up to kRsTile keys by one CTA: every pass in shared memory.
struct RsSmall {
  uint32_t wcnt[kRsWarps][256];
  uint32_t dstart[256];
  int tmp[33];
  uint64_t keys[kRsTile];
  uint32_t vals[kRsTile];
};

__global__ void __launch_bounds__(kRsThreads) k_rs_small(const uint64_t* __restrict__ kin,
                                                         const uint32_t* __restrict__ vin,
                                                         uint64_t* __restrict__ kout,
                                                         uint32_t* __restrict__ vout, int64_t n64,
                                                         RsBits bits, int iota_vals,
                                                         const uint32_t* __restrict__ dn) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RsSmall& S = *reinterpret_cast<RsSmall*>(smem_raw);
  const int n = (int)live_n(n64, dn);
  const bool has_vals = vout != nullptr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lt = lanemask_lt();
  const int rounds = (n + kRsThreads - 1) / kRsThreads;
  const int base = warp * 32 * rounds + lane;  // this thread's keys: every 32nd from here
  for (int x = threadIdx.x; x < n; x += kRsThreads) {
    S.keys[x] = kin[x];
    if (has_vals) S.vals[x] = iota_vals ? (uint32_t)x : vin[x];
  }
  for (int p = 0; p < bits.passes(); ++p) {
    const int shift = bits.shift(p);
    const uint32_t dmask = bits.mask(p);
    for (int x = threadIdx.x; x < kRsWarps * 256; x += kRsThreads) (&S.wcnt[0][0])[x] = 0;
    __syncthreads();
    uint64_t key[kRsItems];
    uint32_t val[kRsItems], loc[kRsItems];
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
      if (r >= rounds) break;
      const int idx = base + r * 32;
      const bool ok = idx < n;
      key[r] = ok ? S.keys[idx] : 0ull;
      val[r] = ok && has_vals ? S.vals[idx] : 0u;
      rank_round(S.wcnt[warp], ok ? digit_of(key[r], shift, dmask) : 256u, lt, loc[r]);
    }
    __syncthreads();
    {
      uint32_t count = 0;
#pragma unroll
      for (int w = 0; w < kRsWarps; ++w) {
        const uint32_t c = S.wcnt[w][threadIdx.x];
        S.wcnt[w][threadIdx.x] = count;
        count += c;
      }
      int tot;
      S.dstart[threadIdx.x] = (uint32_t)block_exclusive_sum((int)count, S.tmp, &tot);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRsItems; ++r) {
      if (r >= rounds) break;
      if (base + r * 32 < n) {
        const uint32_t d = digit_of(key[r], shift, dmask);
        const uint32_t to = S.dstart[d] + S.wcnt[warp][d] + loc[r];
        S.keys[to] = key[r];
        if (has_vals) S.vals[to] = val[r];
      }
    }
    __syncthreads();
  }
  for (int x = threadIdx.x; x < n; x += kRsThreads) {
    kout[x] = S.keys[x];
    if (has_vals) vout[x] = S.vals[x];
  }
}

// --------------------------------------------------------- offset table ----

constexpr int kOffChunk = 4096;
// A thread sums 16 consecutive counts; one word of padding per 16 puts a
// warp's reads in different banks.
__device__ __forceinline__ int off_slot(int x) { return x + (x >> 4); }

// Bound by its writes (4 B per hash) on large tables.  Written straight from
// the scan, 16 words per thread, every store touched 32 sectors: 86 us for
// the 16.7 M hashes of k = 12 and a 2 Mbp genome, 25 us through shared memory.
__global__ void __launch_bounds__(256) k_offsets(const uint64_t* __restrict__ sorted, int64_t n,
                                                 int64_t nhash, uint32_t* __restrict__ off,
                                                 const uint32_t* __restrict__ dn) {
  n = live_n(n, dn);
  __shared__ uint32_t cnt[kOffChunk + kOffChunk / 16];
  __shared__ int64_t rng[2];
  __shared__ int tmp[33];
  const int64_t X0 = (int64_t)blockIdx.x * kOffChunk;
  for (int x = threadIdx.x; x < kOffChunk + kOffChunk / 16; x += 256) cnt[x] = 0;
  if (threadIdx.x < 64) {
    // first record of the chunk and past its last: a warp each, 32 probes at
    // a time
    const uint64_t key = (uint64_t)(X0 + (threadIdx.x >= 32 ? kOffChunk : 0));
    const int lane = threadIdx.x & 31;
    int64_t lo = 0, hi = n;  // hash < key before lo, >= key from hi on
    while (hi > lo) {
      const int64_t step = (hi - lo + 31) / 32;
      const int64_t at = lo + lane * step;
      const unsigned below = __ballot_sync(0xffffffffu, at < hi && (sorted[at < hi ? at : lo] >> 33) < key);
      const int c = __popc(below);  // the probes below key come first
      const int64_t next = lo + c * step;
      if (c > 0) lo = lo + (c - 1) * step + 1;
      if (next < hi) hi = next;
    }
    if (lane == 0) rng[threadIdx.x >> 5] = lo;
  }
  __syncthreads();
  const int64_t R0 = rng[0], R1 = rng[1];
  for (int64_t r = R0 + threadIdx.x; r < R1; r += 256)
    atomicAdd(&cnt[off_slot((int)((sorted[r] >> 33) - (uint64_t)X0))], 1u);
  __syncthreads();
  // exclusive scan of the counts: 16 consecutive ones per thread
  uint32_t* mine = cnt + off_slot(threadIdx.x * 16);
  uint32_t s = 0;
#pragma unroll
  for (int x = 0; x < 16; ++x) s += mine[x];
  int tot;
  uint32_t run = (uint32_t)(R0 + block_exclusive_sum((int)s, tmp, &tot));
#pragma unroll
  for (int x = 0; x < 16; ++x) {
    const uint32_t c = mine[x];
    mine[x] = run;
    run += c;
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < kOffChunk / 256; ++x) {
    const int at = x * 256 + threadIdx.x;
    if (X0 + at < nhash) off[X0 + at] = cnt[off_slot(at)];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) off[nhash] = (uint32_t)n;
}

}  // namespace

int scan_exclusive_u32(sedef_ctx* ctx, const uint32_t* in, uint32_t* out, int64_t n,
                       uint32_t* d_total) {
  cudaStream_t st = ctx_stream(ctx);
  if (n <= 0) {
    if (d_total) SEDEF_CUDA(cudaMemsetAsync(d_total, 0, 4, st));
    return SEDEF_OK;
  }
  const int64_t tiles = (n + kScanTile - 1) / kScanTile;
  if (tiles == 1) {
    SEDEF_KERNEL(ctx, "k_scan_tiles", k_scan_tiles<<<1, kScanThreads, 0, st>>>(in, out, n, nullptr, d_total));
    return SEDEF_OK;
  }
  uint32_t* sums = (uint32_t*)ctx_alloc(ctx, (size_t)tiles * 4);
  uint32_t* soff = (uint32_t*)ctx_alloc(ctx, (size_t)tiles * 4);
  if (!sums || !soff) return SEDEF_ERR_OOM;
  SEDEF_KERNEL(ctx, "k_scan_reduce", k_scan_reduce<<<(int)tiles, kScanThreads, 0, st>>>(in, n, sums));
  SEDEF_TRY(scan_exclusive_u32(ctx, sums, soff, tiles, nullptr));
  SEDEF_KERNEL(ctx, "k_scan_tiles",
               k_scan_tiles<<<(int)tiles, kScanThreads, 0, st>>>(in, out, n, soff, d_total));
  return SEDEF_OK;
}

int radix_sort_u64(sedef_ctx* ctx, const uint64_t* keys_in, const uint32_t* vals_in,
                   uint64_t* keys_out, uint32_t* vals_out, int64_t n, int bit_lo, int bit_hi,
                   const uint32_t* dn) {
  cudaStream_t st = ctx_stream(ctx);
  if (n <= 0) return SEDEF_OK;
  const int passes = (bit_hi - bit_lo + 7) / 8;
  const bool iota = (vals_in == nullptr && vals_out != nullptr);
  if (passes <= 0) {
    SEDEF_CUDA(cudaMemcpyAsync(keys_out, keys_in, (size_t)n * 8, cudaMemcpyDeviceToDevice, st));
    return SEDEF_OK;
  }
  const RsBits bits{bit_lo, bit_hi};
  if (n <= kRsTile) {
    SEDEF_TRY(ensure_smem_attr((const void*)k_rs_small, sizeof(RsSmall)));
    SEDEF_KERNEL(ctx, "k_rs_small",
                 k_rs_small<<<1, kRsThreads, sizeof(RsSmall), st>>>(keys_in, vals_in, keys_out, vals_out,
                                                                    n, bits, iota ? 1 : 0, dn));
    return SEDEF_OK;
  }
  const int64_t ntiles = (n + kRsTile - 1) / kRsTile;
  const size_t head = 64 + (size_t)passes * 256 * 4;
  char* scratch = (char*)ctx_alloc(ctx, head + (size_t)ntiles * 256 * 8);
  uint64_t* ktmp = passes > 1 ? (uint64_t*)ctx_alloc(ctx, (size_t)n * 8) : nullptr;
  uint32_t* vtmp = vals_out && passes > 1 ? (uint32_t*)ctx_alloc(ctx, (size_t)n * 4) : nullptr;
  if (!scratch || (passes > 1 && (!ktmp || (vals_out && !vtmp)))) return SEDEF_ERR_OOM;
  RsScratch sc;
  sc.ticket = (unsigned int*)scratch;
  sc.polls = ctx_sort_polls(ctx);
  sc.hist = (uint32_t*)(scratch + 64);
  sc.status = (unsigned long long*)(scratch + head);
  SEDEF_CUDA(cudaMemsetAsync(scratch, 0, head + (size_t)ntiles * 256 * 8, st));
  const size_t smem = vals_out ? sizeof(RsSmem<true>) : sizeof(RsSmem<false>);
  SEDEF_TRY(ensure_smem_attr((const void*)k_rs_pass<true>, sizeof(RsSmem<true>)));
  SEDEF_TRY(ensure_smem_attr((const void*)k_rs_pass<false>, sizeof(RsSmem<false>)));
  const int64_t sms = ctx_sm_count(ctx);
  const int64_t grid = ntiles < sms * (vals_out ? 3 : 4) ? ntiles : sms * (vals_out ? 3 : 4);
  int64_t hgrid = (n + kRsThreads * 8 - 1) / (kRsThreads * 8);
  if (hgrid > sms * 8) hgrid = sms * 8;
  SEDEF_KERNEL(ctx, "k_rs_hist",
               k_rs_hist<<<(int)hgrid, kRsThreads, 0, st>>>(keys_in, n, bits, sc.hist, dn));
  const uint64_t* ksrc = keys_in;
  const uint32_t* vsrc = vals_in;
  for (int p = 0; p < passes; ++p) {
    const bool to_out = ((passes - 1 - p) % 2) == 0;
    uint64_t* kdst = to_out ? keys_out : ktmp;
    uint32_t* vdst = vals_out ? (to_out ? vals_out : vtmp) : nullptr;
    const int first_iota = (p == 0 && iota) ? 1 : 0;
    if (vals_out)
      SEDEF_KERNEL(ctx, "k_rs_pass",
                   k_rs_pass<true><<<(int)grid, kRsThreads, smem, st>>>(ksrc, vsrc, kdst, vdst, n, bits,
                                                                        p, sc, first_iota, dn));
    else
      SEDEF_KERNEL(ctx, "k_rs_pass",
                   k_rs_pass<false><<<(int)grid, kRsThreads, smem, st>>>(ksrc, vsrc, kdst, vdst, n, bits,
                                                                         p, sc, first_iota, dn));
    ksrc = kdst;
    vsrc = vdst;
  }
  return SEDEF_OK;
}

int build_offsets(sedef_ctx* ctx, const uint64_t* sorted, int64_t n, int k, uint32_t* off,
                  const uint32_t* dn) {
  cudaStream_t st = ctx_stream(ctx);
  const int64_t nhash = int64_t(1) << (2 * k);
  const int64_t chunks = (nhash + kOffChunk - 1) / kOffChunk;
  SEDEF_KERNEL(ctx, "k_offsets", k_offsets<<<(int)chunks, 256, 0, st>>>(sorted, n, nhash, off, dn));
  return SEDEF_OK;
}

}  // namespace sedef
