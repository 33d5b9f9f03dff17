// a1 pack and a2 sketch kernels.
//
// pack: 16 input bytes per thread (one 128-bit load), one packed word per
// thread and one mask/N word per lane pair (warp shuffle), so every global
// access is coalesced.  HBM-bound: 1 B read + 0.5 B written per base.
//
// sketch: a warp takes a stretch of 512 positions, 16 consecutive ones per
// lane, all in registers.  A lane reads two packed words and two 16-bit
// pieces of the mask and N bits; forward codes and reverse complements are
// funnel shifts of the words and of their reversal, eligibility of its 16
// k-mers a few shifts of the bit-vectors.  Window minima come from doubling
// (minima over 1, 2, 4, ... positions, then one combination of two
// overlapping ones), reading the lanes above by shuffles; a window's argmin
// is kept when it differs from the previous window's (winnowing argmins are
// non-decreasing, so this emits each selected position once, in order).  The
// window keys are (hash, reversed offset from the lane's first position), so
// that equal hashes go to the rightmost: 32 bits when the hash has at most
// 24 bits and a window at most 112 positions, else 64.  Eight warps share a
// CTA tile; the eager pass writes its records in the same pass, finding each
// tile's offset by a decoupled look-back over the tiles taken before it; the
// planned (graph) pass and the allocation-free call count, scan and write
// instead.
#include <cstring>

#include "common.cuh"

namespace sedef {

namespace {

__device__ __forceinline__ void classify(uint32_t b, uint32_t& code, uint32_t& masked,
                                         uint32_t& isn) {
  const uint32_t l = b | 0x20u;
  const bool acgt = (l == 'a') | (l == 'c') | (l == 'g') | (l == 't');
  code = acgt ? (((l >> 1) ^ (l >> 2)) & 3u) : 0u;  // a=0 c=1 g=2 t=3
  masked = (b >= 'a' && b <= 'z') ? 1u : 0u;
  isn = acgt ? 0u : 1u;
}

// Four bases at once: a code per byte, and which bytes are not ACGTacgt (a
// non-zero byte in the result).  The code picks the letter it stands for,
// and a byte is a base when it is that letter.
__device__ __forceinline__ uint32_t codes4(uint32_t v, uint32_t& code) {
  const uint32_t u = v | 0x20202020u;
  code = ((u >> 1) ^ (u >> 2)) & 0x03030303u;  // a=0 c=1 g=2 t=3
  const uint32_t pick = __byte_perm(code | (code >> 4), 0, 0x4420);  // a nibble per byte
  return __byte_perm(0x74676361u, 0, pick) ^ u;
}

// A thread classifies its 16 bytes four at a time (one at a time, 17
// instructions a base, was bound by their issue: 3.1 Gbp in 2.78 ms; now 1.00
// ms, 4.65 TB/s read and written).  16 bytes with another one among them are
// gone over once more, four at a time too (one at a time, 200 Mbp with an N in
// every 16 took 0.237 ms, 0.133 this way).
template <bool kAligned>
__global__ void __launch_bounds__(256) k_pack(const uint8_t* __restrict__ seq, int64_t n,
                                              uint32_t* __restrict__ packed,
                                              uint32_t* __restrict__ mask,
                                              uint32_t* __restrict__ nbits) {
  const int64_t nchunk = (n + 15) >> 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nchunk; base += stride) {
    const int64_t c = base + threadIdx.x;
    uint32_t word = 0, m16 = 0, n16 = 0;
    if (c < nchunk) {
      const int64_t p0 = c << 4;
      uint32_t v[4];
      if (kAligned && p0 + 16 <= n) {
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(seq + p0));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
        uint32_t other = 0;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          uint32_t code;
          other |= codes4(v[x], code);
          // the multiplications bring the bytes' 2-bit codes and case bits
          // together in the top byte (no two partial products meet)
          word |= ((code * 0x01041040u) >> 24) << (8 * x);
          m16 |= ((((v[x] >> 5) & 0x01010101u) * 0x01020408u) >> 24) << (4 * x);
        }
        if (other) {
          word = m16 = 0;
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            uint32_t code;
            // a one in each byte that is no base, and in each lowercase letter
            const uint32_t no = __vcmpgtu4(codes4(v[x], code), 0u) & 0x01010101u;
            const uint32_t low = __vcmpgeu4(v[x], 0x61616161u) & __vcmpleu4(v[x], 0x7A7A7A7Au) & 0x01010101u;
            word |= (((code & ~(no * 3u)) * 0x01041040u) >> 24) << (8 * x);
            m16 |= ((low * 0x01020408u) >> 24) << (4 * x);
            n16 |= ((no * 0x01020408u) >> 24) << (4 * x);
          }
        }
      } else {
        for (int x = 0; x < 16; ++x) {
          if (p0 + x >= n) break;
          uint32_t code, ms, isn;
          classify(seq[p0 + x], code, ms, isn);
          word |= code << (2 * x);
          m16 |= ms << x;
          n16 |= isn << x;
        }
      }
    }
    const uint32_t om = __shfl_down_sync(0xffffffffu, m16, 1);
    const uint32_t on = __shfl_down_sync(0xffffffffu, n16, 1);
    if (c < nchunk) {
      packed[c] = word;
      if ((c & 1) == 0) {
        mask[c >> 1] = m16 | (om << 16);
        nbits[c >> 1] = n16 | (on << 16);
      }
    }
  }
}

constexpr int kSkThreads = 256;
constexpr int kSkWarps = kSkThreads / 32;
constexpr int kSkP = 16;                           // positions per lane
constexpr int kSkMaxW = 256;
// Lanes of a warp that own windows: not the first (it gives the window
// before lane 1's first) and not the last ceil((w - 1) / 16), whose windows
// would leave the warp's positions.
__host__ __device__ constexpr int sk_lanes(int w) { return 31 - (w - 1 + kSkP - 1) / kSkP; }
__host__ __device__ constexpr int sk_warp_windows(int w) { return sk_lanes(w) * kSkP; }
// Stretches of one warp in a CTA tile.  Long inputs take four, for a quarter
// of the look-backs; short ones one, for more CTAs.
constexpr int kSkRep = 4;
constexpr int64_t kSkRepBases = int64_t(32) << 20;
__host__ __device__ constexpr int64_t sk_tile_windows(int w, int rep) {
  return (int64_t)sk_warp_windows(w) * kSkWarps * rep;
}
constexpr int sk_rep(int64_t n) { return n >= kSkRepBases ? kSkRep : 1; }
constexpr int kSkStage = 31 * kSkP * kSkRep;       // k-mers a warp can select

__device__ __forceinline__ uint32_t bijective_hash(uint32_t x, int k, uint32_t M) {
  // A permutation of [0, 4^k): xor-shift-right and odd multipliers, all
  // modulo 2^(2k) (2k <= 30 bits, so 32-bit arithmetic is exact mod 2^(2k)).
  x &= M;
  x ^= x >> k;
  x = (x * 0x7F4A7C15u) & M;
  x ^= x >> (k - 1);
  x = (x * 0x6659FD93u) & M;
  x ^= x >> k;
  return x;
}

struct SketchArgs {
  const uint32_t* packed;
  const uint32_t* mask;
  const uint32_t* nbits;
  const int64_t* off;  // nseq + 1 sequence offsets (device)
  int nseq;
  int64_t N;
  int k, w, min_unmasked;
  uint32_t kmask;
  int rep;         // stretches of a warp per CTA tile
  int64_t ntiles;
};

// Single-pass form: each CTA takes tiles in ticket order, publishes its
// tile's record count, and adds up its predecessors' counts (decoupled
// look-back) until one has published its inclusive prefix.  A tile's
// predecessors were all taken before it by CTAs that publish their count
// before they wait on anyone, so every wait ends; it is bounded all the
// same, and a wait that gives up raises *err for the host.
struct LookBack {
  unsigned long long* status;  // per tile: flag (2 bits) and value (62 bits); zeroed
  unsigned int* ticket;        // next tile to take; zeroed
  unsigned long long* total;   // records of all tiles (written by the last tile)
  int* err;                    // set when a wait gives up; zeroed
};

constexpr unsigned long long kLbAggregate = 1ull << 62, kLbPrefix = 2ull << 62;
constexpr unsigned long long kLbValue = (1ull << 62) - 1;
constexpr unsigned int kLbSpins = 1u << 20;  // polls of one predecessor before giving up

// Records before tile `tile`; warp 0 of the CTA calls it once per tile.  The
// warp reads the status of the 256 tiles below its window at once (eight
// independent loads per lane: as many tiles are in flight, so a narrower
// window walks several round trips to the nearest published prefix): the
// nearest tile that has published its inclusive prefix ends the walk, and
// the counts of the tiles above it are summed by the warp.
__device__ long long look_back(const LookBack& lb, int64_t tile, int64_t ntiles,
                               unsigned long long count) {
  constexpr int kWide = 8;
  const int lane = threadIdx.x & 31;
  long long before = 0;
  if (tile > 0) {
    if (lane == 0) st_relaxed_gpu(lb.status + tile, kLbAggregate | count);
    int64_t j = tile - 1;  // the walk's top tile
    unsigned int spins = 0;
    bool done = false;
    while (!done) {
      unsigned long long v[kWide];
#pragma unroll
      for (int x = 0; x < kWide; ++x) {
        const int64_t at = j - x * 32 - lane;
        // below tile 0 reads as a published prefix of zero
        v[x] = at >= 0 ? ld_relaxed_gpu(lb.status + at) : kLbPrefix;
      }
#pragma unroll
      for (int x = 0; x < kWide; ++x) {
        const unsigned long long flag = v[x] & ~kLbValue;
        const unsigned prefix = __ballot_sync(0xffffffffu, flag == kLbPrefix);
        const int p = prefix ? __ffs(prefix) - 1 : 31;  // lanes 0..p take part
        const unsigned need = p == 31 ? 0xffffffffu : ((1u << (p + 1)) - 1u);
        if (__ballot_sync(0xffffffffu, flag == 0) & need) {
          if (++spins > kLbSpins) {
            if (lane == 0) atomicExch(lb.err, 1);
            done = true;
          }
          break;  // read again from this window's top
        }
        spins = 0;
        before += lane <= p ? (long long)(v[x] & kLbValue) : 0;
        if (prefix) {
          done = true;
          break;
        }
        j -= 32;
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
  }
  if (lane == 0) {
    st_relaxed_gpu(lb.status + tile, kLbPrefix | ((unsigned long long)before + count));
    if (tile == ntiles - 1) *lb.total = (unsigned long long)before + count;
  }
  return before;
}

// Window keys: a hash over the reversed offset of its position from the
// lane's first one (so that the rightmost of equal hashes is the least); the
// ineligible key lies above every hash.  A key read from the lane d lanes up
// is rebased by subtracting 16 d.
template <typename K>
struct Key;
template <>
struct Key<uint32_t> {  // 24-bit hashes, offsets up to 127
  static __device__ __forceinline__ uint32_t make(uint32_t h, int off) { return h * 128u + (127u - off); }
  static __device__ __forceinline__ uint32_t none(int off) { return 0x80000000u + (127u - off); }
  static __device__ __forceinline__ bool is_none(uint32_t v) { return (int)v < 0; }
  static __device__ __forceinline__ int off(uint32_t v) { return 127 - (int)(v & 127u); }
};
template <>
struct Key<uint64_t> {
  static __device__ __forceinline__ uint64_t make(uint32_t h, int off) {
    return ((uint64_t)h << 32) | (uint32_t)(0xFFFF - off);
  }
  static __device__ __forceinline__ uint64_t none(int off) { return make(kInfHash, off); }
  static __device__ __forceinline__ bool is_none(uint64_t v) { return (uint32_t)(v >> 32) == kInfHash; }
  static __device__ __forceinline__ int off(uint64_t v) { return 0xFFFF - (int)(uint32_t)v; }
};

// v[x] = the value D positions on (D < 16; the next lane's, rebased, past the end).
template <int D, typename K>
__device__ __forceinline__ void shift_positions(K (&v)[kSkP]) {
  K next[D];
#pragma unroll
  for (int x = 0; x < D; ++x) next[x] = __shfl_down_sync(0xffffffffu, v[x], 1) - (K)kSkP;
#pragma unroll
  for (int x = 0; x < kSkP; ++x) v[x] = x + D < kSkP ? v[x + D] : next[x + D - kSkP];
}

// v[x] = min(v[x], the value D positions on).
template <int D, typename K>
__device__ __forceinline__ void min_positions(K (&v)[kSkP]) {
  K next[D];
#pragma unroll
  for (int x = 0; x < D; ++x) next[x] = __shfl_down_sync(0xffffffffu, v[x], 1) - (K)kSkP;
#pragma unroll
  for (int x = 0; x < kSkP; ++x) v[x] = min(v[x], x + D < kSkP ? v[x + D] : next[x + D - kSkP]);
}

// key[x]: minimum over the w positions from x on.
template <typename K>
__device__ __forceinline__ void window_minima(int w, K (&key)[kSkP]) {
  int len = 1;
  if (w >= 2) min_positions<1>(key), len = 2;
  if (w >= 4) min_positions<2>(key), len = 4;
  if (w >= 8) min_positions<4>(key), len = 8;
  if (w >= 16) min_positions<8>(key), len = 16;
  while (2 * len <= w) {  // whole lanes
#pragma unroll
    for (int x = 0; x < kSkP; ++x)
      key[x] = min(key[x], (K)(__shfl_down_sync(0xffffffffu, key[x], len / kSkP) - (K)len));
    len *= 2;
  }
  const int r = w - len;  // the rest: two overlapping minima
  if (r > 0) {
    K v[kSkP];
#pragma unroll
    for (int x = 0; x < kSkP; ++x) v[x] = key[x];
    if (r & 1) shift_positions<1>(v);
    if (r & 2) shift_positions<2>(v);
    if (r & 4) shift_positions<4>(v);
    if (r & 8) shift_positions<8>(v);
    const int up = r / kSkP;
    if (up > 0) {
#pragma unroll
      for (int x = 0; x < kSkP; ++x) v[x] = __shfl_down_sync(0xffffffffu, v[x], up) - (K)(up * kSkP);
    }
#pragma unroll
    for (int x = 0; x < kSkP; ++x) key[x] = min(key[x], v[x]);
  }
}

// The 2-bit groups of a word in reverse order.
__device__ __forceinline__ uint32_t reverse_pairs(uint32_t v) {
  v = __brev(v);
  return ((v >> 1) & 0x55555555u) | ((v & 0x55555555u) << 1);
}

// kMode 0: count the records of each CTA tile; 1: write them at the tile
// offsets given; 2: one pass, offsets by look-back.
//
// Bound by the integer pipe and the tile's barriers: two warp instructions a
// base at k = 12, w = 16 (the form that hashed into shared memory and took van
// Herk minima from it ran 8.1); on 240 Mbp the pipe is busy 73% of the time,
// and what the warps wait for otherwise is warp 0's look-back between the two
// barriers of a tile (7 of 13 stalled warps).  A lane holds as many positions as its registers
// allow (16 keys and their shifted copies in 64 registers, four CTAs per SM);
// the lanes without windows, two of 32 at w = 16, are the waste.  3.1 Gbp:
// 33.7 -> 9.8 ms, 240 Mbp: 2.6 -> 0.78 ms.  Of that the look-back was most:
// with a 32-tile window, one stretch per warp and the next ticket taken
// before the walk the same kernel took 35.7 ms at 3.1 Gbp.
template <int kMode, typename K>
__global__ void __launch_bounds__(kSkThreads, sizeof(K) == 4 ? 4 : 2) k_sketch(SketchArgs a, uint32_t* __restrict__ tile_count,
                                                          const uint32_t* __restrict__ tile_offset,
                                                          uint64_t* __restrict__ out, int64_t cap,
                                                          LookBack lb) {
  // selected positions from the warp's first one, in order
  __shared__ uint16_t s_stage[kMode == 0 ? 1 : kSkWarps][kMode == 0 ? 1 : kSkStage];
  __shared__ int s_cnt[kSkWarps], s_off[kSkWarps];
  __shared__ long long s_tile, s_base;
  const int k = a.k, w = a.w;
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const int wlanes = sk_lanes(w), wwin = sk_warp_windows(w);
  const uint32_t kmask = a.kmask;
  const int64_t nw16 = (a.N + 15) >> 4;
  const uint16_t* mask16 = reinterpret_cast<const uint16_t*>(a.mask);
  const uint16_t* nbits16 = reinterpret_cast<const uint16_t*>(a.nbits);
  int64_t seg_lo = 0, seg_hi = -1;  // the sequence that held the last stretch's first position
  int64_t tile = blockIdx.x;
  if (kMode == 2) {
    if (threadIdx.x == 0) s_tile = (long long)atomicAdd(lb.ticket, 1u);
    __syncthreads();
    tile = s_tile;
  }
  while (tile < a.ntiles) {
    const int64_t base0 = (tile * kSkWarps + warp) * (int64_t)(wwin * a.rep) - kSkP;
    int n = 0;  // k-mers selected
    for (int rep = 0; rep < a.rep; ++rep) {
      const int64_t base = base0 + rep * wwin, first = base + kSkP;  // first: the first window
      int cnt = 0;
      uint32_t flags = 0;
      K key[kSkP];
      if (first < a.N) {
        if (first < seg_lo || first >= seg_hi) {
          const int s = seq_of(a.off, a.nseq, first);
          seg_lo = a.off[s];
          seg_hi = a.off[s + 1];
        }
        const int64_t p0 = base + lane * kSkP;
        const int64_t wi = p0 >> 4;
        const bool in0 = wi >= 0 && wi < nw16, in1 = wi + 1 < nw16;
        const uint32_t w0 = in0 ? __ldg(a.packed + wi) : 0u;
        const uint32_t w1 = in1 ? __ldg(a.packed + wi + 1) : 0u;
        const uint32_t mk = (in0 ? (uint32_t)__ldg(mask16 + wi) : 0xFFFFu) |
                            ((in1 ? (uint32_t)__ldg(mask16 + wi + 1) : 0xFFFFu) << 16);
        const uint32_t nb = (in0 ? (uint32_t)__ldg(nbits16 + wi) : 0xFFFFu) |
                            ((in1 ? (uint32_t)__ldg(nbits16 + wi + 1) : 0xFFFFu) << 16);
        // bit x: the k-mer at p0 + x holds an N, or (min_unmasked = 1) only
        // masked bases; the shifts reach bit 15 + 14 at most
        uint32_t bad = nb, all = mk;
        {
          int len = 1;
          for (; 2 * len <= k; len *= 2) {
            bad |= bad >> len;
            all &= all >> len;
          }
          bad |= bad >> (k - len);
          all &= all >> (k - len);
        }
        if (a.min_unmasked == 1) {
          bad |= all;
        } else if (a.min_unmasked > 1) {
          const uint32_t kb = (1u << k) - 1u;
#pragma unroll
          for (int x = 0; x < kSkP; ++x)
            if (k - __popc((mk >> x) & kb) < a.min_unmasked) bad |= 1u << x;
        }
        // windows that lie in one sequence; only lanes near a sequence's end
        // look at their positions one by one
        uint32_t ok = 0xFFFFu;
        if (p0 < seg_lo || p0 + kSkP - 1 + w + k - 1 > seg_hi) {
          ok = 0;
          int64_t lo = seg_lo, hi = seg_hi;
          for (int x = 0; x < kSkP; ++x) {
            const int64_t p = p0 + x;
            if (p < 0 || p >= a.N) {
              bad |= 1u << x;
              continue;
            }
            if (p < lo || p >= hi) {
              const int s = seq_of(a.off, a.nseq, p);
              lo = a.off[s];
              hi = a.off[s + 1];
            }
            if (p + k > hi) bad |= 1u << x;
            if (p + w + k - 1 <= hi) ok |= 1u << x;
          }
        }
        const uint32_t r0 = reverse_pairs(w0), r1 = reverse_pairs(w1);
#pragma unroll
        for (int x = 0; x < kSkP; ++x) {
          // forward code: first base most significant; the reverse complement's
          // is the complement with the first base least significant
          const uint32_t f = __funnelshift_l(r1, r0, 2 * x) >> (32 - 2 * k);
          const uint32_t rc = ~__funnelshift_r(w0, w1, 2 * x) & kmask;
          const uint32_t h = bijective_hash(f < rc ? f : rc, k, kmask);
          key[x] = ((bad >> x) & 1u) || f == rc ? Key<K>::none(x) : Key<K>::make(h, x);
        }
        window_minima(w, key);
        // selected: an eligible minimum that is not the previous window's
        const K before = __shfl_up_sync(0xffffffffu, key[kSkP - 1], 1) + (K)kSkP;
        uint32_t valid = 0;
#pragma unroll
        for (int x = 0; x < kSkP; ++x)
          if (!Key<K>::is_none(key[x])) valid |= 1u << x;
        valid &= ok;
        uint32_t same = 0;
#pragma unroll
        for (int x = 0; x < kSkP; ++x)
          if (key[x] == (x ? key[x - 1] : before)) same |= 1u << x;
        const uint32_t vb = __shfl_up_sync(0xffffffffu, valid >> (kSkP - 1), 1);
        flags = valid & ~(same & ((valid << 1) | (vb & 1u)));
        if (lane == 0 || lane > wlanes) flags = 0;
        cnt = __popc(flags);
      }
      const int inc = warp_inclusive_sum(cnt);
      if (kMode != 0) {
        int at = n + inc - cnt;
#pragma unroll
        for (int x = 0; x < kSkP; ++x) {
          if ((flags >> x) & 1u) {
            s_stage[warp][at] = (uint16_t)(rep * wwin + lane * kSkP + Key<K>::off(key[x]));
            ++at;
          }
        }
      }
      n += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) s_cnt[warp] = n;
    __syncthreads();
    if (warp == 0) {
      const int c = lane < kSkWarps ? s_cnt[lane] : 0;
      const int ci = warp_inclusive_sum(c);
      const int total = __shfl_sync(0xffffffffu, ci, 31);
      if (lane < kSkWarps) s_off[lane] = ci - c;
      if (kMode == 0) {
        if (lane == 0) tile_count[tile] = (uint32_t)total;
      } else if (kMode == 1) {
        if (lane == 0) s_base = (long long)tile_offset[tile];
      } else {
        const long long before = look_back(lb, tile, a.ntiles, (unsigned long long)total);
        // the next ticket only now: an earlier one would keep the tiles
        // above it waiting through this look-back
        if (lane == 0) {
          s_base = before;
          s_tile = (long long)atomicAdd(lb.ticket, 1u);
        }
      }
    }
    __syncthreads();
    if (kMode != 0) {
      const int64_t o = s_base + s_off[warp];
      for (int x = lane; x < n; x += 32) {
        // the selected k-mer's hash and strand, from its codes again
        const int64_t p = base0 + s_stage[warp][x];
        const int64_t wi = p >> 4;
        const uint32_t w0 = __ldg(a.packed + wi), w1 = wi + 1 < nw16 ? __ldg(a.packed + wi + 1) : 0u;
        const uint32_t g = __funnelshift_r(w0, w1, 2 * (int)(p & 15)) & kmask;
        const uint32_t f = reverse_pairs(g) >> (32 - 2 * k);
        const uint32_t rc = g ^ kmask;
        const uint32_t h = bijective_hash(f < rc ? f : rc, k, kmask);
        if (o + x < cap) out[o + x] = ((uint64_t)h << 33) | ((uint64_t)p << 1) | (uint64_t)(rc < f ? 1u : 0u);
      }
      __syncwarp();
    }
    tile = kMode == 2 ? s_tile : tile + gridDim.x;
  }
}

// The 32-bit window keys hold a hash of 2k bits and a 7-bit offset.
bool narrow_keys(const Derived& D) { return 2 * D.k <= 24 && D.w <= 112; }

}  // namespace

int launch_pack(sedef_ctx* ctx, const uint8_t* seq, int64_t n, uint32_t* packed, uint32_t* mask,
                uint32_t* nbits) {
  cudaStream_t st = ctx_stream(ctx);
  const int64_t nchunk = (n + 15) / 16;
  int64_t blocks = (nchunk + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (blocks < 1) blocks = 1;
  if (((uintptr_t)seq & 15) == 0)
    SEDEF_KERNEL(ctx, "k_pack", k_pack<true><<<(int)blocks, 256, 0, st>>>(seq, n, packed, mask, nbits));
  else
    SEDEF_KERNEL(ctx, "k_pack", k_pack<false><<<(int)blocks, 256, 0, st>>>(seq, n, packed, mask, nbits));
  return SEDEF_OK;
}

int scan_exclusive_u32(sedef_ctx* ctx, const uint32_t* in, uint32_t* out, int64_t n,
                       uint32_t* d_total);

int run_sketch(sedef_ctx* ctx, const uint32_t* packed, const uint32_t* mask, const uint32_t* nbits,
               const int64_t* h_off, int nseq, const Derived& D, uint64_t* rec, int64_t cap,
               int64_t* nrec, Planned* pl) {
  cudaStream_t st = ctx_stream(ctx);
  const int64_t N = h_off[nseq];
  SketchArgs a;
  a.packed = packed;
  a.mask = mask;
  a.nbits = nbits;
  a.nseq = nseq;
  a.N = N;
  a.k = D.k;
  a.w = D.w;
  a.min_unmasked = D.min_unmasked;
  a.kmask = D.kmask;
  const int64_t nwin = N;  // window starts q in [0, N)
  a.rep = sk_rep(N);
  a.ntiles = (nwin + sk_tile_windows(D.w, a.rep) - 1) / sk_tile_windows(D.w, a.rep);
  int64_t* d_off = (int64_t*)ctx_alloc(ctx, (size_t)(nseq + 1) * 8);
  if (!d_off) return SEDEF_ERR_OOM;
  if (pl) {
    int64_t* h = (int64_t*)host_buf(ctx, pl, (size_t)(nseq + 1) * 8);
    if (!h) return SEDEF_ERR_OOM;
    std::memcpy(h, h_off, (size_t)(nseq + 1) * 8);
    SEDEF_CUDA(cudaMemcpyAsync(d_off, h, (size_t)(nseq + 1) * 8, cudaMemcpyHostToDevice, st));
  } else {
    SEDEF_CUDA(cudaMemcpyAsync(d_off, h_off, (size_t)(nseq + 1) * 8, cudaMemcpyHostToDevice, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));  // h_off is caller memory: copy before returning
  }
  a.off = d_off;
  const bool narrow = narrow_keys(D);
  int64_t grid = a.ntiles;
  const int64_t maxgrid = (int64_t)ctx_sm_count(ctx) * 8;
  if (grid > maxgrid) grid = maxgrid;
  if (!pl) {
    // one pass: record offsets by look-back over the tiles
    if (a.ntiles == 0) {
      *nrec = 0;
      return SEDEF_OK;
    }
    unsigned long long* status = (unsigned long long*)ctx_alloc(ctx, (size_t)(a.ntiles + 4) * 8);
    if (!status) return SEDEF_ERR_OOM;
    LookBack lb;
    lb.status = status + 4;
    lb.ticket = (unsigned int*)status;
    lb.total = status + 1;
    lb.err = (int*)(status + 2);
    SEDEF_CUDA(cudaMemsetAsync(status, 0, (size_t)(a.ntiles + 4) * 8, st));
    if (narrow)
      SEDEF_KERNEL(ctx, "k_sketch",
                   k_sketch<2, uint32_t><<<(int)grid, kSkThreads, 0, st>>>(a, nullptr, nullptr, rec, cap, lb));
    else
      SEDEF_KERNEL(ctx, "k_sketch",
                   k_sketch<2, uint64_t><<<(int)grid, kSkThreads, 0, st>>>(a, nullptr, nullptr, rec, cap, lb));
    unsigned long long* h = (unsigned long long*)ctx_host(ctx, 16);
    if (!h) return SEDEF_ERR_OOM;
    SEDEF_CUDA(cudaMemcpyAsync(h, status + 1, 16, cudaMemcpyDeviceToHost, st));
    SEDEF_CUDA(cudaStreamSynchronize(st));
    if ((int)h[1] != 0) return fail(SEDEF_ERR_TIMEOUT, "sedef_sketch: a tile's offset wait gave up");
    *nrec = (int64_t)h[0];
    if (*nrec > cap) return fail(SEDEF_ERR_CAPACITY, "sedef_sketch: record buffer too small");
    return SEDEF_OK;
  }
  // planned pass (one CUDA graph): count, scan and write, without waits
  // between CTAs; the write pass stores the records below the capacity and the
  // exact total stays on the device
  uint32_t* cnt = (uint32_t*)ctx_alloc(ctx, (size_t)(a.ntiles + 1) * 4);
  uint32_t* toff = (uint32_t*)ctx_alloc(ctx, (size_t)(a.ntiles + 1) * 4);
  if (!cnt || !toff) return SEDEF_ERR_OOM;
  if (narrow)
    SEDEF_KERNEL(ctx, "k_sketch_count",
                 k_sketch<0, uint32_t><<<(int)grid, kSkThreads, 0, st>>>(a, cnt, nullptr, nullptr, 0, LookBack{}));
  else
    SEDEF_KERNEL(ctx, "k_sketch_count",
                 k_sketch<0, uint64_t><<<(int)grid, kSkThreads, 0, st>>>(a, cnt, nullptr, nullptr, 0, LookBack{}));
  SEDEF_TRY(scan_exclusive_u32(ctx, cnt, toff, a.ntiles, toff + a.ntiles));
  pl->n_rec = toff + a.ntiles;
  SEDEF_TRY(plan_check(ctx, pl, toff + a.ntiles, cap, 0));
  *nrec = cap;
  if (narrow)
    SEDEF_KERNEL(ctx, "k_sketch_write",
                 k_sketch<1, uint32_t><<<(int)grid, kSkThreads, 0, st>>>(a, nullptr, toff, rec, cap, LookBack{}));
  else
    SEDEF_KERNEL(ctx, "k_sketch_write",
                 k_sketch<1, uint64_t><<<(int)grid, kSkThreads, 0, st>>>(a, nullptr, toff, rec, cap, LookBack{}));
  return SEDEF_OK;
}

}  // namespace sedef

// ------------------------------------------------ allocation-free sketch --
//
// sedef_sketch_noalloc: the sketch with its scratch (per-tile counts and
// offsets, the sequence offsets) in a fixed static device array instead of
// memory from a context, for callers that must not allocate device memory.
// The array's host-side name is only a stand-in, so its device address is
// looked up once per device with cudaGetSymbolAddress and passed to the
// kernels.

namespace sedef {
namespace {

constexpr int64_t kNoallocMaxBases = int64_t(256) << 20;  // 268,435,456 bases
constexpr int kNoallocMaxSeqs = 4096;
// the widest window has the fewest windows per tile; inputs just below the
// long ones have the most tiles of one stretch
constexpr int64_t kNoallocMaxTiles =
    (kNoallocMaxBases + sk_tile_windows(kSkMaxW, kSkRep) - 1) / sk_tile_windows(kSkMaxW, kSkRep);
static_assert(kNoallocMaxTiles >= (kSkRepBases + sk_tile_windows(kSkMaxW, 1) - 1) / sk_tile_windows(kSkMaxW, 1),
              "the shorter inputs' tiles must fit too");
constexpr size_t kNoallocCountBytes = (size_t)(kNoallocMaxTiles + 1) * 4;
constexpr size_t kNoallocBytes = 2 * kNoallocCountBytes + (size_t)(kNoallocMaxSeqs + 1) * 8;

// Shared by every call in the process and kept between calls; about 1 MB on
// each device that loads the library.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];


// Exclusive scan of n counts by one block (n is at most 34,953 here).
__global__ void __launch_bounds__(1024) k_scan_one_block(const uint32_t* __restrict__ in,
                                                         uint32_t* __restrict__ out, int64_t n) {
  __shared__ int tmp[33];
  const int64_t per = (n + blockDim.x - 1) / blockDim.x;
  const int64_t lo = (int64_t)threadIdx.x * per, hi = min(n, lo + per);
  uint32_t s = 0;
  for (int64_t x = lo; x < hi; ++x) s += in[x];
  int tot;
  uint32_t run = (uint32_t)block_exclusive_sum((int)s, tmp, &tot);
  for (int64_t x = lo; x < hi; ++x) {
    const uint32_t v = in[x];
    out[x] = run;
    run += v;
  }
  if (threadIdx.x == 0) out[n] = (uint32_t)tot;
}

}  // namespace
}  // namespace sedef

extern "C" int sedef_sketch_noalloc(const uint32_t* d_packed, const uint32_t* d_mask,
                                    const uint32_t* d_nbits, const int64_t* h_seq_off,
                                    int32_t nseq, const sedef_params* p, uint64_t* d_rec,
                                    int64_t rec_cap, int64_t* h_nrec, void* stream) {
  using namespace sedef;
  if (!h_nrec) return fail(SEDEF_ERR_INVALID, "h_nrec is NULL");
  *h_nrec = 0;
  Derived D;
  SEDEF_TRY(derive(p, &D));
  if (nseq < 0 || (nseq > 0 && !h_seq_off)) return fail(SEDEF_ERR_INVALID, "bad offsets");
  if (nseq == 0) return SEDEF_OK;
  if (h_seq_off[0] != 0) return fail(SEDEF_ERR_INVALID, "offsets must start at 0");
  for (int s = 0; s < nseq; ++s)
    if (h_seq_off[s + 1] < h_seq_off[s]) return fail(SEDEF_ERR_INVALID, "offsets decrease");
  const int64_t N = h_seq_off[nseq];
  if (N == 0) return SEDEF_OK;
  if (N > kNoallocMaxBases || nseq > kNoallocMaxSeqs)
    return fail(SEDEF_ERR_UNSUPPORTED,
                "sedef_sketch_noalloc: at most 268435456 bases in at most 4096 sequences "
                "(the fixed scratch array); use sedef_sketch for larger inputs");
  if (!d_packed || !d_mask || !d_nbits || (rec_cap > 0 && !d_rec))
    return fail(SEDEF_ERR_INVALID, "NULL buffer");
  int dev = 0;
  SEDEF_CUDA(cudaGetDevice(&dev));
  // The array's device address on the current device.  Looked up on every
  // call (a table lookup once the module is loaded; the first call on a
  // device loads it), so it stays right after a cudaDeviceReset and needs no
  // lock between host threads.  In host code the array's name is only a
  // host-side stand-in, never a device address.
  void* ptr = nullptr;
  {
    const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || !ptr) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
  }
  unsigned char* base = (unsigned char*)ptr;
  uint32_t* cnt = reinterpret_cast<uint32_t*>(base);
  uint32_t* toff = reinterpret_cast<uint32_t*>(base + kNoallocCountBytes);
  int64_t* d_off = reinterpret_cast<int64_t*>(base + 2 * kNoallocCountBytes);
  cudaStream_t st = (cudaStream_t)stream;
  SEDEF_CUDA(cudaMemcpyAsync(d_off, h_seq_off, (size_t)(nseq + 1) * 8, cudaMemcpyHostToDevice, st));
  SketchArgs a;
  a.packed = d_packed;
  a.mask = d_mask;
  a.nbits = d_nbits;
  a.off = d_off;
  a.nseq = nseq;
  a.N = N;
  a.k = D.k;
  a.w = D.w;
  a.min_unmasked = D.min_unmasked;
  a.kmask = D.kmask;
  a.rep = sk_rep(N);
  a.ntiles = (N + sk_tile_windows(D.w, a.rep) - 1) / sk_tile_windows(D.w, a.rep);
  int sms = 0;
  SEDEF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  int64_t grid = a.ntiles < (int64_t)sms * 8 ? a.ntiles : (int64_t)sms * 8;
  if (narrow_keys(D))
    k_sketch<0, uint32_t><<<(int)grid, kSkThreads, 0, st>>>(a, cnt, nullptr, nullptr, 0, LookBack{});
  else
    k_sketch<0, uint64_t><<<(int)grid, kSkThreads, 0, st>>>(a, cnt, nullptr, nullptr, 0, LookBack{});
  count_launch();
  SEDEF_LAUNCHED("k_sketch_count");
  k_scan_one_block<<<1, 1024, 0, st>>>(cnt, toff, a.ntiles);
  count_launch();
  SEDEF_LAUNCHED("k_scan_one_block");
  uint32_t total = 0;
  SEDEF_CUDA(cudaMemcpyAsync(&total, toff + a.ntiles, 4, cudaMemcpyDeviceToHost, st));
  SEDEF_CUDA(cudaStreamSynchronize(st));
  *h_nrec = total;
  if ((int64_t)total > rec_cap) return fail(SEDEF_ERR_CAPACITY, "record buffer too small");
  if (narrow_keys(D))
    k_sketch<1, uint32_t><<<(int)grid, kSkThreads, 0, st>>>(a, nullptr, toff, d_rec, rec_cap, LookBack{});
  else
    k_sketch<1, uint64_t><<<(int)grid, kSkThreads, 0, st>>>(a, nullptr, toff, d_rec, rec_cap, LookBack{});
  count_launch();
  SEDEF_LAUNCHED("k_sketch_write");
  SEDEF_CUDA(cudaStreamSynchronize(st));
  return SEDEF_OK;
}
