// CSR construction by a least-significant-digit radix sort of packed edge
// keys: the CSRs of G and of G' (Section 4.1, 4.3 of arXiv 2404.08299) from an
// edge list, duplicates merged and one self-loop per vertex (Section 3.1,
// 5.1.3). Weights move with their keys; merged duplicates keep the largest.
//
// Key of entry (r, c): r << B | c, B = bits of n - 1, so the key order is the
// CSR order (rows ascending, columns ascending inside a row). Eight key bits
// per pass, ceil(2B / 8) passes; each pass is
//   tile histograms -> one exclusive scan over [digit][tile] -> stable scatter
// with tiles of 4096 keys. The scatter ranks a tile's keys by digit in shared
// memory (warp-level match of equal digits, per-warp counters, in input
// order, so every pass is stable) and writes each digit's run of the tile to
// its global place from a staged copy, so the stores are contiguous runs
// rather than one random store per key. No global atomics, so the result
// and its timing do not depend on how skewed the rows are. The first pass
// reads the edge list and makes the keys (and the self-loop keys) on the
// fly. After the last pass, adjacent equal keys are merged: a count per warp,
// one scan, one emit pass that writes the columns and the row offsets (found
// row-parallel instead when the list is much shorter than n).
#include "internal.cuh"

namespace prdf {

namespace {

constexpr int kRT = 256;              // threads per tile
constexpr int kRK = 16;               // keys per thread
constexpr int kRTile = kRT * kRK;     // 4096 keys per tile
constexpr int kRWarps = kRT / 32;
constexpr int kRBlocks = 3;           // blocks an SM of the scatter
constexpr int kRDigits = 256;
static_assert(kRT == kRDigits, "one digit per thread in the scatter's digit scan");
static_assert(kRTile <= 65536 && kRK % 2 == 0, "ranks are packed two to a word");

struct KeySrc {
  const uint64_t* keys;  // later passes
  const float* w;        // weighted builds: the entries' weights, moved along with the keys
  const int32_t* rows;   // first pass: entry i < m0 is (rows[i], cols[i]),
  const int32_t* cols;   // entry m0 + v is the self-loop (v, v)
  int64_t m0;
  int B;
};

// key of the list's entry i < m0
__device__ __forceinline__ uint64_t list_key(const KeySrc& s, int64_t i) {
  return ((uint64_t)(uint32_t)__ldcs(s.rows + i) << s.B) | (uint64_t)(uint32_t)__ldcs(s.cols + i);
}

template <bool FIRST>
__device__ __forceinline__ uint64_t load_key(const KeySrc& s, int64_t i) {
  if (!FIRST) return __ldcs(reinterpret_cast<const unsigned long long*>(s.keys) + i);
  if (i < s.m0) return list_key(s, i);
  const uint64_t v = (uint64_t)(i - s.m0);
  return (v << s.B) | v;
}

// weight of entry i; 0 marks an added self-loop (given weights are positive)
template <bool FIRST>
__device__ __forceinline__ float load_w(const KeySrc& s, int64_t i) {
  if (FIRST && i >= s.m0) return 0.f;
  return __ldcs(s.w + i);
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Lanes of the warp whose value d (BITS bits) equals this lane's: one ballot
// per bit. Bit 8 marks lanes without a key; full tiles match 8 bits.
template <int BITS>
__device__ __forceinline__ uint32_t match_digit(uint32_t d) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < BITS; ++b) {
    const uint32_t m = __ballot_sync(0xffffffffu, (d >> b) & 1u);
    peers &= ~(m ^ (0u - ((d >> b) & 1u)));  // no select: 3 % of a build
  }
  return peers;
}

// Exclusive scan of one value per thread over a block of kRT threads.
// wsum: kRWarps words of shared memory; the caller syncs before reusing it.
__device__ __forceinline__ uint32_t block_scan_excl(uint32_t v, uint32_t* wsum, uint32_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) wsum[w] = x;
  __syncthreads();
  uint32_t add = 0, all = 0;
#pragma unroll
  for (int k = 0; k < kRWarps; ++k) {
    const uint32_t c = wsum[k];
    add += k < w ? c : 0u;
    all += c;
  }
  if (total) *total = all;
  return x - v + add;
}

// hist[d * ntiles + tile] = number of keys of the tile whose digit is d.
// Counting needs no ranks: a shared-memory atomic per key on the warp's own
// counters (equal digits within a warp are serialised by the hardware).
template <bool FIRST>
__global__ void __launch_bounds__(kRT) k_radix_hist(const KeySrc src, int64_t M, int shift, uint32_t* __restrict__ hist,
                                                     int64_t ntiles) {
  __shared__ uint32_t h[kRWarps][kRDigits];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kRWarps; ++k) h[k][threadIdx.x] = 0;
  const int64_t i0 = (int64_t)blockIdx.x * kRTile + (int64_t)w * (32 * kRK) + lane;
  const int nv = M <= i0 ? 0 : (M - i0 >= 32 * kRK ? kRK : (int)((M - i0 + 31) / 32));
  uint32_t d[kRK];
  if (FIRST && src.B >= 8 && (int64_t)(blockIdx.x + 1) * kRTile <= src.m0) {
    // the first digit is in the column alone
#pragma unroll
    for (int r = 0; r < kRK; ++r) d[r] = (uint32_t)__ldcs(src.cols + i0 + r * 32) & 0xFFu;
  } else {
#pragma unroll
    for (int r = 0; r < kRK; ++r)
      d[r] = r < nv ? (uint32_t)(load_key<FIRST>(src, i0 + r * 32) >> shift) & 0xFFu : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRK; ++r)
    if (r < nv) atomicAdd(&h[w][d[r]], 1u);
  __syncthreads();
  uint32_t c = 0;
#pragma unroll
  for (int k = 0; k < kRWarps; ++k) c += h[k][threadIdx.x];
  hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = c;
}

// Rank of each key among the equal digits before it in its warp's part of the
// tile: earlier rounds (the warp's counter), then lower lanes of the same
// round. FULL: every round of every lane has a key (else rounds r < nv).
template <bool FULL>
__device__ __forceinline__ void rank_keys(const uint64_t (&key)[kRK], int shift, int nv, uint32_t* mine,
                                          uint32_t (&rank)[kRK / 2]) {
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const bool ok = FULL || r < nv;
    const uint32_t d = ok ? (uint32_t)(key[r] >> shift) & 0xFFu : 0x100u;
    const uint32_t peers = match_digit<FULL ? 8 : 9>(d);
    const uint32_t before = (uint32_t)__popc(peers & lt);
    const uint32_t prev = ok ? mine[d] : 0u;
    __syncwarp();
    if (ok && before == 0) mine[d] = prev + (uint32_t)__popc(peers);
    __syncwarp();
    const uint32_t rk = prev + before;
    if (r & 1) rank[r >> 1] |= rk << 16;
    else rank[r >> 1] = rk;
  }
}

// Stable scatter of one tile by digit; goff = exclusive scan of hist. W: the
// weights move with their keys. Bound by shared memory (the data pipe 85 %
// busy: counters by digit and the staged keys are hit at random banks) and by
// issue (60 %, the ballots), not by DRAM (4.0 of 6.7 TB/s). So a digit's start
// is folded into the warps' counters (one random read less a key), and full
// tiles take a branch-free path: all loads are in flight before the first
// key is ranked, and no round tests for a missing key. 285 M keys to two CSRs:
// 28.5 ms before, 24.2 now; the first pass alone 2.6 ms before, its rows and
// columns loaded one key after the other. 512 or 768 threads a tile: 28.2 to
// 30.1; 12 keys a thread and 4 blocks an SM: 24.8; __match_any_sync for the
// ballots: 7 % more.
template <bool FIRST, bool W>
__global__ void __launch_bounds__(kRT, kRBlocks) k_radix_scatter(const KeySrc src, int64_t M, int shift,
                                                                 const int64_t* __restrict__ goff, int64_t ntiles,
                                                                 uint64_t* __restrict__ out,
                                                                 float* __restrict__ wout) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* buf = reinterpret_cast<uint64_t*>(smem_raw);          // kRTile keys
  int64_t* gbase = reinterpret_cast<int64_t*>(buf + kRTile);       // kRDigits
  uint32_t* wcnt = reinterpret_cast<uint32_t*>(gbase + kRDigits);  // kRWarps x kRDigits
  uint32_t* wsum = wcnt + kRWarps * kRDigits;                      // kRWarps
  float* wbuf = reinterpret_cast<float*>(wsum + kRWarps);          // kRTile weights (W)
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kRWarps; ++k) wcnt[k * kRDigits + threadIdx.x] = 0;
  const int64_t t0 = (int64_t)blockIdx.x * kRTile;
  const int64_t i0 = t0 + (int64_t)w * (32 * kRK) + lane;
  // rounds r < nv hold a key of this thread
  const int nv = M <= i0 ? 0 : (M - i0 >= 32 * kRK ? kRK : (int)((M - i0 + 31) / 32));
  uint64_t key[kRK];
  if (FIRST && t0 + kRTile <= src.m0) {
#pragma unroll
    for (int r = 0; r < kRK; ++r) key[r] = list_key(src, i0 + r * 32);
  } else if (!FIRST && t0 + kRTile <= M) {
#pragma unroll
    for (int r = 0; r < kRK; ++r) key[r] = load_key<FIRST>(src, i0 + r * 32);
  } else {
#pragma unroll
    for (int r = 0; r < kRK; ++r) key[r] = r < nv ? load_key<FIRST>(src, i0 + r * 32) : 0ull;
  }
  __syncthreads();
  uint32_t* mine = wcnt + w * kRDigits;
  const bool full = t0 + kRTile <= M;
  uint32_t rank[kRK / 2];  // two 16-bit ranks a word (a rank is below kRTile)
  if (full) rank_keys<true>(key, shift, nv, mine, rank);
  else rank_keys<false>(key, shift, nv, mine, rank);
  float wv[W ? kRK : 1];
  if (W) {
    if (full && (!FIRST || t0 + kRTile <= src.m0)) {
#pragma unroll
      for (int r = 0; r < kRK; ++r) wv[W ? r : 0] = __ldcs(src.w + i0 + r * 32);
    } else {
#pragma unroll
      for (int r = 0; r < kRK; ++r) wv[W ? r : 0] = r < nv ? load_w<FIRST>(src, i0 + r * 32) : 0.f;
    }
  }
  __syncthreads();
  // digit d = this thread: its start inside the tile, and from there each
  // warp's (in warp order)
  {
    const int d = threadIdx.x;
    uint32_t all = 0;
#pragma unroll
    for (int k = 0; k < kRWarps; ++k) all += wcnt[k * kRDigits + d];
    uint32_t at = block_scan_excl(all, wsum, nullptr);
    gbase[d] = goff[(int64_t)d * ntiles + blockIdx.x] - (int64_t)at;
#pragma unroll
    for (int k = 0; k < kRWarps; ++k) {
      const uint32_t c = wcnt[k * kRDigits + d];
      wcnt[k * kRDigits + d] = at;
      at += c;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    if (r < nv) {
      const uint32_t d = (uint32_t)(key[r] >> shift) & 0xFFu;
      const uint32_t at = mine[d] + ((rank[r >> 1] >> (16 * (r & 1))) & 0xFFFFu);
      buf[at] = key[r];
      if (W) wbuf[at] = wv[W ? r : 0];
    }
  }
  __syncthreads();
  const int cnt = (int)(M - t0 < kRTile ? M - t0 : kRTile);
  for (int i = threadIdx.x; i < cnt; i += kRT) {
    const uint64_t k = buf[i];
    const int64_t at = gbase[(k >> shift) & 0xFFu] + i;
    __stcs(reinterpret_cast<unsigned long long*>(out) + at, k);
    if (W) __stcs(wout + at, wbuf[i]);
  }
}

constexpr int kRScatterSmem = kRTile * 8 + kRDigits * 8 + kRWarps * kRDigits * 4 + kRWarps * 4;
constexpr int kRScatterSmemW = kRScatterSmem + kRTile * 4;
static_assert(kRScatterSmem <= kDefaultSmem, "launched without raising the limit");

// ---- merge of equal keys ----
// A warp takes 32 * kRK consecutive sorted keys, 32 per round (coalesced);
// key i is new when it differs from key i - 1, which is the lane below in the
// same round, lane 31 of the round before, or the previous warp's last key.

__device__ __forceinline__ bool new_key(int64_t i, uint64_t key, uint64_t& carry, int lane) {
  uint64_t prev = __shfl_up_sync(0xffffffffu, key, 1);
  if (lane == 0) prev = carry;
  carry = __shfl_sync(0xffffffffu, key, 31);
  return i == 0 || key != prev;
}

__device__ __forceinline__ uint64_t warp_carry_in(const uint64_t* __restrict__ k, int64_t i0) {
  return i0 > 0 ? k[i0 - 1] : ~0ull;  // i0: the warp's first key (lane 0)
}

// cnt[warp] = number of new keys among the warp's 32 * kRK
__global__ void __launch_bounds__(kRT) k_uniq_count(const uint64_t* __restrict__ k, int64_t M, uint32_t* __restrict__ cnt) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * kRT + threadIdx.x) >> 5;
  const int64_t base = gw * (32 * kRK);
  uint64_t key[kRK];
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    key[r] = i < M ? __ldcs(reinterpret_cast<const unsigned long long*>(k) + i) : ~0ull;
  }
  uint64_t carry = base < M ? warp_carry_in(k, base) : ~0ull;
  uint32_t c = 0;
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    const bool f = new_key(i, key[r], carry, lane) && i < M;
    c += (uint32_t)__popc(__ballot_sync(0xffffffffu, f));
  }
  if (lane == 0) cnt[gw] = c;
}

// ---- row offsets of long runs of empty rows ----
// The lane of a key writes the offsets of its row and of the empty rows before
// it, runs of fewer than kGapLane rows that is (and those after the last key).
// Longer runs are left to far_gaps, which a warp that saw one calls in the end:
// the warp writes them, or lists those of kGapWarp rows and more for
// k_fill_gaps, the whole GPU's. One lane took 140 ms for the 16 M rows after the
// last used one (1 M edges; the whole build 145.6 ms, 2.0 now).
constexpr int64_t kGapLane = 64;
constexpr int64_t kGapWarp = 1 << 16;
struct Gap {
  int64_t first, last, pos;  // off[first..last] = pos
};
struct Gaps {
  Gap* list;  // room for n / kGapWarp + 1
  unsigned int* count;
};

// the runs at the warp's keys [base, base + 32 * kRK) of k[0..M), the first new one of which has position pos
__device__ __forceinline__ void far_gaps(const uint64_t* __restrict__ k, int64_t M, int B, int32_t n, int64_t base,
                                      int64_t pos, int64_t* __restrict__ off, const Gaps gaps) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = lanemask_lt();
#pragma unroll 1
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    const uint64_t key = i < M ? k[i] : ~0ull, prev = i > 0 && i < M ? k[i - 1] : ~0ull;
    const bool f = i < M && (i == 0 || key != prev);
    const uint32_t bal = __ballot_sync(0xffffffffu, f);
    const int64_t row = (int64_t)(key >> B);
    // the rows before a new key, and those after the last key
#pragma unroll 1
    for (int after = 0; after < 2; ++after) {
      int64_t first = 1, last = 0, at = 0;
      if (after == 0 && f) {
        first = i == 0 ? 0 : (int64_t)(prev >> B) + 1;
        last = row;
        at = pos + __popc(bal & lt);
      } else if (after == 1 && i == M - 1) {
        first = row + 1;
        last = n;
        at = pos + __popc(bal);
      }
      uint32_t todo = __ballot_sync(0xffffffffu, last - first >= kGapLane);
      while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        const Gap g = {__shfl_sync(0xffffffffu, first, l), __shfl_sync(0xffffffffu, last, l),
                       __shfl_sync(0xffffffffu, at, l)};
        if (g.last - g.first >= kGapWarp) {
          if (lane == 0) gaps.list[atomicAdd(gaps.count, 1u)] = g;
        } else {
          for (int64_t q = g.first + lane; q <= g.last; q += 32) off[q] = g.pos;
        }
      }
    }
    pos += __popc(bal);
  }
}

__global__ void k_fill_gaps(const Gaps gaps, int64_t* __restrict__ off) {
  const unsigned int c = *gaps.count;
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (unsigned int k = 0; k < c; ++k) {
    const Gap g = gaps.list[k];
    for (int64_t q = g.first + tid; q <= g.last; q += step) off[q] = g.pos;
  }
}

// Columns of the unique keys, and off[r] = position of row r's first unique
// key (rows without keys take the next row's start; off[n] = total).
// woff = exclusive scan of the per-warp counts, woff[nw] = total. kt (or null)
// gets the keys of the transposed CSR in this CSR's order, uw (or null, zeros
// on entry) the largest weight bits of each unique key: a plain store where the
// key stands alone, an atomic only among duplicates (one per key before, and
// another pass for the weights of added self-loops: 9.5 ms for 64 M weighted
// edges to two CSRs, 8.2 with the scatter's changes). With urow
// (lists much shorter than n) the row of each unique key goes to urow instead
// and k_offsets_from_rows fills off.
__global__ void __launch_bounds__(kRT) k_uniq_emit(const uint64_t* __restrict__ k, int64_t M, int B, int32_t n,
                                                   const int64_t* __restrict__ woff, int64_t nw,
                                                   int32_t* __restrict__ adj, int64_t* __restrict__ off,
                                                   int32_t* __restrict__ urow, const Gaps gaps,
                                                   uint64_t* __restrict__ kt, const float* __restrict__ w,
                                                   uint32_t* __restrict__ uw) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = ((int64_t)blockIdx.x * kRT + threadIdx.x) >> 5;
  const int64_t base = gw * (32 * kRK);
  const uint32_t lt = lanemask_lt();
  const uint64_t cmask = (1ull << B) - 1;
  uint64_t key[kRK];
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    key[r] = i < M ? __ldcs(reinterpret_cast<const unsigned long long*>(k) + i) : ~0ull;
  }
  uint64_t carry = base < M ? warp_carry_in(k, base) : ~0ull;
  uint32_t wv[kRK];
  if (uw) {
#pragma unroll
    for (int r = 0; r < kRK; ++r) {
      const int64_t i = base + r * 32 + lane;
      wv[r] = i < M ? __float_as_uint(__ldcs(w + i)) : 0u;
    }
  }
  const uint64_t after = base + 32 * kRK < M ? k[base + 32 * kRK] : ~0ull;  // the next warp's first key
  int64_t pos = gw < nw ? woff[gw] : 0;
  bool far = false;
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    uint64_t prev = __shfl_up_sync(0xffffffffu, key[r], 1);
    if (lane == 0) prev = carry;
    carry = __shfl_sync(0xffffffffu, key[r], 31);
    const bool f = i < M && (i == 0 || key[r] != prev);
    const uint32_t bal = __ballot_sync(0xffffffffu, f);
    if (uw) {
      // an entry alone has its weight (an added self-loop 1); of duplicates, cleared before, the largest stays
      // (positive floats order as their bits, and the mark of an added self-loop is 0)
      uint64_t next = __shfl_down_sync(0xffffffffu, key[r], 1);
      const uint64_t over = __shfl_sync(0xffffffffu, r + 1 < kRK ? key[r + 1 < kRK ? r + 1 : 0] : after, 0);
      if (lane == 31) next = over;
      uint32_t* to = uw + pos + __popc(bal & lt);
      if (f && key[r] != next) *to = wv[r] ? wv[r] : __float_as_uint(1.f);
      else if (i < M) atomicMax(to - (f ? 0 : 1), wv[r]);
    }
    if (f) {
      const int64_t p = pos + __popc(bal & lt);
      const int64_t row = (int64_t)(key[r] >> B);
      adj[p] = (int32_t)(key[r] & cmask);
      if (kt) kt[p] = (key[r] & cmask) << B | (uint64_t)row;
      if (urow) {
        urow[p] = (int32_t)row;
      } else {
        const int64_t first = i == 0 ? 0 : (int64_t)(prev >> B) + 1;  // rows after the previous key's
        if (row - first < kGapLane)
          for (int64_t q = first; q <= row; ++q) off[q] = p;
        else
          far = true;
      }
    }
    if (!urow && i == M - 1) {
      const int64_t total = woff[nw], first = (int64_t)(key[r] >> B) + 1;
      if (n - first < kGapLane)
        for (int64_t q = first; q <= n; ++q) off[q] = total;
      else
        far = true;
    }
    pos += __popc(bal);
  }
  if (__any_sync(0xffffffffu, far)) far_gaps(k, M, B, n, base, woff[gw], off, gaps);
}

// off[r] = first position whose row is >= r (urow ascending, length mu): one
// binary search per row, for lists much shorter than n
__global__ void k_offsets_from_rows(const int32_t* __restrict__ urow, int64_t mu, int32_t n, int64_t* __restrict__ off) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r <= n; r += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = mu;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (urow[mid] < r) lo = mid + 1; else hi = mid;
    }
    off[r] = lo;
  }
}

// columns and row offsets of sorted keys without duplicates; a warp takes
// 32 * kRK keys, all loaded before the first is written (one key at a time a
// thread before: 0.73 ms for 285 M keys, 4.6 TB/s)
__global__ void __launch_bounds__(kRT) k_emit(const uint64_t* __restrict__ k, int64_t m, int B, int32_t n,
                                              int32_t* __restrict__ adj, int64_t* __restrict__ off, const Gaps gaps) {
  const uint64_t cmask = (1ull << B) - 1;
  const int lane = threadIdx.x & 31;
  const int64_t base = (((int64_t)blockIdx.x * kRT + threadIdx.x) >> 5) * (32 * kRK);
  if (base >= m) return;
  uint64_t key[kRK];
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    key[r] = i < m ? __ldcs(reinterpret_cast<const unsigned long long*>(k) + i) : ~0ull;
  }
  int64_t row = base > 0 ? (int64_t)(k[base - 1] >> B) : -1;  // of the key before the round's first
  bool far = false;
#pragma unroll
  for (int r = 0; r < kRK; ++r) {
    const int64_t i = base + r * 32 + lane;
    const int64_t mine = i < m ? (int64_t)(key[r] >> B) : n;
    int64_t prev = __shfl_up_sync(0xffffffffu, mine, 1);
    if (lane == 0) prev = row;
    row = __shfl_sync(0xffffffffu, mine, 31);
    if (i < m) adj[i] = (int32_t)(key[r] & cmask);
    // rows after the previous key's start here; past the last key (i = m) they are empty and end there
    if (i <= m) {
      if (mine - (prev + 1) < kGapLane)
        for (int64_t q = prev + 1; q <= mine; ++q) off[q] = i;
      else
        far = true;
    }
  }
  if (base + 32 * kRK == m && lane == 31) {  // no lane had i = m
    if (n - (row + 1) < kGapLane)
      for (int64_t q = row + 1; q <= n; ++q) off[q] = m;
    else
      far = true;
  }
  if (__any_sync(0xffffffffu, far)) far_gaps(k, m, B, n, base, base, off, gaps);
}

template <bool FIRST>
int radix_pass(const KeySrc& src, int64_t M, int shift, uint64_t* out, float* wout, DBuf<uint32_t>& hist,
               DBuf<int64_t>& goff, int64_t ntiles, Workspace& ws, cudaStream_t s) {
  k_radix_hist<FIRST><<<(unsigned)ntiles, kRT, 0, s>>>(src, M, shift, hist.p, ntiles);
  PRDF_LAUNCH_CHECK();
  PRDF_TRY(exclusive_scan_u32(hist.p, ntiles * kRDigits, goff.p, ws, s));
  if (wout) {
    // above the default limit, which each device keeps for itself: set before every launch
    PRDF_CUDA(cudaFuncSetAttribute(k_radix_scatter<FIRST, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   kRScatterSmemW));
    k_radix_scatter<FIRST, true><<<(unsigned)ntiles, kRT, kRScatterSmemW, s>>>(src, M, shift, goff.p, ntiles, out, wout);
  } else {
    k_radix_scatter<FIRST, false><<<(unsigned)ntiles, kRT, kRScatterSmem, s>>>(src, M, shift, goff.p, ntiles, out,
                                                                               nullptr);
  }
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

}  // namespace

bool radix_build_applies(int32_t n, int64_t m0, const float* w, bool allow_skip, bool self_loops) {
  const int64_t M = m0 + (self_loops ? n : 0);
  return !w && !allow_skip && M > 0 && M < (1ll << 32);
}

bool radix_pair_applies(int32_t n, int64_t m0, bool self_loops) {
  const int64_t M = m0 + (self_loops ? n : 0);
  return M > 0 && M < (1ll << 32) && M * 16 >= (int64_t)n;
}

namespace {

// The CSR of the list, and with `in` that of its transpose: the first CSR's
// unique entries, in its order, are a list sorted by row, so a stable sort by
// column alone (half the passes) gives the transposed CSR with its rows in
// order.
int build_radix(int32_t n, int64_t m0, const int32_t* rows, const int32_t* cols, const float* w, bool self_loops,
                Csr& out, Csr* in, Workspace& ws, cudaStream_t s) {
  const int64_t M = m0 + (self_loops ? n : 0);
  int B = 1;
  while (B < 31 && ((int64_t)1 << B) < (int64_t)n) ++B;  // ids < n <= 2^B
  const int passes = (2 * B + 7) / 8;
  const int64_t ntiles = (M + kRTile - 1) / kRTile;
  DBuf<uint64_t> ka, kb;
  DBuf<float> wa, wb;
  DBuf<uint32_t> hist;
  DBuf<int64_t> goff;
  PRDF_TRY(ka.alloc((size_t)M, s));
  PRDF_TRY(kb.alloc((size_t)M, s));
  if (w) {
    PRDF_TRY(wa.alloc((size_t)M, s));
    PRDF_TRY(wb.alloc((size_t)M, s));
  }
  PRDF_TRY(hist.alloc((size_t)(ntiles * kRDigits), s));
  PRDF_TRY(goff.alloc((size_t)(ntiles * kRDigits + 1), s));
  KeySrc src;
  src.keys = nullptr;
  src.w = w;
  src.rows = rows;
  src.cols = cols;
  src.m0 = m0;
  src.B = B;
  uint64_t* cur = ka.p;
  uint64_t* nxt = kb.p;
  float* wcur = wa.p;
  float* wnxt = wb.p;
  PRDF_TRY(radix_pass<true>(src, M, 0, cur, wcur, hist, goff, ntiles, ws, s));
  auto swap = [](auto& a, auto& b) {
    auto t = a;
    a = b;
    b = t;
  };
  for (int p = 1; p < passes; ++p) {
    src.keys = cur;
    src.w = wcur;
    PRDF_TRY(radix_pass<false>(src, M, 8 * p, nxt, wnxt, hist, goff, ntiles, ws, s));
    swap(cur, nxt);
    swap(wcur, wnxt);
  }
  // merge equal keys
  const int64_t nw = ntiles * kRWarps;
  DBuf<uint32_t> wcnt;
  DBuf<int64_t> woff;
  PRDF_TRY(wcnt.alloc((size_t)nw, s));
  PRDF_TRY(woff.alloc((size_t)nw + 1, s));
  k_uniq_count<<<(unsigned)ntiles, kRT, 0, s>>>(cur, M, wcnt.p);
  PRDF_LAUNCH_CHECK();
  PRDF_TRY(exclusive_scan_u32(wcnt.p, nw, woff.p, ws, s));
  PRDF_CUDA(cudaMemcpyAsync(ws.host_i64, woff.p + nw, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  PRDF_CUDA(cudaStreamSynchronize(s));
  const int64_t m = ws.host_i64[0];
  const size_t room = (size_t)(m > 0 ? m : 1);
  out.m = m;
  PRDF_TRY(out.off.alloc((size_t)n + 1, s));
  PRDF_TRY(out.adj.alloc(room, s));
  if (w) {
    PRDF_TRY(out.w.alloc(room, s));
    PRDF_CUDA(cudaMemsetAsync(out.w.p, 0, sizeof(float) * (size_t)m, s));
  } else {
    out.w.release();
  }
  // a list much shorter than n leaves long runs of empty rows: their offsets
  // are found row-parallel instead of by the lanes that emit the keys
  const bool sparse = M * 16 < (int64_t)n;
  DBuf<Gap> gap_list;
  DBuf<unsigned int> gap_count;
  PRDF_TRY(gap_list.alloc((size_t)(n / kGapWarp + 1), s));
  PRDF_TRY(gap_count.alloc(1, s));
  const Gaps gaps{gap_list.p, gap_count.p};
  PRDF_CUDA(cudaMemsetAsync(gap_count.p, 0, sizeof(unsigned int), s));
  DBuf<int32_t> urow;
  if (sparse) PRDF_TRY(urow.alloc(room, s));
  k_uniq_emit<<<(unsigned)ntiles, kRT, 0, s>>>(cur, M, B, n, woff.p, nw, out.adj.p, out.off.p,
                                               sparse ? urow.p : nullptr, gaps, in ? nxt : nullptr, wcur,
                                               w ? reinterpret_cast<uint32_t*>(out.w.p) : nullptr);
  if (sparse) k_offsets_from_rows<<<grid_for((int64_t)n + 1, kRT), kRT, 0, s>>>(urow.p, out.m, n, out.off.p);
  else if (n >= kGapWarp) k_fill_gaps<<<grid_for(n, 8 * kRT, kSMs * 8), kRT, 0, s>>>(gaps, out.off.p);
  PRDF_LAUNCH_CHECK();
  if (!in) return PRDF_OK;
  swap(cur, nxt);  // the transposed keys
  in->m = m;
  PRDF_TRY(in->off.alloc((size_t)n + 1, s));
  PRDF_TRY(in->adj.alloc(room, s));
  if (w) PRDF_TRY(in->w.alloc(room, s));
  else in->w.release();
  const int half = (B + 7) / 8;
  for (int p = 0; p < half; ++p) {
    // the weights go from the first CSR's, through the buffers, to the second's
    src.keys = cur;
    src.w = p == 0 ? out.w.p : wcur;
    float* to = p == half - 1 ? in->w.p : wnxt;
    PRDF_TRY(radix_pass<false>(src, m, B + 8 * p, nxt, to, hist, goff, (m + kRTile - 1) / kRTile, ws, s));
    swap(cur, nxt);
    swap(wcur, wnxt);
  }
  PRDF_CUDA(cudaMemsetAsync(gap_count.p, 0, sizeof(unsigned int), s));
  k_emit<<<(unsigned)((m + kRTile - 1) / kRTile), kRT, 0, s>>>(cur, m, B, n, in->adj.p, in->off.p, gaps);
  if (n >= kGapWarp) k_fill_gaps<<<grid_for(n, 8 * kRT, kSMs * 8), kRT, 0, s>>>(gaps, in->off.p);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

}  // namespace

int build_csr_radix(int32_t n, int64_t m0, const int32_t* rows, const int32_t* cols, bool self_loops, Csr& out,
                    Workspace& ws, cudaStream_t s) {
  return build_radix(n, m0, rows, cols, nullptr, self_loops, out, nullptr, ws, s);
}

int build_csr_pair_radix(int32_t n, int64_t m0, const int32_t* rows, const int32_t* cols, const float* w,
                         bool self_loops, Csr& out, Csr& in, Workspace& ws, cudaStream_t s) {
  return build_radix(n, m0, rows, cols, w, self_loops, out, &in, ws, s);
}

}  // namespace prdf
