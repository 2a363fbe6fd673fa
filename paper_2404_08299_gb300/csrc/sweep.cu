// Synchronous, pull-based rank sweeps (Alg. update of arXiv 2404.08299) for
// Static (Eq. 1, every vertex) and DF / DF-P (Eq. 1 / Eq. 2 on the affected
// vertices, with prune and expand flags), the expansion rounds between them
// (Alg. affected), and the loop around both, in FP64 and in FP32.
//
// One persistent kernel runs a whole loop: k_rank_loop is launched
// cooperatively with as many blocks as fit the GPU, every sweep and every
// expansion round is one phase of it, and a grid barrier separates phases.
// Before, each in-degree class of each sweep was a kernel of its own inside a
// CUDA graph (eight launches a sweep, up to eight more an expansion round,
// and a graph to build anew after every batch update).
//
// State: x[u] = R[u] / |out(u)|, so a sweep gathers one value per in-edge.
// The sweeps run on the class-contiguous numbering (relabel.cu): class c is
// the id range [begin, end). A class is cut into units of rows that warps
// fetch from a counter, long rows first, so that the tail of one class is
// filled with the work of the next. A unit goes through batches of 32 rows
// (the affected ones only, in DF / DF-P): groups of G lanes (G = 4, 8, 16, 32
// by class) sum the batch's rows one after the other, each group keeping the
// sum of its s-th row in its s-th lane, and the epilogue then runs once with
// a row in every lane. The epilogue costs some hundred instructions, FP64
// ones among them (which GB300 issues at about 1.6 a clock per SM whatever
// the number of active lanes), so it is shared by 32 rows instead of running
// in one lane per row.
//
// The L-inf change of the sweep is reduced per block and with one atomic max
// per block on the bit pattern of a non-negative value; rank writes stay one
// plain store per vertex.
#include <cstring>

#include "internal.cuh"

namespace prdf {

namespace {

// Two blocks of 512 threads per SM at 64 registers: the sweeps are bound by
// the latency and the rate of their gathers, so resident warps matter more
// than registers, and few blocks keep the grid barrier short.
constexpr int kThreads = 512;
constexpr int kMinBlocks = 2;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxWords = 8;  // a unit holds at most 8 x 32 rows

// ------------------------------------------------------ precision traits ----

// gathered state: coherent loads (the buffers are written in the same kernel,
// a grid barrier earlier), kept in L2 (evict-last)
__device__ __forceinline__ uint64_t ld_state(const double* p, uint64_t pol) {
  uint64_t v;
  asm volatile("ld.global.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ uint32_t ld_state(const float* p, uint64_t pol) {
  uint32_t v;
  asm volatile("ld.global.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ float ld_const(const float* p, uint64_t pol) {
  float v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
  return v;
}

// Exact accumulator (4 x 32-bit words, 2^-124 resolution).
struct AccExact {
  Fix4 v;
  __device__ __forceinline__ void add(uint64_t xb) { v.add(xb); }
  // add_w1: only for terms with in_w1 (the common window, three-word add)
  __device__ __forceinline__ static bool in_w1(uint64_t xb) { return Fix4::in_w1(xb); }
  __device__ __forceinline__ void add_w1(uint64_t xb) { v.add_w1(xb); }
  template <int G>
  __device__ __forceinline__ void group_reduce() { v.template group_reduce<G>(); }
  __device__ __forceinline__ double value() const { return v.to_double(); }
  __device__ __forceinline__ uint4 pack() const { return make_uint4(v.w0, v.w1, v.w2, v.w3); }
  __device__ __forceinline__ void merge(const uint4& p) { v.add4(p.x, p.y, p.z, p.w); }
};

// plain FP64 additions
struct AccPlain {
  double v = 0;
  __device__ __forceinline__ void add(uint64_t xb) { v += bitsd(xb); }
  __device__ __forceinline__ static bool in_w1(uint64_t) { return true; }
  __device__ __forceinline__ void add_w1(uint64_t xb) { v += bitsd(xb); }
  template <int G>
  __device__ __forceinline__ void group_reduce() {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  }
  __device__ __forceinline__ double value() const { return v; }
  __device__ __forceinline__ uint4 pack() const {
    const uint64_t b = dbits(v);
    return make_uint4((uint32_t)b, (uint32_t)(b >> 32), 0u, 0u);
  }
  __device__ __forceinline__ void merge(const uint4& p) { v += bitsd(((uint64_t)p.y << 32) | p.x); }
};

// FP32 sum compensated by Kahan-Babuska (TwoSum of every term, errors summed
// separately): value = s + e
struct AccKahan {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void addf(float y) {
    const float t = s + y;
    const float bp = t - s;
    e += (s - (t - bp)) + (y - bp);
    s = t;
  }
  __device__ __forceinline__ void add(uint32_t b) { addf(__uint_as_float(b)); }
  __device__ __forceinline__ static bool in_w1(uint32_t) { return true; }
  __device__ __forceinline__ void add_w1(uint32_t b) { addf(__uint_as_float(b)); }
  __device__ __forceinline__ void merge2(float s2, float e2) {
    addf(s2);
    e += e2;
  }
  template <int G>
  __device__ __forceinline__ void group_reduce() {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const float s2 = __shfl_xor_sync(kFull, s, o);
      const float e2 = __shfl_xor_sync(kFull, e, o);
      merge2(s2, e2);
    }
  }
  __device__ __forceinline__ float value() const { return s + e; }
  __device__ __forceinline__ uint4 pack() const {
    return make_uint4(__float_as_uint(s), __float_as_uint(e), 0u, 0u);
  }
  __device__ __forceinline__ void merge(const uint4& p) { merge2(__uint_as_float(p.x), __uint_as_float(p.y)); }
};

template <class A>
struct Prec64 {
  using Real = double;
  using Bits = uint64_t;
  using Acc = A;
};
using PExact = Prec64<AccExact>;
using PPlain = Prec64<AccPlain>;
struct PKahan {
  using Real = float;
  using Bits = uint32_t;
  using Acc = AccKahan;
};

// Exact integer value of an out-degree held as a double (an integer below
// 2^53), decoded from its bit pattern on the integer pipes; 0 for 0.
__device__ __forceinline__ uint64_t degree_of(double d) {
  const uint64_t b = dbits(d);
  const int e = (int)(b >> 52) - 1023;
  const uint64_t mant = (b & 0x000FFFFFFFFFFFFFull) | (1ull << 52);
  return e >= 0 ? mant >> (52 - e) : 0ull;
}
__device__ __forceinline__ uint64_t degree_of(float d) { return (uint64_t)d; }

// What a warp carries through a sweep: largest |r - R[v]|, (FP32) largest r,
// out-edges put into deltaN, affected vertices seen.
struct Tally {
  uint64_t dmax = 0;
  uint32_t rmax = 0;
  uint64_t fw = 0;
  unsigned int aff = 0;
};

// ---------------------------------------------------------- per sweep ----
template <class P>
struct Ctx {
  const typename P::Real* x;
  typename P::Real* xn;
  LoopSlot* slot;  // this sweep's
  uint64_t pf, pl;
  int lane;
};

// Frontier entries of one vertex: one per kFrontChunk out-edges.
__device__ __forceinline__ unsigned int front_entries(uint64_t deg) {
  return (unsigned int)((deg + kFrontChunk - 1) / kFrontChunk);
}

// The lanes with flag set append their vertices to the frontier list (all
// lanes call it): warp-aggregated, one entry per kFrontChunk out-edges.
__device__ __forceinline__ void append_frontier(bool flag, int32_t v, uint64_t deg, unsigned int* count, int2* list,
                                                int lane) {
  if (!__any_sync(kFull, flag)) return;
  const unsigned int c = flag ? front_entries(deg) : 0u;
  unsigned int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  unsigned int base = 0;
  if (lane == 31) base = atomicAdd(count, incl);
  base = __shfl_sync(kFull, base, 31) + incl - c;
  for (unsigned int k = 0; k < c; ++k) list[base + k] = make_int2(v, (int)k);
}

// Vertex epilogue: Eq. 1 (Static, DF) or Eq. 2 (DF-P), prune / expand flags,
// next x, and this vertex's |r - R[v]| into the tally. GB300's FP64 pipe is
// narrow, so the FP64 form keeps to what needs FP64 rounding; the maximum and
// the comparisons run on the bit patterns of the non-negative doubles
// (integer instructions, the same order as the FP64 comparison; a negative
// threshold's pattern is negative as int64, so it orders below every
// non-negative value, as in FP64). Returns whether v joins deltaN.
template <bool DYN>
__device__ __forceinline__ bool finish(const SweepArgs<double>& a, const Ctx<PExact>& c, int32_t v, double sum,
                                       double xself, bool dn_old, Tally& t, uint64_t& deg) {
  const double d = ld_stream_f64(a.deg + v, c.pf);
  const double iv = ld_stream_f64(a.inv + v, c.pf);
  double r;
  if (DYN && a.prune) {
    // Eq. 2: the self-loop term is solved in closed form (factor precomputed per vertex)
    r = ld_stream_f64(a.kf + v, c.pf) * (a.c0 + a.alpha * (sum - xself));
  } else {
    r = fma(a.alpha, sum, a.c0);  // Eq. 1
  }
  // |r - R[v]| with R[v] = x[v] * |out(v)| of the previous iteration, one rounding
  const double dr = fabs(fma(xself, -d, r));
  bool front = false;
  if (DYN) {
    const uint64_t rb = dbits(r), ob = dbits(xself * d), drb = dbits(dr);
    const double m = bitsd(rb > ob ? rb : ob);  // max(r, R[v])
    const int64_t tp = (int64_t)dbits(a.tau_p * m);
    const int64_t tf = a.tau_f == a.tau_p ? tp : (int64_t)dbits(a.tau_f * m);
    if (a.prune && (int64_t)drb <= tp) a.dV[v] = 0;
    // deltaN holds exactly this sweep's expand set: set or cleared for every vertex
    front = (int64_t)drb > tf;
    if (front != dn_old) a.dN[v] = front ? 1 : 0;
    if (front) {
      deg = degree_of(d);
      t.fw += deg;
    }
    a.wrote[v] = 1;
  }
  c.xn[v] = r * iv;
  const uint64_t db = dbits(dr);
  t.dmax = db > t.dmax ? db : t.dmax;
  return front;
}
template <bool DYN>
__device__ __forceinline__ bool finish(const SweepArgs<double>& a, const Ctx<PPlain>& c, int32_t v, double sum,
                                       double xself, bool dn_old, Tally& t, uint64_t& deg) {
  const Ctx<PExact> e{c.x, c.xn, c.slot, c.pf, c.pl, c.lane};
  return finish<DYN>(a, e, v, sum, xself, dn_old, t, deg);
}
// the same in FP32, with Alg. update's prune and expand tests evaluated in FP32
template <bool DYN>
__device__ __forceinline__ bool finish(const SweepArgs<float>& a, const Ctx<PKahan>& c, int32_t v, float sum,
                                       float xself, bool dn_old, Tally& t, uint64_t& deg) {
  const float d = ld_const(a.deg + v, c.pf);
  const float iv = ld_const(a.inv + v, c.pf);
  const float rold = xself * d;
  float r;
  if (DYN && a.prune) r = ld_const(a.kf + v, c.pf) * fmaf(a.alpha, sum - xself, a.c0);  // Eq. 2
  else r = fmaf(a.alpha, sum, a.c0);                                                      // Eq. 1
  const float dr = fabsf(r - rold);
  bool front = false;
  if (DYN) {
    const float m = fmaxf(r, rold);
    if (a.prune && dr <= a.tau_p * m) a.dV[v] = 0;
    front = dr > a.tau_f * m;
    if (front != dn_old) a.dN[v] = front ? 1 : 0;
    if (front) {
      deg = degree_of(d);
      t.fw += deg;
    }
    a.wrote[v] = 1;
  }
  c.xn[v] = r * iv;
  const uint32_t db = __float_as_uint(dr), rb = __float_as_uint(r);
  t.dmax = db > (uint32_t)t.dmax ? db : t.dmax;
  t.rmax = rb > t.rmax ? rb : t.rmax;
  return front;
}

__device__ __forceinline__ double as_real(uint64_t b) { return bitsd(b); }
__device__ __forceinline__ float as_real(uint32_t b) { return __uint_as_float(b); }

// DF / DF-P: an unaffected vertex keeps its rank; its slot in xn is stale
// only if the previous sweep wrote it (then copy it through). It is not in
// this sweep's expand set, so its deltaN flag is cleared (the sweep keeps
// deltaN exact without a separate clearing pass).
template <class P>
__device__ __forceinline__ void skip_vertex(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int32_t v, bool wr,
                                            bool dn) {
  if (wr) {
    c.xn[v] = as_real(ld_state(c.x + v, c.pl));
    a.wrote[v] = 0;
  }
  if (dn) a.dN[v] = 0;
}

// The rows of one unit, [vb, ve) with at most 256 rows. Static: all of them.
// DF / DF-P: the affected ones, compacted over the whole unit (the flags of
// 256 rows are read at once, a bit mask per 32 rows is kept in the lanes), so
// that a batch is 32 affected rows however thinly they are spread; the others
// are copied through.
template <class P, bool DYN>
struct UnitRows {
  int64_t vb;
  int nact;
  uint32_t mdv, mdn;  // lane i: affected / deltaN bits of rows vb + 32 i ..
  int excl;           // lane i: affected rows before word i

  __device__ __forceinline__ UnitRows(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t vb_, int64_t ve,
                                      Tally& t)
      : vb(vb_), mdv(0), mdn(0), excl(0) {
    if (!DYN) {
      nact = (int)(ve - vb);
      return;
    }
    uint32_t mwr = 0;
    uint8_t dv[kMaxWords], wr[kMaxWords], dn[kMaxWords];
#pragma unroll
    for (int i = 0; i < kMaxWords; ++i) {
      const int64_t v = vb + 32 * i + c.lane;
      const bool in = v < ve;
      dv[i] = in ? a.dV[v] : (uint8_t)0;
      wr[i] = in ? a.wrote[v] : (uint8_t)0;
      dn[i] = in ? a.dN[v] : (uint8_t)0;
    }
#pragma unroll
    for (int i = 0; i < kMaxWords; ++i) {
      const uint32_t b0 = __ballot_sync(kFull, dv[i] != 0), b1 = __ballot_sync(kFull, wr[i] != 0),
                     b2 = __ballot_sync(kFull, dn[i] != 0);
      if (c.lane == i) {
        mdv = b0;
        mwr = b1;
        mdn = b2;
      }
    }
    // unaffected rows with something to undo
    uint32_t todo = __ballot_sync(kFull, ((mwr | mdn) & ~mdv) != 0);
    while (todo) {
      const int i = __ffs(todo) - 1;
      todo &= todo - 1;
      const uint32_t w = __shfl_sync(kFull, mwr & ~mdv, i), d = __shfl_sync(kFull, mdn & ~mdv, i);
      const bool bw = (w >> c.lane) & 1u, bd = (d >> c.lane) & 1u;
      if (bw || bd) skip_vertex(a, c, (int32_t)(vb + 32 * i + c.lane), bw, bd);
    }
    const int cnt = __popc(mdv);
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < kMaxWords; o <<= 1) {
      const int u = __shfl_up_sync(kFull, incl, o);
      if (c.lane >= o) incl += u;
    }
    excl = incl - cnt;
    nact = __shfl_sync(kFull, incl, kMaxWords - 1);
    if (c.lane == 0) t.aff += (unsigned int)nact;
  }

  // the k-th row (0 <= k < nact; any k on lanes that hold no row) and its deltaN flag
  __device__ __forceinline__ int32_t row(int k, bool& dn) const {
    if (!DYN) {
      dn = false;
      return (int32_t)(vb + k);
    }
    int w = 0, before = 0;
#pragma unroll
    for (int i = 1; i < kMaxWords; ++i) {
      const int e = __shfl_sync(kFull, excl, i);
      if (e <= k) {
        w = i;
        before = e;
      }
    }
    const uint32_t m = __shfl_sync(kFull, mdv, w);
    const uint32_t d = __shfl_sync(kFull, mdn, w);
    int r = k - before;  // the r-th set bit of m
    int pos = 0;
#pragma unroll
    for (int half = 16; half > 0; half >>= 1) {
      const int low = __popc((m >> pos) & ((1u << half) - 1u));
      if (r >= low) {
        r -= low;
        pos += half;
      }
    }
    dn = (d >> pos) & 1u;
    return (int32_t)(vb + 32 * w + pos);
  }
};

// One row per lane, its offsets known: the epilogue of a batch.
template <class P, bool DYN>
__device__ __forceinline__ void finish_batch(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, bool have,
                                             int32_t v, typename P::Real sum, typename P::Real xself, bool dn,
                                             Tally& t) {
  bool front = false;
  uint64_t deg = 0;
  if (have) front = finish<DYN>(a, c, v, sum, xself, dn, t, deg);
  if (DYN && a.expand) append_frontier(front, v, deg, &c.slot->nlist, a.list, c.lane);
}

// Sum of the gathered terms of one step into acc: one vote picks the
// three-word add when every gathered term of the warp's step is in the common
// window.
template <class P, int U>
__device__ __forceinline__ void add_terms(typename P::Acc& acc, const int32_t (&u)[U],
                                          const typename P::Bits (&xv)[U]) {
  bool w1 = true;
#pragma unroll
  for (int k = 0; k < U; ++k) w1 = w1 && (u[k] < 0 || P::Acc::in_w1(xv[k]));
  if (__all_sync(kFull, w1)) {
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (u[k] >= 0) acc.add_w1(xv[k]);
  } else {
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (u[k] >= 0) acc.add(xv[k]);
  }
}

// Four entries of a row, positions j .. j + 3 (a multiple of four) of the
// sequence at base (16-byte aligned), those outside [lo, hi) masked by -1.
__device__ __forceinline__ int4 load4(const int32_t* base, int j, int hi, uint64_t pf) {
  return j < hi ? ld_stream_i32x4(base + j, pf) : make_int4(-1, -1, -1, -1);
}
__device__ __forceinline__ void mask4(const int4& q, int j, int lo, int hi, int32_t (&u)[4]) {
  u[0] = (j + 0 >= lo && j + 0 < hi) ? q.x : -1;
  u[1] = (j + 1 >= lo && j + 1 < hi) ? q.y : -1;
  u[2] = (j + 2 >= lo && j + 2 < hi) ? q.z : -1;
  u[3] = (j + 3 >= lo && j + 3 < hi) ? q.w : -1;
}

// G lanes per row, a 16-byte index load each per step. The row's entries are
// read from the 16-byte boundary below its first one (positions in a row are
// 32-bit, counted from that boundary). While the gathers of one step are in
// flight the indices of the next step load: the next chunk of the same rows,
// or the first chunk of the groups' next rows, whose offsets are already in
// the lanes, so a step waits for one round trip. The offsets of the next
// batch load before the batch.
template <class P, int G, bool DYN>
__device__ __forceinline__ void unit_group(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t vb,
                                           int64_t ve, Tally& t) {
  using Bits = typename P::Bits;
  constexpr int NG = 32 / G;
  const int lane = c.lane, sub = lane & (G - 1), src0 = lane & ~(G - 1);
  const UnitRows<P, DYN> rows(a, c, vb, ve, t);
  const int nact = rows.nact;
  if (nact == 0) return;

  // lane's row of the batch at k0: group g takes rows g * S .. g * S + S - 1
  struct Batch {
    int32_t v;  // row, its deltaN flag in the sign bit
    int len;
    int64_t b;
  };
  auto steps = [&](int k0) { return ((nact - k0 < 32 ? nact - k0 : 32) + NG - 1) / NG; };
  auto in_batch = [&](int k0) {
    const int S = steps(k0);
    return sub < S && (lane / G) * S + sub < (nact - k0 < 32 ? nact - k0 : 32);
  };
  auto load_batch = [&](int k0) {
    Batch r;
    const bool have = in_batch(k0);
    bool dn;
    const int32_t v = rows.row(have ? k0 + (lane / G) * steps(k0) + sub : 0, dn);
    r.v = dn ? (v | INT32_MIN) : v;
    r.b = 0;
    r.len = 0;
    if (have) {
      r.b = ld_stream_i64(a.off + v, c.pf);
      r.len = (int)(ld_stream_i64(a.off + v + 1, c.pf) - r.b);
    }
    return r;
  };

  Batch cur = load_batch(0);
  for (int k0 = 0; k0 < nact; k0 += 32) {
    Batch nxt = cur;
    if (k0 + 32 < nact) nxt = load_batch(k0 + 32);
    const int S = steps(k0);
    typename P::Acc saved, acc;
    bool hit = false, myhit = false;
    // the group's row: entries [lo, hi) from base; this lane's position j
    int64_t rb = __shfl_sync(kFull, cur.b, src0);
    int lo = (int)(rb & 3), hi = lo + __shfl_sync(kFull, cur.len, src0), j = 4 * sub;
    const int32_t* base = a.adj + (rb & ~(int64_t)3);
    int4 q = load4(base, j, hi, c.pf);
    for (int s = 0; s < S;) {
      int32_t u[4];
      mask4(q, j, lo, hi, u);
      Bits xv[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) xv[k] = u[k] >= 0 ? ld_state(c.x + u[k], c.pl) : Bits(0);
      // the next step's indices
      const bool more = __any_sync(kFull, j - 4 * sub + 4 * G < hi);
      if (more) {
        j += 4 * G;
        lo = 0;
      } else {
        const int src = src0 + s + 1;  // (past the last row: any lane, no entries)
        rb = __shfl_sync(kFull, cur.b, src & 31);
        const int len = __shfl_sync(kFull, cur.len, src & 31);
        lo = (int)(rb & 3);
        hi = s + 1 < S ? lo + len : 0;
        j = 4 * sub;
        base = a.adj + (rb & ~(int64_t)3);
      }
      q = load4(base, j, hi, c.pf);
      if (G < 32 && !a.self_loops) {
        const int32_t rv = __shfl_sync(kFull, cur.v, src0 + s) & INT32_MAX;
#pragma unroll
        for (int k = 0; k < 4; ++k) myhit = myhit || u[k] == rv;
      }
      add_terms<P>(acc, u, xv);
      if (!more) {
        acc.template group_reduce<G>();
        if (sub == s) saved = acc;
        acc = typename P::Acc();
        if (G < 32 && !a.self_loops) {
          // graphs without self-loops on every vertex: x[v] counts only when the row holds v
          const uint32_t m = __ballot_sync(kFull, myhit) >> src0;
          if (sub == s) hit = (m & ((1u << (G & 31)) - 1u)) != 0;
          myhit = false;
        }
        ++s;
      }
    }
    const bool have = in_batch(k0);
    const int32_t v = cur.v & INT32_MAX;
    const Bits xs = have && (G == 32 || a.self_loops || hit) ? ld_state(c.x + v, c.pl) : Bits(0);
    finish_batch<P, DYN>(a, c, have, v, saved.value(), as_real(xs), cur.v < 0, t);
    cur = nxt;
  }
}

// One row per lane, U indices in flight (short rows).
template <class P, int U, bool DYN>
__device__ __forceinline__ void unit_thread(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t vb, int64_t ve,
                                         Tally& t) {
  using Bits = typename P::Bits;
  const UnitRows<P, DYN> rows(a, c, vb, ve, t);
  const int nact = rows.nact;
  if (nact == 0) return;
  struct Row {
    int32_t v;
    int len;
    int64_t b;
    bool have, dn;
  };
  auto load_row = [&](int k0) {
    Row r;
    r.have = k0 + c.lane < nact;
    r.v = rows.row(r.have ? k0 + c.lane : 0, r.dn);
    r.b = 0;
    r.len = 0;
    if (r.have) {
      r.b = ld_stream_i64(a.off + r.v, c.pf);
      r.len = (int)(ld_stream_i64(a.off + r.v + 1, c.pf) - r.b);
    }
    return r;
  };
  auto load_idx = [&](const Row& r, int32_t (&u)[U]) {
#pragma unroll
    for (int k = 0; k < U; ++k) u[k] = k < r.len ? ld_stream_i32(a.adj + r.b + k, c.pf) : -1;
  };
  // offsets two batches ahead, indices one ahead
  Row cur = load_row(0), nxt;
  int32_t u[U];
  load_idx(cur, u);
  nxt.have = false;
  nxt.len = 0;
  nxt.b = 0;
  nxt.v = 0;
  nxt.dn = false;
  if (32 < nact) nxt = load_row(32);
  for (int k0 = 0; k0 < nact; k0 += 32) {
    Bits xv[U];
#pragma unroll
    for (int k = 0; k < U; ++k) xv[k] = u[k] >= 0 ? ld_state(c.x + u[k], c.pl) : Bits(0);
    const Bits xs = cur.have ? ld_state(c.x + cur.v, c.pl) : Bits(0);
    int32_t un[U];
    load_idx(nxt, un);
    Row far = nxt;
    far.have = false;
    far.len = 0;
    if (k0 + 64 < nact) far = load_row(k0 + 64);
    typename P::Acc acc;
    bool hit = false;
#pragma unroll
    for (int k = 0; k < U; ++k) hit = hit || u[k] == cur.v;
    add_terms<P>(acc, u, xv);
    // rest of a row longer than U (rows that grew past their class's bound in a batch update)
    for (int j = U; j < cur.len; ++j) {
      const int32_t w = ld_stream_i32(a.adj + cur.b + j, c.pf);
      acc.add(ld_state(c.x + w, c.pl));
      hit = hit || w == cur.v;
    }
    const Bits xself = (a.self_loops || hit) ? xs : Bits(0);
    finish_batch<P, DYN>(a, c, cur.have, cur.v, acc.value(), as_real(xself), cur.dn, t);
    cur = nxt;
    nxt = far;
#pragma unroll
    for (int k = 0; k < U; ++k) u[k] = un[k];
  }
}

// The class of in-degree <= 1 on a graph with all self-loops: the row is [v],
// so the in-neighbour sum is the single term x[v], exactly, and no offsets or
// indices are read (a vertex that gained in-edges in a batch update has its
// bit in multi and reads its row).
template <class P, bool DYN>
__device__ __forceinline__ void unit_self(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t vb, int64_t ve,
                                       Tally& t) {
  using Bits = typename P::Bits;
  const UnitRows<P, DYN> rows(a, c, vb, ve, t);
  const int nact = rows.nact;
  for (int k0 = 0; k0 < nact; k0 += 32) {
    const bool have = k0 + c.lane < nact;
    bool dn;
    const int32_t v = rows.row(have ? k0 + c.lane : 0, dn);
    const Bits xs = have ? ld_state(c.x + v, c.pl) : Bits(0);
    typename P::Real sum = as_real(xs);
    if (a.multi && have && ((a.multi[v >> 5] >> (v & 31)) & 1u)) {
      typename P::Acc acc;
      const int64_t e = a.off[v + 1];
      for (int64_t j = a.off[v]; j < e; ++j) acc.add(ld_state(c.x + a.adj[j], c.pl));
      sum = acc.value();
    }
    finish_batch<P, DYN>(a, c, have, v, sum, as_real(xs), dn, t);
  }
}

// One 1024-edge chunk of a row of the highest in-degree class. The warp that
// finishes the last chunk of a row adds the row's partial sums and finishes
// the vertex. With exact accumulation the partials are integers, so the
// result is the same bits as any other split; the compensated FP32 partials
// are added in chunk order by lanes and a fixed shuffle tree, so every run
// gives the same bits. A hub's flags change only in its finishing warp, which
// runs after every chunk's warp has read them, or (unaffected hubs) in the
// warp of its first chunk, which leaves dV alone.
template <class P, bool DYN>
__device__ __forceinline__ void unit_hub(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t ch, Tally& t) {
  using Bits = typename P::Bits;
  const int lane = c.lane;
  const int64_t h = a.hub.chunk_hub[ch];
  const int32_t v = (int32_t)(a.hub.begin + h);
  const int64_t jb = a.hub.chunk_j0[ch];
  const int64_t first = a.hub.hub_first[h], last = a.hub.hub_first[h + 1];
  if (DYN) {
    const bool skip = __shfl_sync(kFull, lane == 0 ? (int)(a.dV[v] == 0) : 0, 0) != 0;
    if (skip) {
      if (ch == first && lane == 0) skip_vertex(a, c, v, a.wrote[v] != 0, a.dN[v] != 0);
      return;
    }
    if (ch == first && lane == 0) t.aff += 1;
  }
  const int64_t row_e = a.off[v + 1];
  const int64_t je = jb + kHubChunk < row_e ? jb + kHubChunk : row_e;
  typename P::Acc acc;
  const int lo0 = (int)(jb & 3), hi = lo0 + (int)(je - jb);
  const int32_t* base = a.adj + (jb & ~(int64_t)3);
  int4 q = load4(base, 4 * lane, hi, c.pf);
  for (int j = 4 * lane; j - 4 * lane < hi; j += 128) {
    int32_t u[4];
    mask4(q, j, lo0, hi, u);
    Bits xv[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) xv[k] = u[k] >= 0 ? ld_state(c.x + u[k], c.pl) : Bits(0);
    q = load4(base, j + 128, hi, c.pf);
    add_terms<P>(acc, u, xv);
  }
  acc.template group_reduce<32>();
  unsigned int done = 0;
  if (last - first > 1) {
    if (lane == 0) {
      __stcg(a.hub_part + ch, acc.pack());
      __threadfence();
      done = atomicAdd(a.hub_done + h, 1u) + 1;
    }
    done = __shfl_sync(kFull, done, 0);
    if (done != (unsigned int)(last - first)) return;
    if (lane == 0) a.hub_done[h] = 0;
    __threadfence();
    acc = typename P::Acc();
    for (int64_t k = first + lane; k < last; k += 32) acc.merge(__ldcg(a.hub_part + k));
    acc.template group_reduce<32>();
  }
  const bool have = lane == 0;
  const Bits xs = have ? ld_state(c.x + v, c.pl) : Bits(0);
  finish_batch<P, DYN>(a, c, have, v, acc.value(), as_real(xs), DYN && have && a.dN[v] != 0, t);
}

// -------------------------------------------------------------- phases ----

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

// Barrier over the whole (co-resident) grid: every block adds one arrival and
// waits until all of this barrier's are in. The wait is bounded: past the
// limit (minutes; no sweep takes that long) the block flags the loop as timed
// out and gives up, and so does every other block when it sees the flag.
// Returns false after a timeout.
constexpr unsigned long long kSpinLimit = 1ull << 28;

__device__ bool grid_barrier(LoopCtl* ctl, unsigned long long& target) {
  __shared__ int s_ok;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&ctl->bar, 1ull);
    int ok = 1;
    unsigned long long spins = 0;
    while (ld_acquire(&ctl->bar) < target) {
      if (++spins > kSpinLimit || ((spins & 1023) == 0 && *(volatile int*)&ctl->timeout)) {
        *(volatile int*)&ctl->timeout = 1;
        ok = 0;
        break;
      }
      if (spins > 256) __nanosleep(100);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// the slot of sweep it: a ring of kLoopRing in the whole-loop kernel, one a
// sweep from it_first on in the host-driven loop (slot 0: the sweep before)
template <class Real>
__device__ __forceinline__ LoopSlot* slot_of(const SweepArgs<Real>& a, int it) {
  return a.slot + (a.mode == kLoopAll ? (it & (kLoopRing - 1)) : it - a.it_first + 1);
}

template <class P, bool DYN>
__device__ __forceinline__ void sweep(const SweepArgs<typename P::Real>& a, int it) {
  Ctx<P> c;
  c.x = (it & 1) ? a.xb : a.xa;
  c.xn = (it & 1) ? a.xa : a.xb;
  c.slot = slot_of(a, it);
  c.pf = policy_evict_first();
  c.pl = policy_evict_last();
  c.lane = threadIdx.x & 31;
  Tally t;
  // first unit by position (consecutive units on different SMs), the rest from the counter
  const unsigned int nw = gridDim.x * kWarps;
  unsigned int u = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  while (u < a.units) {
    unsigned int nx = 0;
    if (c.lane == 0) nx = atomicAdd(&c.slot->units, 1u);
    if (u < (unsigned int)a.hub.nchunk) {
      unit_hub<P, DYN>(a, c, u, t);
    } else {
      int k = 0;
      while (k + 1 < a.ncls && u >= a.cls[k + 1].unit0) ++k;
      const SweepClass& cl = a.cls[k];
      const int64_t vb = cl.begin + (int64_t)(u - cl.unit0) * cl.rows;
      const int64_t ve = vb + cl.rows < cl.end ? vb + cl.rows : cl.end;
      switch (cl.kind) {
        case kRowSelf: unit_self<P, DYN>(a, c, vb, ve, t); break;
        case kRowThread: unit_thread<P, 4, DYN>(a, c, vb, ve, t); break;
        case kRow4: unit_group<P, 4, DYN>(a, c, vb, ve, t); break;
        case kRow8: unit_group<P, 8, DYN>(a, c, vb, ve, t); break;
        case kRow16: unit_group<P, 16, DYN>(a, c, vb, ve, t); break;
        default: unit_group<P, 32, DYN>(a, c, vb, ve, t); break;
      }
    }
    u = nw + __shfl_sync(kFull, nx, 0);
  }
  // block maxima and sums
  __shared__ unsigned long long s_max, s_fw;
  __shared__ unsigned int s_r, s_aff;
  if (threadIdx.x == 0) {
    s_max = 0;
    s_fw = 0;
    s_r = 0;
    s_aff = 0;
  }
  __syncthreads();
  const uint64_t dm = warp_max_u64(t.dmax);
  if (c.lane == 0 && dm) atomicMax(&s_max, (unsigned long long)dm);
  if (sizeof(typename P::Real) == 4) {
    const uint32_t rm = __reduce_max_sync(kFull, t.rmax);
    if (c.lane == 0 && rm) atomicMax(&s_r, rm);
  }
  if (DYN) {
    const uint64_t f = (uint64_t)warp_sum_i64((int64_t)t.fw);
    if (c.lane == 0 && f) atomicAdd(&s_fw, (unsigned long long)f);
    if (c.lane == 0 && t.aff) atomicAdd(&s_aff, t.aff);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sizeof(typename P::Real) == 8) {
      if (s_max) atomicMax(&c.slot->resid, s_max);
    } else {
      uint32_t* r = reinterpret_cast<uint32_t*>(&c.slot->resid);
      if (s_max) atomicMax(r, (uint32_t)s_max);
      if (s_r) atomicMax(r + 1, s_r);
    }
    if (DYN && s_fw) atomicAdd(&c.slot->fw, s_fw);
    if (DYN && it == 0 && s_aff) atomicAdd(&a.ctl->aff0, s_aff);
  }
}

// stop rule on a sweep's residual word: FP64, L-inf change <= tol; FP32, max|dR| <= tol * max R
__device__ __forceinline__ bool stopped(unsigned long long resid, double tol) { return bitsd(resid) <= tol; }
__device__ __forceinline__ bool stopped(unsigned long long resid, float tol) {
  return __uint_as_float((uint32_t)resid) <= tol * __uint_as_float((uint32_t)(resid >> 32));
}

// Push form of an expansion round from the frontier list the sweep (or the
// initial marking) left: dV[w] = 1 for every out-neighbour w. A warp takes up
// to 32 entries and walks their edges as one sequence, so short rows share a
// step; a long row is several entries (kFrontChunk edges each) on different
// warps. A flag already set is not stored again.
template <class Real>
__device__ void push_round(const SweepArgs<Real>& a, const unsigned int* count) {
  const int lane = threadIdx.x & 31;
  const unsigned int total = __ldcg(count);
  const unsigned int nw = gridDim.x * kWarps;
  const unsigned int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const unsigned int per = (total + nw - 1) / nw;
  const unsigned int epw = per < 1 ? 1 : (per > 32 ? 32 : per);
  for (unsigned int base = w * epw; base < total; base += nw * epw) {
    int64_t b = 0;
    unsigned int len = 0;
    if ((unsigned int)lane < epw && base + lane < total) {
      const int2 en = __ldcg(a.list + base + lane);
      const int64_t rb = a.ooff[en.x] + (int64_t)en.y * kFrontChunk, re = a.ooff[en.x + 1];
      b = rb;
      len = (unsigned int)(re - rb < kFrontChunk ? re - rb : kFrontChunk);
    }
    unsigned int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int x = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += x;
    }
    const unsigned int excl = incl - len;
    const unsigned int edges = __shfl_sync(kFull, incl, 31);
    constexpr int kU = 4;
    for (unsigned int e0 = 0; e0 < edges; e0 += 32 * kU) {
      int32_t t[kU];
#pragma unroll
      for (int k = 0; k < kU; ++k) {
        const unsigned int e = e0 + 32 * k + lane;
        int lo = 0;  // the last entry that starts at or before e
#pragma unroll
        for (int half = 16; half > 0; half >>= 1) {
          const unsigned int s = __shfl_sync(kFull, excl, lo + half);
          if (s <= e) lo += half;
        }
        const int64_t rb = __shfl_sync(kFull, b, lo);
        const unsigned int st = __shfl_sync(kFull, excl, lo);
        t[k] = e < edges ? __ldg(a.oadj + rb + (e - st)) : -1;
      }
      uint8_t f[kU];
#pragma unroll
      for (int k = 0; k < kU; ++k) f[k] = t[k] >= 0 ? a.dV[t[k]] : (uint8_t)1;
#pragma unroll
      for (int k = 0; k < kU; ++k)
        if (!f[k]) a.dV[t[k]] = 1;
    }
  }
}

// Pull form over G' (the same marks, since w is an out-neighbour of u exactly
// when u is an in-neighbour of w): a vertex outside dV joins it when an
// in-neighbour is in the frontier. Only w's own thread (or warp) reads or
// writes dV[w]; the scan stops at the first frontier in-neighbour. Rows below
// pull_warp_b take a thread each, the others a warp.
template <class Real>
__device__ void pull_round(const SweepArgs<Real>& a) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * kWarps;
  const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  for (int64_t w = a.pull_warp_b + warp; w < a.n; w += nw) {
    if (__shfl_sync(kFull, lane == 0 ? (int)a.dV[w] : 0, 0)) continue;
    const int64_t b = a.off[w], e = a.off[w + 1];
    for (int64_t j0 = b; j0 < e; j0 += 32) {
      const int64_t j = j0 + lane;
      const bool hit = j < e && a.dN[a.adj[j]];
      if (__any_sync(kFull, hit)) {
        if (lane == 0) a.dV[w] = 1;
        break;
      }
    }
  }
  for (int64_t w = warp * 32 + lane; w < a.pull_warp_b; w += nw * 32) {
    if (a.dV[w]) continue;
    const int64_t e = a.off[w + 1];
    for (int64_t j = a.off[w]; j < e; ++j)
      if (a.dN[a.adj[j]]) {
        a.dV[w] = 1;
        break;
      }
  }
}

// The expansion round after a sweep: pull when the frontier's out-edges
// exceed fthr, else push.
template <class Real>
__device__ __forceinline__ void expand_round(const SweepArgs<Real>& a, LoopSlot* slot) {
  if (__ldcg(&slot->fw) > a.fthr) pull_round(a);
  else push_round(a, &slot->nlist);
}

// mode kLoopAll: the whole loop (cooperative launch): [initial push], then
// sweep, barrier, stop test, [expansion, barrier] until the stop rule holds or
// max_iter sweeps ran. The other modes run one phase of iteration it0 as a
// launch of its own (the host-driven loop): a phase past convergence exits at
// once.
template <class P, bool DYN>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_rank_loop(const __grid_constant__ SweepArgs<typename P::Real> a) {
  if (a.mode == kLoopPush) {
    if (DYN) push_round(a, &a.ctl->nlist0);
    return;
  }
  if (a.mode == kLoopSweep) {
    if (a.it0 > 0 && stopped(__ldcg(&slot_of(a, a.it0 - 1)->resid), a.tol)) return;
    sweep<P, DYN>(a, a.it0);
    return;
  }
  if (a.mode == kLoopExpand) {
    LoopSlot* sl = slot_of(a, a.it0);
    if (DYN && !stopped(__ldcg(&sl->resid), a.tol)) expand_round(a, sl);
    return;
  }
  unsigned long long target = 0;
  if (DYN && a.init_push) {
    push_round(a, &a.ctl->nlist0);
    if (!grid_barrier(a.ctl, target)) return;
  }
  for (int it = 0;; ++it) {
    sweep<P, DYN>(a, it);
    if (!grid_barrier(a.ctl, target)) return;
    LoopSlot* sl = slot_of(a, it);
    const unsigned long long resid = __ldcg(&sl->resid);
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (stopped(resid, a.tol) || it + 1 >= a.max_iter) {
      if (first) {
        a.ctl->iters = it + 1;
        a.ctl->resid = resid;
      }
      return;
    }
    // the slot of sweep it + 2, which the sweep before this one used: a
    // barrier separates both from here
    if (first) *slot_of(a, it + 2) = LoopSlot();
    if (DYN && a.expand) {
      expand_round(a, sl);
      if (!grid_barrier(a.ctl, target)) return;
    }
  }
}

// Effective sources of a batch into dN and the first frontier list, targets
// of effective deletions into dV (initialAffected, Alg. affected, in the
// sweep numbering).
__global__ void k_mark_batch(const int32_t* __restrict__ del_src, const int32_t* __restrict__ del_dst,
                             const uint8_t* __restrict__ del_mask, int64_t n_del, const int32_t* __restrict__ ins_src,
                             const uint8_t* __restrict__ ins_mask, int64_t n_ins, const int32_t* __restrict__ inv,
                             const int64_t* __restrict__ ooff, uint8_t* __restrict__ dV, uint8_t* __restrict__ dN,
                             LoopCtl* __restrict__ ctl, int2* __restrict__ list) {
  const int lane = threadIdx.x & 31;
  const int64_t tot = n_del + n_ins, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; base < tot; base += stride) {
    const int64_t i = base + lane;
    int32_t u = -1;
    if (i < n_del) {
      if (!del_mask || del_mask[i]) {
        u = inv[del_src[i]];
        dV[inv[del_dst[i]]] = 1;
      }
    } else if (i < tot) {
      if (!ins_mask || ins_mask[i - n_del]) u = inv[ins_src[i - n_del]];
    }
    // first to set the flag appends the vertex (flags are read by words: the array is padded to them)
    bool mine = false;
    if (u >= 0) {
      const uint32_t bit = 1u << (8 * (u & 3));
      mine = !(atomicOr(reinterpret_cast<uint32_t*>(dN + (u & ~3)), bit) & bit);
    }
    const uint64_t deg = mine ? (uint64_t)(ooff[u + 1] - ooff[u]) : 0;
    append_frontier(mine, u, deg, &ctl->nlist0, list, lane);
  }
}

// Kernel shape of class c by its upper degree bound; the last class runs in
// hub chunks and the one before it a warp per row.
int class_kind(const PartThr& t, int c, bool self_loops) {
  const int C = t.n + 1;
  if (c == C - 2 && C >= 3) return kRowWarp;
  const int64_t hi = t.thr[c];
  if (hi <= 1 && self_loops) return kRowSelf;
  if (hi <= 4) return kRowThread;
  if (hi <= 16) return kRow4;
  if (hi <= 32) return kRow8;
  if (hi <= 128) return kRow16;
  return kRowWarp;
}

template <class P, bool DYN>
struct Launcher {
  using Args = SweepArgs<typename P::Real>;
  // co-resident blocks of the loop kernel on the current device
  static int max_blocks(int* out) {
    auto k = k_rank_loop<P, DYN>;
    int dev = 0, sms = 0, per = 0;
    PRDF_CUDA(cudaGetDevice(&dev));
    PRDF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // almost no shared memory: the unified L1 / shared storage goes to L1, which
    // holds the gathered x of the hottest sources (a preference the driver
    // declines is not an error)
    if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 0) != cudaSuccess) cudaGetLastError();
    PRDF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kThreads, 0));
    if (per < 1 || sms < 1) {
      set_error("the sweep kernel does not fit this device");
      return PRDF_ECUDA;
    }
    *out = per * sms;
    return PRDF_OK;
  }

  // units of rows per class, long rows first
  static int plan(Args& a, const PartThr& t, const int64_t* cb, int max_b) {
    const int C = t.n + 1;
    const int64_t n = cb[C];
    const double warps = (double)max_b * kWarps;
    // a unit's share of the sweep: about an eighth of a warp's work, at least
    // two short steps, at most a few thousand edges
    double target = ((double)a.m + 6.0 * (double)n) / (warps * 8.0);
    if (target < 96) target = 96;
    if (target > 4096) target = 4096;
    int64_t units = a.hub.nchunk;
    a.ncls = 0;
    for (int c = C - 2; c >= 0; --c) {
      const int64_t cnt = cb[c + 1] - cb[c];
      if (cnt <= 0) continue;
      const int kind = class_kind(t, c, a.self_loops != 0);
      const double lo = c > 0 ? (double)t.thr[c - 1] + 1 : 1, hi = (double)t.thr[c];
      const double deg = (lo + hi) / 2 < 2.5 * lo ? (lo + hi) / 2 : 2.5 * lo;
      const int least = kind == kRowWarp ? 1 : kind == kRow16 ? 2 : kind == kRow8 ? 4 : kind == kRow4 ? 8 : 32;
      int rows = least;
      while (rows < 32 * kMaxWords && 2 * rows * (deg + 6) <= target) rows *= 2;
      SweepClass& k = a.cls[a.ncls++];
      k.begin = cb[c];
      k.end = cb[c + 1];
      k.unit0 = (uint32_t)units;
      k.rows = rows;
      k.kind = kind;
      units += (cnt + rows - 1) / rows;
    }
    if (units >= (int64_t)UINT32_MAX / 2) {
      set_error("too many work units");
      return PRDF_EINVAL;
    }
    a.units = (uint32_t)units;
    return PRDF_OK;
  }

  static int run(Args a, const PartThr& t, const int64_t* cb, cudaStream_t s) {
    int max_b = 0;
    PRDF_TRY(max_blocks(&max_b));
    PRDF_TRY(plan(a, t, cb, max_b));
    // few units: few blocks, and a shorter barrier
    int64_t blocks = ((int64_t)a.units + kWarps - 1) / kWarps;
    if (blocks > max_b) blocks = max_b;
    if (blocks < 1) blocks = 1;
    if (a.mode != kLoopAll) {
      k_rank_loop<P, DYN><<<(unsigned)(a.mode == kLoopSweep ? blocks : max_b), kThreads, 0, s>>>(a);
      PRDF_LAUNCH_CHECK();
      return PRDF_OK;
    }
    void* args[] = {&a};
    PRDF_CUDA(cudaLaunchCooperativeKernel((const void*)k_rank_loop<P, DYN>, dim3((unsigned)blocks), dim3(kThreads),
                                          args, 0, s));
    return PRDF_OK;
  }
};

}  // namespace

int launch_rank_loop(const SweepArgs<double>& a, const PartThr& t, const int64_t* cb, bool exact, bool dynamic,
                     cudaStream_t s) {
  if (exact) return dynamic ? Launcher<PExact, true>::run(a, t, cb, s) : Launcher<PExact, false>::run(a, t, cb, s);
  return dynamic ? Launcher<PPlain, true>::run(a, t, cb, s) : Launcher<PPlain, false>::run(a, t, cb, s);
}

int launch_rank_loop(const SweepArgs<float>& a, const PartThr& t, const int64_t* cb, bool dynamic, cudaStream_t s) {
  return dynamic ? Launcher<PKahan, true>::run(a, t, cb, s) : Launcher<PKahan, false>::run(a, t, cb, s);
}

int launch_mark_batch(const int32_t* del_src, const int32_t* del_dst, const uint8_t* del_mask, int64_t n_del,
                      const int32_t* ins_src, const uint8_t* ins_mask, int64_t n_ins, const int32_t* inv,
                      const int64_t* ooff, uint8_t* dV, uint8_t* dN, LoopCtl* ctl, int2* list, cudaStream_t s) {
  if (n_del + n_ins == 0) return PRDF_OK;
  k_mark_batch<<<grid_for(n_del + n_ins, 256), 256, 0, s>>>(del_src, del_dst, del_mask, n_del, ins_src, ins_mask,
                                                           n_ins, inv, ooff, dV, dN, ctl, list);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

}  // namespace prdf
