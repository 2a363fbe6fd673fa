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

#include "loop.cuh"

namespace prdf {

namespace {

// Two blocks of 512 threads per SM at 64 registers: the sweeps are bound by
// the latency and the rate of their gathers, so resident warps matter more
// than registers, and few blocks keep the grid barrier short. (1024 x 1 and
// 256 x 4 within 1 %; 256 x 5 at 51 registers: 4096^2 grid 13.1 against 14.1
// ms, but 2^16 R-MAT 1.41 against 1.25 and the 2^20 stream window 3.51 against
// 3.33 ms; 384 x 4 at 42: 2^24 R-MAT 66.9 against 60.2 ms.)
//
// What bounds a sweep: the L1's handling of its 8-byte gathers. At 2^22 (69 M
// edges) one sweep takes 227 us with 62 M L1 sector misses, 0.88 a clock per
// SM, where uniform gathers reach 0.92; it took 357 us as eight class kernels.
// In FP32 186 us with 54 M misses, 0.93 a clock.
constexpr int kThreads = 512;
constexpr int kMinBlocks = 2;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxRows = 256;  // rows of a unit at most

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
  static constexpr bool kAnyOrder = true;  // the sum does not depend on the order of the terms
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
  static constexpr bool kAnyOrder = false;
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
  static constexpr bool kAnyOrder = false;
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
// The same of an FP32 out-degree: below 2^24 a float holds every integer, from there on the row's offsets are read (a
// rounded degree would leave the row's last out-edges out of its frontier entries).
__device__ __forceinline__ uint64_t degree_of(float d, const int64_t* ooff, int32_t v) {
  return d < 16777216.f || !ooff ? (uint64_t)d : (uint64_t)(__ldg(ooff + v + 1) - __ldg(ooff + v));
}

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

// What the epilogue of a vertex reads besides its sum: out-degree and its
// inverse, (DF-P) the Eq. 2 factor, (DF / DF-P) the deltaN flag.
template <class Real>
struct Own {
  Real d, iv, kf;
  uint8_t dn;
};
__device__ __forceinline__ double ld_const(const double* p, uint64_t pol) { return ld_stream_f64(p, pol); }
template <class P, bool DYN>
__device__ __forceinline__ Own<typename P::Real> load_own(const SweepArgs<typename P::Real>& a, const Ctx<P>& c,
                                                          bool have, int32_t v) {
  Own<typename P::Real> w;
  w.d = w.iv = w.kf = 0;
  w.dn = 0;
  if (have) {
    w.d = ld_const(a.deg + v, c.pf);
    w.iv = ld_const(a.inv + v, c.pf);
    if (DYN) {
      if (a.prune) w.kf = ld_const(a.kf + v, c.pf);
      w.dn = a.dN[v];
    }
  }
  return w;
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
                                       double xself, const Own<double>& w, Tally& t, uint64_t& deg) {
  const double d = w.d, iv = w.iv;
  const bool dn_old = w.dn != 0;
  double r;
  if (DYN && a.prune) {
    // Eq. 2: the self-loop term is solved in closed form (factor precomputed per vertex)
    r = w.kf * (a.c0 + a.alpha * (sum - xself));
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
                                       double xself, const Own<double>& w, Tally& t, uint64_t& deg) {
  const Ctx<PExact> e{c.x, c.xn, c.slot, c.pf, c.pl, c.lane};
  return finish<DYN>(a, e, v, sum, xself, w, t, deg);
}
// the same in FP32, with Alg. update's prune and expand tests evaluated in FP32
template <bool DYN>
__device__ __forceinline__ bool finish(const SweepArgs<float>& a, const Ctx<PKahan>& c, int32_t v, float sum,
                                       float xself, const Own<float>& w, Tally& t, uint64_t& deg) {
  const float d = w.d, iv = w.iv;
  const bool dn_old = w.dn != 0;
  const float rold = xself * d;
  float r;
  if (DYN && a.prune) r = w.kf * fmaf(a.alpha, sum - xself, a.c0);  // Eq. 2
  else r = fmaf(a.alpha, sum, a.c0);                                                      // Eq. 1
  const float dr = fabsf(r - rold);
  bool front = false;
  if (DYN) {
    const float m = fmaxf(r, rold);
    if (a.prune && dr <= a.tau_p * m) a.dV[v] = 0;
    front = dr > a.tau_f * m;
    if (front != dn_old) a.dN[v] = front ? 1 : 0;
    if (front) {
      deg = degree_of(d, a.ooff, v);
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

// The k-th row of a class: every vertex of it (Static), or the k-th affected
// one (DF / DF-P, listed by the scan phase), with its deltaN flag.
template <class P, bool DYN>
__device__ __forceinline__ int32_t row_at(const SweepArgs<typename P::Real>& a, int64_t k) {
  return DYN ? __ldcg(a.act + k) : (int32_t)k;
}

// One row per lane, its offsets known: the epilogue of a batch.
template <class P, bool DYN>
__device__ __forceinline__ void finish_batch(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, bool have,
                                             int32_t v, typename P::Real sum, typename P::Real xself,
                                             const Own<typename P::Real>& w, Tally& t) {
  bool front = false;
  uint64_t deg = 0;
  if (have) front = finish<DYN>(a, c, v, sum, xself, w, t, deg);
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

// Sums of up to 32 rows, one after the other by groups of G lanes; row s of a
// group is described by its lane s (b: first entry, len, and v when the graph
// has vertices without self-loop), S rows at most per group. A 16-byte index
// load a lane and step: the row's entries are read from the 16-byte boundary
// below its first one (positions in a row are 32-bit, counted from that
// boundary). While the gathers of one step are in flight the indices of the
// next step load: the next chunk of the same rows, or the first chunk of the
// groups' next rows, whose offsets are already in the lanes, so a step waits
// for one round trip. On return lane s of each group holds the sum of row s
// in saved (and in hit whether the row holds v itself).
template <class P, int G>
__device__ __forceinline__ void sum_rows(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int S, int64_t b,
                                         int len, int32_t v, typename P::Acc& saved, bool& hit) {
  using Bits = typename P::Bits;
  const int lane = c.lane, sub = lane & (G - 1), src0 = lane & ~(G - 1);
  typename P::Acc acc;
  bool myhit = false;
  // the group's row: entries [lo, hi) from base; this lane's position j
  int64_t rb = __shfl_sync(kFull, b, src0);
  int lo = (int)(rb & 3), hi = lo + __shfl_sync(kFull, len, src0), j = 4 * sub;
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
      const int src = (src0 + s + 1) & 31;  // (past the last row: any lane, no entries)
      rb = __shfl_sync(kFull, b, src);
      const int l = __shfl_sync(kFull, len, src);
      lo = (int)(rb & 3);
      hi = s + 1 < S ? lo + l : 0;
      j = 4 * sub;
      base = a.adj + (rb & ~(int64_t)3);
    }
    q = load4(base, j, hi, c.pf);
    if (G < 32 && !a.self_loops) {
      const int32_t rv = __shfl_sync(kFull, v, src0 + s) & INT32_MAX;
#pragma unroll
      for (int k = 0; k < 4; ++k) myhit = myhit || u[k] == rv;
    }
    add_terms<P>(acc, u, xv);
    if (!more) {
      acc.template group_reduce<G>();
      if (sub == s) saved = acc;
      acc = typename P::Acc();
      if (G < 32 && !a.self_loops) {
        const uint32_t m = __ballot_sync(kFull, myhit) >> src0;
        if (sub == s) hit = (m & ((1u << (G & 31)) - 1u)) != 0;
        myhit = false;
      }
      ++s;
    }
  }
}

// The other way to sum a batch: a row per lane, eight entries a step in two
// 16-byte loads from the boundary below the row's first entry, the next step's
// entries loading while this one's are gathered. No lanes idle past a group's
// row and nothing to meet by shuffles, but the index loads touch a line per
// lane.
template <class P>
__device__ __forceinline__ void sum_lane_rows(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t b,
                                              int len, int32_t v, typename P::Acc& acc, bool& hit) {
  using Bits = typename P::Bits;
  const int lo = (int)(b & 3), hi = len > 0 ? lo + len : 0;
  const int32_t* base = a.adj + (b & ~(int64_t)3);
  auto load = [&](int j) { return j < hi ? ld_stream_i32x4(base + j, c.pf) : make_int4(-1, -1, -1, -1); };
  int4 q0 = load(0), q1 = load(4);
  for (int j = 0; __any_sync(kFull, j < hi); j += 8) {
    int32_t u[8];
    {
      int32_t t[4];
      mask4(q0, j, lo, hi, t);
#pragma unroll
      for (int k = 0; k < 4; ++k) u[k] = t[k];
      mask4(q1, j + 4, lo, hi, t);
#pragma unroll
      for (int k = 0; k < 4; ++k) u[4 + k] = t[k];
    }
    Bits xv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) xv[k] = u[k] >= 0 ? ld_state(c.x + u[k], c.pl) : Bits(0);
    q0 = load(j + 8);
    q1 = load(j + 12);
    if (!a.self_loops) {
#pragma unroll
      for (int k = 0; k < 8; ++k) hit = hit || u[k] == v;
    }
    add_terms<P>(acc, u, xv);
  }
}

// Rows that outgrew their class. Batch updates keep the numbering until 1/64 of
// the edges have changed, so a row of a short class can grow to that many
// entries, and a lane or a small group would walk it for longer than the rest
// of the sweep takes. The classes below a warp per row leave rows above these
// lengths out of their batches and set the warp's flag; sum_grown takes them by
// the whole warp after the unit. 100 K in-edges added to a row of 1 / 2 / 6 / 20 /
// 60 on 8.9 M edges, a solve of 76 sweeps: 1401 / 1972 / 714 / 169 / 88 ms when
// the batch summed them, 40.2 / 40.9 / 40.2 / 41.0 / 40.3 ms now, 38.7 with the
// row numbered as what it is. A flag in shared memory and a second pass, as
// registers for it in the batch loops cost every solve (a 4096^2 grid 13.5 ms
// without, 14.2 summed within the batch, 13.2 this way).
constexpr int kGrown = 128;     // no class of 4, 8 or 16 lanes per row is made for longer rows
constexpr int kGrownLane = 16;  // the same for a lane per row
__device__ __forceinline__ volatile int* grown_flag() {
  __shared__ int flag[kWarps];
  return flag + (threadIdx.x >> 5);
}
template <class Row>
__device__ __forceinline__ void leave_grown(Row& r, int limit) {
  if (r.len > limit) {
    *grown_flag() = 1;
    r.v = -1;
    r.len = 0;
  }
}

// A unit: the rows at positions [kb, ke) of a class, G lanes per row, in
// batches of up to 32. The offsets of the next batch and the row ids of the
// one after it load before the batch.
template <class P, int G, bool DYN>
__device__ __forceinline__ void unit_group(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t kb,
                                           int64_t ke, Tally& t) {
  using Bits = typename P::Bits;
  constexpr int NG = 32 / G;
  const int lane = c.lane, sub = lane & (G - 1);
  const int nact = (int)(ke - kb);
  struct Batch {
    int32_t v;
    int len;
    int64_t b;
  };
  // lane's row of the batch at k0: group g takes rows g * S .. g * S + S - 1
  auto steps = [&](int k0) { return ((nact - k0 < 32 ? nact - k0 : 32) + NG - 1) / NG; };
  auto in_batch = [&](int k0) {
    const int S = steps(k0);
    return sub < S && (lane / G) * S + sub < (nact - k0 < 32 ? nact - k0 : 32);
  };
  auto load_v = [&](int k0) {
    return k0 < nact && in_batch(k0) ? row_at<P, DYN>(a, kb + k0 + (lane / G) * steps(k0) + sub) : -1;
  };
  auto load_off = [&](int32_t v) {
    Batch r;
    r.v = v;
    r.b = 0;
    r.len = 0;
    if (v >= 0) {
      r.b = ld_stream_i64(a.off + v, c.pf);
      r.len = (int)(ld_stream_i64(a.off + v + 1, c.pf) - r.b);
    }
    return r;
  };

  int32_t vn = load_v(32);
  Batch cur = load_off(load_v(0));
  if (G < 32) leave_grown(cur, kGrown);
  for (int k0 = 0; k0 < nact; k0 += 32) {
    const Batch nxt = load_off(vn);
    vn = load_v(k0 + 64);
    const bool have = cur.v >= 0;
    const Own<typename P::Real> own = load_own<P, DYN>(a, c, have, cur.v);
    typename P::Acc saved;
    bool hit = false;
    // rows of 5 to 32 entries: a row per lane when the batch fills most lanes
    // (static solves, a row per lane against a group per row: 2^24 R-MAT 58.6 ->
    // 57.6 ms, 4096^2 grid 21.8 -> 14.1 ms, mixed 2^22 13.5 -> 13.0 ms; rows of 33
    // to 128 lose, 58.8 ms, their index loads then cost as much as the gathers);
    // small batches of a small graph keep the groups (2^16: 1.07 against 1.25 ms).
    // In DF / DF-P a row's place in the list, and with it the size of its batch,
    // changes from run to run, so sums that depend on the order of their terms
    // take one form whatever the batch (as fast as by size, DF-P and DT on 2^16 to
    // 2^24; groups throughout: DT of a 2^22 grid 14.7 against 12.4 ms)
    constexpr bool kOneForm = DYN && !P::Acc::kAnyOrder;
    if (G <= 8 && (kOneForm || nact - k0 >= 24))
      sum_lane_rows<P>(a, c, cur.b, cur.len, cur.v, saved, hit);
    else
      sum_rows<P, G>(a, c, steps(k0), cur.b, cur.len, cur.v, saved, hit);
    // graphs without self-loops on every vertex: x[v] counts only when the row
    // holds v (rows of a warp or more always took x[v])
    const Bits xs = have && (G == 32 || a.self_loops || hit) ? ld_state(c.x + cur.v, c.pl) : Bits(0);
    finish_batch<P, DYN>(a, c, have, cur.v, saved.value(), as_real(xs), own, t);
    cur = nxt;
    if (G < 32) leave_grown(cur, kGrown);
  }
}

// The rows of [kb, ke) above `limit` entries, one after the other. (A graph
// that had a batch has every self-loop.)
template <class P, bool DYN>
__device__ __forceinline__ void sum_grown(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t kb,
                                          int64_t ke, int limit, Tally& t) {
  for (int64_t k0 = kb; k0 < ke; k0 += 32) {
    int32_t v = 0;
    int64_t b = 0;
    int len = 0;
    if (k0 + c.lane < ke) {
      v = row_at<P, DYN>(a, k0 + c.lane);
      b = a.off[v];
      len = (int)(a.off[v + 1] - b);
    }
    const bool far = len > limit;
    const uint32_t m = __ballot_sync(kFull, far);
    if (!m) continue;
    const Own<typename P::Real> own = load_own<P, DYN>(a, c, far, v);
    typename P::Acc saved;
    bool hit = false;
    sum_rows<P, 32>(a, c, 32 - __clz(m), b, far ? len : 0, 0, saved, hit);
    const typename P::Bits xs = far ? ld_state(c.x + v, c.pl) : typename P::Bits(0);
    finish_batch<P, DYN>(a, c, far, v, saved.value(), as_real(xs), own, t);
  }
}

// A unit of chunks of the long rows (the chunk table), a warp per chunk one
// after the other. A row of one chunk is finished like any other. The chunks
// of a longer row leave their sums in hub_part; the warp that sums the last
// of them (an arrival counter per row) adds the row's partial sums and
// finishes the vertex. With exact accumulation the partials are integers, so
// the result is the same bits as any other split; the compensated FP32
// partials are added in chunk order by lanes and a fixed shuffle tree, so
// every run gives the same bits. DF / DF-P: a row's flags change only in its
// finishing warp, which runs after every chunk's warp has read them, or
// (unaffected rows) in the warp of its first chunk, which leaves dV alone.
template <class P, bool DYN>
__device__ __forceinline__ void unit_chunks(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t cb,
                                            int cnt, Tally& t) {
  using Bits = typename P::Bits;
  const int lane = c.lane;
  SweepChunk k = {};
  if (lane < cnt) {
    const int4* p = reinterpret_cast<const int4*>(a.chunks + cb + lane);
    const int4 p0 = __ldg(p), p1 = __ldg(p + 1);
    k.j0 = (int64_t)(((uint64_t)(uint32_t)p0.y << 32) | (uint32_t)p0.x);
    k.len = p0.z;
    k.v = p0.w;
    k.first = p1.x;
    k.parts = p1.y;
    k.row = p1.z;
  }
  int64_t ch = cb + lane;
  int nact = cnt;
  bool have = lane < cnt;
  if (DYN) {
    const bool act = have && a.dV[k.v] != 0;
    if (have && ch == k.first) {
      if (act) t.aff += 1;
      else skip_vertex(a, c, k.v, a.wrote[k.v] != 0, a.dN[k.v] != 0);
    }
    // affected chunks to the first lanes
    const uint32_t m = __ballot_sync(kFull, act);
    nact = __popc(m);
    if (nact == 0) return;
    int src = 0;
    uint32_t rest = m;
    for (int i = 0; i < nact; ++i) {
      const int l = __ffs(rest) - 1;
      rest &= rest - 1;
      if (lane == i) src = l;
    }
    k.j0 = __shfl_sync(kFull, k.j0, src);
    k.len = __shfl_sync(kFull, k.len, src);
    k.v = __shfl_sync(kFull, k.v, src);
    k.first = __shfl_sync(kFull, k.first, src);
    k.parts = __shfl_sync(kFull, k.parts, src);
    k.row = __shfl_sync(kFull, k.row, src);
    ch = cb + src;
    have = lane < nact;
  }
  const Own<typename P::Real> own = load_own<P, DYN>(a, c, have, k.v);
  typename P::Acc saved;
  bool hit = false;
  sum_rows<P, 32>(a, c, nact, k.j0, k.len, 0, saved, hit);
  bool fin = have;
  if (have && k.parts > 1) {
    __stcg(a.hub_part + ch, saved.pack());
    __threadfence();
    fin = atomicAdd(a.hub_done + k.row, 1u) + 1 == (unsigned int)k.parts;
    if (fin) a.hub_done[k.row] = 0;
    __threadfence();
  }
  uint32_t need = __ballot_sync(kFull, fin && have && k.parts > 1);
  __syncwarp();
  while (need) {
    const int l = __ffs(need) - 1;
    need &= need - 1;
    const int first = __shfl_sync(kFull, k.first, l), parts = __shfl_sync(kFull, k.parts, l);
    typename P::Acc acc;
    for (int i = lane; i < parts; i += 32) acc.merge(__ldcg(a.hub_part + first + i));
    acc.template group_reduce<32>();
    if (lane == l) saved = acc;
  }
  const Bits xs = fin ? ld_state(c.x + k.v, c.pl) : Bits(0);
  finish_batch<P, DYN>(a, c, fin, k.v, saved.value(), as_real(xs), own, t);
}

// One row per lane, U indices in flight (short rows).
template <class P, int U, bool DYN>
__device__ __forceinline__ void unit_thread(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t kb,
                                            int64_t ke, Tally& t) {
  using Bits = typename P::Bits;
  const int nact = (int)(ke - kb);
  struct Row {
    int32_t v;
    int len;
    int64_t b;
  };
  auto load_v = [&](int k0) { return k0 + c.lane < nact ? row_at<P, DYN>(a, kb + k0 + c.lane) : -1; };
  auto load_off = [&](int32_t v) {
    Row r;
    r.v = v;
    r.b = 0;
    r.len = 0;
    if (v >= 0) {
      r.b = ld_stream_i64(a.off + v, c.pf);
      r.len = (int)(ld_stream_i64(a.off + v + 1, c.pf) - r.b);
    }
    return r;
  };
  auto load_idx = [&](const Row& r, int32_t (&u)[U]) {
#pragma unroll
    for (int k = 0; k < U; ++k) u[k] = k < r.len ? __ldg(a.adj + r.b + k) : -1;
  };
  // row ids three batches ahead, offsets two, indices one
  const int32_t v0 = load_v(0), v1 = load_v(32);
  int32_t vf = load_v(64);
  Row cur = load_off(v0), nxt = load_off(v1);
  leave_grown(cur, kGrownLane);
  int32_t u[U];
  load_idx(cur, u);
  for (int k0 = 0; k0 < nact; k0 += 32) {
    const bool have = cur.v >= 0;
    Bits xv[U];
#pragma unroll
    for (int k = 0; k < U; ++k) xv[k] = u[k] >= 0 ? ld_state(c.x + u[k], c.pl) : Bits(0);
    const Bits xs = have ? ld_state(c.x + cur.v, c.pl) : Bits(0);
    const Own<typename P::Real> own = load_own<P, DYN>(a, c, have, cur.v);
    int32_t un[U];
    load_idx(nxt, un);
    const Row far = load_off(vf);
    vf = load_v(k0 + 96);
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
    finish_batch<P, DYN>(a, c, have, cur.v, acc.value(), as_real(xself), own, t);
    cur = nxt;
    leave_grown(cur, kGrownLane);
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
__device__ __forceinline__ void unit_self(const SweepArgs<typename P::Real>& a, const Ctx<P>& c, int64_t kb,
                                          int64_t ke, Tally& t) {
  using Bits = typename P::Bits;
  int32_t vn = kb + c.lane < ke ? row_at<P, DYN>(a, kb + c.lane) : 0;
  for (int64_t k0 = kb; k0 < ke; k0 += 32) {
    bool have = k0 + c.lane < ke;
    const int32_t v = vn;
    vn = k0 + 32 + c.lane < ke ? row_at<P, DYN>(a, k0 + 32 + c.lane) : 0;
    const Bits xs = have ? ld_state(c.x + v, c.pl) : Bits(0);
    const Own<typename P::Real> own = load_own<P, DYN>(a, c, have, v);
    typename P::Real sum = as_real(xs);
    if (a.multi && have && ((a.multi[v >> 5] >> (v & 31)) & 1u)) {
      const int64_t b = a.off[v], e = a.off[v + 1];
      if (e - b > kGrownLane) {
        *grown_flag() = 1;
        have = false;
      } else {
        typename P::Acc acc;
        for (int64_t j = b; j < e; ++j) acc.add(ld_state(c.x + a.adj[j], c.pl));
        sum = acc.value();
      }
    }
    finish_batch<P, DYN>(a, c, have, v, sum, as_real(xs), own, t);
  }
}

// -------------------------------------------------------------- phases ----

// the slot of sweep it: a ring of kLoopRing in the whole-loop kernel, one a
// sweep from it_first on in the host-driven loop (slot 0: the sweep before)
template <class Real>
__device__ __forceinline__ LoopSlot* slot_of(const SweepArgs<Real>& a, int it) {
  return a.slot + (a.mode == kLoopAll ? (it & (kLoopRing - 1)) : it - a.it_first + 1);
}

// Units of a sweep: the chunk units, then each class cut by `rows`. Classes
// without rows have no units.
struct Plan {
  uint32_t unit0[kMaxCls];
  int64_t begin[kMaxCls], end[kMaxCls];
  int rows[kMaxCls];
  uint32_t chunk_units, total;
  bool counted;
};

// Cuts the classes (Static: whole, DF / DF-P: their affected rows) into units
// of about a quarter of a warp's share of the sweep, at least a full batch of
// short rows and at most a few thousand edges (so that a unit's start-up
// latency is paid for, and the last units of a sweep are short). A half / a
// quarter / an eighth / a sixteenth: 2^20 stream window 3.70 / 3.36 / 3.51 /
// 3.95 ms, mixed solve at 2^22 13.6 / 13.5 / 13.6 / 14.7 ms. Least cost of 96 /
// 512 / 768 / 1024: 2^16 R-MAT 1.08 / 0.90 / 0.92 / 0.92 ms, 512^2 grid 1.37 /
// 1.11 / 0.70 / 0.71, DF-P on a 2^20 R-MAT 3.1 / 3.1 / 3.5 / 3.5.
// Lane k of the block's first warp takes class k.
template <bool DYN, class Real>
__device__ __forceinline__ void make_plan(const SweepArgs<Real>& a, const LoopSlot* slot, Plan* plan) {
  if (threadIdx.x < 32) {
    const int k = threadIdx.x;
    const bool in = k < a.ncls;
    const int64_t cnt = !in ? 0 : DYN ? (int64_t)__ldcg(&slot->act[k]) : a.cls[k].end - a.cls[k].begin;
    const unsigned int nchunk = a.nchunk ? (unsigned int)__ldg(a.nchunk) : 0u;
    const float per = in ? a.cls[k].deg + 6.f : 0.f;
    float cost = (float)cnt * per;
    if (k == 31) cost = (float)nchunk * (float)a.chunk_size;
    const float all = warp_sum_f32(cost);
    float target = all / (4.f * (float)(gridDim.x * kWarps));
    // rows of more than 128 edges: units of very different length
    const bool uneven = nchunk > 0 || __any_sync(kFull, in && cnt > 0 && a.cls[k].kind == kRowWarp);
    target = fminf(fmaxf(target, uneven ? 512.f : 768.f), 4096.f);
    int rows = in ? a.cls[k].least : 1;
    while (rows < kMaxRows && 2.f * rows * per <= target) rows *= 2;
    const unsigned int units = (unsigned int)((cnt + rows - 1) / rows);
    unsigned int incl = units;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int x = __shfl_up_sync(kFull, incl, o);
      if (k >= o) incl += x;
    }
    const unsigned int cu = (nchunk + a.chunks_per_unit - 1) / a.chunks_per_unit;
    if (in) {
      plan->unit0[k] = cu + incl - units;
      plan->begin[k] = DYN ? a.cls[k].list : a.cls[k].begin;
      plan->end[k] = plan->begin[k] + cnt;
      plan->rows[k] = rows;
    }
    if (k == 31) {
      plan->chunk_units = cu;
      plan->total = cu + incl;
      const float warps = (float)(gridDim.x * kWarps);
      plan->counted = (float)(cu + incl) > 4.f * warps && all > (uneven ? 2048.f : 8192.f) * warps;
    }
  }
  __syncthreads();
}

// bins of the 129..4096 class in DF / DF-P: without them a long row listed late
// sets the sweep's end (DT on 50 M edges 10.4 against 9.2 ms)
constexpr int64_t kLong0 = 2048, kLong1 = 1024, kLong2 = 512;

// DF / DF-P: lists the affected rows of every class outside the chunk table,
// in id order within a stretch of 1024 (a.act + class begin, counts in the
// sweep's slot), and copies the unaffected ones through. A sweep then works
// on full batches of affected rows, however thinly they are spread, at the
// cost of one pass over the flag bytes.
template <class P>
__device__ __forceinline__ void scan(const SweepArgs<typename P::Real>& a, int it) {
  Ctx<P> c;
  c.x = (it & 1) ? a.xb : a.xa;
  c.xn = (it & 1) ? a.xa : a.xb;
  c.slot = slot_of(a, it);
  c.pf = policy_evict_first();
  c.pl = policy_evict_last();
  c.lane = threadIdx.x & 31;
  const int lane = c.lane;
  const int64_t nw = (int64_t)gridDim.x * kWarps;
  const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  unsigned int aff = 0;
  const bool parts = a.ncls > 0 && a.cls[0].part == 0;
  const int64_t n = parts ? a.cls[0].begin : a.scan_end;
  if (parts) {
    // rows of 129 to 4096 edges: by length, so that the sweep can start with
    // the longest; few vertices, so 32 rows a step spread them over the warps
    for (int64_t v0 = n + warp * 32; v0 < a.scan_end; v0 += nw * 32) {
      const int64_t v = v0 + lane;
      int part = -1;
      if (v < a.scan_end) {
        const bool dv = a.dV[v] != 0, wr = a.wrote[v] != 0, dn = a.dN[v] != 0;
        const int64_t len = __ldg(a.off + v + 1) - __ldg(a.off + v);
        if (dv) part = len > kLong0 ? 0 : len > kLong1 ? 1 : len > kLong2 ? 2 : 3;
        else if (wr || dn) skip_vertex(a, c, (int32_t)v, wr, dn);
      }
      uint32_t b[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) b[p] = __ballot_sync(kFull, part == p);
      const uint32_t all = b[0] | b[1] | b[2] | b[3];
      if (!all) continue;
      if (lane == 0) aff += __popc(all);
      const uint32_t mine = lane == 0 ? b[0] : lane == 1 ? b[1] : lane == 2 ? b[2] : b[3];
      unsigned int at = 0;
      if (lane < 4 && mine) at = atomicAdd(&c.slot->act[lane], (unsigned int)__popc(mine));
      at = __shfl_sync(kFull, at, part < 0 ? 0 : part);
      const uint32_t same = __shfl_sync(kFull, mine, part < 0 ? 0 : part);
      if (part >= 0) a.act[a.cls[part].list + at + __popc(same & ((1u << lane) - 1u))] = (int32_t)v;
    }
  }
  for (int64_t v0 = warp * a.scan_rows; v0 < n; v0 += nw * a.scan_rows) {
    // lane's word: rows v0 + 32 lane ..
    uint32_t mdv = 0, mwr = 0, mdn = 0;
    const int64_t w0 = v0 + 32 * lane;
    if (32 * lane < a.scan_rows && w0 < n) {
      const uint4 f[6] = {*reinterpret_cast<const uint4*>(a.dV + w0),    *reinterpret_cast<const uint4*>(a.dV + w0 + 16),
                          *reinterpret_cast<const uint4*>(a.wrote + w0), *reinterpret_cast<const uint4*>(a.wrote + w0 + 16),
                          *reinterpret_cast<const uint4*>(a.dN + w0),    *reinterpret_cast<const uint4*>(a.dN + w0 + 16)};
      // four flag bytes (0 or 1) to four bits
      auto bits4 = [](uint32_t x) { return ((x * 0x10204080u) >> 28) & 0xFu; };
      auto bits16 = [&](const uint4& q) {
        return bits4(q.x) | bits4(q.y) << 4 | bits4(q.z) << 8 | bits4(q.w) << 12;
      };
      const uint32_t in = n - w0 >= 32 ? kFull : (1u << (int)(n - w0)) - 1u;
      mdv = (bits16(f[0]) | bits16(f[1]) << 16) & in;
      mwr = (bits16(f[2]) | bits16(f[3]) << 16) & in;
      mdn = (bits16(f[4]) | bits16(f[5]) << 16) & in;
    }
    uint32_t todo = __ballot_sync(kFull, ((mwr | mdn) & ~mdv) != 0);
    while (todo) {
      const int i = __ffs(todo) - 1;
      todo &= todo - 1;
      const uint32_t w = __shfl_sync(kFull, mwr & ~mdv, i), d = __shfl_sync(kFull, mdn & ~mdv, i);
      const bool bw = (w >> lane) & 1u, bd = (d >> lane) & 1u;
      if (bw || bd) skip_vertex(a, c, (int32_t)(v0 + 32 * i + lane), bw, bd);
    }
    if (!__any_sync(kFull, mdv != 0)) continue;
    aff += __popc(mdv);
    for (int k = 0; k < a.ncls; ++k) {  // (one class, but for the stretches that hold a class bound)
      const int64_t cb = a.cls[k].begin - v0, ce = a.cls[k].end - v0;
      if (ce <= 0 || cb >= a.scan_rows || a.cls[k].part >= 0) continue;
      // rows of this class among the word's: bits [lo, hi)
      const int lo = (int)(cb - 32 * lane < 0 ? 0 : cb - 32 * lane > 32 ? 32 : cb - 32 * lane);
      const int hi = (int)(ce - 32 * lane < 0 ? 0 : ce - 32 * lane > 32 ? 32 : ce - 32 * lane);
      uint32_t m = mdv;
      m &= lo >= 32 ? 0u : kFull << lo;
      m &= hi >= 32 ? kFull : (1u << hi) - 1u;
      const int cnt = __popc(m);
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += x;
      }
      unsigned int base = 0;
      if (lane == 31 && incl) base = atomicAdd(&c.slot->act[k], (unsigned int)incl);
      base = __shfl_sync(kFull, base, 31);
      int32_t* out = a.act + a.cls[k].list + base;
      uint32_t some = __ballot_sync(kFull, m != 0);
      while (some) {
        const int i = __ffs(some) - 1;
        some &= some - 1;
        const uint32_t w = __shfl_sync(kFull, m, i);
        const int at = __shfl_sync(kFull, incl - cnt, i);
        if ((w >> lane) & 1u) out[at + __popc(w & ((1u << lane) - 1u))] = (int32_t)(v0 + 32 * i + lane);
      }
    }
  }
  if (it == 0) {
    aff = __reduce_add_sync(kFull, aff);
    if (lane == 0 && aff) atomicAdd(&a.ctl->aff0, aff);
  }
}

template <class P, bool DYN>
__device__ __forceinline__ void sweep(const SweepArgs<typename P::Real>& a, int it, const Plan* plan) {
  Ctx<P> c;
  c.x = (it & 1) ? a.xb : a.xa;
  c.xn = (it & 1) ? a.xa : a.xb;
  c.slot = slot_of(a, it);
  c.pf = policy_evict_first();
  c.pl = policy_evict_last();
  c.lane = threadIdx.x & 31;
  if (c.lane == 0) *grown_flag() = 0;
  __syncwarp();
  Tally t;
  // First unit by position (consecutive units on different SMs). The others
  // come from a counter, or by position again where units are few or the sweep
  // is short: the counter is one address, and thousands of warps asking at
  // once wait for one another longer than a short sweep lasts (2^16 R-MAT,
  // counter from more than one unit a warp on: 1.21 against 1.02 ms; none up to
  // 16 units a warp: mixed solve at 2^22 16.0 against 13.4 ms). Without long
  // rows the units are alike and position serves longer sweeps too: FP32
  // frontier sweeps of a 1024^2 grid 4.1 against 3.5 ms; with them it does not
  // (2^20 R-MAT, counter from a cost of 2048 / 4096 a warp on: 4.4 / 5.0 ms).
  const unsigned int nw = gridDim.x * kWarps;
  const bool counted = plan->counted;
  for (unsigned int u = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; u < plan->total;) {
    unsigned int nx = u;
    if (counted && c.lane == 0) nx = atomicAdd(&c.slot->units, 1u);
    if (u < plan->chunk_units) {
      const unsigned int nchunk = (unsigned int)__ldg(a.nchunk);
      const unsigned int cb = u * a.chunks_per_unit;
      const unsigned int cnt = nchunk - cb < a.chunks_per_unit ? nchunk - cb : a.chunks_per_unit;
      unit_chunks<P, DYN>(a, c, cb, (int)cnt, t);
    } else {
      int k = 0;
      while (k + 1 < a.ncls && u >= plan->unit0[k + 1]) ++k;
      const int64_t kb = plan->begin[k] + (int64_t)(u - plan->unit0[k]) * plan->rows[k];
      const int64_t ke = kb + plan->rows[k] < plan->end[k] ? kb + plan->rows[k] : plan->end[k];
      switch (a.cls[k].kind) {
        case kRowSelf: unit_self<P, DYN>(a, c, kb, ke, t); break;
        case kRowThread: unit_thread<P, 4, DYN>(a, c, kb, ke, t); break;
        case kRow4: unit_group<P, 4, DYN>(a, c, kb, ke, t); break;
        case kRow8: unit_group<P, 8, DYN>(a, c, kb, ke, t); break;
        case kRow16: unit_group<P, 16, DYN>(a, c, kb, ke, t); break;
        default: unit_group<P, 32, DYN>(a, c, kb, ke, t); break;
      }
      __syncwarp();
      if (*grown_flag()) {  // (the unit is looked up again, so that nothing is kept over it)
        int q = 0;
        while (q + 1 < a.ncls && u >= plan->unit0[q + 1]) ++q;
        const int64_t gb = plan->begin[q] + (int64_t)(u - plan->unit0[q]) * plan->rows[q];
        const int64_t ge = gb + plan->rows[q] < plan->end[q] ? gb + plan->rows[q] : plan->end[q];
        sum_grown<P, DYN>(a, c, gb, ge, a.cls[q].kind <= kRowThread ? kGrownLane : kGrown, t);
        __syncwarp();
        *grown_flag() = 0;
        __syncwarp();
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
    const unsigned int af = __reduce_add_sync(kFull, t.aff);  // (each lane counted the rows of its own chunks)
    if (c.lane == 0 && af) atomicAdd(&s_aff, af);
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
// step (entries of a step's length and more one by one: 8.2 -> 4.0 ms for DF-P
// with push rounds alone, 6000 edges on a 2^20 R-MAT); a long row is several
// entries (kFrontChunk edges each) on different warps. A flag already set is not
// stored again.
template <class Real>
__device__ void push_round(const SweepArgs<Real>& a, const unsigned int* count) {
  const int lane = threadIdx.x & 31;
  const unsigned int total = __ldcg(count);
  const unsigned int nw = gridDim.x * kWarps;
  const unsigned int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const unsigned int per = (total + nw - 1) / nw;
  const unsigned int epw = per < 1 ? 1 : (per > 32 ? 32 : per);
  // (entries nw apart: neighbours in the list are of one class and of like length)
  for (unsigned int base = w; base < total; base += nw * epw) {
    int64_t b = 0;
    unsigned int len = 0;
    if ((unsigned int)lane < epw && base + lane * nw < total) {
      const int2 en = __ldcg(a.list + base + lane * nw);
      const int64_t rb = a.ooff[en.x] + (int64_t)en.y * kFrontChunk, re = a.ooff[en.x + 1];
      b = rb;
      len = (unsigned int)(re - rb < kFrontChunk ? re - rb : kFrontChunk);
    }
    constexpr int kU = 4;
    // entries that fill a step each on their own, without a search for an edge's entry
    uint32_t alone = __ballot_sync(kFull, len >= 32 * kU);
    while (alone) {
      const int l = __ffs(alone) - 1;
      alone &= alone - 1;
      const int32_t* row = a.oadj + __shfl_sync(kFull, b, l);
      const unsigned int cnt = __shfl_sync(kFull, len, l);
      for (unsigned int e0 = lane; e0 < cnt; e0 += 32 * kU) {
        int32_t t[kU];
        uint8_t f[kU];
#pragma unroll
        for (int k = 0; k < kU; ++k) t[k] = e0 + 32 * k < cnt ? __ldg(row + e0 + 32 * k) : -1;
#pragma unroll
        for (int k = 0; k < kU; ++k) f[k] = t[k] >= 0 ? a.dV[t[k]] : (uint8_t)1;
#pragma unroll
        for (int k = 0; k < kU; ++k)
          if (!f[k]) a.dV[t[k]] = 1;
      }
    }
    if (len >= 32 * kU) len = 0;
    unsigned int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int x = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += x;
    }
    const unsigned int excl = incl - len;
    const unsigned int edges = __shfl_sync(kFull, incl, 31);
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
// in-neighbour is in the frontier. Only w's own lanes read or write dV[w]; the
// scan of a row stops at its first frontier in-neighbour. A warp takes the
// rows of a class outside dV among 32, G lanes per row with four entries each
// in flight (a lane per row and serial loads before: the longest rows of 128
// entries set the round's time).
template <class Real, int G>
__device__ __forceinline__ void pull_rows(const SweepArgs<Real>& a, int64_t vb, int64_t ve, int64_t warp, int64_t nw,
                                          uint64_t pf) {
  const int lane = threadIdx.x & 31, sub = lane & (G - 1), grp = lane / G;
  constexpr int NG = 32 / G;
  // rows a warp looks at together: 32, or fewer where that leaves warps without
  // any (it walks them one after the other: 40 rows of 50 K entries on two warps
  // took 9.7 ms a call, 32 rows a warp whatever their number, 1.1 now)
  const int64_t share = (ve - vb + nw - 1) / nw;
  const int per = share >= 32 ? 32 : share > NG ? (int)share : NG;
  int64_t v = vb + warp * per + lane;
  bool out = lane < per && v < ve && a.dV[v] == 0;
  for (int64_t v0 = vb + warp * per; v0 < ve; v0 += nw * per) {
    v = v0 + lane;
    uint32_t m = __ballot_sync(kFull, out);
    const int64_t w = v + nw * per;  // the next rows' flags load ahead
    out = lane < per && w < ve && a.dV[w] == 0;
    if (!m) continue;
    int64_t b = 0;
    int len = 0;
    if ((m >> lane) & 1u) {
      b = ld_stream_i64(a.off + v, pf);
      len = (int)(ld_stream_i64(a.off + v + 1, pf) - b);
    }
    while (m) {
      // the next NG rows, one per group
      int r = -1;
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        const int l = m ? __ffs(m) - 1 : -1;
        m &= m - 1;  // (0 stays 0)
        if (g == grp) r = l;
      }
      const int64_t rb = __shfl_sync(kFull, b, r < 0 ? 0 : r);
      const int rl = __shfl_sync(kFull, len, r < 0 ? 0 : r);
      const int lo = (int)(rb & 3);
      const int32_t* base = a.adj + (rb & ~(int64_t)3);
      int hi = r < 0 ? 0 : lo + rl;
      bool hit = false;
      for (int j = 4 * sub; __any_sync(kFull, j - 4 * sub < hi); j += 4 * G) {
        int32_t u[4];
        mask4(load4(base, j, hi, pf), j, lo, hi, u);
        uint8_t f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] = u[k] >= 0 ? a.dN[u[k]] : (uint8_t)0;
        const uint32_t any = __ballot_sync(kFull, (f[0] | f[1] | f[2] | f[3]) != 0);
        const uint32_t mine = G == 32 ? any : (any >> (lane & ~(G - 1))) & ((1u << (G & 31)) - 1u);
        if (mine) {
          hit = true;
          hi = 0;  // this group is done
        }
      }
      if (hit && sub == 0) a.dV[v0 + r] = 1;
    }
  }
}

// one vertex of the in-degree <= 1 class
template <class Real>
__device__ __forceinline__ void pull_self(const SweepArgs<Real>& a, int64_t v) {
  if (a.dV[v]) return;
  bool hit = a.dN[v] != 0;
  if (!hit && a.multi && ((a.multi[v >> 5] >> (v & 31)) & 1u)) {
    const int64_t e = a.off[v + 1];
    for (int64_t j = a.off[v]; j < e && !hit; ++j) hit = a.dN[a.adj[j]] != 0;
  }
  if (hit) a.dV[v] = 1;
}

template <class Real>
__device__ void pull_round(const SweepArgs<Real>& a) {
  const int lane = threadIdx.x & 31;
  const uint64_t pf = policy_evict_first();
  const int64_t nw = (int64_t)gridDim.x * kWarps;
  const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  pull_rows<Real, 32>(a, a.scan_end, a.n, warp, nw, pf);
  for (int k = 0; k < a.ncls; ++k) {
    const SweepClass& cl = a.cls[k];
    if (cl.part > 0) continue;  // (the class's other parts list the same rows)
    switch (cl.kind) {
      case kRowSelf:
        // the row is [v], so v joins when it is in the frontier itself: 16 flags
        // at a time inside the class, its ragged ends and the vertices that
        // gained in-edges one by one
        {
          const int64_t wb = (cl.begin + 15) >> 4, we = cl.end >> 4;
          for (int64_t w = wb + warp * 32 + lane; w < we; w += nw * 32) {
            const uint4 d = reinterpret_cast<const uint4*>(a.dV)[w], f = reinterpret_cast<const uint4*>(a.dN)[w];
            const uint4 o = make_uint4(d.x | f.x, d.y | f.y, d.z | f.z, d.w | f.w);
            if (o.x != d.x || o.y != d.y || o.z != d.z || o.w != d.w) reinterpret_cast<uint4*>(a.dV)[w] = o;
            if (a.multi && ((a.multi[w >> 1] >> (16 * (w & 1))) & 0xFFFFu))
              for (int64_t v = 16 * w; v < 16 * w + 16; ++v) pull_self(a, v);
          }
          if (warp == 0) {
            const int64_t b0 = cl.begin, b1 = wb * 16 < cl.end ? wb * 16 : cl.end;
            for (int64_t v = b0 + lane; v < b1; v += 32) pull_self(a, v);
            const int64_t e0 = we * 16 > b1 ? we * 16 : b1;
            for (int64_t v = e0 + lane; v < cl.end; v += 32) pull_self(a, v);
          }
        }
        break;
      case kRowThread:
      case kRow4: pull_rows<Real, 4>(a, cl.begin, cl.end, warp, nw, pf); break;
      case kRow8: pull_rows<Real, 8>(a, cl.begin, cl.end, warp, nw, pf); break;
      case kRow16: pull_rows<Real, 16>(a, cl.begin, cl.end, warp, nw, pf); break;
      default: pull_rows<Real, 32>(a, cl.begin, cl.end, warp, nw, pf); break;
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
// max_iter sweeps ran (the last of them expands too). The other modes run one phase of iteration it0 as a
// launch of its own (the host-driven loop): a phase past convergence exits at
// once.
template <class P, bool DYN>
__global__ void __launch_bounds__(kThreads, kMinBlocks) k_rank_loop(const __grid_constant__ SweepArgs<typename P::Real> a) {
  __shared__ Plan plan;
  if (a.mode == kLoopPush) {
    if (DYN) push_round(a, &a.ctl->nlist0);
    return;
  }
  if (a.mode == kLoopScan || a.mode == kLoopSweep) {
    if (a.it0 > 0 && stopped(__ldcg(&slot_of(a, a.it0 - 1)->resid), a.tol)) return;
    if (a.mode == kLoopScan) {
      if (DYN) scan<P>(a, a.it0);
      return;
    }
    make_plan<DYN>(a, slot_of(a, a.it0), &plan);
    sweep<P, DYN>(a, a.it0, &plan);
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
  if (!DYN) make_plan<DYN>(a, a.slot, &plan);
  for (int it = 0;; ++it) {
    LoopSlot* sl = slot_of(a, it);
    if (DYN) {
      scan<P>(a, it);
      if (!grid_barrier(a.ctl, target)) return;
      make_plan<DYN>(a, sl, &plan);
    }
    sweep<P, DYN>(a, it, &plan);
    if (!grid_barrier(a.ctl, target)) return;
    const unsigned long long resid = __ldcg(&sl->resid);
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    const bool done = stopped(resid, a.tol);
    if (done || it + 1 >= a.max_iter) {
      if (first) {
        a.ctl->iters = it + 1;
        a.ctl->resid = resid;
      }
      // a loop cut off by max_iter leaves the affected set of a next sweep, as after every sweep that did not converge
      if (DYN && a.expand && !done) expand_round(a, sl);
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

// Chunk table: a row is cut into ceil(len / size) chunks (one when empty).
__global__ void k_chunk_count(const int64_t* __restrict__ off, int64_t begin, int64_t rows, int size, int above,
                              uint32_t* __restrict__ cnt) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < rows; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t d = off[begin + i + 1] - off[begin + i];
    cnt[i] = above > 0 ? (d > above ? (uint32_t)((d + size - 1) / size) : 0u)
                       : (d > 0 ? (uint32_t)((d + size - 1) / size) : 1u);
  }
}

__global__ void k_chunk_fill(const int64_t* __restrict__ off, int64_t begin, int64_t rows, int size,
                             const int64_t* __restrict__ first, SweepChunk* __restrict__ chunks) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = warp; i < rows; i += nwarps) {
    const int64_t b = off[begin + i], e = off[begin + i + 1], f = first[i];
    const int parts = (int)(first[i + 1] - f);
    for (int p = lane; p < parts; p += 32) {
      const int64_t j0 = b + (int64_t)p * size;
      SweepChunk k;
      k.j0 = j0;
      k.len = (int)(e - j0 < size ? e - j0 : size);
      k.v = (int32_t)(begin + i);
      k.first = (int32_t)f;
      k.parts = parts;
      k.row = (int32_t)i;
      k.pad = 0;
      chunks[f + p] = k;
    }
  }
}

// Kernel shape of class c by its upper degree bound; the last class runs in
// chunks and the one before it a warp per row (or in chunks).
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

  // classes outside the chunk table, long rows first
  static void classes(Args& a, const PartThr& t, const int64_t* cb) {
    a.ncls = 0;
    a.scan_end = cb[a.chunk_class];
    int64_t extra = a.n;  // lists of the parts of the longest rows follow the n first entries
    for (int c = a.chunk_class - 1; c >= 0; --c) {
      const int64_t cnt = cb[c + 1] - cb[c];
      if (cnt <= 0) continue;
      const double lo = c > 0 ? (double)t.thr[c - 1] + 1 : 1, hi = (double)t.thr[c];
      SweepClass k;
      k.begin = cb[c];
      k.end = cb[c + 1];
      k.list = cb[c];
      k.kind = class_kind(t, c, a.self_loops != 0);
      k.deg = (float)((lo + hi) / 2 < 2.5 * lo ? (lo + hi) / 2 : 2.5 * lo);
      k.least = k.kind == kRowWarp ? 1 : k.kind == kRow16 ? 2 : k.kind == kRow8 ? 4 : k.kind == kRow4 ? 8 : 32;
      k.part = -1;
      if (DYN && c == a.chunk_class - 1 && k.kind == kRowWarp) {
        const float deg[4] = {1.4f * kLong0, 1.4f * kLong1, 1.4f * kLong2, 250.f};
        for (int p = 0; p < 4; ++p) {
          k.part = p;
          k.deg = deg[p];
          k.list = p < 3 ? extra : cb[c];
          if (p < 3) extra += cnt;
          a.cls[a.ncls++] = k;
        }
        continue;
      }
      a.cls[a.ncls++] = k;
    }
  }

  static int run(Args a, const PartThr& t, const int64_t* cb, cudaStream_t s) {
    int max_b = 0;
    PRDF_TRY(max_blocks(&max_b));
    classes(a, t, cb);
    // small graphs: few blocks, and a shorter barrier
    int64_t blocks = ((a.m + 8 * (int64_t)a.n) / 64 + kWarps - 1) / kWarps;
    if (blocks > max_b) blocks = max_b;
    if (blocks < 1) blocks = 1;
    // rows a warp scans at a time: 1024, fewer when that leaves warps idle
    a.scan_rows = 1024;
    while (a.scan_rows > 32 && a.scan_end < (int64_t)a.scan_rows * blocks * kWarps) a.scan_rows /= 2;
    if (a.mode != kLoopAll) {
      k_rank_loop<P, DYN><<<(unsigned)blocks, kThreads, 0, s>>>(a);
      PRDF_LAUNCH_CHECK();
      return PRDF_OK;
    }
    void* args[] = {&a};
    return launch_coop((const void*)k_rank_loop<P, DYN>, blocks, kThreads, args, s);
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

int build_chunks(const int64_t* off, int64_t begin, int64_t n, int64_t m, int size, int above, SweepChunks& t,
                 Workspace& ws, cudaStream_t s) {
  t.rows = n - begin;
  t.max_chunks = 0;
  if (t.rows <= 0) {
    t.rows = 0;
    return PRDF_OK;
  }
  PRDF_TRY(t.cnt.reserve((size_t)t.rows, s));
  PRDF_TRY(t.first.reserve((size_t)t.rows + 1, s));
  k_chunk_count<<<grid_for(t.rows, 256), 256, 0, s>>>(off, begin, t.rows, size, above, t.cnt.p);
  PRDF_LAUNCH_CHECK();
  PRDF_TRY(exclusive_scan_u32(t.cnt.p, t.rows, t.first.p, ws, s));
  if (above > 0) {
    // the K-column calls keep a partial sum per chunk and column: room for as
    // many chunks as there are (2^22 vertices, K = 64: 158 K chunks, 81 MB; the
    // bound m / above + m / size would be 859 K, 440 MB)
    PRDF_CUDA(cudaMemcpyAsync(ws.host_i64, t.first.p + t.rows, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    PRDF_CUDA(cudaStreamSynchronize(s));
    t.max_chunks = ws.host_i64[0];
  } else {
    // the rank sweep's 16 bytes a chunk: room for the most there can be, so that a call after a batch waits for nothing
    t.max_chunks = t.rows + m / size + 1;
  }
  if (t.max_chunks >= INT32_MAX) {
    set_error("too many row chunks");
    return PRDF_EINVAL;
  }
  PRDF_TRY(t.chunks.reserve((size_t)(t.max_chunks > 0 ? t.max_chunks : 1), s));
  k_chunk_fill<<<grid_for(t.rows * 32, 256), 256, 0, s>>>(off, begin, t.rows, size, t.first.p, t.chunks.p);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
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
