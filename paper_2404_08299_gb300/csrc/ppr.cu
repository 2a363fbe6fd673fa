// K-column weighted personalised PageRank (an extension of Eq. 1 and
// Alg. static): R[:, c] = alpha * P^T R[:, c] + (1 - alpha) * S[:, c] with the
// row-stochastic P_uv = w_uv / sum_k w_uk, for K personalisation columns at
// once. State is row-major [n, Kp] in the class-contiguous numbering, Kp = K
// rounded up to a multiple of four (padding columns stay zero), so one index
// and weight fetch serves a tile of columns, four of them per lane.
//
// FP32 sweeps sum the products of up to four edges with FMAs and fold each
// such sum into a compensated pair (TwoSum), so the rounding error does not
// grow with the row length. (Eight at a time lose most of what follows a large
// product in a row of eight; four cost 1 % of the K = 32 forward and backward
// and nothing at K = 64.) The FP64 stage is mixed-precision
// iterative refinement: an FP64 sweep computes the Jacobi step T(R) and the
// residual T(R) - R; an FP32 solve of E = alpha P^T E + residual gives the
// correction. The stop rule is the same as Static's: the L-inf change of an
// FP64 Jacobi step <= tol.
//
// One persistent kernel per solve (k_ppr_loop, a cooperative launch), as in
// sweep.cu: units of rows and row chunks of every column tile, a grid barrier
// between sweeps, the stop test on the device. What bounds a sweep is the
// 16-byte gathers of the rows of R (K * 4 bytes per edge through L2), so the
// kernel is built to keep them in flight: the indices and weights of the next
// step load (one per lane, handed round by shuffles; in narrow FP32 tiles four
// per lane, the same in every lane of a row) while this step's gathers are on
// their way, across row and chunk bounds. At 2^22 and K = 64 (69 M edges, 17.8
// GB of gathered rows) an FP32 sweep takes 2.3 ms; four kernels per sweep with
// unpipelined loads took 3.07 ms.
#include <cstring>

#include "loop.cuh"

namespace prdf {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kFull = 0xffffffffu;
// K of 1 or 2: 2 lanes a row in units of at most this mean length, else 4. (2 up to a mean of 4 and 8 lanes above it
// left most lanes without an edge on rows of 5 to 20. K = 2, ms a solve, FP64 and mixed: 10^6-vertex grid 22.3 -> 5.4
// and 11.1 -> 3.9, 8.7 M random edges 21.8 -> 7.1 and 9.2 -> 5.3, 2^22 R-MAT 59.4 -> 47.6 and 39.2 -> 35.)
constexpr int64_t kShortMean = 20;

// Compensated FP32 sum (s + e): TwoSum folds each term's rounding error into e.
struct Dot2 {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float y) {
    const float t = s + y;
    const float bp = t - s;
    e += (s - (t - bp)) + (y - bp);
    s = t;
  }
  __device__ __forceinline__ void merge(const Dot2& o) {
    add(o.s);
    e += o.e;
  }
  __device__ __forceinline__ float value() const { return s + e; }
  __device__ __forceinline__ Dot2 shfl_xor(int o) const {
    Dot2 x;
    x.s = __shfl_xor_sync(kFull, s, o);
    x.e = __shfl_xor_sync(kFull, e, o);
    return x;
  }
};
// Plain FP64 sum (fixed order: edges of a slot, then slots, then chunks).
struct Sum64 {
  double s = 0;
  __device__ __forceinline__ void merge(const Sum64& o) { s += o.s; }
  __device__ __forceinline__ double value() const { return s; }
  __device__ __forceinline__ Sum64 shfl_xor(int o) const {
    Sum64 x;
    x.s = __shfl_xor_sync(kFull, s, o);
    return x;
  }
};

// Column accumulator: products go to b; fold() ends a block of at most four
// of them; sum(folded) is the total (folded: any block was ended before).
struct Col32 {
  using Sum = Dot2;
  Dot2 d;
  float b = 0.f;
  __device__ __forceinline__ void prod(float p, float r) { b = fmaf(p, r, b); }
  __device__ __forceinline__ void fold() {
    d.add(b);
    b = 0.f;
  }
  // a whole block at once
  template <class R>
  __device__ __forceinline__ void block(const float (&p)[4], const R (&r)[4], int q) {
    float x = p[0] * r[0].v[q];
#pragma unroll
    for (int k = 1; k < 4; ++k) x = fmaf(p[k], r[k].v[q], x);
    d.add(x);
  }
  __device__ __forceinline__ Dot2 sum(bool folded) {
    if (!folded) {
      d.s = b;
      d.e = 0.f;
    } else {
      d.add(b);
    }
    return d;
  }
};
struct Col64 {
  using Sum = Sum64;
  Sum64 d;
  __device__ __forceinline__ void prod(double p, double r) { d.s = fma(p, r, d.s); }
  __device__ __forceinline__ void fold() {}
  __device__ __forceinline__ Sum64 sum(bool) const { return d; }
};

template <class T>
struct Traits;
template <>
struct Traits<float> {
  using Col = Col32;
  static constexpr int kU = 4;          // gathers of a lane in flight (8: spills, 223 against 215 ms a solve)
  static constexpr int kMinBlocks = 4;  // 64 registers (3 blocks: 248 against 211 ms, 5: 239)
};
template <>
struct Traits<double> {
  using Col = Col64;
  static constexpr int kU = 4;
  static constexpr int kMinBlocks = 2;  // 128 registers (3 blocks spill: K = 5 on 0.7 M edges 3.03 against 2.86 ms)
};

template <class T, int Q>
struct Vec {
  T v[Q];
};

// Q columns of a row, one load (two for four doubles): coherent, as R is
// written in the same kernel, a grid barrier earlier. Q is 4 (a row stride that
// is a multiple of four: every K above 2, the columns past K are the row's zero
// padding), or the whole row of K = 1 or 2. Nothing is read and zeros are
// returned when `on` is false.
template <int Q>
__device__ __forceinline__ void ld_row(const float* src, bool on, Vec<float, Q>& r) {
#pragma unroll
  for (int q = 0; q < Q; ++q) r.v[q] = 0.f;
  if (!on) return;
  if constexpr (Q == 4)
    asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(r.v[0]), "=f"(r.v[1]), "=f"(r.v[2]), "=f"(r.v[3])
                 : "l"(src));
  else if constexpr (Q == 2)
    asm volatile("ld.global.v2.f32 {%0,%1}, [%2];" : "=f"(r.v[0]), "=f"(r.v[1]) : "l"(src));
  else
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(r.v[0]) : "l"(src));
}
template <int Q>
__device__ __forceinline__ void ld_row(const double* src, bool on, Vec<double, Q>& r) {
#pragma unroll
  for (int q = 0; q < Q; ++q) r.v[q] = 0.0;
  if (!on) return;
  if constexpr (Q == 1)
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(r.v[0]) : "l"(src));
  else
    asm volatile("ld.global.v2.f64 {%0,%1}, [%2];" : "=d"(r.v[0]), "=d"(r.v[1]) : "l"(src));
  if constexpr (Q == 4) asm volatile("ld.global.v2.f64 {%0,%1}, [%2];" : "=d"(r.v[2]), "=d"(r.v[3]) : "l"(src + 2));
}
template <int Q>
__device__ __forceinline__ void st_row(float* dst, const float* v) {
  if constexpr (Q == 4) *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
  else if constexpr (Q == 2) *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
  else *dst = v[0];
}
template <int Q>
__device__ __forceinline__ void st_row(double* dst, const double* v) {
  if constexpr (Q == 1) *dst = v[0];
  else *reinterpret_cast<double2*>(dst) = make_double2(v[0], v[1]);
  if constexpr (Q == 4) reinterpret_cast<double2*>(dst)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ float ld_weight(const float* p, uint64_t pol) {
  float v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ double ld_weight(const double* p, uint64_t pol) { return ld_stream_f64(p, pol); }
// four weights from a 16-byte boundary
__device__ __forceinline__ void ld_weights4(const float* p, uint64_t pol, float (&w)[4]) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
      : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3])
      : "l"(p), "l"(pol));
}

// Largest |T(R) - R| and |T(R)| a thread saw (bits).
struct Peak {
  uint64_t d = 0;
  uint32_t r = 0;
  __device__ __forceinline__ void see(float diff, float val) {
    const uint32_t a = __float_as_uint(fabsf(diff)), b = __float_as_uint(fabsf(val));
    d = a > (uint32_t)d ? a : d;
    r = b > r ? b : r;
  }
  __device__ __forceinline__ void see(double diff, double) {
    const uint64_t a = dbits(fabs(diff));
    d = a > d ? a : d;
  }
};

template <class T>
struct Ctx {
  const T* R;     // this lane's columns of row 0 of the current iterate
  T* Rn;          // the next iterate
  uint64_t pf;
  int lane, col;
  bool colok;     // the lane has columns
};

template <int Q, class T>
__device__ __forceinline__ void gather(const Ctx<T>& c, int K, int32_t u, bool on, Vec<T, Q>& r) {
  ld_row<Q>(c.R + (int64_t)u * K, on && c.colok, r);
}

// The teleport and the previous R of a lane's columns of a vertex.
template <class T, int Q>
struct Own {
  Vec<T, Q> s, old;
};
template <class T, int Q>
__device__ __forceinline__ void load_own(const PprArgs<T>& a, const Ctx<T>& c, int32_t v, Own<T, Q>& w) {
  const bool on = c.colok;
  // right-hand side row: dense, or (srow) the compact row of v, none when v has no teleport mass
  const int64_t sr = !on ? -1 : a.srow ? (int64_t)__ldg(a.srow + v) : (int64_t)v;
  ld_row<Q>(c.R + (int64_t)v * a.K, on, w.old);
  ld_row<Q>(a.S + (sr >= 0 ? sr : 0) * a.K + c.col, sr >= 0, w.s);
}

// New values of a lane's columns of vertex v from their sums: Eq. 1 with the
// teleport S, the change against the previous R, and (FP64) the residual.
template <class T, int Q>
__device__ __forceinline__ void finish_row(const PprArgs<T>& a, const Ctx<T>& c, int32_t v, const T* sum,
                                           const Own<T, Q>& w, Peak& pk) {
  if (!c.colok) return;
  const int64_t o = (int64_t)v * a.K + c.col;
  T t[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    t[q] = fma(a.alpha, sum[q], a.beta * w.s.v[q]);
    pk.see(t[q] - w.old.v[q], t[q]);
  }
  st_row<Q>(c.Rn + o, t);
  if (sizeof(T) == 8 && a.res32) {
    float d[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) d[q] = (float)((t[q] - w.old.v[q]) * a.inv_beta);
    st_row<Q>(a.res32 + o, d);
  }
}

// Rows of at most a few hundred edges: LPE lanes (a slot) per row, kSlots rows
// side by side, [vb, ve) in steps of kSlots. A slot's lanes hold a window of
// the row's indices and weights (kE edges) and hand them round by shuffles.
// The next window (of the same rows, or of the slots' next rows, whose offsets
// are known a step ahead) loads while this one's rows are gathered.
template <class T, int LPE>
__device__ __forceinline__ void unit_rows(const PprArgs<T>& a, const Ctx<T>& c, int32_t vb, int32_t ve, Peak& pk) {
  constexpr int kSlots = 32 / LPE;
  constexpr int kEpl = LPE >= 16 ? 1 : LPE >= 8 ? 2 : 4;  // window edges per lane
  constexpr int kE = kEpl * LPE;
  constexpr int U = 4;
  const int sub = c.lane & (LPE - 1), slot = c.lane / LPE, slot0 = c.lane & ~(LPE - 1);
  // (rows above row_max are in the chunk table: length -1, nothing to do)
  auto load_off = [&](int32_t v, int64_t& b, int& len) {
    b = 0;
    len = -1;
    if (v < ve && v >= 0) {  // (v + kSlots may pass the largest id)
      b = ld_stream_i64(a.off + v, c.pf);
      const int64_t d = ld_stream_i64(a.off + v + 1, c.pf) - b;
      len = d <= a.row_max ? (int)d : -1;
    }
  };
  int32_t u[kEpl];
  T p[kEpl];
  auto load_win = [&](int64_t b, int rem) {
#pragma unroll
    for (int i = 0; i < kEpl; ++i) {
      const int e = sub + LPE * i;
      u[i] = e < rem ? ld_stream_i32(a.adj + b + e, c.pf) : 0;
      p[i] = e < rem ? ld_weight(a.P + b + e, c.pf) : T(0);
    }
  };
  int64_t b, bn;
  int32_t v = vb + slot;
  int rem, ln;
  load_off(v, b, rem);
  load_win(b, rem);
  load_off(v + kSlots, bn, ln);
  typename Traits<T>::Col acc[4];
  bool todo = rem >= 0;
  for (int32_t v0 = vb; v0 < ve;) {
    const int here = rem < kE ? rem : kE;
    const int most = __reduce_max_sync(kFull, here);
    const bool more = __any_sync(kFull, rem > kE);
    int32_t cu[kEpl];
    T cp[kEpl];
#pragma unroll
    for (int i = 0; i < kEpl; ++i) {
      cu[i] = u[i];
      cp[i] = p[i];
    }
    Vec<T, 4> r[U];
#pragma unroll
    for (int k = 0; k < U; ++k)
      gather<4>(c, a.K, __shfl_sync(kFull, cu[k / LPE], slot0 + k % LPE), k < here, r[k]);
    // the next window
    const int32_t vdone = v;
    const bool done = todo;
    if (more) {
      b += kE;
      rem = rem > kE ? rem - kE : 0;
      load_win(b, rem);
    } else {
      v += kSlots;
      b = bn;
      rem = ln;
      todo = ln >= 0;
      load_win(b, rem);
      load_off(v + kSlots, bn, ln);
    }
#pragma unroll
    for (int e0 = 0; e0 < kE; e0 += U) {
      if (e0 >= most) break;
      if constexpr (sizeof(T) == 4) {
        // (no partial block is kept from step to step: K = 32 on 17 M edges 130.3 -> 128.6, 10^6-vertex grid 17.7 -> 16.9 ms)
        T w[U];
#pragma unroll
        for (int k = 0; k < U; ++k) w[k] = __shfl_sync(kFull, cp[(e0 + k) / LPE], slot0 + (e0 + k) % LPE);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q].block(w, r, q);
      } else {
#pragma unroll
        for (int k = 0; k < U; ++k) {
          // FP64 products are what a step is short of, and an instruction costs its 32 lanes whatever they hold:
          // those past the longest row are left out (K = 8 on 17 M edges: 37.3 -> 34.2 ms)
          if (k > 0 && e0 + k >= most) break;
          const T w = __shfl_sync(kFull, cp[(e0 + k) / LPE], slot0 + (e0 + k) % LPE);
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[q].prod(w, r[k].v[q]);
        }
      }
      if (e0 + U < kE && e0 + U < most) {
#pragma unroll
        for (int k = 0; k < U; ++k) {
          const int e = e0 + U + k;
          gather<4>(c, a.K, __shfl_sync(kFull, cu[e / LPE], slot0 + e % LPE), e < here, r[k]);
        }
      }
    }
    if (!more) {
      if (done) {
        T t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) t[q] = acc[q].d.value();
        Own<T, 4> own;
        load_own<T, 4>(a, c, vdone, own);
        finish_row<T, 4>(a, c, vdone, t, own, pk);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = typename Traits<T>::Col();
      v0 += kSlots;
    }
  }
}

// The same rows for FP32 tiles of up to 16 columns (LPE lanes a row, 1, 2 or
// 4): every lane of a slot loads the row's next four indices and weights
// itself, one 16-byte load each (from the 16-byte boundary at or before the
// row, so the first and last may hold neighbours' entries: adj and the weights
// end in padding), which leaves out the window's registers and its shuffles.
// The indices of the next step load while this step's gathers are on their
// way; the weights come with the gathers. The
// block of four products goes straight into the compensated pair. Ms a mixed
// solve, windows and this form: 10^6-vertex grid K = 4 5.8 and 4.1, K = 8 6.5
// and 5.6, K = 16 11.9 and 9.8; 8.7 M random edges 8.2 and 5.7, 8.7 and 7.2, 14.7
// and 12.8; 2^22 R-MAT 51.8 and 41.0, 54.3 and 51.8, 88.9 and 83.0. At 32
// columns and above the windows' loads, one entry a lane, are the cheaper ones.
// (The teleport and the previous rank load with the step's gathers; with one
// lane a row that cost more: K = 4 on the random edges 6.53 against 6.43.)
template <int LPE>
__device__ __forceinline__ void unit_rows_direct(const PprArgs<float>& a, const Ctx<float>& c, int32_t vb, int32_t ve,
                                                 Peak& pk) {
  constexpr int kSlots = 32 / LPE;
  const int slot = c.lane / LPE;
  auto load_off = [&](int32_t v, int64_t& b, int& len) {
    b = 0;
    len = -1;
    if (v < ve && v >= 0) {
      b = ld_stream_i64(a.off + v, c.pf);
      const int64_t d = ld_stream_i64(a.off + v + 1, c.pf) - b;
      len = d <= a.row_max ? (int)d : -1;
    }
  };
  int32_t v = vb + slot;
  int64_t b, bn;
  int len, ln;
  load_off(v, b, len);
  load_off(v + kSlots, bn, ln);
  int j = -(int)(b & 3);  // the step's first entry, counted from the row's
  int4 u = make_int4(0, 0, 0, 0);
  if (j < len) u = ld_stream_i32x4(a.adj + b + j, c.pf);
  Dot2 acc[4];
  float w[4] = {};
  for (int32_t v0 = vb; v0 < ve;) {
    Vec<float, 4> r[4];
    const int32_t id[4] = {u.x, u.y, u.z, u.w};
    if (j < len) ld_weights4(a.P + b + j, c.pf, w);
#pragma unroll
    for (int k = 0; k < 4; ++k) gather<4>(c, a.K, id[k], j + k >= 0 && j + k < len, r[k]);
    j += 4;
    const bool more = __any_sync(kFull, j < len);
    const int32_t vdone = v;
    const bool fin = len >= 0 && !more;
    Own<float, 4> own;
    if (LPE > 1 && fin) load_own<float, 4>(a, c, vdone, own);
    if (!more) {
      v += kSlots;
      b = bn;
      len = ln;
      j = -(int)(b & 3);
      load_off(v + kSlots, bn, ln);
    }
    if (j < len) u = ld_stream_i32x4(a.adj + b + j, c.pf);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float x = w[0] * r[0].v[q];
#pragma unroll
      for (int k = 1; k < 4; ++k) x = fmaf(w[k], r[k].v[q], x);
      acc[q].add(x);
    }
    if (more) continue;
    if (fin) {
      if (LPE == 1) load_own<float, 4>(a, c, vdone, own);
      float t[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) t[q] = acc[q].value();
      finish_row<float, 4>(a, c, vdone, t, own, pk);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = Dot2();
    v0 += kSlots;
  }
}

// The same rows where a lane holds whole rows of R (K of 1 or 2): G lanes per
// row, each with its own edges, so no index or weight is handed round, and the
// lanes' sums meet at the row's end. With a lane per four columns half of the
// lanes and three of four products were idle: K = 1 on 69 M edges, mixed 51.3
// ms a solve before, 28.9 now; FP64 101.5 (four kernels a sweep) and 44.0. At
// K = 4 the form above is the faster one (FP64 on 8.7 M edges 16.6 against 19.0
// ms).
template <class T, int Q, int G>
__device__ __forceinline__ void unit_rows_narrow(const PprArgs<T>& a, const Ctx<T>& c, int32_t vb, int32_t ve,
                                                 Peak& pk) {
  constexpr int kSlots = 32 / G;
  constexpr int U = 4;       // edges of a lane a step
  constexpr int kE = U * G;
  const int sub = c.lane & (G - 1), slot = c.lane / G;
  auto load_off = [&](int32_t v, int64_t& b, int& len) {
    b = 0;
    len = -1;
    if (v < ve && v >= 0) {
      b = ld_stream_i64(a.off + v, c.pf);
      const int64_t d = ld_stream_i64(a.off + v + 1, c.pf) - b;
      len = d <= a.row_max ? (int)d : -1;
    }
  };
  int32_t u[U];
  T p[U];
  auto load_win = [&](int64_t b, int rem) {
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int e = sub + G * i;
      u[i] = e < rem ? ld_stream_i32(a.adj + b + e, c.pf) : 0;
      p[i] = e < rem ? ld_weight(a.P + b + e, c.pf) : T(0);
    }
  };
  int64_t b, bn;
  int32_t v = vb + slot;
  int rem, ln;
  load_off(v, b, rem);
  load_win(b, rem);
  load_off(v + kSlots, bn, ln);
  typename Traits<T>::Col acc[Q];
  bool folded = false;
  for (int32_t v0 = vb; v0 < ve;) {
    const bool more = __any_sync(kFull, rem > kE);
    Vec<T, Q> r[U];
    T cp[U];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      gather<Q>(c, a.K, u[i], sub + G * i < rem, r[i]);
      cp[i] = p[i];
    }
    const int32_t vdone = v;
    const bool fin = !more && rem >= 0 && sub == 0;
    Own<T, Q> own;
    if (fin) load_own<T, Q>(a, c, vdone, own);
    if (more) {
      b += kE;
      rem = rem > kE ? rem - kE : (rem >= 0 ? 0 : -1);
      load_win(b, rem);
    } else {
      v += kSlots;
      b = bn;
      rem = ln;
      load_win(b, rem);
      load_off(v + kSlots, bn, ln);
    }
#pragma unroll
    for (int i = 0; i < U; ++i)
#pragma unroll
      for (int q = 0; q < Q; ++q) acc[q].prod(cp[i], r[i].v[q]);
    if (more) {
#pragma unroll
      for (int q = 0; q < Q; ++q) acc[q].fold();
      folded = true;
      continue;
    }
    T t[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      typename Traits<T>::Col::Sum x = acc[q].sum(folded);
#pragma unroll
      for (int o = 1; o < G; o <<= 1) x.merge(x.shfl_xor(o));
      t[q] = x.value();
      acc[q] = typename Traits<T>::Col();
    }
    if (fin) finish_row<T, Q>(a, c, vdone, t, own, pk);
    folded = false;
    v0 += kSlots;
  }
}

// sums of the slots of a warp meet in every slot (a fixed tree)
template <class Sum, int LPE, int Q>
__device__ __forceinline__ void merge_slots(Sum* t) {
#pragma unroll
  for (int o = LPE; o < 32; o <<= 1)
#pragma unroll
    for (int q = 0; q < Q; ++q) t[q].merge(t[q].shfl_xor(o));
}

__device__ __forceinline__ void ld_part(const Dot2* p, Dot2& x) {
  const float2 f = __ldcg(reinterpret_cast<const float2*>(p));
  x.s = f.x;
  x.e = f.y;
}
__device__ __forceinline__ void ld_part(const Sum64* p, Sum64& x) { x.s = __ldcg(reinterpret_cast<const double*>(p)); }

// Chunks of long rows (the chunk table), up to 32 a unit, a warp per chunk one
// after the other, the slots striding over its edges. A row of one chunk is
// finished at once; of a longer row the warp that sums the last chunk (an
// arrival counter per row and tile) adds the row's partial sums in chunk order
// and finishes it.
template <class T, int LPE, int Q>
__device__ __forceinline__ void unit_chunks(const PprArgs<T>& a, const Ctx<T>& c, int64_t cb, int cnt, int tile_no,
                                            Peak& pk) {
  using Sum = typename Traits<T>::Col::Sum;
  constexpr int kSlots = 32 / LPE;
  constexpr int U = Traits<T>::kU;
  constexpr int W = LPE >= U ? 1 : U / LPE;  // 32-edge windows a step
  constexpr int kE = 32 * W;                 // edges a step
  constexpr int kPer = kE / kSlots;          // of them a slot's
  const int lane = c.lane, sub = lane & (LPE - 1), slot = lane / LPE;
  // lane l: chunk cb + l
  int64_t j0 = 0;
  int len = 0;
  int32_t kv = 0;
  if (lane < cnt) {
    const int4 p0 = __ldg(reinterpret_cast<const int4*>(a.chunks + cb + lane));
    j0 = (int64_t)(((uint64_t)(uint32_t)p0.y << 32) | (uint32_t)p0.x);
    len = p0.z;
    kv = p0.w;
  }
  int32_t u[W];
  T p[W];
  auto load_win = [&](int64_t b, int rem) {
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const int e = lane + 32 * i;
      u[i] = e < rem ? ld_stream_i32(a.adj + b + e, c.pf) : 0;
      p[i] = e < rem ? ld_weight(a.P + b + e, c.pf) : T(0);
    }
  };
  int64_t b = __shfl_sync(kFull, j0, 0);
  int rem = __shfl_sync(kFull, len, 0);
  load_win(b, rem);
  typename Traits<T>::Col acc[Q];
  for (int s = 0; s < cnt;) {
    int32_t cu[W];
    T cp[W];
#pragma unroll
    for (int i = 0; i < W; ++i) {
      cu[i] = u[i];
      cp[i] = p[i];
    }
    const int here = rem < kE ? rem : kE;
    const bool more = rem > kE;  // the same on every lane
    Vec<T, Q> r[U];
    // slot's i-th edge of the step is edge i * kSlots + slot
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int e = i * kSlots + slot;
      gather<Q>(c, a.K, __shfl_sync(kFull, cu[(i * kSlots) / 32], e & 31), e < here, r[i]);
    }
    if (more) {
      b += kE;
      rem -= kE;
    } else {
      const int nx = s + 1 < cnt ? s + 1 : 0;
      b = __shfl_sync(kFull, j0, nx);
      rem = __shfl_sync(kFull, len, nx);
      if (s + 1 >= cnt) rem = 0;
    }
    load_win(b, rem);
#pragma unroll
    for (int i0 = 0; i0 < kPer; i0 += U) {
      if (i0 * kSlots >= here && i0 > 0) break;
#pragma unroll
      for (int i = 0; i < U; ++i) {
        if (sizeof(T) == 8 && i > 0 && (i0 + i) * kSlots >= here) break;
        const T w = __shfl_sync(kFull, cp[((i0 + i) * kSlots) / 32], ((i0 + i) * kSlots + slot) & 31);
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[q].prod(w, r[i].v[q]);
      }
#pragma unroll
      for (int q = 0; q < Q; ++q) acc[q].fold();
      if (i0 + U < kPer && (i0 + U) * kSlots < here) {
#pragma unroll
        for (int i = 0; i < U; ++i) {
          const int e = (i0 + U + i) * kSlots + slot;
          gather<Q>(c, a.K, __shfl_sync(kFull, cu[((i0 + U + i) * kSlots) / 32], e & 31), e < here, r[i]);
        }
      }
    }
    if (more) continue;
    Sum t[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      t[q] = acc[q].sum(true);
      acc[q] = typename Traits<T>::Col();
    }
    merge_slots<Sum, LPE, Q>(t);
    const int4 rec = __ldg(reinterpret_cast<const int4*>(a.chunks + cb + s) + 1);  // first, parts, row
    const int parts = rec.y;
    const int32_t v = __shfl_sync(kFull, kv, s);
    bool fin = true;
    if (parts > 1) {
      Sum* part = reinterpret_cast<Sum*>(a.part) + (int64_t)tile_no * a.max_chunks * (Q * LPE);
      const int first = rec.x, row = rec.z;
      if (slot == 0) {
#pragma unroll
        for (int q = 0; q < Q; ++q) part[(cb + s) * (Q * LPE) + Q * sub + q] = t[q];
      }
      __threadfence();
      __syncwarp();
      unsigned int n = 0;
      if (lane == 0) n = atomicAdd(a.done + (int64_t)tile_no * a.chunk_rows + row, 1u) + 1;
      n = __shfl_sync(kFull, n, 0);
      fin = n == (unsigned int)parts;
      if (fin) {
        if (lane == 0) a.done[(int64_t)tile_no * a.chunk_rows + row] = 0;
        __threadfence();
#pragma unroll
        for (int q = 0; q < Q; ++q) t[q] = Sum();
        for (int i = slot; i < parts; i += kSlots) {
#pragma unroll
          for (int q = 0; q < Q; ++q) {
            Sum x;
            ld_part(part + (int64_t)(first + i) * (Q * LPE) + Q * sub + q, x);
            t[q].merge(x);
          }
        }
        merge_slots<Sum, LPE, Q>(t);
      }
    }
    if (fin && slot == 0) {
      T sum[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q) sum[q] = t[q].value();
      Own<T, Q> own;
      load_own<T, Q>(a, c, v, own);
      finish_row<T, Q>(a, c, v, sum, own, pk);
    }
    ++s;
  }
}

template <class T>
__device__ __forceinline__ LoopSlot* slot_of(const PprArgs<T>& a, int it) {
  return a.slot + (a.mode == kLoopAll ? (it & (kLoopRing - 1)) : it - a.it_first + 1);
}

__device__ __forceinline__ bool stopped(unsigned long long resid, double tol) { return bitsd(resid) <= tol; }
__device__ __forceinline__ bool stopped(unsigned long long resid, float tol) {
  return __uint_as_float((uint32_t)resid) <= tol * __uint_as_float((uint32_t)(resid >> 32));
}

// LPE lanes of four columns each side by side (Q = 4); LPE = 1: a lane has the
// whole row, Q columns (FP32: 1, 2 or 4, FP64: 1 or 2).
template <class T, int LPE, int Q>
__device__ __forceinline__ void ppr_sweep(const PprArgs<T>& a, int it) {
  Ctx<T> c;
  const T* R = (it & 1) ? a.Rb : a.Ra;
  c.Rn = (it & 1) ? a.Ra : a.Rb;
  c.pf = policy_evict_first();
  c.lane = threadIdx.x & 31;
  LoopSlot* slot = slot_of(a, it);
  Peak pk;
  const unsigned int nw = gridDim.x * kWarps;
  const unsigned int nchunk = a.nchunk ? (unsigned int)__ldg(a.nchunk) : 0u;
  const unsigned int cu = (nchunk + a.chunks_per_unit - 1) / a.chunks_per_unit;
  const unsigned int ru = (unsigned int)((a.n + a.rows_per_unit - 1) / a.rows_per_unit);
  const unsigned int per_tile = cu + ru;
  const unsigned int total = per_tile * a.tiles;
  // Many units are handed out by a counter, one address for the whole GPU. Units of one step of rows (eight a warp at
  // most, by the rule of run_tile) are over before the next number comes: mixed on grids, counted and by position, 3.6 *
  // 10^5 vertices K = 8 2.98 and 2.56 ms, 0.9 * 10^5 K = 32 2.87 and 2.45.
  constexpr unsigned int kStep = Q == 4 ? 32 / LPE : 16;
  const bool counted = total > 4 * nw && (a.rows_per_unit > kStep || total > 8 * nw);
  for (unsigned int x = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; x < total;) {
    unsigned int nx = x;
    if (counted && c.lane == 0) nx = atomicAdd(&slot->units, 1u);
    // the chunks of every tile first (long work), then the rows of every tile
    const bool chunk = x < cu * a.tiles;
    const unsigned int y = chunk ? x : x - cu * a.tiles;
    const unsigned int per = chunk ? cu : ru;
    const int tile_no = (int)(y / per);
    const unsigned int un = y - (unsigned int)tile_no * per;
    c.col = tile_no * (Q * LPE) + Q * (c.lane & (LPE - 1));
    c.colok = c.col < a.K;
    c.R = R + c.col;
    if (chunk) {
      const unsigned int cb = un * a.chunks_per_unit;
      const unsigned int cnt = nchunk - cb < a.chunks_per_unit ? nchunk - cb : a.chunks_per_unit;
      unit_chunks<T, LPE, Q>(a, c, cb, (int)cnt, tile_no, pk);
    } else {
      // from the highest class down: long rows first
      const int64_t ve = a.n - (int64_t)un * a.rows_per_unit;
      const int64_t vb = ve > a.rows_per_unit ? ve - a.rows_per_unit : 0;
      if constexpr (sizeof(T) == 4 && Q == 4 && LPE <= 4) {
        unit_rows_direct<LPE>(a, c, (int32_t)vb, (int32_t)ve, pk);
      } else if constexpr (LPE > 1) {
        unit_rows<T, LPE>(a, c, (int32_t)vb, (int32_t)ve, pk);
      } else {
        const int64_t len = __ldg(a.off + ve) - __ldg(a.off + vb);
        if (len <= kShortMean * (ve - vb)) unit_rows_narrow<T, Q, 2>(a, c, (int32_t)vb, (int32_t)ve, pk);
        else unit_rows_narrow<T, Q, 4>(a, c, (int32_t)vb, (int32_t)ve, pk);
      }
    }
    x = nw + __shfl_sync(kFull, nx, 0);
  }
  __shared__ unsigned long long s_d;
  __shared__ unsigned int s_r;
  if (threadIdx.x == 0) {
    s_d = 0;
    s_r = 0;
  }
  __syncthreads();
  const uint64_t d = warp_max_u64(pk.d);
  const uint32_t r = __reduce_max_sync(kFull, pk.r);
  if (c.lane == 0) {
    if (d) atomicMax(&s_d, (unsigned long long)d);
    if (r) atomicMax(&s_r, r);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sizeof(T) == 8) {
      if (s_d) atomicMax(&slot->resid, s_d);
    } else {
      uint32_t* w = reinterpret_cast<uint32_t*>(&slot->resid);
      if (s_d) atomicMax(w, (uint32_t)s_d);
      if (s_r) atomicMax(w + 1, s_r);
    }
  }
}

// The whole solve (kLoopAll, cooperative launch) or one sweep of the
// host-driven loop.
template <class T, int LPE, int Q>
__global__ void __launch_bounds__(kThreads, Traits<T>::kMinBlocks) k_ppr_loop(const __grid_constant__ PprArgs<T> a) {
  if (a.mode == kLoopSweep) {
    if (a.it0 > 0 && stopped(__ldcg(&slot_of(a, a.it0 - 1)->resid), a.tol)) return;
    ppr_sweep<T, LPE, Q>(a, a.it0);
    return;
  }
  unsigned long long target = 0;
  for (int it = 0;; ++it) {
    ppr_sweep<T, LPE, Q>(a, it);
    if (!grid_barrier(a.ctl, target)) return;
    const unsigned long long resid = __ldcg(&slot_of(a, it)->resid);
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (stopped(resid, a.tol) || it + 1 >= a.max_iter) {
      if (first) {
        a.ctl->iters = it + 1;
        a.ctl->resid = resid;
      }
      return;
    }
    if (first) *slot_of(a, it + 2) = LoopSlot();  // as in sweep.cu
  }
}

// Edge gradient of L = sum_c G_c . R_c with respect to w_uv (out-slot j of
// renumbered row i, vertex u = perm[i], target v = adj[j]):
//   dL/dw_uv = (1 / W_u) * sum_c R[u, c] * (alpha * lambda[v, c] - (lambda[u, c] - G[u, c]))
// using sum_k P_uk lambda[k] = (lambda[u] - G[u]) / alpha. The per-row constant
// b_u = sum_c R[u, c] * (lambda[u, c] - G[u, c]) is formed once per row.
template <int L>
__global__ void k_grad_rows(const double* __restrict__ lam, const double* __restrict__ Gs, double g_scale,
                            const double* __restrict__ Rr, int32_t n, int K, double* __restrict__ bu) {
  const int sub = threadIdx.x & (L - 1);
  const int64_t row0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / L;
  const int64_t step = ((int64_t)gridDim.x * blockDim.x) / L;
  const int64_t last = ((int64_t)n + step - 1) / step * step;
  for (int64_t i = row0; i < last; i += step) {  // (the same trip count on every lane)
    double b = 0;
    if (i < n)
      for (int c = sub; c < K; c += L) b = fma(Rr[i * K + c], lam[i * K + c] - g_scale * Gs[i * K + c], b);
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) b += __shfl_xor_sync(kFull, b, o);
    if (sub == 0 && i < n) bu[i] = b;
  }
}

// A warp takes kGradChunk consecutive out-slots; L lanes (a slot) per edge,
// columns over the lanes, L edges of a slot at a time, whose dot products meet
// by exchanging halves (fewer additions than one per edge and level: FP64
// additions are what this kernel is short of after its multiplications). The
// rows of long and short vertices cost the same per edge (a lane per edge and a
// warp per row before: a serial walk over the columns, and the longest row's
// walk at the end).
constexpr int64_t kGradChunk = 512;
template <int L>
__global__ void __launch_bounds__(256) k_grad_w(const int64_t* __restrict__ off, const int32_t* __restrict__ adj,
                                                const int32_t* __restrict__ perm, const int64_t* __restrict__ orig_off,
                                                const double* __restrict__ lam, const double* __restrict__ bu,
                                                const double* __restrict__ Rr, const double* __restrict__ W, int32_t n,
                                                int64_t m, int K, double alpha, double* __restrict__ grad_w) {
  constexpr int kSlots = 32 / L;
  const int lane = threadIdx.x & 31, sub = lane & (L - 1), slot = lane / L;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t p0 = warp * kGradChunk; p0 < m; p0 += nwarps * kGradChunk) {
    const int64_t pe = p0 + kGradChunk < m ? p0 + kGradChunk : m;
    // row of the slot's first edge: the last r with off[r] <= p
    int64_t r = 0, z = n;
    while (z - r > 1) {
      const int64_t mid = (r + z) >> 1;
      if (off[mid] <= p0 + slot * L) r = mid; else z = mid;
    }
    for (int64_t q0 = p0; q0 < pe; q0 += kSlots * L) {
      double d[L];
      int64_t row[L];
#pragma unroll
      for (int k = 0; k < L; ++k) {
        const int64_t p = q0 + slot * L + k;
        d[k] = 0;
        row[k] = -1;
        if (p < pe) {
          int steps = 0;
          while (off[r + 1] <= p && steps < 8) {
            ++r;
            ++steps;
          }
          if (off[r + 1] <= p) {  // past a run of empty rows
            int64_t a = r, b = n;
            while (b - a > 1) {
              const int64_t mid = (a + b) >> 1;
              if (off[mid] <= p) a = mid; else b = mid;
            }
            r = a;
          }
          row[k] = r;
          const double* Lv = lam + (int64_t)adj[p] * K;
          const double* Ru = Rr + r * K;
          if ((K & 1) == 0) {
            for (int c = 2 * sub; c < K; c += 2 * L) {
              const double2 x = __ldg(reinterpret_cast<const double2*>(Ru + c));
              const double2 y = __ldg(reinterpret_cast<const double2*>(Lv + c));
              d[k] = fma(x.x, y.x, d[k]);
              d[k] = fma(x.y, y.y, d[k]);
            }
          } else {
            for (int c = sub; c < K; c += L) d[k] = fma(__ldg(Ru + c), __ldg(Lv + c), d[k]);
          }
        }
      }
      // lane sub of the slot ends with the sum of its edge sub
      int have = L;
#pragma unroll
      for (int o = 1; o < L; o <<= 1) {
        have >>= 1;
        const bool hi = sub & o;
#pragma unroll
        for (int k = 0; k < L / 2; ++k) {
          if (k < have) {
            const double keep = hi ? d[2 * k + 1] : d[2 * k], give = hi ? d[2 * k] : d[2 * k + 1];
            d[k] = keep + __shfl_xor_sync(kFull, give, o);
          }
        }
      }
      const int64_t p = q0 + slot * L + sub;
      int64_t rw = row[0];
#pragma unroll
      for (int k = 1; k < L; ++k)
        if (sub == k) rw = row[k];
      if (rw >= 0 && p < pe)
        grad_w[orig_off[perm[rw]] + (p - off[rw])] = (alpha * d[0] - bu[rw]) * (1.0 / W[rw]);
    }
  }
}

// rows of a [n, K] matrix with a non-zero entry (flag per row)
__global__ void k_row_nonzero(const double* __restrict__ S, int64_t n, int K, uint32_t* __restrict__ flag) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < n; v += nwarps) {
    bool nz = false;
    for (int c = lane; c < K; c += 32) nz = nz || S[v * K + c] != 0.0;
    nz = __any_sync(0xffffffffu, nz);
    if (lane == 0) flag[v] = nz ? 1u : 0u;
  }
}

// srow[v] = compact row of v or -1; Sc64 / Sc32 (FP64 / FP32) get the non-zero rows, and R32 (zero on
// entry) the FP32 rows at their place
__global__ void k_row_compact(const double* __restrict__ S, int64_t n, int K, const uint32_t* __restrict__ flag,
                              const int64_t* __restrict__ pos, int32_t* __restrict__ srow, double* __restrict__ Sc64,
                              float* __restrict__ Sc32, float* __restrict__ R32) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = warp; v < n; v += nwarps) {
    const bool nz = flag[v] != 0;
    const int64_t r = nz ? pos[v] : -1;
    if (lane == 0) srow[v] = (int32_t)r;
    if (!nz) continue;
    for (int c = lane; c < K; c += 32) {
      const double x = S[v * K + c];
      Sc64[r * K + c] = x;
      Sc32[r * K + c] = (float)x;
      if (R32) R32[v * K + c] = (float)x;
    }
  }
}

__global__ void k_add_correction(double* __restrict__ R, const float* __restrict__ E, int64_t cnt) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
    R[i] += (double)E[i];
}

__global__ void k_narrow(const double* __restrict__ x, int64_t cnt, float* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}

__global__ void k_widen_n(const float* __restrict__ y, int64_t cnt, double* __restrict__ x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = (double)y[i];
}

template <class T, int LPE, int Q>
int run_tile(PprArgs<T> a, int64_t n, cudaStream_t s) {
  auto k = k_ppr_loop<T, LPE, Q>;
  int dev = 0, sms = 0, per = 0;
  PRDF_CUDA(cudaGetDevice(&dev));
  PRDF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  PRDF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kThreads, 0));
  if (per < 1 || sms < 1) {
    set_error("the K-column kernel does not fit this device");
    return PRDF_ECUDA;
  }
  const int max_b = per * sms;
  constexpr int kSlots = Q == 4 ? 32 / LPE : 16;
  a.tiles = (a.K + Q * LPE - 1) / (Q * LPE);
  // rows of a unit: about an eighth of a warp's share, a few steps at least
  int64_t rows = kSlots;
  while (rows < 8 * kSlots && rows * 8 * (int64_t)max_b * kWarps < n * a.tiles) rows *= 2;
  a.rows_per_unit = (int)rows;
  // four chunks a unit on large graphs (K = 64 at 2^22: 218 against 222 ms), one
  // where that leaves warps idle (K = 32 at 2^19, 8.9 M edges: 35 against 53 ms)
  a.chunks_per_unit = a.m >= (1ll << 25) ? 4 : 1;
  const int64_t work = (a.n / rows + 1 + a.max_chunks / a.chunks_per_unit + 1) * a.tiles;
  if (work * 2 >= (int64_t)UINT32_MAX) {
    set_error("too many work units");
    return PRDF_EINVAL;
  }
  int64_t blocks = (work + kWarps - 1) / kWarps;
  if (blocks > max_b) blocks = max_b;
  if (a.mode != kLoopAll) {
    k<<<(unsigned)blocks, kThreads, 0, s>>>(a);
    PRDF_LAUNCH_CHECK();
    return PRDF_OK;
  }
  void* args[] = {&a};
  return launch_coop((const void*)k, blocks, kThreads, args, s);
}

template <class T>
int run_ppr(const PprArgs<T>& a, int tile, int64_t n, cudaStream_t s) {
  if (a.K == 1) return run_tile<T, 1, 1>(a, n, s);
  if (a.K == 2) return run_tile<T, 1, 2>(a, n, s);
  if constexpr (sizeof(T) == 4)
    if (a.K == 4) return run_tile<T, 1, 4>(a, n, s);
  switch (tile) {
    case 8: return run_tile<T, 2, 4>(a, n, s);
    case 16: return run_tile<T, 4, 4>(a, n, s);
    case 32: return run_tile<T, 8, 4>(a, n, s);
    default: return run_tile<T, 16, 4>(a, n, s);
  }
}

}  // namespace

int launch_ppr_loop(const PprArgs<float>& a, int tile, int64_t n, cudaStream_t s) { return run_ppr(a, tile, n, s); }
int launch_ppr_loop(const PprArgs<double>& a, int tile, int64_t n, cudaStream_t s) { return run_ppr(a, tile, n, s); }

int launch_grad_w(const int64_t* off, const int32_t* adj, const int32_t* perm, const int64_t* orig_off,
                  const double* lam, const double* Gs, double g_scale, const double* Rr, const double* W, int32_t n,
                  int64_t m, int K, double alpha, double* grad_w, cudaStream_t s) {
  DBuf<double> bu;
  PRDF_TRY(bu.alloc((size_t)n, s));
  const int grid = grid_for((m + kGradChunk - 1) / kGradChunk * 32, 256);
  if (K > 8)
    k_grad_rows<8><<<grid_for((int64_t)n * 8, 256), 256, 0, s>>>(lam, Gs, g_scale, Rr, n, K, bu.p);
  else
    k_grad_rows<2><<<grid_for((int64_t)n * 2, 256), 256, 0, s>>>(lam, Gs, g_scale, Rr, n, K, bu.p);
  // Lanes per edge: as few as keep the gathered rows of lambda in flight, since every lane past the columns is idle
  // and the lanes' sums cost additions. Gradient part, ms, 8 lanes -> 2: R-MAT 2^19 (8 M edges) K = 12 0.78 -> 0.45,
  // K = 32 1.05 -> 0.82; 12 M edges in rows of 200 0.90 -> 0.49, 1.23 -> 0.89; 8 -> 4 at K = 64: 1.66 -> 1.47.
  if (K > 32)
    k_grad_w<4><<<grid, 256, 0, s>>>(off, adj, perm, orig_off, lam, bu.p, Rr, W, n, m, K, alpha, grad_w);
  else
    k_grad_w<2><<<grid, 256, 0, s>>>(off, adj, perm, orig_off, lam, bu.p, Rr, W, n, m, K, alpha, grad_w);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

int ppr_sparse_rhs(const double* S, int64_t n, int K, Workspace& ws, PprSparseRhs* out, float* R32, cudaStream_t s) {
  out->rows = 0;
  DBuf<uint32_t> flag;
  DBuf<int64_t> pos;
  PRDF_TRY(flag.alloc((size_t)n, s));
  PRDF_TRY(pos.alloc((size_t)n + 1, s));
  k_row_nonzero<<<grid_for(n * 32, kThreads), kThreads, 0, s>>>(S, n, K, flag.p);
  PRDF_LAUNCH_CHECK();
  PRDF_TRY(exclusive_scan_u32(flag.p, n, pos.p, ws, s));
  PRDF_CUDA(cudaMemcpyAsync(ws.host_i64, pos.p + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  PRDF_CUDA(cudaStreamSynchronize(s));
  const int64_t rows = ws.host_i64[0];
  if (rows * 4 > n) return PRDF_OK;  // dense enough: keep the dense form
  PRDF_TRY(out->srow.reserve((size_t)n, s));
  PRDF_TRY(out->Sc64.reserve((size_t)(rows > 0 ? rows : 1) * K, s));
  PRDF_TRY(out->Sc32.reserve((size_t)(rows > 0 ? rows : 1) * K, s));
  if (R32) PRDF_CUDA(cudaMemsetAsync(R32, 0, sizeof(float) * (size_t)n * K, s));
  k_row_compact<<<grid_for(n * 32, kThreads), kThreads, 0, s>>>(S, n, K, flag.p, pos.p, out->srow.p, out->Sc64.p,
                                                                out->Sc32.p, R32);
  PRDF_LAUNCH_CHECK();
  out->rows = rows;
  return PRDF_OK;
}

int ppr_add_correction(double* R, const float* E, int64_t cnt, cudaStream_t s) {
  k_add_correction<<<grid_for(cnt, kThreads), kThreads, 0, s>>>(R, E, cnt);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

int ppr_narrow(const double* x, int64_t cnt, float* y, cudaStream_t s) {
  k_narrow<<<grid_for(cnt, kThreads), kThreads, 0, s>>>(x, cnt, y);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

int ppr_widen(const float* y, int64_t cnt, double* x, cudaStream_t s) {
  k_widen_n<<<grid_for(cnt, kThreads), kThreads, 0, s>>>(y, cnt, x);
  PRDF_LAUNCH_CHECK();
  return PRDF_OK;
}

}  // namespace prdf
