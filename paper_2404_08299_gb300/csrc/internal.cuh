// Internal declarations shared by the translation units of libprdf.
#pragma once

#include "common.cuh"

namespace prdf {

constexpr int kMaxThr = 7;  // at most eight degree classes

struct PartThr {
  int n = 0;                    // number of thresholds (classes = n + 1)
  int64_t thr[kMaxThr] = {0, 0, 0, 0, 0, 0, 0};
};

// Scratch reused across calls on one graph. Calls on a graph do not overlap.
struct Workspace {
  DBuf<int64_t> scan;       // tile sums of the device-wide scan
  DBuf<int64_t> part_cnt;   // per-tile class counts of the partition
  DBuf<int64_t> part_base;  // their exclusive scan
  int64_t* host_i64 = nullptr;  // pinned host scratch, kHostSlots entries
  static constexpr int kHostSlots = 64;
  int init();
  ~Workspace();
};

// Exclusive prefix sums: out[i] = sum(in[0..i)), out[n] = total.
int exclusive_scan_u32(const uint32_t* in, int64_t n, int64_t* out, Workspace& ws, cudaStream_t s);
int exclusive_scan_i64(const int64_t* in, int64_t n, int64_t* out, Workspace& ws, cudaStream_t s);

// Alg. partition over the rows of a CSR (degree = off[v+1] - off[v]).
int partition_by_degree(const int64_t* off, int64_t n, const PartThr& t, int32_t* P, int64_t* counts_host,
                        Workspace& ws, cudaStream_t s);
// Stable partition of a list of vertex ids (in = NULL: 0..n-1) by the degree
// classes of off; desc puts the highest class first. P may not alias in.
int partition_list(const int64_t* off, const int32_t* in, int64_t n, const PartThr& t, bool desc, int32_t* P,
                   int64_t* counts_host, Workspace& ws, cudaStream_t s);

constexpr int kAdjPad = 4;

// A device CSR with optional float weights.
struct Csr {
  DBuf<int64_t> off;  // n + 1
  DBuf<int32_t> adj;  // m (+ kAdjPad in the sweep numbering: 16-byte loads may reach past the last entry)
  DBuf<float> w;      // m or empty
  int64_t m = 0;
};

// Build a CSR of unique{(rows[i], cols[i])} (plus one self-loop per row if
// self_loops), rows sorted ascending. Entries with a negative row or column
// are skipped when allow_skip is set, otherwise they are an error. Weights
// (optional) of merged duplicates: maximum; added self-loops: 1.0.
int build_csr(int32_t n, int64_t m0, const int32_t* rows, const int32_t* cols, const float* w, bool self_loops,
              bool allow_skip, Csr& out, Workspace& ws, cudaStream_t s);
// Both CSRs of a list without skipped entries.
int build_csr_pair(int32_t n, int64_t m0, const int32_t* src, const int32_t* dst, const float* w, bool self_loops,
                   Csr& out, Csr& in, Workspace& ws, cudaStream_t s);
bool radix_pair_applies(int32_t n, int64_t m0, bool self_loops);
int build_csr_pair_radix(int32_t n, int64_t m0, const int32_t* rows, const int32_t* cols, const float* w,
                         bool self_loops, Csr& out, Csr& in, Workspace& ws, cudaStream_t s);
// The same CSR by a radix sort of packed (row, column) keys (radix_build.cu):
// unweighted lists without skipped entries, m0 + n < 2^32; ids already checked.
bool radix_build_applies(int32_t n, int64_t m0, const float* w, bool allow_skip, bool self_loops);
int build_csr_radix(int32_t n, int64_t m0, const int32_t* rows, const int32_t* cols, bool self_loops, Csr& out,
                    Workspace& ws, cudaStream_t s);

// Batch update of one CSR with set semantics (Sec. 3.3): out gets rows
// (old \ D) u I in column order, merged without re-sorting (batch_update.cu).
// D: (del_rows[i], del_cols[i]), self-loops ignored; I: (ins_rows[i],
// ins_cols[i]) with weights ins_w when old is weighted (duplicates and
// re-inserted surviving edges keep the maximum). Equal to a rebuild when
// every row of old holds its own vertex. Keyed form (key, store not null):
// old's entries are ordered by key[entry], the batch's columns are keys, an
// added column c is stored as store[c], and a deletion (r, c) is a self-loop
// when key[r] == c.
int update_csr(int32_t n, const Csr& old, const int32_t* del_rows, const int32_t* del_cols, int64_t n_del,
               const int32_t* ins_rows, const int32_t* ins_cols, const float* ins_w, int64_t n_ins, Csr& out,
               Workspace& ws, cudaStream_t s, const int32_t* key, const int32_t* store);
// The same for the CSRs of G and G' (old[k] with the lists b[k]) together.
struct BatchLists {
  const int32_t *del_rows, *del_cols;
  int64_t n_del;
  const int32_t *ins_rows, *ins_cols;
  int64_t n_ins;
};
int update_csr_pair(int32_t n, const Csr* old, const BatchLists* b, const float* ins_w, Csr* out, Workspace& ws,
                    cudaStream_t s, const int32_t* key = nullptr, const int32_t* store = nullptr);

// The graph renumbered so that each in-degree class is a contiguous id range
// (new id i = vertex perm[i], perm being the in-degree partition).
struct Relabel {
  bool valid = false;
  PartThr thr;                       // in-degree classes the numbering follows
  int64_t count[kMaxThr + 1] = {};   // class sizes; class c is ids [sum(count[<c]), +count[c])
  DBuf<int32_t> perm;                // new -> old
  DBuf<int32_t> inv;                 // old -> new
  Csr in, out;                       // G' and G in the new numbering
  DBuf<double> degd, inv_deg;        // |out(i)| and 1/|out(i)| in the new numbering
  DBuf<double> kf;                   // Eq. 2 factor 1 / (1 - alpha / |out(i)|) for kf_alpha
  double kf_alpha = -1;              // alpha kf was made for (< 0: none)
  DBuf<int32_t> pout;                // out-degree partition of `out` (new ids), for marking
  int64_t pout_count[kMaxThr + 1] = {};
  bool pout_valid = false;
  uint64_t version = 0;              // bumped on every rebuild and every batch update
  // Batch updates keep the numbering: in and out are updated in place (rows
  // stay ordered by original id), so a vertex's degree may leave its class
  // bounds. Every kernel handles rows of any length; the one exception is the
  // class of in-degree <= 1, whose kernel reads no row: a vertex of that class
  // that gains an in-edge gets its bit in multi (one bit per vertex, cleared by
  // the next renumbering) and takes the general path.
  DBuf<uint32_t> multi;
  int64_t multi_count = 0;           // vertices with their bit set
  int64_t drift = 0;                 // batch entries applied since the numbering was made
};

constexpr int kHubChunk = 1024;  // edges of a chunk of the rank sweeps's longest rows

// ---- the rank loop (sweep.cu) ----

// Row shapes of a class of the sweep: a lane per row (no gather: in-degree <=
// 1, the row is [v]), a lane per row, 4, 8 or 16 lanes per row, a warp per row.
enum RowKind { kRowSelf = 0, kRowThread, kRow4, kRow8, kRow16, kRowWarp };

// A class of the sweep: its rows, their shape, about how long they are, and
// the fewest rows a unit of work takes. In DF / DF-P the affected rows are
// listed from act + list on; the rows of the warp-per-row class are listed in
// four parts by their length (entries k .. k + 3, parts 0 to 3, longest first).
struct SweepClass {
  int64_t begin, end, list;
  float deg;
  int least, kind, part;  // part: -1 whole class
};
constexpr int kMaxCls = kMaxThr + 4;

// A chunk of a long row of the sweep: entries [j0, j0 + len) of vertex v;
// chunks [first, first + parts) are the row's, row its index in the table.
struct alignas(16) SweepChunk {
  int64_t j0;
  int32_t len, v;
  int32_t first, parts, row, pad;
};
// Owner of the chunk table of the sweep's long rows [begin, n) of G'.
struct SweepChunks {
  int64_t rows = 0, max_chunks = 0;
  int first_class = 0, size = 0, above = 0;
  DBuf<uint32_t> cnt;
  DBuf<int64_t> first;       // rows + 1: exclusive scan of the chunk counts, first[rows] = number of chunks
  DBuf<SweepChunk> chunks;
  DBuf<uint4> part;          // partial sum of a chunk
  DBuf<uint32_t> done;       // chunks of a row that arrived
  uint64_t version = 0;      // numbering version it was built for
  bool valid = false;
};

// Counters of one sweep and its expansion round.
struct LoopSlot {
  unsigned long long resid;  // FP64: L-inf change (bits); FP32: low word max |dR|, high word max R (bits)
  unsigned long long fw;     // out-edges of the vertices the sweep put into deltaN
  unsigned int units;        // units handed out beyond the first of each warp
  unsigned int nlist;        // frontier entries
  unsigned int act[kMaxCls];  // DF / DF-P: affected rows of each class
};
constexpr int kLoopRing = 4;  // slots of the whole-loop kernel (a power of two)

// State and result of a loop.
struct LoopCtl {
  unsigned long long bar;    // arrivals at the grid barrier
  unsigned long long resid;  // residual word of the last sweep
  int iters;                 // sweeps run
  int timeout;               // a block gave up waiting at the grid barrier
  unsigned int nlist0;       // frontier entries of the initial marking
  unsigned int aff0;         // affected vertices at the first sweep
};

enum LoopMode { kLoopAll = 0, kLoopScan, kLoopSweep, kLoopExpand, kLoopPush };

// A frontier entry (v, k) stands for out-edges [k, k + 1) * kFrontChunk of v.
constexpr int kFrontChunk = 1024;

// Arguments of the rank loop, Real = double (FP64 sweeps) or float (FP32
// stage of the mixed-precision solves).
template <class Real>
struct SweepArgs {
  const int64_t* off;      // in-CSR offsets of G'
  const int32_t* adj;      // in-CSR sources (padded: 16-byte loads may reach past the last entry)
  Real* xa;                // x[u] = R[u] / |out(u)|; even sweeps read xa and write xb
  Real* xb;
  const Real* deg;         // |out(v)| (self-loop included)
  const Real* inv;         // 1 / |out(v)|
  const Real* kf;          // DF-P: 1 / (1 - alpha / |out(v)|) (Eq. 2's self-loop factor)
  Real alpha, c0;          // damping, (1 - alpha) / n
  Real tol;                // FP64: stop at L-inf change <= tol; FP32: at max |dR| <= tol * max R
  int self_loops;          // every vertex has exactly one self-loop (graph built with PRDF_ADD_SELF_LOOPS)
  const uint32_t* multi;   // null, or a bit per vertex: set for the in-degree <= 1 classes' vertices that
                           // gained in-edges since the numbering was made (they read their row)
  int64_t m;               // in-edges
  int32_t n;
  int max_iter;
  int mode, it0, it_first; // LoopMode; single phases: the iteration, and the one slot[1] stands for
  LoopSlot* slot;
  LoopCtl* ctl;
  // chunk table of the classes from chunk_class on: a partial sum per chunk
  // and an arrival counter (zero between sweeps) per row
  const SweepChunk* chunks;
  const int64_t* nchunk;   // number of chunks (device), null: none
  int chunk_class, chunk_size;
  uint32_t chunks_per_unit;
  uint4* hub_part;
  uint32_t* hub_done;
  // the other classes (filled by the launcher)
  SweepClass cls[kMaxCls];
  int ncls;
  // DF / DF-P / DT
  uint8_t* dV;             // affected flags (read; cleared on prune)
  uint8_t* dN;             // expand flags (set when the change exceeds tau_f)
  uint8_t* wrote;          // 1 where this vertex's slot in xn was written by the previous sweep
  Real tau_f, tau_p;
  int prune;               // DF-P (Eq. 2, prune) or DF (Eq. 1)
  int expand;              // an expansion round after each sweep
  int init_push;           // the marked batch's frontier list is expanded before the first sweep
  const int64_t* ooff;     // G (push form)
  const int32_t* oadj;
  int2* list;              // frontier entries of the round (room for n + m / kFrontChunk + 1)
  unsigned long long fthr; // the round runs in pull form when the frontier's out-edges exceed this
  int32_t* act;            // affected rows of the classes (SweepClass::list)
  int64_t scan_end;        // rows outside the chunk table
  int scan_rows;           // of them a warp scans at a time (a power of two, 32 to 1024)
};
int launch_rank_loop(const SweepArgs<double>& a, const PartThr& t, const int64_t* cb, bool exact, bool dynamic,
                     cudaStream_t s);
int launch_rank_loop(const SweepArgs<float>& a, const PartThr& t, const int64_t* cb, bool dynamic, cudaStream_t s);
// Chunk table of the rows [begin, n) longer than `above` entries (above = 0: of every row). With above > 0 the number of
// chunks is read back (max_chunks is exact), else the table has room for the most there can be.
int build_chunks(const int64_t* off, int64_t begin, int64_t n, int64_t m, int size, int above, SweepChunks& t,
                 Workspace& ws, cudaStream_t s);
// initialAffected (Alg. affected) in the sweep numbering: dV, dN and the frontier list of the first push
// (dN padded to whole 32-bit words)
int launch_mark_batch(const int32_t* del_src, const int32_t* del_dst, const uint8_t* del_mask, int64_t n_del,
                      const int32_t* ins_src, const uint8_t* ins_mask, int64_t n_ins, const int32_t* inv,
                      const int64_t* ooff, uint8_t* dV, uint8_t* dN, LoopCtl* ctl, int2* list, cudaStream_t s);

// K-column personalised PageRank (ppr.cu): one solve of
// R = alpha A R + beta S (A over the rows of off / adj / P), or one sweep of
// it. T = float (FP32 sweeps) or double (FP64 Jacobi steps), row-major
// [n, K] in the class-contiguous numbering; K here is the row stride
// (padded_cols).
template <class T>
struct PprArgs {
  const int64_t* off;
  const int32_t* adj;
  const T* P;              // P_uv of the slot
  T* Ra;                   // even sweeps read Ra and write Rb
  T* Rb;
  const T* S;              // right-hand side [n, K] (teleport, or residual / (1 - alpha))
  const int32_t* srow;     // null: S is dense; else S holds compact rows and row v is S[srow[v]] (-1: zero)
  float* res32;            // FP64: (T(R) - R) / (1 - alpha) in FP32, or null
  int K, tiles;
  T alpha, beta, inv_beta; // alpha, 1 - alpha, 1 / (1 - alpha)
  T tol;                   // FP32: stop at max|dR| <= tol * max|R|; FP64: at max|dR| <= tol
  int64_t m;               // entries of the CSR
  int max_iter, mode, it0, it_first;  // as in SweepArgs
  LoopSlot* slot;
  LoopCtl* ctl;
  // the n rows of at most row_max entries one by one, the others in the chunk table
  int64_t n;
  int row_max;
  int rows_per_unit;
  const SweepChunk* chunks;
  const int64_t* nchunk;
  int64_t max_chunks, chunk_rows;
  uint32_t chunks_per_unit;
  void* part;              // [tiles][max_chunks][tile] partial sums
  uint32_t* done;          // [tiles][chunk_rows] arrivals, zero between sweeps
};
int launch_ppr_loop(const PprArgs<float>& a, int tile, int64_t n, cudaStream_t s);
int launch_ppr_loop(const PprArgs<double>& a, int tile, int64_t n, cudaStream_t s);
// row stride of the K-column state: a multiple of four columns (16-byte FP32
// rows), except for one or two columns
inline int padded_cols(int K) { return K <= 2 ? K : (K + 3) & ~3; }

// Sparse teleport: the rows of S (double [n, K]) with a non-zero entry. When
// at most n / 4 rows are non-zero, srow[v] gets v's compact row (-1 for none),
// Sc64 / Sc32 the rows in FP64 / FP32, R32 (float [n, K]) the FP32 matrix
// (the iteration's start R = S) and rows their count; otherwise rows = 0 and
// the dense form is kept. Sweeps then read 4 bytes per vertex instead of the
// vertex's whole teleport row.
struct PprSparseRhs {
  int64_t rows = 0;
  DBuf<int32_t> srow;
  DBuf<double> Sc64;
  DBuf<float> Sc32;
};
int ppr_sparse_rhs(const double* S, int64_t n, int K, Workspace& ws, PprSparseRhs* out, float* R32, cudaStream_t s);
int ppr_add_correction(double* R, const float* E, int64_t cnt, cudaStream_t s);
int launch_grad_w(const int64_t* off, const int32_t* adj, const int32_t* perm, const int64_t* orig_off,
                  const double* lam, const double* Gs, double g_scale, const double* Rr, const double* W, int32_t n,
                  int64_t m, int K, double alpha, double* grad_w, cudaStream_t s);
int ppr_narrow(const double* x, int64_t cnt, float* y, cudaStream_t s);
int ppr_widen(const float* y, int64_t cnt, double* x, cudaStream_t s);

// Alg. affected kernels (frontier.cu). map (nullable): vertex id -> flag index.
int launch_initial_affected(const int32_t* del_src, const int32_t* del_dst, const uint8_t* del_mask, int64_t n_del,
                            const int32_t* ins_src, const uint8_t* ins_mask, int64_t n_ins, const int32_t* map,
                            uint8_t* dV, uint8_t* dN, cudaStream_t s);
// expandAffected over the out-degree partition. dF (nullable): also mark in
// dF every vertex that was not yet in dV (one round of Dynamic Traversal's
// reachability closure). fl (optional scratch): a frontier of at most fl.cap
// vertices is listed and expanded from the list, without the partition
// kernels' scan of every vertex.
struct FrontList {
  int32_t* list = nullptr;      // cap entries
  unsigned int* cnt = nullptr;  // one counter
  unsigned int cap = 0;
};
int launch_expand(const int64_t* off, const int32_t* adj, const int32_t* P, const int64_t* cb, int nclass,
                  const uint8_t* dN, uint8_t* dV, uint8_t* dF, cudaStream_t s, const FrontList& fl = FrontList());
int count_flags(const uint8_t* f, int64_t n, unsigned long long* dev_out, cudaStream_t s);

}  // namespace prdf

// The graph handle of the C ABI.
struct prdf_graph {
  int32_t n = 0;
  bool weighted = false;
  bool self_loops = true;           // every vertex has exactly one self-loop
  cudaStream_t stream = nullptr;
  prdf::Csr csr[2];                  // [PRDF_OUT] = G, [PRDF_IN] = G' in original ids (see orig_valid)
  bool orig_valid = true;            // false after a batch update until ensure_orig()
  // in-CSR slot of each out-CSR slot (original ids), kept until the edges change; for set_weights
  prdf::DBuf<uint32_t> in_slot;
  bool in_slot_valid = false;
  int64_t m = 0;                     // edges of G (self-loops included)
  prdf::PartThr thr[2];              // class thresholds per CSR
  prdf::DBuf<int32_t> P[2];          // partitions
  int64_t pcount[2][prdf::kMaxThr + 1] = {};
  bool pvalid[2] = {false, false};
  prdf::Workspace ws;
  // solver scratch
  prdf::DBuf<double> xa, xb;
  prdf::SweepChunks sweep_chunks;     // chunk table of the rank sweeps
  prdf::SweepChunks ppr_chunks_in, ppr_chunks_out;  // of G' (K-column forward) and of G (adjoint)
  prdf::DBuf<double> ppr_part;        // K-column calls: partial sum of a chunk and column
  prdf::DBuf<uint32_t> ppr_done;      // and arrivals per row and tile
  prdf::DBuf<float> ya, yb, degf, invf;  // FP32 stage state and degrees (class-contiguous numbering)
  prdf::DBuf<float> kf32;                // FP32 stage of DF-P: Eq. 2 factor
  prdf::DBuf<uint8_t> dV, dN, wrote;
  prdf::DBuf<uint8_t> dF;  // Dynamic Traversal: next frontier of the closure
  prdf::DBuf<unsigned long long> counter;
  prdf::DBuf<unsigned long long> chk;  // input checks: bad-id flag, bad-rank flag, rank sum (double bits)
  prdf::DBuf<prdf::LoopCtl> loop_ctl;    // state of a rank loop
  prdf::DBuf<prdf::LoopSlot> loop_slots; // its per-sweep counters
  prdf::DBuf<int2> loop_list;            // DF / DF-P: frontier entries of an expansion round
  prdf::DBuf<int32_t> loop_act;          // DF / DF-P / DT: affected rows of a sweep
  prdf::DBuf<int32_t> flist;             // DT: a small frontier listed for its closure round (frontier.cu)
  prdf::DBuf<unsigned int> fcnt;         // its size
  prdf::Relabel rl;                  // class-contiguous copy used by the sweeps
  // weighted graphs: transition probabilities P_uv = w_uv / sum_k w_uk
  bool ppr_valid = false;
  prdf::DBuf<double> wsum;           // sum of out-weights per vertex (sweep numbering)
  prdf::DBuf<double> pin64;          // P on the in-edge slots of rl.in
  prdf::DBuf<float> pin32;  // m + kAdjPad, the padding zero, as pout32
  prdf::DBuf<double> pout64;         // P on the out-edge slots of rl.out (adjoint)
  prdf::DBuf<float> pout32;
  // K-column scratch
  prdf::DBuf<double> S64, R64a, R64b;
  prdf::PprSparseRhs ppr_rhs;        // compact teleport rows of the last forward call (rows = 0: dense)
  prdf::DBuf<float> S32, R32a, R32b;
};

namespace prdf {
int build_relabelled(prdf_graph* g, cudaStream_t s);
int build_ppr_weights(prdf_graph* g, cudaStream_t s);
// the weights of the original-id CSRs into the sweep numbering's (rows in place)
int permute_weights(prdf_graph* g, cudaStream_t s);
// The CSRs of G and G' in original ids, derived from the sweep numbering's
// copies when a batch update has changed those (rows come out sorted, as the
// numbering keeps each row in original-id order).
int ensure_orig(prdf_graph* g, cudaStream_t s);
// |out(i)| and 1 / |out(i)| of the sweep numbering from its out-CSR (drops the cached Eq. 2 factor)
int update_degrees(prdf_graph* g, cudaStream_t s);
// the same, and the cached Eq. 2 factor, for the rows of the cnt vertices a[] (original ids) only
int update_degrees_of(prdf_graph* g, const int32_t* a, int64_t cnt, cudaStream_t s);
}
