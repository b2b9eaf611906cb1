// Task tables shared by the host planner (plan.cpp) and the persistent
// kernel (stiles_kernel.cu).
//
// A plan is a flat list of fine-block tasks in claim order. Every task writes
// one output block of at most FB x FB doubles:
//     acc = sum over its segments  op(A_s) * op(B_s)          (FP64)
// followed by an epilogue (Op) that combines acc with an input block and, for
// POTRF / TRSM / TRTRI, a triangular solve in shared memory. The paper's tile
// operations (Sec. III-A; Algorithms 2 and 3) are split into such tasks over
// FB x FB sub-blocks of the b x b tiles.
//
// Dependencies are counters in device memory: a task lists (counter, need)
// pairs to wait for and the counters it increments when done (the producer /
// consumer flags of Algorithm 3, one per block or block panel instead of one
// per tile).
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define STILES_HD __host__ __device__
#else
#define STILES_HD
#endif

namespace stiles {

constexpr int FB = 64;  // fine block order (rows and columns of one task's output)
constexpr int kCtasPerSm = 2;  // persistent CTAs (workers) per SM

// Buffer ids, stored in the top bits of a 64-bit element offset.
enum Buf : int { BUF_A = 0, BUF_L = 1, BUF_S = 2, BUF_W = 3, BUF_P = 4 };
constexpr int BUF_SHIFT = 60;
constexpr int64_t OFF_MASK = (int64_t(1) << BUF_SHIFT) - 1;
inline int64_t mkref(int buf, int64_t off) { return (int64_t(buf) << BUF_SHIFT) | off; }

enum Op : uint8_t {
  OP_UPD = 0,       // out = cin - acc
  OP_POTRF = 1,     // out = chol(cin - acc)           (square, lower; zero above the diagonal); aux = its
                    // columns divided by their pivots (below the diagonal) and 1 / L_jj (on it)
  OP_TRSM_RLT = 2,  // out = (cin - acc) * T^{-T}      (T lower n x n, given by aux as OP_POTRF leaves it)
  OP_TRTRI = 3,     // out = T^{-1}                    (T = aux, lower m x m; zero above)
  OP_STORE = 5,     // out = acc, or -acc (TF_NEG)
  OP_NEG = 6,       // out = -acc
  OP_SYMUPD = 7,    // out = cin - acc and its transpose into the mirror block (aux)
  OP_PREP = 8,      // served requests: one tile column of A from the shape's base values and the
                    // request's (rho, tau): band entries x rho, arrow entries as they are,
                    // diagonal tau + rho rb[i] + ra[i] (rb / ra = band / arrow absolute row sums)
  OP_ZERO = 9,      // the zrows x n block above out (L's strict upper part in a diagonal tile's
                    // block column) set to zero; off the factorization's critical path
  OP_SPLIT = 11,    // digit / piece planes of one vector group of a tile (see "Planes" below)
  OP_JOIN = 10,     // no work: one dependency point for many waiters (a tile column of L final)
};

// How a task's output block is divided among CTAs (each part runs as its own
// queue entry; the last part to finish releases the task's successors).
enum PartMode : uint8_t {
  PM_FULL = 0,   // one part: the whole block
  PM_ROWS2 = 1,  // rows [0,32) and [32,64)
  PM_QUAD4 = 2,  // the four 32 x 32 quadrants
  PM_TRI3 = 3,   // quadrants (0,0), (1,0), (1,1): a diagonal block's lower part
  PM_ROWS4 = 4,  // rows [0,16), [16,32), ..
  PM_ROWS8 = 6,  // rows [0,8), [8,16), ..
  PM_ROWS4F = 11, // rows [0,4), [4,8), ..
  PM_GRID16 = 7, // a grid of at most 4 x 4 sub-tiles of at most 16 x 16 (parts = row tiles x column tiles)
  PM_COLS2 = 9,  // columns [0,32) and [32,64) (products from planes)
  PM_SPLIT = 10, // OP_SPLIT: 16 vectors x 512 of K
  PM_TRI16 = 8,  // the sub-tiles of that grid on or below the diagonal of a square block, row by row
};

// Arithmetic of a task's block products (its epilogue is always FP64).
enum Precision : uint8_t {
  PREC_FP64 = 0,   // FP64 FMA pipe
  PREC_EMU64 = 1,  // split-precision emulated FP64: 8 fixed-point digits of 8 bits per operand (fp16
                   // planes) against per-row / per-column exponents, products on the tensor cores
  PREC_FP32X = 2,  // FP32-class: each operand's FP32 value as three bf16 pieces, products on the
                   // tensor cores with FP32 sums
};

// Task flags.
enum TaskFlag : uint8_t {
  TF_SYM_DIAG = 1,  // OP_SYMUPD on a diagonal block (mirror inside the block)
  TF_URGENT = 2,    // on the critical path: queued ahead of the buckets
  TF_CORNER = 4,    // OP_PREP of the arrow corner column
  TF_PLANES = 8,    // products from planes: the segments' operands are BUF_P refs
  TF_KCONT = 16,    // OP_SPLIT: K is the contiguous dimension of the source tile
  TF_BSIDE = 32,    // OP_SPLIT: planes of a right-hand operand
  TF_NEG = 64,      // OP_STORE: out = -acc
  TF_SMALL = 128,   // reduced-precision product of a matrix of small tiles (padding left out)
};

// Planes. The reduced-precision products of phase 2 read their operands as 16-bit
// planes (8 fp16 digits for emulated FP64, 3 bf16 pieces for the FP32-class mode)
// that OP_SPLIT tasks have written once, in the layout the tensor core reads, so a
// product part is bulk copies and MMAs with no conversion. A plane group holds
// 64 vectors (rows of a left-hand operand, columns of a right-hand one) and the
// whole K of one tile, K padded to stages of 16:
//   emulated FP64: int32 exponent of vector v in K chunk ch (512 of K) at
//   [64 ch + v], then the stages; FP32-class: the stages alone.
// A stage is NP planes x 64 vectors x 16 K in core matrices of 8 x 8;
// left-hand: plane order of the MMA's row stacks, 64 vectors each; right-hand:
// two halves of 32 vectors, planes in order.
// Offsets in BUF_P count units of 16 bytes.
constexpr int kPlaneChunk = 512;  // K per exponent (two stretches of the 256 that cells sum exactly)
constexpr int kPlaneK = 16;       // K per stage
STILES_HD inline int plane_count(int prec) { return prec == PREC_EMU64 ? 8 : 3; }
STILES_HD inline int64_t plane_stages(int k) { return (k + kPlaneK - 1) / kPlaneK; }
STILES_HD inline int64_t plane_chunks(int k) { return (k + kPlaneChunk - 1) / kPlaneChunk; }
STILES_HD inline int64_t plane_head(int prec, int k) { return prec == PREC_EMU64 ? 16 * plane_chunks(k) : 0; }
STILES_HD inline int64_t plane_group(int prec, int k) {  // units of one group
  return plane_head(prec, k) + plane_stages(k) * 128 * plane_count(prec);
}

// The count of stages a CTA has run, kept below 128: stage g is in slot g % slots and
// phase g / slots of its barriers, of which the parity counts, for 4 or 8 slots, and
// whether there was a phase before.
STILES_HD inline uint32_t stage_count(uint32_t n) { return n < 64 ? n : 64 + n % 64; }

// Sub-tile of part q of an m x n block (rm or cn <= 0: nothing to do).
struct Sub {
  int r0, c0, rm, cn;
};

STILES_HD inline Sub part_sub(int pmode, int m, int n, int q) {
  Sub s{0, 0, m, n};
  int dim = 0;  // sub-tile order of the grid modes
  switch (pmode) {
    case PM_ROWS2: s.r0 = 32 * q; s.rm = 32; break;
    case PM_ROWS4: s.r0 = 16 * q; s.rm = 16; break;
    case PM_ROWS8: s.r0 = 8 * q; s.rm = 8; break;
    case PM_ROWS4F: s.r0 = 4 * q; s.rm = 4; break;
    case PM_COLS2: s.c0 = 32 * q; s.cn = 32; break;
    case PM_QUAD4: dim = 32; s.r0 = 32 * (q & 1); s.c0 = 32 * (q >> 1); break;
    case PM_TRI3: dim = 32; s.r0 = q == 0 ? 0 : 32; s.c0 = q == 2 ? 32 : 0; break;
    case PM_GRID16: {
      const int pr = (m + 15) / 16;
      dim = 16;
      s.r0 = 16 * (q % pr);
      s.c0 = 16 * (q / pr);
      break;
    }
    case PM_TRI16: {
      const int r = q >= 6 ? 3 : q >= 3 ? 2 : q >= 1 ? 1 : 0;
      dim = 16;
      s.r0 = 16 * r;
      s.c0 = 16 * (q - r * (r + 1) / 2);
      break;
    }
    default: break;
  }
  if (dim) s.rm = s.cn = dim;
  if (s.rm > m - s.r0) s.rm = m - s.r0;
  if (s.cn > n - s.c0) s.cn = n - s.c0;
  return s;
}

struct Seg {       // acc += op(A) (m x k) * op(B) (k x n)
  int64_t a, b;    // buffer refs (mkref) of element (0,0) of the stored operands
  int32_t lda, ldb;
  int32_t k;       // inner length
  int32_t trans;   // bit 0: op(A) = A^T ; bit 1: op(B) = B^T
};

struct Wait {
  int32_t ctr;
  int32_t need;    // wait until counter >= need
};

struct Task {        // 80 bytes
  int64_t out;       // ref of the output block
  int64_t cin;       // ref of the input block (OP_UPD/POTRF/TRSM_RLT/SYMUPD) or -1
  int64_t aux;       // ref of the triangular block (TRSM/TRTRI) or the mirror block (SYMUPD) or -1
  int32_t ldo, ldc, ldx;
  int16_t m, n;      // output rows / columns (<= FB)
  int32_t seg0, nseg;
  int32_t succ0, nsucc;  // its successors: succ[succ0 .. succ0 + nsucc) (who counts it off them: counts_parts)
  int32_t diag;      // POTRF: index of its logdet partial sum
  int32_t zrows;     // ZERO: rows above the block in its tile column to zero (L's strict upper part)
  int32_t gcol;      // POTRF: 0-based global column of the block's first pivot
  uint8_t op;        // op, flags, parts and pmode share one aligned 32-bit word (read on
  uint8_t flags;     // their own by the finisher of a predecessor); flags: TaskFlag bits
  uint8_t parts;     // 1..16 queue entries (see PartMode)
  uint8_t pmode;
  uint8_t prec;      // Precision of the block products
};
static_assert(sizeof(Task) == 80 && offsetof(Task, op) % 4 == 0, "task layout");

// ---- bounds of a task's accesses -----------------------------------------
// The buffers of a launch: doubles in each of A, L, Sigma, scratch tiles, which of
// them are there (a bit each), units of planes, logdet slots.
struct Bounds {
  int64_t doubles;
  unsigned present;
  int64_t plane_units;
  int ndiag;
};
STILES_HD inline bool ref_in(const Bounds& b, int64_t ref, int64_t lo, int64_t hi) {  // [ref + lo, ref + hi]
  const int buf = (int)(ref >> BUF_SHIFT);
  const int64_t off = ref & OFF_MASK;
  return ref >= 0 && buf < 4 && ((b.present >> buf) & 1) && off + lo >= 0 && off + hi < b.doubles;
}
STILES_HD inline bool planes_in(const Bounds& b, int64_t ref, int64_t len) {
  return ref >= 0 && (ref >> BUF_SHIFT) == BUF_P && (ref & OFF_MASK) + len <= b.plane_units;
}

// What is wrong with part q of a task (every kind but OP_PREP): an access outside the
// launch's buffers, or a part mode that its kernel does not take; null if nothing is.
// The host validates whole tables with it, the self-checking device build every
// part before it runs.
STILES_HD inline const char* part_fault(const Task& t, int q, const Seg* segs, const Bounds& b) {
  if (t.op == OP_JOIN) return t.parts != 1 || t.nseg != 0 ? "join with work" : nullptr;  // no access
  if (t.m < 1 || t.n < 1 || t.m > FB || t.n > FB || t.op > OP_SPLIT || t.op == OP_PREP) return "unknown task";
  if (t.op == OP_SPLIT) {
    const int64_t left = t.zrows - t.gcol, most = kPlaneChunk * (int64_t)(t.parts / 4), kc = left < most ? left : most;
    const bool kcont = t.flags & TF_KCONT;
    return t.parts % 4 || t.gcol % kPlaneChunk || kc < 1 || t.prec == PREC_FP64 || most - kPlaneChunk >= left ||
                   !ref_in(b, t.cin, 0,
                           kcont ? (t.m - 1) * (int64_t)t.ldc + kc - 1 : t.m - 1 + (kc - 1) * (int64_t)t.ldc) ||
                   !planes_in(b, t.out, plane_group(t.prec, t.zrows))
               ? "split out of bounds"
               : nullptr;
  }
  if (t.op == OP_ZERO)  // zrows x n above the block
    return t.parts != 1 || t.nseg != 0 || t.zrows < 1 ||
                   !ref_in(b, t.out, -(int64_t)t.zrows, -1 + (int64_t)(t.n - 1) * t.ldo)
               ? "zeroed rows out of bounds"
               : nullptr;
  const Sub s = part_sub(t.pmode, t.m, t.n, q);
  if ((t.pmode == PM_TRI16 || t.pmode == PM_TRI3) && t.m != t.n) return "triangle parts on a block that is not square";
  if (t.prec != PREC_FP64 && (t.pmode != PM_COLS2 || s.cn > 32)) return "reduced-precision part other than 64 x 32";
  if (t.prec != PREC_FP64 && t.op != OP_UPD && t.op != OP_NEG && t.op != OP_STORE && t.op != OP_SYMUPD)
    return "reduced precision on a triangular task";
  if (t.prec != PREC_FP64 && (t.flags & TF_NEG)) return "negated reduced-precision store";
  if (s.rm <= 0 || s.cn <= 0) return nullptr;
  const int r0 = s.r0, c0 = s.c0, r1 = r0 + s.rm - 1, c1 = c0 + s.cn - 1;
  for (int g = t.seg0; g < t.seg0 + t.nseg; ++g) {
    const Seg x = segs[g];
    if (x.k <= 0) return "empty segment";
    if (t.flags & TF_PLANES) {
      const int64_t len = plane_group(t.prec, x.k);
      if (t.prec == PREC_FP64 || !planes_in(b, x.a, len) || !planes_in(b, x.b, len)) return "planes out of bounds";
      continue;
    }
    const int64_t amax = (x.trans & 1) ? (x.k - 1) + (int64_t)r1 * x.lda : r1 + (int64_t)(x.k - 1) * x.lda;
    const int64_t amin = (x.trans & 1) ? (int64_t)r0 * x.lda : r0;
    const int64_t bmax = (x.trans & 2) ? c1 + (int64_t)(x.k - 1) * x.ldb : (x.k - 1) + (int64_t)c1 * x.ldb;
    const int64_t bmin = (x.trans & 2) ? c0 : (int64_t)c0 * x.ldb;
    if (!ref_in(b, x.a, amin, amax)) return "segment A out of bounds";
    if (!ref_in(b, x.b, bmin, bmax)) return "segment B out of bounds";
  }
  if (!ref_in(b, t.out, r0 + (int64_t)c0 * t.ldo, r1 + (int64_t)c1 * t.ldo)) return "output out of bounds";
  const bool cin = t.op == OP_UPD || t.op == OP_POTRF || t.op == OP_TRSM_RLT || t.op == OP_SYMUPD;
  if (cin && !ref_in(b, t.cin, r0 + (int64_t)c0 * t.ldc, r1 + (int64_t)c1 * t.ldc)) return "input out of bounds";
  const int tri = t.op == OP_TRSM_RLT || t.op == OP_POTRF ? t.n : t.op == OP_TRTRI ? t.m : 0;  // order of aux
  if (tri && !ref_in(b, t.aux, 0, (tri - 1) + (int64_t)(tri - 1) * t.ldx)) return "T out of bounds";
  if (t.op == OP_SYMUPD && !(t.flags & TF_SYM_DIAG) && !ref_in(b, t.aux, c0 + (int64_t)r0 * t.ldx, c1 + (int64_t)r1 * t.ldx))
    return "mirror out of bounds";
  if (t.op == OP_POTRF && (t.diag < 0 || t.diag >= b.ndiag)) return "logdet slot out of range";
  return nullptr;
}

}  // namespace stiles

#ifndef __CUDACC_RTC__
#include <vector>

namespace stiles {

enum PlanKind : int { PLAN_FACTOR = 0, PLAN_SELINV = 1, PLAN_FUSED = 2 };

// Tuning code of a plan (bit fields; 0 = the defaults). It changes how work is
// cut into tasks, never what is computed: bits 2-5 only re-partition output
// blocks among CTAs (bit-identical results), bits 0-1 regroup the factor's
// update terms (the same sums, rounded at other points).
//   bits 0-1  factor: source block columns per update task for tile columns
//             older than k-1 (0: 8, 1: 4, 2: 16, 3: 32)
//   bits 2-3  phase 2: parts of an off-diagonal Sigma block task
//             (0: four 32 x 32 quadrants, 1: two 32-row halves, 2: whole block)
//   bits 4-5  factor: parts of the newest update of an off-diagonal block
//             (0: four quadrants, 1: whole block)
//   bit 6     reduced-precision plans: the block updates inside a diagonal
//             tile (the SYRK / GEMM steps of that tile's POTRF) also run in
//             the reduced precision (0: they stay FP64, so that the whole
//             diagonal-tile POTRF is true FP64). This one changes rounding.
enum : int { kTuneBits = 7 };
inline int tune_chunk_old(int t) { const int v[4] = {8, 4, 16, 32}; return v[t & 3]; }
inline int tune_p2_split(int t) { return (t >> 2) & 3; }
inline int tune_upd_split(int t) { return (t >> 4) & 3; }
inline bool tune_lower_diag(int t) { return (t >> 6) & 1; }
inline bool tune_valid(int t) { return t >= 0 && t < (1 << kTuneBits) && tune_p2_split(t) <= 2 && tune_upd_split(t) <= 1; }

struct Shape {
  int nt, b, w, a;  // w already clipped to nt-1
  int prec = PREC_FP64;  // precision of the off-diagonal bulk products (Precision)
  int tune = 0;          // tuning code (see above)
  int sel0 = 0;          // selected inversion of tile columns >= sel0 only (their phase 1 and 2)
  bool planes = false;   // reduced precisions: phase-2 products from planes
  bool coarse = false;   // FP64 tasks in at most four parts (the same results, fewer queue slots)
};

// Whether the phase-2 products of a (reduced-precision) shape read planes: a rule
// on its sizes, with its reasons at the definition.
bool use_planes(const Shape& s);
// Units of 16 bytes that they take, beside the scratch tiles.
int64_t plane_units(const Shape& s);
// Whether buffers of `doubles` doubles (A, L, Sigma and the scratch tiles) and the
// planes go into a device of `device_bytes`, a sixteenth of which is left to tables and
// the runtime: a matrix that fills the device runs without planes, as it has to.
inline bool planes_fit(int64_t doubles, int64_t units, int64_t device_bytes) {
  return 32 * doubles + 16 * units <= device_bytes / 16 * 15;
}

// A task with few successors is counted off them by each of its parts as it
// finishes (one atomic per successor and part, no join of the parts on the
// critical path); one with many by the last of its parts.
constexpr int kPartSucc = 16;
STILES_HD inline bool counts_parts(const Task& t) { return t.nsucc <= kPartSucc; }

// Dynamic schedule: a task becomes ready when the last part of its last
// predecessor finishes (device counter rem[t], initialised to rem0[t]) and is
// pushed into the bucket of its queue position (by bottom level);
// workers pop from the earliest non-empty bucket. Buckets hold kTasksPerBucket
// consecutive tasks of that order.
constexpr int kTasksPerBucket = 64;
constexpr int kMaxParts = 16;  // parts of one task; a queue entry is kMaxParts * task + part
constexpr int kMaxTasks = (1 << 27) - 1;  // entries stay positive 32-bit integers

// Trace: a record per part on the device, four per task for the caller: record r is
// the one of the parts r, r + 4, .. that completed the task, else their last to end.
constexpr int kTraceWords = 4;
constexpr unsigned long long kTraceLast = 1ull << 9;  // in a record's last word
inline void trace_records(const unsigned long long* parts, unsigned long long* out) {
  for (int r = 0; r < 4; ++r) {
    const unsigned long long* best = parts + kTraceWords * r;
    for (int q = r + 4; q < kMaxParts; q += 4) {
      const unsigned long long* x = parts + kTraceWords * q;
      const bool last = x[3] & kTraceLast, best_last = best[3] & kTraceLast;
      if (last != best_last ? last : x[2] > best[2]) best = x;
    }
    for (int i = 0; i < kTraceWords; ++i) out[kTraceWords * r + i] = best[i];
  }
}

struct Plan {
  int64_t plane_units = 0;  // BUF_P: units of 16 bytes (0: no product reads planes)
  std::vector<Task> tasks;  // in queue order
  std::vector<Seg> segs;
  std::vector<Wait> waits;  // counter form of the dependencies (host checks)
  std::vector<int32_t> sigs;
  std::vector<int64_t> wait_off;  // waits of task t: waits[wait_off[t] .. wait_off[t+1])
  std::vector<int64_t> sig_off;   // signalled counters of task t: sigs[sig_off[t] .. sig_off[t+1])
  std::vector<int32_t> indeg;     // predecessors per task
  std::vector<int32_t> rem0;      // device counter's start value: predecessors, those that count parts by their parts
  std::vector<int32_t> succ_off;  // successors: succ[succ_off[t] .. succ_off[t+1])
  std::vector<int32_t> succ;
  std::vector<int32_t> soff;      // slots of bucket b: [soff[b], soff[b+1]) (one per part)
  std::vector<int32_t> slots0;    // initial bucket slots: ready tasks at the front, -1 elsewhere
  std::vector<int32_t> tail0;     // initial ready parts per bucket
  std::vector<int32_t> uslots0;   // initial urgent queue (ready urgent parts first, -1 elsewhere)
  int32_t urgent_parts = 0;       // capacity of the urgent queue
  int32_t urgent_tail0 = 0;
  int32_t nbuckets = 0;
  int32_t nctr = 0;         // dependency counters used
  int32_t ndiag = 0;        // logdet partial sums (one per POTRF task)
  double flops = 0;         // algorithmic flops (tile-operation convention)
  double flops_lowered = 0; // the part of them run as block products in the plan's reduced precision
  long long tile_gemms = 0; // phase-2 (tile, tile) products
  double cp_ns = 0;         // critical path of the estimated task graph
  double makespan_ns = 0;   // list-schedule makespan on `workers` workers
};

// Packed band+arrow layout (see include/stiles.h).
struct Layout {
  int nt, b, w, a;
  int64_t colstride;
  explicit Layout(const Shape& s)
      : nt(s.nt), b(s.b), w(s.w), a(s.a), colstride((int64_t)(1 + s.w) * s.b * s.b + (int64_t)s.a * s.b) {}
  int rows(int i) const { return i == nt ? a : b; }
  int last() const { return a > 0 ? nt : nt - 1; }
  int nsub(int k) const { return k >= nt ? 0 : (nt - 1 - k < w ? nt - 1 - k : w); }
  int64_t doubles() const { return (int64_t)nt * colstride + (int64_t)a * a; }
  int64_t tile(int i, int k) const {
    if (k == nt) return (int64_t)nt * colstride;
    if (i == nt) return (int64_t)k * colstride + (int64_t)(1 + w) * b * b;
    return (int64_t)k * colstride + (int64_t)(i - k) * b * b;
  }
  int nblk(int i) const { return (rows(i) + FB - 1) / FB; }
  int bdim(int i, int r) const { int m = rows(i) - r * FB; return m < FB ? m : FB; }
  int64_t blk(int i, int k, int r, int c) const { return tile(i, k) + (int64_t)r * FB + (int64_t)c * FB * rows(i); }
  void structure(int k, std::vector<int>& out) const {
    out.clear();
    if (k >= nt) return;
    for (int i = k + 1; i <= k + nsub(k); ++i) out.push_back(i);
    if (a > 0) out.push_back(nt);
  }
};

// 32-bit words of a launch's scheduler state (laid out in stiles_device.h).
inline size_t sched_state_ints(int ntasks, int nbuckets, int nslots, int ucap) {
  const int ngroups = (nbuckets + 31) / 32, nsuper = (ngroups + 31) / 32;
  return 2 * (size_t)ntasks + (size_t)nslots + 3 * (size_t)nbuckets + (size_t)ngroups +
         (size_t)nsuper + (size_t)(ucap > 0 ? ucap : 1) + 32;
}
inline size_t sched_state_ints(const Plan& p) {
  return sched_state_ints((int)p.tasks.size(), p.nbuckets, (int)p.slots0.size(), p.urgent_parts);
}

// Build the task table of one plan kind, ordered by bottom level; workers > 0:
// also the makespan of its list schedule on so many workers (statistics).
// Returns 0 or a negative stiles status code.
int build_plan(const Shape& s, PlanKind kind, int workers, Plan* out);

// The fused table of a shape for a scratch of `limit` bytes that its ordinary table
// exceeds: without planes, then with fewer parts as well. `w_bytes`: of the scratch
// tiles, which the scheduler state follows. STILES_ERR_TOO_LARGE if none fits.
int build_small_plan(Shape s, size_t w_bytes, size_t limit, Plan* out);

// Consistency check of a task table: every wait names an existing counter
// that enough tasks signal, and every such producer precedes the waiter in
// claim order (the condition under which claim-order execution cannot
// deadlock). Returns 0 or STILES_ERR_PLAN.
int check_plan(const Plan& p);

// Host emulation of a launch of the plan (bounds of every access, queue
// capacities, every task released once). Returns 0 or STILES_ERR_PLAN.
int validate_plan(const Plan& p, const Shape& s, int kind);
// The same with an explicit buffer length (doubles in each of A, L, Sigma and
// the scratch's packed part), for batch plans.
int validate_plan_len(const Plan& p, int64_t buf_doubles, int kind);
// Host race check of a plan (see plan.cpp); plant = 1 plants a race first.
int race_check_plan(const Plan& p, int64_t buf_doubles, int plant, bool serve = false);

// Fused task table of one shape for the request server: as the fused plan,
// plus one OP_PREP task per tile column that writes the request's A (in the
// L buffer) from the shape's base values; every task that reads a block of A
// waits for the PREP of its tile column, and the PREP tasks are the only
// roots. PREP fields: out = tile column slot (BUF_L), cin = the same slot of
// the base values (BUF_A), aux = rb of the column's first row (BUF_A; ra
// follows rb at distance gcol = n), ldo = b, ldc = a, ldx = present
// sub-diagonal tiles, zrows = w, diag = first row of the column.
int build_serve_template(const Shape& s, int workers, Plan* out);

// One fused (factor + selected inversion) task table for a batch of
// independent matrices: matrix m's tiles live at offset base[m] (doubles) of
// each of the shared A, L, Sigma and scratch buffers; its tasks, counters and
// logdet slots are renumbered into one table and ordered by one list
// schedule over all of them, so the small matrices fill the GPU beside the
// critical paths of the large ones. diag_base[m] .. diag_base[m+1] are the
// logdet / pivot slots of matrix m. Returns 0 or a negative status code.
int build_batch_plan(const std::vector<Shape>& shapes, const std::vector<int64_t>& base, int workers, Plan* out,
                     std::vector<int32_t>* diag_base);

}  // namespace stiles
#endif
