// Block POTRF: the in-place Cholesky factorization of one block of at most
// FB x FB in shared memory by the 128 threads of a CTA. A header of its own so
// that the host tests run it too (with the CUDA names it uses supplied, warp
// after warp in a chosen order between two block barriers).
#pragma once
#include <cstdint>

#include "plan.h"

namespace stiles {

constexpr int LDS = FB + 1;    // padded shared-memory row length (doubles)
constexpr int NTHREADS = 128;  // 4 warps: one per SM sub-partition

// In-place lower Cholesky of the n x n block X (n <= FB, padded with the
// identity to a multiple of 4) in panels of 4 columns, as L = M D^1/2: a pivot
// d_j gives the multipliers m_ij = a_ij / d_j, the later columns take
// a_ik -= m_ij a_kj, and the columns are scaled by d_j^-1/2 only when they are
// stored. What bounds it: an FP64 warp instruction holds its sub-partition's
// pipe for 64 cycles whatever its active lanes, so the pivot chain is counted
// in the FP64 instructions of the warp that runs it, and the trailing update
// (43.7k multiply-adds: 22k cycles over the four pipes) in packed elements.
// Hence
//   * 1 / d is formed in integers (recip_fixed, ~145 cycles, an rsqrt takes
//     380), beside the FP64 pipe; a pivot then costs a multiply and a
//     multiply-add on the chain;
//   * a panel runs in registers, a row per lane (its 4 pivot rows in lanes
//     0-3 of every warp that takes part, so no warp waits for another); four
//     columns keep the multiply-adds inside the panel (6) off the chain, eight
//     (28) took 2.5 times as long per panel;
//   * the trailing update takes a panel at a time; the next panel's own columns
//     take it in the next panel's registers, so that one barrier a panel is
//     enough and the next panel runs while the other warps, and then its own,
//     apply the rest (batches of 32 2 x 2 elements of the packed lower triangle,
//     shared out by their FP64 time; single elements claimed from a counter,
//     their rows found by a division, took three times as long).
// A block POTRF task takes 47 us in the median (43 to 52, the 10th and 90th percentiles)
// on a GPU that runs a factorization alone, (60, 256, 2, 50), 66 us beside the parts of
// n = 24,640 in emulated FP64 (stamped: 94k cycles): 5k until the block is in shared
// memory, 3k the first panel, 5.7k for each of the first eight of the fifteen steps and
// 2.9k for each of the last seven (the first have trailing updates of up to 13 batches, a
// panel alone is about 2.8k), 1.4k the scales, 7.4k the stores, 8k until the successors
// are released, 3k for the logdet after that. Factor and logdet of (60, 250, 2, 50):
// 36.6 ms with a column and a barrier per step and the other links of the chain as they
// were, 17.3 ms now.

constexpr int PNB = 4;           // panel width
constexpr int PROWS = 32 - PNB;  // rows below the panel's own per warp
constexpr int PMS = PNB + 1;     // row length of a multiplier buffer
// shared memory beside X (doubles from the start of the dynamic region)
constexpr int PT_M = 0;                       // two multiplier buffers, FB x PMS
constexpr int PT_PIV = PT_M + 2 * FB * PMS;   // pivots d_j
constexpr int PT_RS = PT_PIV + FB;            // scale of column j
constexpr int PT_DIAG = PT_RS + FB;           // L_jj
constexpr int PT_RCP = PT_DIAG + FB;          // 1 / L_jj
constexpr int PT_TRI = PT_RCP + FB;           // a panel's own rows left of their diagonal (row length PNB)
constexpr int PT_END = PT_TRI + FB * PNB;
// a panel's time in batches of the trailing update (16 multiply-adds of 64 cycles)
constexpr int PBATCH = 2;

// ceil(2^20 / w): e / w = (e * kInv20[w]) >> 20 for the e < 1600 walked here
struct Inv20 {
  uint32_t v[FB + 1];
  constexpr Inv20() : v{} {
    for (int w = 1; w <= FB; ++w) v[w] = ((1u << 20) + w - 1) / w;
  }
};
__constant__ const Inv20 kInv20{};

// 1 / |d| of a normal d with biased exponent in [1, 2043], correctly rounded
// but for rare cases (error below 0.51 ulp, from an estimate off by two units in its
// last place too; exact for a power of two). Newton's iteration in fixed point
// from a single-precision estimate q / 2^24 of 1 / m, d = m 2^e, m in [1, 2):
// with M = 2^52 m the residual e1 = 1 - m q / 2^24 = (2^76 - M q) / 2^76 is
// below 2^-21 and exact in 64 bits; 1 / m = q / 2^24 (1 + e1 + e1^2) to 2^-63.
#ifdef __CUDACC__
__device__ __forceinline__ float recip_estimate(float f) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  return r;
}
#endif
__device__ __forceinline__ double recip_fixed(double d) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
  const int e = (int)((bits >> 52) & 0x7ff);
  const unsigned long long M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const float f = __uint_as_float(0x3f800000u | (uint32_t)((bits >> 29) & 0x7fffffu));
  const float r = fminf(fmaxf(recip_estimate(f), 0.5f), 0.99999994f);  // the exponent of [1/2, 1)
  const uint32_t q = (__float_as_uint(r) & 0x7fffffu) | 0x800000u;
  const long long E = (long long)(0ull - M * (unsigned long long)q);
  const int Eh = (int)(E >> 24);
  const long long S = E + (((long long)Eh * Eh) >> 28);
  // 2^63 / m, truncated: 2^63 - 1 for m = 1, so it is rounded without a sign
  const unsigned long long Y = ((unsigned long long)q << 39) + (unsigned long long)(((S >> 16) * (long long)q) >> 21);
  return __longlong_as_double(((long long)(2044 - e) << 52) + (long long)((Y + 512) >> 10));
}

__device__ __forceinline__ bool recip_range(double d) {  // recip_fixed's range
  const unsigned e = (unsigned)((__double_as_longlong(d) >> 52) & 0x7ff);
  return e - 1u <= 2042u;
}

// Panel j0 .. j0 + 3 in registers: lanes 0-3 hold the panel's own rows, the
// others rows j0 + 28 cw + lane of warp cw. Writes the (unscaled) panel columns
// back to X, the multipliers to M and the pivots. A pivot whose reciprocal
// leaves the normal range (zero, subnormal, above 2^1020, not finite) has its
// column scaled by d^-1/2 at once (m = l), and a 1 left in its scale slot: the
// panel is then done again that way.
// The panel before (its multipliers Mp, columns j0 - 4 ..) has updated every column
// but this panel's: that update is applied here first (16 multiply-adds a row).
// Every warp of the panel reads the panel's own rows of X and no barrier orders those
// reads before warp 0's end, so their eliminated values go to `tri`, which nothing
// reads before the last block barrier: no word of shared memory is written by one warp
// and read by another between two barriers.
__device__ __forceinline__ void potrf_panel(double* X, double* M, const double* Mp, double* piv, double* rs, double* tri,
                                            int j0, int n, int cw) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int row = j0 + (lane < PNB ? lane : PROWS * cw + lane);
  const bool own = row < n;
  double a[PNB], a0[PNB], m[PNB], d[PNB], fin[PNB];
#pragma unroll
  for (int k = 0; k < PNB; ++k) a[k] = own ? X[row * LDS + j0 + k] : 0.0;
  double mr[PNB], up[PNB][PNB];
#pragma unroll
  for (int k = 0; k < PNB; ++k) mr[k] = j0 > 0 && own ? Mp[row * PMS + k] : 0.0;
#pragma unroll
  for (int c = 0; c < PNB; ++c)
#pragma unroll
    for (int k = 0; k < PNB; ++k) up[c][k] = j0 > 0 ? X[(j0 + c) * LDS + j0 - PNB + k] : 0.0;
#pragma unroll
  for (int k = 0; k < PNB; ++k) a[0] = fma(-mr[k], up[0][k], a[0]);
  bool range = true;
#pragma unroll
  for (int j = 0; j < PNB; ++j) {
    fin[j] = 0.0;
    d[j] = __shfl_sync(FULL, a[j], j);
    const double rd = recip_fixed(d[j]);
    range = range && recip_range(d[j]);
    if (j == 0) {  // the other columns' update runs on the FP64 pipe beside the first reciprocal
#pragma unroll
      for (int c = 1; c < PNB; ++c)
#pragma unroll
        for (int k = 0; k < PNB; ++k) a[c] = fma(-mr[k], up[c][k], a[c]);
#pragma unroll
      for (int k = 0; k < PNB; ++k) a0[k] = a[k];
    }
    double u[PNB];
#pragma unroll
    for (int k = j + 1; k < PNB; ++k) u[k] = __shfl_sync(FULL, a[j], k);
    m[j] = a[j] * rd;
#pragma unroll
    for (int k = j + 1; k < PNB; ++k) a[k] = fma(-m[j], u[k], a[k]);
  }
  if (!range) {
#pragma unroll
    for (int k = 0; k < PNB; ++k) a[k] = a0[k];
#pragma unroll
    for (int j = 0; j < PNB; ++j) {
      d[j] = __shfl_sync(FULL, a[j], j);
      const bool in = recip_range(d[j]);
      fin[j] = in ? 0.0 : 1.0;
      if (!in) a[j] *= rsqrt(d[j]);
      m[j] = in ? a[j] * recip_fixed(d[j]) : a[j];
#pragma unroll
      for (int k = j + 1; k < PNB; ++k) a[k] = fma(-m[j], __shfl_sync(FULL, a[j], k), a[k]);
    }
  }
  if (own && lane >= PNB) {
#pragma unroll
    for (int k = 0; k < PNB; ++k) {
      M[row * PMS + k] = m[k];
      X[row * LDS + j0 + k] = a[k];
    }
  } else if (cw == 0 && lane < PNB) {
#pragma unroll
    for (int k = 0; k < PNB; ++k)
      if (k < lane) tri[row * PNB + k] = a[k];
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < PNB; ++k) {
        piv[j0 + k] = d[k];
        rs[j0 + k] = fin[k];
      }
    }
  }
}

// 2 x 2 elements (rows r, r + 1; columns c, c + 1) of a trailing update by the
// panel at j0: X[r][c] -= sum_k M[r][k] X[c][j0 + k]. Elements above the
// diagonal are computed and not stored. load / apply: the operands of the next
// batch are read while the pipe works on this one.
struct PotrfTile {
  double x[2][2], m[2][PNB], u[2][PNB];
  int at;  // of (r, c); -1: none
  bool diag;
  __device__ __forceinline__ void load(const double* X, const double* M, int j0, int r, int c, bool own) {
    at = own ? r * LDS + c : -1;
    diag = r == c;
    const double *Xr = X + (own ? r * LDS + c : 0), *Mr = M + (own ? r * PMS : 0), *Xc = X + (own ? c * LDS : 0) + j0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int t = 0; t < 2; ++t) x[i][t] = Xr[i * LDS + t];
#pragma unroll
      for (int k = 0; k < PNB; ++k) m[i][k] = Mr[i * PMS + k];
#pragma unroll
      for (int k = 0; k < PNB; ++k) u[i][k] = Xc[i * LDS + k];
    }
  }
  __device__ __forceinline__ void apply(double* X) {
#pragma unroll
    for (int k = 0; k < PNB; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int t = 0; t < 2; ++t) x[i][t] = fma(-m[i][k], u[t][k], x[i][t]);
    if (at >= 0) {
      X[at] = x[0][0];
      if (!diag) X[at + 1] = x[0][1];
      X[at + LDS] = x[1][0];
      X[at + LDS + 1] = x[1][1];
    }
  }
};

// The factorization of X; `S` is the staging region. On return (after a block
// barrier) L = X diag(scale): column j times S[PT_RS + j], whose diagonal
// entry is S[PT_DIAG + j] and its reciprocal S[PT_RCP + j].
__device__ __noinline__ void potrf_smem(double* X, double* S, int n) {
  static_assert(FB % PNB == 0 && FB - PNB <= 3 * PROWS, "panels; three warps hold a panel's rows");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double *piv = S + PT_PIV, *rs = S + PT_RS, *tri = S + PT_TRI;
  const int np = (n + PNB - 1) / PNB * PNB;
  for (int e = tid; e < (np - n) * np; e += NTHREADS) {  // identity rows up to a whole panel
    const int r = n + e / np, c = e % np;
    X[r * LDS + c] = r == c ? 1.0 : 0.0;
  }
  __syncthreads();
  if (warp == 0 || (warp < 3 && PNB + PROWS * warp < np)) potrf_panel(X, S + PT_M, nullptr, piv, rs, tri, 0, np, warp);
  for (int j0 = 0; j0 + PNB < np; j0 += PNB) {
    const int j1 = j0 + PNB, j2 = j1 + PNB, pb = j0 / PNB;
    const double* M = S + PT_M + (pb & 1) * FB * PMS;
    double* Mn = S + PT_M + ((pb & 1) ^ 1) * FB * PMS;
    __syncthreads();
    // warps 0 .. npw - 1 hold the panel's rows
    const int npw = 1 + (j1 + PNB + PROWS < np) + (j1 + PNB + 2 * PROWS < np);
    if (warp < npw) potrf_panel(X, Mn, M, piv, rs, tri, j1, np, warp);
    // columns j2 .. np - 1: the lower triangle in 2 x 2 elements, h of them
    // wide (even), line a (a + 1 of them) folded with line h - 1 - a; every
    // warp gets the same time, the panel's warps less by the panel
    const int h = (np - j2) / 2, w1 = h + 1, ne = h / 2 * w1, nbatch = (ne + 31) / 32;
    const int mine = max(0, (nbatch + PBATCH * npw) / 4 - PBATCH), others = nbatch - npw * mine;
    const int each = npw == 1 ? (others + 2) / 3 : npw == 2 ? (others + 1) / 2 : others;
    int b = warp < npw ? others + mine * warp : each * (warp - npw);
    const int b1 = warp < npw ? b + mine : min(others, b + each);
    const uint32_t inv = kInv20.v[w1];
    auto load_batch = [&](PotrfTile& t, int bb) {
      const int e = 32 * bb + lane, i = (int)((e * inv) >> 20), kk = e - i * w1;
      const bool low = kk <= i;
      t.load(X, M, j0, j2 + 2 * (low ? i : h - 1 - i), j2 + 2 * (low ? kk : kk - i - 1), e < ne);
    };
    if (b < b1) {
      PotrfTile t0, t1;
      load_batch(t0, b);
#pragma unroll 1
      for (;;) {
        load_batch(t1, min(b + 1, b1 - 1));
        t0.apply(X);
        if (++b >= b1) break;
        load_batch(t0, min(b + 1, b1 - 1));
        t1.apply(X);
        if (++b >= b1) break;
      }
    }
  }
  __syncthreads();
  if (tid < n) {
    const double d = piv[tid];
    const double r = rsqrt(d);
    S[PT_DIAG + tid] = d * r;
    S[PT_RCP + tid] = r;
    rs[tid] = rs[tid] == 0.0 ? r : 1.0;
    for (int k = 0; k < tid % PNB; ++k) X[tid * LDS + tid / PNB * PNB + k] = tri[tid * PNB + k];
  }
  __syncthreads();
}

}  // namespace stiles
