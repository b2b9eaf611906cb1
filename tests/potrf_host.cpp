// The block POTRF of csrc/block_potrf.cuh on the host, for tests: 128 fibers
// stand for its threads. Between two block barriers the warps run one after
// the other, in an order that the caller chooses (as if every other warp were
// late), and a warp's lanes run up to each shuffle in turn. A result that
// depends on the order shows a race between warps.
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#define __device__
#define __constant__
#define __forceinline__ inline
#define __noinline__

struct Dim {
  unsigned x;
};
static Dim threadIdx;

static inline long long __double_as_longlong(double v) {
  long long r;
  memcpy(&r, &v, 8);
  return r;
}
static inline double __longlong_as_double(long long v) {
  double r;
  memcpy(&r, &v, 8);
  return r;
}
static inline uint32_t __float_as_uint(float v) {
  uint32_t r;
  memcpy(&r, &v, 4);
  return r;
}
static inline float __uint_as_float(uint32_t v) {
  float r;
  memcpy(&r, &v, 4);
  return r;
}
static inline double rsqrt(double v) { return 1.0 / std::sqrt(v); }
using std::fma;
using std::max;
using std::min;

void __syncthreads();
double __shfl_sync(unsigned mask, double v, int src);

namespace stiles {
static int estimate_ulp = 0;  // added to the last place of the single-precision estimate
static inline float recip_estimate(float f) { return __uint_as_float(__float_as_uint(1.0f / f) + estimate_ulp); }
}  // namespace stiles

#include "block_potrf.cuh"

namespace {

constexpr int kThreads = stiles::NTHREADS, kStack = 1 << 16;
enum State { RUN, SHUFFLE, BARRIER, DONE };
ucontext_t scheduler, fiber[kThreads];
std::vector<char> stacks;
State state[kThreads];
double slot[kThreads];
int current;
double *blockX, *blockS;
int blockN;

void yield(State s) {
  state[current] = s;
  swapcontext(&fiber[current], &scheduler);
}

void body() {
  stiles::potrf_smem(blockX, blockS, blockN);
  yield(DONE);
}

void resume(int t) {
  current = t;
  threadIdx.x = (unsigned)t;
  state[t] = RUN;
  swapcontext(&scheduler, &fiber[t]);
}

}  // namespace

void __syncthreads() { yield(BARRIER); }

double __shfl_sync(unsigned, double v, int src) {
  slot[current] = v;
  yield(SHUFFLE);  // every lane has stored its value
  const double r = slot[current / 32 * 32 + src % 32];
  yield(SHUFFLE);  // every lane has read
  return r;
}

// Factors the lower triangle of the n x n column-major A. order: the warps'
// order, four digits. L (lower, column-major) and the pivots' 1 / L_jj.
// Returns 0, or 1 if a shuffle was not reached by its whole warp.
extern "C" int potrf_host(const double* A, int n, int order, double* L, double* rcp) {
  using namespace stiles;
  std::vector<double> X(FB * LDS, std::nan("")), S(PT_END, std::nan(""));
  for (int c = 0; c < n; ++c)
    for (int r = 0; r < n; ++r) X[r * LDS + c] = A[r + c * n];
  blockX = X.data();
  blockS = S.data();
  blockN = n;
  stacks.resize((size_t)kThreads * kStack);
  for (int t = 0; t < kThreads; ++t) {
    getcontext(&fiber[t]);
    fiber[t].uc_stack.ss_sp = stacks.data() + (size_t)t * kStack;
    fiber[t].uc_stack.ss_size = kStack;
    fiber[t].uc_link = &scheduler;
    makecontext(&fiber[t], body, 0);
    state[t] = RUN;
  }
  for (;;) {
    for (int o = order, k = 0; k < 4; ++k, o /= 10) {
      const int w0 = 32 * (o % 10);
      while (state[w0] == RUN || state[w0] == SHUFFLE) {
        for (int t = w0; t < w0 + 32; ++t) resume(t);
        for (int t = w0; t < w0 + 32; ++t)
          if (state[t] != state[w0]) return 1;
      }
    }
    if (std::all_of(state, state + kThreads, [](State s) { return s == DONE; })) break;
    if (!std::all_of(state, state + kThreads, [](State s) { return s == BARRIER; })) return 1;
    for (int t = 0; t < kThreads; ++t) state[t] = RUN;
  }
  for (int c = 0; c < n; ++c) {
    rcp[c] = S[PT_RCP + c];
    for (int r = 0; r < n; ++r)
      L[r + c * n] = r < c ? 0.0 : r == c ? S[PT_DIAG + c] : X[r * LDS + c] * S[PT_RS + c];
  }
  return 0;
}

// 1 / |d| from an estimate off by `ulp` units in the last place.
extern "C" double recip_host(double d, int ulp) {
  stiles::estimate_ulp = ulp;
  const double r = stiles::recip_fixed(d);
  stiles::estimate_ulp = 0;
  return r;
}
