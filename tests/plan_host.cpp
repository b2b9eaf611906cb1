// Planner internals for host tests, built together with csrc/plan.cpp.
#include "plan.h"

#include <string.h>

using namespace stiles;

static Shape shape(int nt, int b, int w, int a, int prec) {
  Shape s{nt, b, w < nt - 1 ? w : nt - 1, a, prec, 0};
  s.planes = use_planes(s);
  return s;
}

// Scratch bytes of the fused plan that a fixed scratch of `limit` bytes takes
// (tiles, planes, scheduler state), or -1 if none fits. most: the finest-cut
// plan's bytes.
extern "C" long long fixed_scratch(int nt, int b, int w, int a, int prec, long long limit, long long* most) {
  const Shape s = shape(nt, b, w, a, prec);
  const size_t w_bytes = ((size_t)Layout(s).doubles() * 8 + 255) / 256 * 256;
  Plan p;
  if (build_plan(s, PLAN_FUSED, 0, &p)) return -2;
  *most = (long long)(w_bytes + 16 * (size_t)p.plane_units + 4 * sched_state_ints(p));
  if (*most <= limit) return *most;
  if (build_small_plan(s, w_bytes, (size_t)limit, &p)) return -1;
  return validate_plan(p, s, PLAN_FUSED) ? -3 : (long long)(w_bytes + 4 * sched_state_ints(p));
}

extern "C" long long plane_bytes(int nt, int b, int w, int a, int prec) { return 16 * plane_units(shape(nt, b, w, a, prec)); }
extern "C" int planes_go_in(long long doubles, long long plane_bytes, long long device) {
  return planes_fit(doubles, plane_bytes / 16, device);
}

extern "C" void trace_pick(const unsigned long long* parts, unsigned long long* out) { trace_records(parts, out); }

extern "C" unsigned stages_run(unsigned before, unsigned used) { return stage_count(before + used); }

// Plants one fault in the fused plan's tasks that work on planes, and counts the
// parts in which the part check (that of the self-checking device build) finds it.
// which: 0 none, 1 a split's planes past the end, 2 a split's source past the end, 3 a
// product's planes past the end, 4 a product's output, 5 its input block, 6 its mirror, 7 TF_NEG on a reduced-precision
// store (whose epilogue does not negate).
extern "C" int plane_faults(int nt, int b, int w, int a, int prec, int which) {
  const Shape s = shape(nt, b, w, a, prec);
  Plan p;
  if (build_plan(s, PLAN_FUSED, 0, &p) || !p.plane_units) return -1;
  const int64_t n = Layout(s).doubles();
  const Bounds all{n, 15, p.plane_units, p.ndiag};
  for (Task& t : p.tasks) {
    const bool split = t.op == OP_SPLIT, product = t.flags & TF_PLANES;
    if (which == 1 && split) t.out = mkref(BUF_P, p.plane_units - plane_group(t.prec, t.zrows) + 1);
    if (which == 2 && split) t.cin = mkref((int)(t.cin >> BUF_SHIFT), n - 1);
    if (which == 3 && product) p.segs[t.seg0].b = mkref(BUF_P, p.plane_units);
    if (which == 4 && product) t.out = mkref(BUF_S, n - 1);
    if (which == 5 && product && t.op == OP_SYMUPD) t.cin = mkref(BUF_S, n - 1);
    if (which == 6 && product && t.op == OP_SYMUPD && !(t.flags & TF_SYM_DIAG)) t.aux = mkref(BUF_S, n - 1);
    if (which == 7 && t.op == OP_STORE && t.prec != PREC_FP64) t.flags |= TF_NEG;
  }
  int found = 0;
  for (const Task& t : p.tasks)
    for (int q = 0; q < t.parts; ++q) found += part_fault(t, q, p.segs.data(), all) != nullptr;
  return found;
}

// Two splits without an order between them. apart: of their groups (units of 16 bytes;
// the first at `apart`, the second at 0, 64 vectors x 16 of K each). Returns the race
// check's verdict.
extern "C" int two_splits(int prec, int apart) {
  Plan p;
  const int64_t group = plane_group(prec, kPlaneK);
  p.plane_units = group + apart;
  for (int k = 0; k < 2; ++k) {
    Task t;
    memset(&t, 0, sizeof(t));
    t.op = OP_SPLIT;
    t.out = mkref(BUF_P, k == 0 ? apart : 0);
    t.cin = mkref(BUF_S, 0);
    t.aux = -1;
    t.ldc = t.m = FB;
    t.n = 1;
    t.zrows = kPlaneK;
    t.parts = 4;
    t.pmode = PM_SPLIT;
    t.prec = (uint8_t)prec;
    p.tasks.push_back(t);
  }
  p.succ_off.assign(3, 0);
  return race_check_plan(p, FB * kPlaneK, 0);
}
