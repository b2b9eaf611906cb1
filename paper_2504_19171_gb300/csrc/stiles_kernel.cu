// Persistent dependency-driven kernel for tiled Cholesky and two-phase
// selected inversion on GB300 (sm_103a).
//
// Two CTAs per SM (each 4 warps) run task parts until every part of the plan
// has been executed. A task becomes ready when its last predecessor finishes
// (per-task predecessor counters, decremented by the finishing task: the
// device form of Algorithm 3's "WaitForTile / SignalTileReady" flags); the
// finisher pushes its parts into a queue, and idle workers claim parts with
// fetch-and-add on availability counters. Static plans queue parts in
// buckets of the host's critical-path order behind an urgent FIFO for the
// factorization's frontier; the request server (serve mode) uses three FIFO
// rings and activates new requests from a host-mapped inbox while it runs.
// Every wait is bounded by %globaltimer and ends the launch with a TIMEOUT
// status instead of hanging.
//
// FP64 has no tensor-core path on GB300 (tcgen05 has no f64 kind), so the
// FP64 block products run on the FP64 FMA pipe: 2 DFMA per clock per SM,
// reached with 4 warps. Each task stages FB x KC panels of its operands in
// shared memory (L2-only loads, so data published by other SMs is never read
// from a stale L1 line) and accumulates up to a 64 x 64 block in registers
// (4 x 8 per thread). The reduced-precision modes replace the products of
// the bulk tasks by split-precision digit products on the tensor cores
// (tcgen05 MMAs from shared memory into tensor memory): 8 fixed-point digits
// per operand for emulated FP64, 3 bf16 pieces for the FP32-class mode. In the
// end-to-end call the matrix may live in page-locked host memory (read over the host link by the tasks that first
// load each block) and every final Sigma write is repeated into a host
// buffer, so the transfers overlap the computation.
#include <cuda/atomic>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <mutex>

#include "block_potrf.cuh"
#include "plan.h"
#include "stiles_device.h"
#include "tcgen05.cuh"

namespace stiles {

constexpr int KC = 32;  // K chunk staged in shared memory
static_assert(PT_END <= 2 * KC * LDS, "the block POTRF's data fits in the staging region");

__device__ __forceinline__ double* resolve(const KParams& p, int64_t ref) {
  return p.buf[ref >> BUF_SHIFT] + (ref & OFF_MASK);
}

// Task-table reads. A request server rewrites table ranges (copy engine)
// while the kernel runs; a worker reads a task only after the acquire load of
// the queue slot that delivered it, which is ordered after the host's
// publication (system-scope release / acquire on the inbox, then release /
// acquire through the queues), so plain loads see the new rows. (Loading
// whole rows with L2-only vector loads instead costs registers the block
// products need.)
__device__ __forceinline__ Task load_task(const KParams& p, int t) { return p.tasks[t]; }

__device__ __forceinline__ Seg load_seg(const KParams& p, int g) { return p.segs[g]; }

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int load_relaxed_flag(int* a) {
  return cuda::atomic_ref<int, cuda::thread_scope_device>(*a).load(cuda::memory_order_relaxed);
}

__device__ __forceinline__ int load_acquire_i(const int* a) {
  return cuda::atomic_ref<int, cuda::thread_scope_device>(*const_cast<int*>(a)).load(cuda::memory_order_acquire);
}

__device__ __forceinline__ void store_release_i(int* a, int v) {
  cuda::atomic_ref<int, cuda::thread_scope_device>(*a).store(v, cuda::memory_order_release);
}

// Host-mapped memory (request server control block).
__device__ __forceinline__ int load_acquire_sys(const int* a) {
  return cuda::atomic_ref<int, cuda::thread_scope_system>(*const_cast<int*>(a)).load(cuda::memory_order_acquire);
}

__device__ __forceinline__ void store_release_sys(unsigned* a, unsigned v) {
  cuda::atomic_ref<unsigned, cuda::thread_scope_system>(*a).store(v, cuda::memory_order_release);
}

// Record a TIMEOUT (first error wins) and stop every worker.
__device__ void raise_timeout(const KParams& p, long long where) {
  if (atomicCAS(&p.st->code, 0, STILES_DEV_TIMEOUT) == 0) p.st->info = (unsigned long long)where;
  atomicExch(&p.st->abort, 1);
}

// Record the first violation of a table or queue invariant (what, task,
// part) and stop every worker (STILES_DEV_CHECK, reported as a plan error).
__device__ void check_fail(const KParams& p, int what, long long t, int q) {
  if (atomicCAS(&p.st->code, 0, STILES_DEV_CHECK) == 0)
    p.st->info = ((unsigned long long)(t & 0xffffffffll) << 16) | ((unsigned long long)q << 8) | (unsigned)what;
  atomicExch(&p.st->abort, 1);
}

#ifdef STILES_CHECKED
// Self-checking build: every invariant below is checked.
#define STILES_CHECK(cond, what, t, q) \
  do {                                  \
    if (!(cond)) check_fail(p, what, t, q); \
  } while (0)
#else
#define STILES_CHECK(cond, what, t, q) \
  do {                                  \
  } while (0)
#endif

// Order of the scheduler's memory operations. A part's writes are released by
// one fence of the finishing warp (its block barrier made them that warp's
// past), after which relaxed atomics count it off; whoever brings a counter to
// zero fences again (it takes on the other finishers' writes) and publishes
// queue slots with relaxed stores. A worker takes a slot with an acquire load,
// and its block barrier passes that on to the other warps.
__device__ __forceinline__ void fence_dev() { cuda::atomic_thread_fence(cuda::memory_order_acq_rel, cuda::thread_scope_device); }

__device__ __forceinline__ void store_relaxed_i(int* a, int v) {
  cuda::atomic_ref<int, cuda::thread_scope_device>(*a).store(v, cuda::memory_order_relaxed);
}

__device__ __forceinline__ int add_relaxed_i(int* a, int v) {
  return cuda::atomic_ref<int, cuda::thread_scope_device>(*a).fetch_add(v, cuda::memory_order_relaxed);
}

// The word of a task row that a releaser needs (op, flags, parts, pmode).
struct TaskWord {
  uint32_t w;
  __device__ __forceinline__ int op() const { return (int)(w & 0xffu); }
  __device__ __forceinline__ int flags() const { return (int)((w >> 8) & 0xffu); }
  __device__ __forceinline__ int parts() const { return (int)((w >> 16) & 0xffu); }
};
static_assert(offsetof(Task, flags) == offsetof(Task, op) + 1 && offsetof(Task, parts) == offsetof(Task, op) + 2,
              "task word");

// Plain load, as load_task (a request server's rows are ordered by the
// acquire of the slot that delivered a task of the same request).
__device__ __forceinline__ TaskWord load_task_word(const KParams& p, int t) {
  return {*reinterpret_cast<const uint32_t*>(&p.tasks[t].op)};
}

__device__ void serve_push(const KParams& p, int t, TaskWord tw, int q0);

// Push parts q0 .. of a ready task (one slot per part, value kMaxParts t +
// part, so that the parts run on different CTAs): urgent tasks into their
// FIFO, the others into the bucket of their queue position. The slots are
// reserved (tail), stored, and only then counted as available. The caller has
// fenced.
__device__ __forceinline__ void push_task(const KParams& p, int t, TaskWord tw, int q0) {
  if (p.serve) {
    serve_push(p, t, tw, q0);
    return;
  }
  const int parts = tw.parts() - q0;
  if (parts <= 0) return;
  // The queue capacities are checked in every build (one compare on an
  // atomic path): a table that would overflow a queue stops the launch with
  // a check failure instead of writing past the slots.
  if (tw.flags() & TF_URGENT) {
    const int pos = add_relaxed_i(p.q.lo + 8, parts);
    if (pos + parts > p.ucap) {
      check_fail(p, 1, t, 0);
      return;
    }
    for (int q = 0; q < parts; ++q) store_relaxed_i(p.q.uslots + pos + q, kMaxParts * t + q0 + q);
    atomicAdd(p.q.lo + 24, parts);
    return;
  }
  const int b = t / kTasksPerBucket;
  if (b >= p.nbuckets || t < 0) {
    check_fail(p, 2, t, 0);
    return;
  }
  const int s0 = p.soff[b], cap = p.soff[b + 1] - s0;
  const int pos = add_relaxed_i(p.q.tail + b, parts);
  if (pos + parts > cap) {
    check_fail(p, 3, t, 0);
    return;
  }
  for (int q = 0; q < parts; ++q) store_relaxed_i(p.q.slots + s0 + pos + q, kMaxParts * t + q0 + q);
  atomicAdd(p.q.avail + b, parts);
  atomicAdd(p.q.gcnt + (b >> 5), parts);
  atomicAdd(p.q.scnt + (b >> 10), parts);
}

// Lane 0: wait for the store of a claimed queue slot (its pusher reserved it
// before counting it available, and stores it right after). Returns the
// item, or -1 on abort / budget expiry.
__device__ int wait_slot(const KParams& p, int* slot, unsigned long long start) {
  int t = load_acquire_i(slot);
  while (t < 0) {
    if (load_relaxed_flag(&p.st->abort)) return -1;
    if (gtimer() - start > (unsigned long long)p.budget_ns) {
      raise_timeout(p, -1);
      return -1;
    }
    __nanosleep(32);
    t = load_acquire_i(slot);
  }
  return t;
}

// Lane 0: claim one available part of a queue (avail / head pair) without a
// compare-and-swap retry loop: many idle workers contending for the same
// bucket each cost two fetch-and-adds, not a round trip per lost race. The
// caller has just read avail > 0. False if nothing was available; else `pos` is the
// claimed slot's index (a ring's grows over the launch, past 2^31 too).
__device__ __forceinline__ bool claim(int* avail, int* head, unsigned& pos) {
  if (atomicSub(avail, 1) <= 0) {
    atomicAdd(avail, 1);
    return false;
  }
  pos = (unsigned)atomicAdd(head, 1);
  return true;
}

// Pause of a worker that found nothing. The first half of the grid (one CTA
// per SM) looks again at once, the second half after a longer pause: with few
// ready parts they go to different SMs, whose FP64 pipes they then do not
// share, and fewer workers contend for them.
__device__ __forceinline__ void idle_pause() { __nanosleep(blockIdx.x * 2 < gridDim.x ? 20 : 600); }

// ---- request server: three FIFO rings (urgent, other factor tasks, rest) ---
// Ring entries are reserved (tail), stored, then counted available, like the
// buckets; a popped entry is reset to -1 so the ring can wrap (its capacity
// exceeds the parts that can be ready at once).
__device__ void serve_push(const KParams& p, int t, TaskWord tw, int q0) {
  const int parts = tw.parts() - q0, op = tw.op();
  if (parts <= 0) return;
  const bool factor = op == OP_UPD || op == OP_POTRF || op == OP_TRSM_RLT || op == OP_PREP;
  const ServeRing& R = p.sv.ring[(tw.flags() & TF_URGENT) ? 0 : factor ? 1 : 2];
  const unsigned pos = (unsigned)atomicAdd(R.ctr, parts);
  for (int q = 0; q < parts; ++q) {
    int* slot = R.slots + ((pos + q) & R.mask);
    const unsigned long long start = gtimer();
    while (load_acquire_i(slot) != -1) {  // the previous lap's entry not yet taken: bounded wait
      if (load_relaxed_flag(&p.st->abort)) return;
      if (gtimer() - start > (unsigned long long)p.budget_ns) {
        raise_timeout(p, t);
        return;
      }
      __nanosleep(64);
    }
    store_release_i(slot, kMaxParts * t + q0 + q);
  }
  atomicAdd(R.ctr + 16, parts);
}

// Warp 0: activate inbox record `idx`: its value parameters, then its root
// tasks into the rings (lanes in parallel).
__device__ void serve_activate(const KParams& p, int idx) {
  const int lane = threadIdx.x & 31;
  const ServeRec* rec = &p.sv.ctl->inbox[idx % kServeInbox];
  int slot = 0, root0 = 0, nroots = 0;
  if (lane == 0) {
    const volatile ServeRec* vr = rec;
    slot = vr->slot;
    root0 = vr->root0;
    nroots = vr->nroots;
    p.sv.req_param[2 * slot] = vr->rho;
    p.sv.req_param[2 * slot + 1] = vr->tau;
    p.sv.req_seq[slot] = vr->seq;
    __threadfence();
  }
  root0 = __shfl_sync(0xffffffffu, root0, 0);
  nroots = __shfl_sync(0xffffffffu, nroots, 0);
  __syncwarp();
  for (int i = lane; i < nroots; i += 32) {
    const int t = __ldcg(p.sv.roots + root0 + i);
    push_task(p, t, load_task_word(p, t), 0);
  }
}

// Idle worker of a request server: a ready part of the highest non-empty
// ring, or -1 to stop. One round of loads per look (the abort flag and the
// three rings' counts, one lane each); the host-mapped words (inbox, stop),
// whose reads cross the host link, are looked at by a few workers on every
// round and by the others on every eighth.
__device__ int serve_pop(const KParams& p, unsigned long long deadline) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const bool watcher = blockIdx.x < 8;
  for (unsigned round = 0;; ++round) {
    int* word = lane == 0 ? &p.st->abort : p.sv.ring[min(max(lane - 1, 0), 2)].ctr + 16;
    const int v = lane < 4 ? load_relaxed_flag(word) : 0;
    if (__shfl_sync(FULL, v, 0)) return -1;
    unsigned ready = __ballot_sync(FULL, lane >= 1 && lane < 4 && v > 0);
    while (ready) {
      const int r = __ffs(ready) - 2;
      ready &= ready - 1;
      int got = -3;
      if (lane == 0) {
        const ServeRing& R = p.sv.ring[r];
        unsigned h = 0;
        if (claim(R.ctr + 16, R.ctr + 8, h)) {
          int* slot = R.slots + (h & R.mask);
          got = wait_slot(p, slot, gtimer());
          if (got >= 0) store_relaxed_i(slot, -1);
        }
      }
      got = __shfl_sync(FULL, got, 0);
      if (got != -3) return got;
    }
    if (watcher || (round & 7) == 1) {
      int rec = -3;
      if (lane == 0) {
        const int seen = load_relaxed_flag(p.sv.inbox_seen);
        if (seen < load_acquire_sys(&p.sv.ctl->inbox_count)) {
          if (atomicCAS(p.sv.inbox_seen, seen, seen + 1) == seen) rec = seen;
        } else if (load_acquire_sys(&p.sv.ctl->stop)) {
          rec = -1;
        } else if (gtimer() > deadline) {
          raise_timeout(p, -2);
          rec = -1;
        }
      }
      rec = __shfl_sync(FULL, rec, 0);
      if (rec == -1) return -1;
      if (rec >= 0) {
        serve_activate(p, rec);
        continue;
      }
    }
    __nanosleep(watcher ? 20 : 300);
  }
}

// Warp 0 pops a ready task part: the urgent queue first, then the earliest
// bucket (queue order) with an available part. Lane 0 claims and broadcasts,
// so the warp stays uniform. One look costs one round of loads, each lane its
// own word: the abort flag, the urgent queue's count, lo, the first 29
// top-level counts (the buckets' own in a plan of at most 29, else the groups'
// or super-groups'), and the heads of the 32 buckets from lo on (to move lo).
// Returns kMaxParts * task + part, or -1 when every part has been popped, the
// launch was aborted, or the wait budget of this call expired (TIMEOUT;
// checked on every pass of the loop).
__device__ int pop_task(const KParams& p, unsigned long long deadline) {
  if (p.serve) return serve_pop(p, deadline);
  const unsigned FULL = 0xffffffffu;
  constexpr int kTop = 29;
  const int lane = threadIdx.x & 31;
  const int nb = p.nbuckets, ngroups = (nb + 31) / 32, nsuper = (ngroups + 31) / 32;
  const int level = nb <= kTop ? 0 : ngroups <= kTop ? 1 : 2;  // counts looked at first
  int* const top = level == 0 ? p.q.avail : level == 1 ? p.q.gcnt : p.q.scnt;
  const int ntop = level == 0 ? nb : level == 1 ? ngroups : nsuper;
  const unsigned long long start = lane == 0 ? gtimer() : 0ull;
  int l = 0;
  for (;;) {
    int* word = lane == 0 ? &p.st->abort : lane == 1 ? p.q.lo + 24 : lane == 2 ? p.q.lo : top + min(lane - 3, ntop - 1);
    const bool used = lane < 3 || lane - 3 < ntop;
    const int hb = l + lane;
    const int v = used ? load_relaxed_flag(word) : 0;
    const int head = hb < nb ? load_relaxed_flag(p.q.head + hb) : 0;
    if (__shfl_sync(FULL, v, 0)) return -1;
    if (__shfl_sync(FULL, v, 1) > 0) {  // urgent parts
      int got = -3;
      if (lane == 0) {
        unsigned uh = 0;
        if (!claim(p.q.lo + 24, p.q.lo + 16, uh)) {
          // another worker was faster
        } else if (uh >= (unsigned)p.ucap) {  // claimed past the urgent queue (checked in every build)
          check_fail(p, 4, uh, 0);
          got = -1;
        } else {
          got = wait_slot(p, p.q.uslots + uh, start);
        }
      }
      got = __shfl_sync(FULL, got, 0);
      if (got != -3) return got;
    }
    int got = -3;  // -3: nothing found, -1: stop, >= 0: item
    // claim from the ready buckets of a 32-bucket group, in order
    auto try_buckets = [&](unsigned rm, int base) {
      while (rm && got == -3) {
        const int bb = base + __ffs(rm) - 1;
        rm &= rm - 1;
        if (lane == 0) {
          unsigned h = 0;
          if (claim(p.q.avail + bb, p.q.head + bb, h)) {
            atomicSub(p.q.gcnt + (bb >> 5), 1);
            atomicSub(p.q.scnt + (bb >> 10), 1);
            const int s0 = p.soff[bb];
            if (h >= (unsigned)(p.soff[bb + 1] - s0)) {  // claimed past the bucket (checked in every build)
              check_fail(p, 5, bb, 0);
              got = -1;
            } else {
              got = wait_slot(p, p.q.slots + s0 + h, start);
            }
          }
        }
        got = __shfl_sync(FULL, got, 0);
      }
    };
    auto try_groups = [&](unsigned gm, int base) {  // groups in order, the buckets of each
      while (gm && got == -3) {
        const int gi = base + __ffs(gm) - 1;
        gm &= gm - 1;
        const int b = gi * 32 + lane;
        try_buckets(__ballot_sync(FULL, b < nb && load_relaxed_flag(p.q.avail + b) > 0), gi * 32);
      }
    };
    auto try_supers = [&](unsigned sm, int base) {  // super-groups in order, the groups of each
      while (sm && got == -3) {
        const int si = base + __ffs(sm) - 1;
        sm &= sm - 1;
        const int g = si * 32 + lane;
        try_groups(__ballot_sync(FULL, g < ngroups && load_relaxed_flag(p.q.gcnt + g) > 0), si * 32);
      }
    };
    const unsigned tm = __ballot_sync(FULL, lane >= 3 && v > 0) >> 3;
    if (level == 0) try_buckets(tm, 0);
    else if (level == 1) try_groups(tm, 0);
    else try_supers(tm, 0);
    if (level == 2)
      for (int sbase = kTop; sbase < nsuper && got == -3; sbase += 32) {
        const int sg = sbase + lane;
        try_supers(__ballot_sync(FULL, sg < nsuper && load_relaxed_flag(p.q.scnt + sg) > 0), sbase);
      }
    if (got != -3) return got;
    // nothing claimed: move lo past finished buckets (finished is permanent,
    // so atomicMax is safe), stop once every part was popped, else back off
    const bool fin = hb >= nb || head >= p.soff[hb + 1] - p.soff[hb];
    const unsigned unf = __ballot_sync(FULL, !fin);
    const int nfin = unf ? __ffs(unf) - 1 : 32;
    const int seen = __shfl_sync(FULL, v, 2);
    if (nfin > 0 && l < nb && lane == 0 && l + nfin > seen) atomicMax(p.q.lo, l + nfin);
    const int next = max(seen, l < nb ? min(l + nfin, nb) : l);
    if (next >= nb) {  // every bucket popped: the urgent parts too?
      const int u = lane < 2 ? load_relaxed_flag(p.q.lo + 16 + 4 * lane) : 0;
      if (__shfl_sync(FULL, u, 0) + __shfl_sync(FULL, u, 1) >= p.ucap) return -1;
    }
    int stop = 0;
    if (lane == 0 && gtimer() - start > (unsigned long long)p.budget_ns) {
      raise_timeout(p, (long long)seen * kTasksPerBucket);
      stop = 1;
    }
    if (__shfl_sync(FULL, stop, 0)) return -1;
    if (next != l) {
      l = next;
      continue;
    }
    idle_pause();
  }
}

// Warp 0, after a part (of a task that counts parts) or the last part of a task
// finished and its writes were fenced: count it off every successor and queue
// those that became ready. `first` / `word`: this lane's successor (-1: none) and its
// task word, read ahead while the part ran. Of the urgent tasks released, one
// part is kept for this worker (a one-part task, the block POTRF, before any
// other): it starts without a trip through the queue. Returns that part or -1.
__device__ int release_successors(const KParams& p, const Task& tk, int first, TaskWord word) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int keep = -1;
  const int aborted = load_relaxed_flag(&p.st->abort);  // looked at below, after the counts' round trip
  int next = 32 + lane < tk.nsucc ? __ldcg(p.succ + tk.succ0 + 32 + lane) : -1;
  for (int q = lane; q - lane < tk.nsucc; q += 32) {
    int s = first;
    TaskWord tw = word;
    if (q >= 32) {
      s = next;
      if (s >= 0) tw = load_task_word(p, s);  // in flight with the count below
      next = q + 32 < tk.nsucc ? __ldcg(p.succ + tk.succ0 + q + 32) : -1;
    }
    STILES_CHECK(s < p.ntasks, 6, s, 0);
    bool ready = false;
    if (s >= 0) ready = add_relaxed_i(p.q.rem + s, -1) == 1;
    const bool urgent = ready && (tw.flags() & TF_URGENT);
    int q0 = 0;
    if (keep < 0) {
      const unsigned one = __ballot_sync(FULL, urgent && tw.parts() == 1), any = __ballot_sync(FULL, urgent);
      const int who = one ? __ffs(one) - 1 : any ? __ffs(any) - 1 : -1;
      if (who >= 0) {
        keep = kMaxParts * __shfl_sync(FULL, s, who);
        q0 = lane == who;
        if (lane == 0 && !p.serve) atomicAdd(p.q.lo + 20, 1);
      }
    }
    if (ready) {
      fence_dev();
      push_task(p, s, tw, q0);
    }
  }
  __syncwarp();
  return aborted ? -1 : keep;
}

// Lane 0 of warp 0, once a task's last part is complete in every respect:
// count it; the last task of a served request signals the host.
__device__ void account_task(const KParams& p, int t) {
  atomicAdd(&p.st->done, 1ull);
  if (!p.serve) return;
  const int slot = __ldcg(p.sv.treq + t);
  if (atomicSub(p.sv.req_left + slot, 1) == 1) {
    __threadfence_system();
    store_release_sys(&p.sv.ctl->done_seq[slot], __ldcg(p.sv.req_seq + slot));
  }
}

// OP_PREP (request server): tile column of A from the shape's base values and
// the request's (rho, tau): band entries x rho, arrow entries unchanged,
// diagonal tau + rho rb[i] + ra[i]. Every output element is written once.
__device__ void run_prep(const KParams& p, const Task& tk, int t) {
  const int slot = __ldcg(p.sv.treq + t);
  const double rho = __ldcg(p.sv.req_param + 2 * slot), tau = __ldcg(p.sv.req_param + 2 * slot + 1);
  if (rho != rho) return;  // a request with explicit values: its A was copied into place
  double* O = resolve(p, tk.out);
  const double* B = resolve(p, tk.cin);
  const double* rb = resolve(p, tk.aux);
  const double* ra = rb + tk.gcol;
  const int b = tk.ldo, a = tk.ldc;
  if (tk.flags & TF_CORNER) {  // arrow x arrow: entries unchanged, diagonal rebuilt
    for (int e = threadIdx.x; e < a * a; e += NTHREADS) {
      const int r = e % a, c = e / a;
      O[e] = r == c ? tau + rho * rb[r] + ra[r] : __ldg(B + e);
    }
    return;
  }
  const int64_t bb = (int64_t)b * b, band = (1 + (int64_t)tk.ldx) * bb;
  for (int64_t e = threadIdx.x; e < band; e += NTHREADS) {  // diagonal tile, then the sub-diagonal tiles
    const int r = (int)(e % b);
    const bool dg = e < bb && r == (int)(e / b);
    O[e] = dg ? tau + rho * rb[r] + ra[r] : rho * __ldg(B + e);
  }
  const int64_t arrow0 = (1 + (int64_t)tk.zrows) * bb;  // the arrow tile (a x b) is copied
  for (int64_t e = threadIdx.x; e < (int64_t)a * b; e += NTHREADS) O[arrow0 + e] = __ldg(B + arrow0 + e);
}

// acc[i][j] += sum over the task's segments of op(A)[r0 + tx + 16 i, :] op(B)[:, c0 + ty + 8 j]
// with 128 threads as a 16 x 8 grid (tx = tid % 16, ty = tid / 16): a
// (16 TM) x (8 TN) sub-tile, staged KC columns of K at a time in shared
// memory through L2-only loads.
// (the 16 x 16 parts of critical paths: 64 at a time, every load of a stage in
// flight at once, in rows of 17 values).
template <int TM, int TN>
__device__ __forceinline__ void accumulate(const KParams& p, const Task& tk, const Sub& sb, double (&acc)[TM][TN],
                                           double* As, double* Bs) {
  constexpr int RM = 16 * TM, CN = 8 * TN;
  constexpr bool SMALL = TM == 1 && TN == 2;
  constexpr int KC = SMALL ? 64 : stiles::KC, LDS = SMALL ? 17 : stiles::LDS;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ntm = (sb.rm + 15) / 16, ntn = (sb.cn + 7) / 8;
  const bool full = ntm == TM && ntn == TN;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
  for (int s = 0; s < tk.nseg; ++s) {
    const Seg g = load_seg(p, tk.seg0 + s);
    const bool ta = g.trans & 1, tb = g.trans & 2;
    // op(A)[r0 + i, k] and op(B)[k, c0 + j]
    const double* A = resolve(p, g.a) + (ta ? (int64_t)sb.r0 * g.lda : (int64_t)sb.r0);
    const double* B = resolve(p, g.b) + (tb ? (int64_t)sb.c0 : (int64_t)sb.c0 * g.ldb);
    for (int k0 = 0; k0 < g.k; k0 += KC) {
      const int kc = min(KC, g.k - k0);
      // each batch of loads is in flight before its shared-memory stores
      constexpr int NA = RM * KC / NTHREADS, NB = CN * KC / NTHREADS;
      constexpr int BA = NA < 8 ? NA : 8, BB = NB < 8 ? NB : 8;
#pragma unroll
      for (int u0 = 0; u0 < NA; u0 += BA) {
        double v[BA];
#pragma unroll
        for (int u = 0; u < BA; ++u) {
          const int e = tid + (u0 + u) * NTHREADS;
          int i, kk;
          if (!ta) { i = e % RM; kk = e / RM; } else { kk = e % KC; i = e / KC; }
          v[u] = (i < sb.rm && kk < kc)
                     ? __ldcg(ta ? A + (int64_t)(k0 + kk) + (int64_t)i * g.lda : A + (int64_t)i + (int64_t)(k0 + kk) * g.lda)
                     : 0.0;
        }
#pragma unroll
        for (int u = 0; u < BA; ++u) {
          const int e = tid + (u0 + u) * NTHREADS;
          int i, kk;
          if (!ta) { i = e % RM; kk = e / RM; } else { kk = e % KC; i = e / KC; }
          As[kk * LDS + i] = v[u];
        }
      }
#pragma unroll
      for (int u0 = 0; u0 < NB; u0 += BB) {
        double v[BB];
#pragma unroll
        for (int u = 0; u < BB; ++u) {
          const int e = tid + (u0 + u) * NTHREADS;
          int j, kk;
          if (tb) { j = e % CN; kk = e / CN; } else { kk = e % KC; j = e / KC; }
          v[u] = (j < sb.cn && kk < kc)
                     ? __ldcg(tb ? B + (int64_t)j + (int64_t)(k0 + kk) * g.ldb : B + (int64_t)(k0 + kk) + (int64_t)j * g.ldb)
                     : 0.0;
        }
#pragma unroll
        for (int u = 0; u < BB; ++u) {
          const int e = tid + (u0 + u) * NTHREADS;
          int j, kk;
          if (tb) { j = e % CN; kk = e / CN; } else { kk = e % KC; j = e / KC; }
          Bs[kk * LDS + j] = v[u];
        }
      }
      __syncthreads();
      // (every FP64 instruction holds the pipe for 64 cycles: the rows, columns
      // and K steps that pad a ragged part are left out)
      if (full) {
#pragma unroll 1
        for (int k1 = 0; k1 < kc; k1 += 8)
#pragma unroll
          for (int kk = k1; kk < k1 + 8; ++kk) {
            double a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk * LDS + tx + 16 * i];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk * LDS + ty + 8 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
              for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
          }
      } else {
#pragma unroll 1
        for (int kk = 0; kk < kc; ++kk) {
          double a[TM], b[TN];
#pragma unroll
          for (int i = 0; i < TM; ++i) a[i] = As[kk * LDS + tx + 16 * i];
#pragma unroll
          for (int j = 0; j < TN; ++j) b[j] = Bs[kk * LDS + ty + 8 * j];
#pragma unroll
          for (int i = 0; i < TM; ++i)
            if (i < ntm) {
#pragma unroll
              for (int j = 0; j < TN; ++j)
                if (j < ntn) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
      }
      __syncthreads();
    }
  }
}

// ---- split-precision block products on the tensor cores (tcgen05) -------
//
// Error-free splitting in the manner of Ozaki, Ogita, Oishi and Rump. Emulated
// FP64: every vector (row of op(A), column of op(B)) gets, per stretch of K, the
// biased exponent of its largest entry; each entry becomes a signed fixed-point
// integer X relative to that exponent, |X| < 2^62 (the largest entry keeps its
// 53-bit significand, and so does every entry down to 2^-9 of it), written as 8
// balanced base-2^8 digits d_t in [-128, 128), X = sum_t d_t 2^(8 (7 - t)), which
// fp16 holds exactly. Digit products of levels t + u <= 7 are kept (36 of 64; the
// dropped levels weigh below 2^-56 of the leading product). FP32-class: no shared
// exponent; every entry becomes its FP32 value (rounded to nearest) written as
// three bf16 pieces that keep their own exponents (piece_pairs), the 8 products
// of levels <= 3 accumulate in FP32.
//
// A part is 64 x 32 outputs. Its MMAs have M = 128: two planes of A (64 rows)
// stacked. Emulated FP64: stack g (planes g, g + 4 in rows 0-63, 64-127) times
// the first 32 (8 - g) columns of [B_0 | .. | B_7] into TMEM columns from 32 g:
// cell (p, c) collects the pairs of level 4 p + c, at most 4 per K, so its FP32
// sum is an integer of magnitude at most 2^24, exact, for 256 of K. 8 levels of
// 32 columns are the 256 TMEM columns of each of two CTAs per SM. FP32-class:
// planes 0, 1 stacked times [B_0 | B_1 | B_2] into columns 0-95, plane 2 times
// [B_0 | B_1] into 96-159: every plane pair sums in a cell of its own, over up to
// 4096 of K. Then the cells are drained: read, combined per output (exactly, for
// emulated FP64) and added to the part's FP64 result in registers.
// Non-finite operands make their row or column NaN (emulated FP64: biased
// exponent 0x7ff; FP32-class: NaN pieces, also beyond the FP32 range).
//
// Operands reach shared memory in one of two ways, in the same layout:
//   * run_planes: phase 2's operands, each read by many products, are split once
//     into planes in global memory (OP_SPLIT) and copied in whole stages;
//   * run_tc: a part loads its operands 64 of K at a time into registers, takes
//     the exponents there and writes the digits itself (factor updates, TRMM).

__device__ __forceinline__ int biased_exp(double v) {
  return (int)((__double_as_longlong(v) >> 52) & 0x7ff);
}

constexpr uint32_t TC_COLS = 256;   // TMEM columns per CTA (two CTAs per SM share 512)

// Per-CTA state of the tensor path (static shared memory of the kernel).
constexpr int PL_SLOTS = 8;         // staging slots of a product from planes, at most
struct TcShared {
  uint64_t pfull[PL_SLOTS];   // products from planes: a slot's copies have landed
  uint64_t pempty[PL_SLOTS];  // ... its MMAs are done
  uint64_t pdone;             // every MMA issued before is done
  uint32_t pstage;       // stages this CTA has run so far (stage_count): stage g is slot g % NST, phase g / NST
  uint32_t pdone_n;      // phases of pdone
  uint32_t tmem;         // TMEM base address of this CTA's TC_COLS columns
};


// Signed fixed-point value of v relative to the biased exponent emax of its row
// or column (emax >= its own), rounded to nearest: the row maximum maps to
// [2^61, 2^62).
__device__ __forceinline__ unsigned long long fixed_point(double v, int emax) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int e = (int)((bits >> 52) & 0x7ff);
  const int d = max(emax, 1) - max(e, 1);
  const unsigned long long m = d > 62 ? 0ull : (bits & 0xFFFFFFFFFFFFFull) | ((unsigned long long)(e != 0) << 52);
  const unsigned long long X = (((m << 11) >> (1 + min(d, 62))) + 1) >> 1;
  const unsigned long long s = 0ull - (bits >> 63);  // all ones for a negative value
  return (X ^ s) - s;
}

// The 8 digits (balanced, base 2^8) of a pair of K-adjacent values (v0 at k, v1
// at k + 1) as packed fp16 pairs: w[t] = d_t(v0) | d_t(v1) << 16. With 128 added
// to every digit they are the bytes of the fixed-point value plus the bias C, top
// byte first; a byte under 0x64 is the fp16 value 1024 + byte, and one packed
// subtraction of 1152 leaves the digits exactly (two permutes and one subtraction
// per pair and digit; through FP32 and bf16 it took five instructions).
__device__ __forceinline__ void digit_pairs(double v0, double v1, int emax, uint32_t (&w)[8]) {
  constexpr unsigned long long C = 0x8080808080808080ull;
  const unsigned long long y0 = fixed_point(v0, emax) + C, y1 = fixed_point(v1, emax) + C;
  const uint32_t h0[2] = {(uint32_t)y0, (uint32_t)(y0 >> 32)}, h1[2] = {(uint32_t)y1, (uint32_t)(y1 >> 32)};
  const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1152
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t lo = __byte_perm(h0[h], h1[h], 0x5140), hi = __byte_perm(h0[h], h1[h], 0x7362);  // byte pairs 0, 1; 2, 3
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const uint32_t u = __byte_perm(b < 2 ? lo : hi, 0x64646464u, b & 1 ? 0x4342 : 0x4140);
      const __half2 f = __hsub2(*reinterpret_cast<const __half2*>(&u), bias);
      w[7 - (4 * h + b)] = *reinterpret_cast<const uint32_t*>(&f);  // digit t is byte 7 - t
    }
  }
}

// FP32-class operands: the value rounded to nearest FP32 (ties away from
// zero), built from the double's bits without an FP64 instruction: half a
// unit of the 23rd fraction bit is added to the bit pattern (a carry moves
// into the exponent as it should), then sign, exponent rebiased and the top
// 23 fraction bits are taken. Below the FP32 normal range it is zero, above
// it infinity; an infinity or NaN in gives NaN.
__device__ __forceinline__ uint32_t fp32_bits_of(double v) {
  const unsigned long long b0 = (unsigned long long)__double_as_longlong(v), b = b0 + (1ull << 28);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, sgn = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ff);
  // exponent and the top 23 fraction bits, rebiased
  uint32_t r = __funnelshift_l(lo, hi & 0x7fffffffu, 3) - ((1023u - 127u) << 23);
  r = e < 1023 - 126 ? 0u : e > 1023 + 127 ? 0x7f800000u : r;
  return ((b0 >> 52) & 0x7ff) == 0x7ff ? 0x7fc00000u : sgn | r;
}

// The FP32 values of a pair of K-adjacent operands (v0 at k, v1 at k + 1) as
// three bf16 pieces each, packed in pairs like digit_pairs: piece t is the
// value left after pieces < t, truncated to its top 8 significant bits, so
// the three pieces sum to the FP32 value exactly and each keeps its own
// exponent. The fourth plane is zero.
__device__ __forceinline__ void piece_pairs(double v0, double v1, uint32_t (&w)[4]) {
  float r0 = __uint_as_float(fp32_bits_of(v0)), r1 = __uint_as_float(fp32_bits_of(v1));
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    const uint32_t p0 = __float_as_uint(r0) & 0xffff0000u, p1 = __float_as_uint(r1) & 0xffff0000u;
    w[t] = __byte_perm(p0, p1, 0x7632);
    r0 -= __uint_as_float(p0);
    r1 -= __uint_as_float(p1);
  }
  w[3] = 0u;
}

// Bounded wait for phase `parity` of a staging barrier (all threads).
__device__ bool tc_wait(const KParams& p, uint32_t mbar, uint32_t parity) {
  if (tc::mbar_test(mbar, parity)) return true;
  const unsigned long long t0 = gtimer();
  while (!tc::mbar_test(mbar, parity)) {
    if (gtimer() - t0 > (unsigned long long)p.budget_ns) {
      raise_timeout(p, -3);
      return false;
    }
  }
  return true;
}

template <int S>
struct PlaneFmt {
  static constexpr int NP = S == 8 ? 8 : 3;              // planes
  static constexpr int A_BYTES = 64 * kPlaneK * 2 * NP;  // a stage of a left-hand group
  static constexpr int B_BYTES = A_BYTES / 2;            // half a stage of a right-hand group
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int NST = S == 8 ? 4 : 8;             // staging slots
  // K that cells sum: exactly (emulated FP64), or with FP32 rounding
  static constexpr int KMAX = S == 8 ? 256 : 4096;
  static_assert(NST <= PL_SLOTS, "slots");
};
constexpr int PL_STAGE_BYTES = 4 * PlaneFmt<8>::STAGE;
static_assert(8 * PlaneFmt<4>::STAGE + 4096 <= PL_STAGE_BYTES, "an MMA of plane 2 reads one plane beyond its stage");
constexpr int PL_XCH_OFF = PL_STAGE_BYTES;            // exchange between the warps of two lane blocks
constexpr int PL_XCH_BYTES = 64 * 8 * 3 * 8;          // 64 rows x 8 columns x (high, low; low)
constexpr int PL_EXP_OFF = PL_XCH_OFF + PL_XCH_BYTES;  // exponents: 32 columns; run_tc's partial ones
constexpr int PL_SMEM_BYTES = PL_EXP_OFF + (32 + 4 * 96) * 4;
constexpr uint32_t PL_LBO = 128, PL_SBO = 256;        // K- and row-adjacent core matrices of a stage

// One thread: the MMAs of one stage (16 of K) at shared address a0, adding to the
// cells or (acc = false) starting them.
template <int S>
__device__ __forceinline__ void stage_mmas(uint32_t tmem, uint32_t a0, bool acc) {
  const uint64_t bd = tc::smem_desc(a0 + PlaneFmt<S>::A_BYTES, PL_LBO, PL_SBO);
  if constexpr (S == 8) {
#pragma unroll
    for (int g = 0; g < 4; ++g)
      tc::mma_f16(tmem + 32 * g, tc::smem_desc(a0 + g * 4096, PL_LBO, PL_SBO), bd, tc::idesc_f16_f32(128, 32 * (8 - g)),
                   g > 0 || acc ? 1u : 0u);
  } else {
    tc::mma_f16(tmem, tc::smem_desc(a0, PL_LBO, PL_SBO), bd, tc::idesc_bf16_f32(128, 96), acc ? 1u : 0u);
    tc::mma_f16(tmem + 96, tc::smem_desc(a0 + 4096, PL_LBO, PL_SBO), bd, tc::idesc_bf16_f32(128, 64), acc ? 1u : 0u);
  }
}

// (H 2^32 + Lo) 2^k2 as a double, rounded once (|H 2^32 + Lo| < 2^76), without an
// FP64 instruction (a conversion holds the pipe like a multiply-add, and the drains
// would keep it from the block POTRFs). All 96 bits are kept up to the rounding:
// with the low 16 rounded off first, half the integer work and 0.5 to 3 % of a
// pass, the error of the n = 122,944 matrix was 3.3e-15 where one rounding gives
// 1.4e-15.
// `slow` is set when the result leaves the normal range (scaled_sum_any then).
__device__ __forceinline__ double scaled_sum(long long H, long long Lo, int k2, bool& slow) {
  const long long t = H + (Lo >> 32);  // the sum is t 2^32 + the low word of Lo
  const unsigned long long sign = (unsigned long long)(t >> 63);  // all ones for a negative sum
  const uint32_t mlo = ((uint32_t)Lo ^ (uint32_t)sign) - (uint32_t)sign;
  const unsigned long long mhi = ((unsigned long long)t ^ sign) + (sign != 0 && mlo == 0 ? 1 : 0);
  const bool far = mhi == 0;
  const unsigned long long top = far ? mlo : mhi;
  const uint32_t low = far ? 0u : mlo;
  const int lz = __clzll((long long)top);
  // top bit set (mhi < 2^45, so lz is 19 or more and the shift of low below 46)
  const unsigned long long norm = (top << (lz & 63)) | (((unsigned long long)low << 32) >> ((64 - lz) & 63));
  const unsigned long long mant = (norm >> 11) + ((norm >> 10) & 1ull);  // 2^52 .. 2^53
  const int e = (63 - lz) + (far ? 0 : 32) + k2 + 1023;                  // biased exponent
  slow = slow || (top != 0 && (unsigned)(e - 1) >= 0x7fdu);
  const unsigned long long bits = (((unsigned long long)(unsigned)(e - 1) << 52) + mant) | (sign << 63);
  return top == 0 ? 0.0 : __longlong_as_double((long long)bits);
}
__device__ __noinline__ double scaled_sum_any(long long H, long long Lo, int k2) {
  return ldexp(fma((double)H, 4294967296.0, (double)Lo), k2);
}

// acc += cell 2^sh for an integer-valued FP32 cell. SMALL (at most 64 of K, so
// |cell| <= 2^22): adding 3 2^22 leaves the integer in the low mantissa bits, so
// the sum runs on the bit patterns (a conversion runs at a quarter of the rate)
// and kCellBias takes the patterns' constant part back out of four levels.
constexpr long long kCellBias = 0x4B400000ll * ((1ll << 24) + (1ll << 16) + (1ll << 8) + 1);
template <bool SMALL>
__device__ __forceinline__ void add_cell(long long& acc, uint32_t cell, int sh) {
  const float f = __uint_as_float(cell);
  const int v = SMALL ? __float_as_int(f + 12582912.0f) : __float2int_rn(f);
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(v), "r"(1 << sh));
}

// Read the cells and add the part's sums of this stretch of K to r16. er: the
// biased exponent of the thread's row, cexp: of the 32 columns (shared memory;
// emulated FP64). SMALL: at most 64 of K in the cells.
// rows, cols: the part's. Unless WHOLE, a group of columns or a warp's 32 rows beyond
// them is left out: with all of them drained, parts of small tiles took 4 to 7k cycles
// more; the tests for it in every part cost (28, 1024, 4, 64) in emulated FP64 2 %.
// Each warp reads the cells of all 32 columns in its lane block (warps 0, 1: the
// low levels / planes 0 and 2; warps 2, 3: the high levels / plane 1), 4 columns
// of the other side's, handed over through shared memory, and 4 of its own at a
// time. The loop is not unrolled (r16 is rotated instead, back in place after its
// four steps): straight-line code of this size ran at the instruction cache's
// rate, 13k cycles a drain (n = 122,944 in emulated FP64: 345 against 321 ms, with
// the splits of run_tc, which had the same fault).
template <int S, bool SMALL, bool WHOLE>
__device__ __forceinline__ void drain_cells(uint32_t tmem, uint8_t* xch, int er, const int* cexp, int rows, int cols,
                                            double (&r16)[16]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int side = warp >> 1, row = 32 * (warp & 1) + lane;
  const uint32_t trow = tmem + ((uint32_t)(32 * warp) << 16);
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    if (WHOLE || 4 * i < cols) {
      uint8_t* buf = xch + (i & 1) * (PL_XCH_BYTES / 2);  // free since the barrier of the step before
      // this warp's columns and the other side's that lie in the part (warp-uniform)
      const bool live = 32 * (warp & 1) < rows;
      const bool own = WHOLE || (live && 16 * side + 4 * i < cols);
      const bool other = WHOLE || (live && 16 * (1 - side) + 4 * i < cols);
      if constexpr (S == 8) {
        constexpr int kScale = 2044 + 2 * 62 - 8 * 7;
        long long* xhl = reinterpret_cast<long long*>(buf);  // [4 c][64 r] x (hi, lo) for side 1
        long long* xlo = xhl + 2 * 4 * 64;                    // [4 c][64 r] lo for side 0
        // level sums of 4 columns from col: hi (levels 0-3), lo (levels 4-7)
        auto sums = [&](int col, long long (&hi)[4], long long (&lo)[4]) {
#pragma unroll
          for (int x = 0; x < 4; ++x) hi[x] = lo[x] = SMALL ? -kCellBias : 0;
          if (side == 0) {
            uint32_t cell[8][4];
            tc::ld_cells(trow + col, cell);
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
              for (int x = 0; x < 4; ++x) {
                if (c <= 3) add_cell<SMALL>(hi[x], cell[c][x], 8 * (3 - c));
                else add_cell<SMALL>(lo[x], cell[c][x], 8 * (7 - c));
              }
          } else {
            uint32_t cell[4][4];
            tc::ld_cells(trow + col, cell);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
              for (int x = 0; x < 4; ++x) add_cell<SMALL>(lo[x], cell[c][x], 8 * (3 - c));
          }
        };
        long long hi[4], lo[4];
        if (other) {
          sums(16 * (1 - side) + 4 * i, hi, lo);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int e = x * 64 + row;
            if (side == 0) {
              xhl[2 * e] = hi[x];
              xhl[2 * e + 1] = lo[x];
            } else {
              xlo[e] = lo[x];
            }
          }
        }
        __syncthreads();
        if (own) {
          sums(16 * side + 4 * i, hi, lo);
          bool slow = false;
          double v[4];
          int k2[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int e = x * 64 + row, ec = cexp[16 * side + 4 * i + x];
            hi[x] = side == 0 ? hi[x] : xhl[2 * e];
            lo[x] += side == 0 ? xlo[e] : xhl[2 * e + 1];
            k2[x] = max(er, 1) + max(ec, 1) - kScale;
            v[x] = scaled_sum(hi[x], lo[x], k2[x], slow);
            if (er == 0x7ff || ec == 0x7ff) v[x] = __longlong_as_double(0x7ff8000000000000ll);
          }
          if (slow) {
#pragma unroll
            for (int x = 0; x < 4; ++x)
              if (v[x] == v[x]) v[x] = scaled_sum_any(hi[x], lo[x], k2[x]);
          }
#pragma unroll
          for (int x = 0; x < 4; ++x) r16[x] += v[x];
        }
      } else {
        float* x0 = reinterpret_cast<float*>(buf);  // [4 c][64 r] plane 0, then plane 2, for side 1
        float* x1 = x0 + 2 * 4 * 64;                // [4 c][64 r] plane 1, for side 0
        auto pieces = [&](int col, float (&v)[4], float (&v2)[4]) {  // lane block's sums of 4 columns
          uint32_t cell[8][4];
          tc::ld_cells(trow + col, cell);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            v[x] = ((0.0f + __uint_as_float(cell[0][x])) + __uint_as_float(cell[1][x])) + __uint_as_float(cell[2][x]);
            v2[x] = (0.0f + __uint_as_float(cell[3][x])) + __uint_as_float(cell[4][x]);
          }
        };
        float v[4], v2[4];
        if (other) {
          pieces(16 * (1 - side) + 4 * i, v, v2);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int e = x * 64 + row;
            if (side == 0) {
              x0[e] = v[x];
              x0[4 * 64 + e] = v2[x];
            } else {
              x1[e] = v[x];
            }
          }
        }
        __syncthreads();
        if (own) {
          pieces(16 * side + 4 * i, v, v2);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int e = x * 64 + row;
            const float p0 = side == 0 ? v[x] : x0[e], p1 = side == 0 ? x1[e] : v[x], p2 = side == 0 ? v2[x] : x0[4 * 64 + e];
            r16[x] += (double)(((0.0f + p0) + p1) + p2);
          }
        }
      }
    }
    double t[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) t[x] = r16[x];
#pragma unroll
    for (int x = 0; x < 12; ++x) r16[x] = r16[x + 4];
#pragma unroll
    for (int x = 0; x < 4; ++x) r16[12 + x] = t[x];
  }
}

// Epilogue of a 64 x 32 part from its result in registers (the thread mapping of
// run_planes); smem: the staging region, free.
__device__ __forceinline__ void store_part(const KParams& p, const Task& tk, int q, double* smem, double (&r16)[16]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int side = warp >> 1, row = 32 * (warp & 1) + lane;
  const int c0 = 32 * q + 16 * side;
  const int m = tk.m, n = tk.n;
  double* O = resolve(p, tk.out);
  if (tk.op != OP_SYMUPD) {  // OP_UPD, OP_STORE, OP_NEG
    double* Om = tk.op == OP_NEG && p.smirror ? p.smirror + (O - p.buf[BUF_S]) : nullptr;
    if (tk.op == OP_UPD) {
      const double* C = resolve(p, tk.cin);
      double v[16];
#pragma unroll
      for (int x = 0; x < 16; ++x)
        v[x] = row < m && c0 + x < n ? __ldcg(C + row + (int64_t)(c0 + x) * tk.ldc) : 0.0;
#pragma unroll
      for (int x = 0; x < 16; ++x) r16[x] = v[x] - r16[x];
    }
#pragma unroll
    for (int x = 0; x < 16; ++x)
      if (row < m && c0 + x < n) {
        const double v = tk.op == OP_NEG ? -r16[x] : r16[x];
        O[row + (int64_t)(c0 + x) * tk.ldo] = v;
        if (Om) Om[row + (int64_t)(c0 + x) * tk.ldo] = v;
      }
    return;
  }
  // OP_SYMUPD: cin - acc, and its transpose into the mirror position (inside the
  // block for a diagonal one, whose part above the diagonal is left out)
  const double* C = resolve(p, tk.cin);
  const bool dblk = tk.flags & TF_SYM_DIAG;
  double* M = dblk ? O : resolve(p, tk.aux);
  const int ldm = dblk ? tk.ldo : tk.ldx;
  double* Om = p.smirror ? p.smirror + (O - p.buf[BUF_S]) : nullptr;
  double* Mm = p.smirror ? p.smirror + (M - p.buf[BUF_S]) : nullptr;
  double v[16];  // (every load in flight before the first subtraction)
#pragma unroll
  for (int x = 0; x < 16; ++x) {
    const bool in = row < m && c0 + x < n && (!dblk || row >= c0 + x);
    v[x] = in ? __ldcg(C + row + (int64_t)(c0 + x) * tk.ldc) : 0.0;
  }
#pragma unroll
  for (int x = 0; x < 16; ++x) v[x] -= r16[x];
  double* X = smem;  // [64 rows][33]: the staging region, every copy of which has been used
#pragma unroll
  for (int x = 0; x < 16; ++x) {
    X[row * 33 + 16 * side + x] = v[x];
    if (row < m && c0 + x < n && (!dblk || row >= c0 + x)) {
      O[row + (int64_t)(c0 + x) * tk.ldo] = v[x];
      if (Om) Om[row + (int64_t)(c0 + x) * tk.ldo] = v[x];
    }
  }
  __syncthreads();
  for (int e = tid; e < 64 * 32; e += NTHREADS) {
    const int c = e % 32, r = e / 32, cc = 32 * q + c;
    if (r < m && cc < n && (!dblk || r > cc)) {
      M[cc + (int64_t)r * ldm] = X[r * 33 + c];
      if (Mm) Mm[cc + (int64_t)r * ldm] = X[r * 33 + c];
    }
  }
}

// The 64 x 32 sub-tile (columns 32 q ..) of a product task from planes, and its
// epilogue. Thread (warp, lane) owns row 32 (warp & 1) + lane, columns
// 16 (warp >> 1) + 0..15 of it. Thread 32 copies, thread 0 multiplies: one
// thread doing both waits for the MMAs of the stage before in between. What bounds
// it, stamped at an inner length of 1088 in a loaded launch: in emulated FP64 the
// drains, 59k of 120k cycles (11.7k per 256 of K), then the MMAs, whose pipe the SM's
// two CTAs share, with 7.5k cycles of waiting for copies; in the FP32-class mode the
// MMAs, 31k of 45k cycles, with 9.6k of waiting and one drain of 4.5k. (L2 is at 19 %
// of its rate over the selected inversion of (10, 1024, 4, 64).) Such a part takes 65
// us in emulated FP64, 26 in the FP32-class mode; 146 and 64 us for half the outputs
// when each part split its operands itself.
template <int S>
__device__ __noinline__ void run_planes(const KParams& p, const Task& tk, int q, double* smem, TcShared& ts) {
  using F = PlaneFmt<S>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int row = 32 * (warp & 1) + lane;
  uint8_t* stage = reinterpret_cast<uint8_t*>(smem);
  const uint32_t stage_a = tc::smem_addr(stage);
  double r16[16];
#pragma unroll
  for (int x = 0; x < 16; ++x) r16[x] = 0.0;
  int* cexp = reinterpret_cast<int*>(stage + PL_EXP_OFF);
  const uint32_t base = ts.pstage;  // this part's stages are base, base + 1, ..
  const bool copier = tid == 32;
  // copies: a cursor over the stages of all segments
  int ls = 0, lk = 0;
  uint32_t issued = 0, used = 0;  // stages copied / multiplied by this part
  Seg lseg = load_seg(p, tk.seg0);
  auto issue = [&]() {  // the next stage into its slot, once the MMAs that last read it are done
    const uint32_t g = base + issued, slot = g % F::NST;
    if (g >= F::NST && !tc_wait(p, tc::smem_addr(&ts.pempty[slot]), (g / F::NST - 1) & 1)) return false;
    const int nst = (lseg.k + kPlaneK - 1) / kPlaneK, nch = (lseg.k + kPlaneChunk - 1) / kPlaneChunk;
    const int64_t head = S == 8 ? 256 * (int64_t)nch : 0;
    const uint8_t* A = p.planes + 16 * (lseg.a & OFF_MASK) + head + (int64_t)lk * F::A_BYTES;
    const uint8_t* B = p.planes + 16 * (lseg.b & OFF_MASK) + head + (int64_t)lk * F::A_BYTES + q * F::B_BYTES;
    const uint32_t bar = tc::smem_addr(&ts.pfull[slot]), dst = stage_a + slot * F::STAGE;
    tc::expect_tx(bar, F::STAGE);
    tc::bulk_load(dst, A, F::A_BYTES, bar);
    tc::bulk_load(dst + F::A_BYTES, B, F::B_BYTES, bar);
    ++issued;
    if (++lk == nst) {
      lk = 0;
      if (++ls < tk.nseg) lseg = load_seg(p, tk.seg0 + ls);
    }
    return true;
  };
  tc::fence_smem_to_async();  // earlier tasks' shared-memory accesses before the copies' writes
  __syncthreads();
  if (copier) {
    tc::fence_global_async();  // the planes' writes (this task was released after them)
    for (int x = 0; x < F::NST && ls < tk.nseg; ++x)
      if (!issue()) break;
  }
  uint32_t ndone = ts.pdone_n;
  int kacc = 0;
  bool ok = true;
  for (int s = 0; s < tk.nseg && ok; ++s) {
    const Seg gs = load_seg(p, tk.seg0 + s);
    const int nst = (gs.k + kPlaneK - 1) / kPlaneK;
    const int* ea = reinterpret_cast<const int*>(p.planes + 16 * (gs.a & OFF_MASK));
    const int* eb = reinterpret_cast<const int*>(p.planes + 16 * (gs.b & OFF_MASK));
    // runs of stages between drains: K chunks of one exponent cut where the
    // cells' exact range ends; FP32-class: 4096 of K, counted in steps of 32
    for (int st0 = 0; st0 < nst && ok;) {
      int st1;
      bool drain, fresh = true;
      if constexpr (S == 8) {
        st1 = min(nst, st0 + F::KMAX / kPlaneK);
        drain = true;
      } else {
        const int room = (F::KMAX - kacc) / 32;
        fresh = kacc == 0;
        st1 = min(nst, st0 + 2 * room);
        kacc += (st1 - st0 + 1) / 2 * 32;
        drain = (s == tk.nseg - 1 && st1 == nst) || kacc + 32 > F::KMAX;
      }
      const uint32_t end = used + (uint32_t)(st1 - st0);
      if (copier)  // up to the slots that the run's last MMAs free (those after the drain's wait)
        while (ls < tk.nseg && issued + 1 < end + F::NST && issue()) {}
      if (tid == 0) {
        bool go = true;
        for (uint32_t x = used; x < end; ++x) {
          const uint32_t g = base + x, slot = g % F::NST;
          if (!tc_wait(p, tc::smem_addr(&ts.pfull[slot]), (g / F::NST) & 1)) {
            go = false;  // pdone is not committed: every thread's wait for it runs out too
            break;
          }
          tc::fence_after_sync();
          stage_mmas<S>(ts.tmem, stage_a + slot * F::STAGE, !(fresh && x == used));
          tc::commit(tc::smem_addr(&ts.pempty[slot]));
        }
        if (drain && go) tc::commit(tc::smem_addr(&ts.pdone));
      }
      used = end;
      const int first = st0;
      st0 = st1;
      if (!drain) continue;
      kacc = 0;
      int er = 0;
      if constexpr (S == 8) {  // this chunk's exponents, in flight while the MMAs finish
        const int ch = first / (kPlaneChunk / kPlaneK);
        er = __ldcg(ea + 64 * ch + row);
        if (warp == 3) cexp[lane] = __ldcg(eb + 64 * ch + 32 * q + lane);  // (read after the barrier below)
      }
      __syncwarp();
      ok = tc_wait(p, tc::smem_addr(&ts.pdone), ndone & 1);
      ++ndone;
      ok = !__syncthreads_or(!ok);
      if (!ok) break;
      tc::fence_after_sync();
      if (copier)  // every slot is free: the next stages load while the cells are read
        while (ls < tk.nseg && issued < end + F::NST && issue()) {}
      drain_cells<S, false, true>(ts.tmem, stage + PL_XCH_OFF, er, cexp, tk.m, tk.n - 32 * q, r16);
      tc::fence_before_sync();
      __syncthreads();  // TMEM and exchange reads done before the next MMAs
    }
  }
  if (!ok) {  // timed out: the copies in flight must land before the part ends (again bounded waits)
    if (copier)
      for (uint32_t g = base + (issued > F::NST ? issued - F::NST : 0); g != base + issued; ++g)
        tc_wait(p, tc::smem_addr(&ts.pfull[g % F::NST]), (g / F::NST) & 1);
    __syncthreads();
    return;
  }
  if (tid == 0) {  // (read again only after the next part's first barrier)
    ts.pstage = stage_count(base + used);  // (counted on, it wraps after an hour or more in a server)
    ts.pdone_n = ndone;
  }
  store_part(p, tk, q, smem, r16);
}

// 8 K-adjacent values of one vector from P (`step` apart), zero from the n-th on.
// Contiguous ones are read in pairs where `pairs` says that P is 16-byte aligned
// (single 8-byte loads fetch each 32-byte sector four times: a lane per vector).
__device__ __forceinline__ void load_octet(const double* P, int64_t step, bool pairs, int n, double (&x)[8]) {
  if (pairs && n >= 8) {
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const double2 v = __ldcg(reinterpret_cast<const double2*>(P) + y);
      x[2 * y] = v.x;
      x[2 * y + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int y = 0; y < 8; ++y) x[y] = y < n ? __ldcg(P + (int64_t)y * step) : 0.0;
  }
}
__device__ __forceinline__ bool pairs_ok(const double* P, int ld) { return ((((uintptr_t)P) & 15) | (ld & 1)) == 0; }

// A chunk of a part's inner length: at most four stages from segment s, K k0 on. In
// emulated FP64 of one segment (it has one exponent per vector); in the FP32-class mode
// whole segments after it too while they fit, as long as the cells may go on summing
// (kacc of K so far): with a chunk per segment of 16 of K the parts of tiles of 16 took
// 7k cycles more per segment.
// x[3 h + 0], x[3 h + 1], x[3 h + 2]: the K octet warp + 4 h of rows lane and lane + 32
// of op(A) and of column lane of op(B).
struct TcChunk {
  int nst, kadd;  // stages; what the chunk adds to kacc
  int s, k0;      // the next chunk's start
};
// octet h: K from k on of segment g, `left` of it to the segment's (or chunk's) end
__device__ __forceinline__ void tc_octets(const KParams& p, const Task& tk, const Seg& g, int k, int left, int q, int h,
                                          double (&x)[6][8]) {
  const int lane = threadIdx.x & 31;
  const bool ta = g.trans & 1, tb = g.trans & 2;
  const int64_t sa = ta ? 1 : g.lda, sb = tb ? g.ldb : 1;
  const double* A = resolve(p, g.a) + (int64_t)k * sa;
  const double* B = resolve(p, g.b) + (int64_t)k * sb + (int64_t)(32 * q) * (tb ? 1 : g.ldb);
  const bool va = ta && pairs_ok(A, g.lda), vb = !tb && pairs_ok(B, g.ldb);
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int v = lane + 32 * u;
    load_octet(A + (int64_t)v * (ta ? g.lda : 1), sa, va, v < tk.m ? left : 0, x[3 * h + u]);
  }
  load_octet(B + (int64_t)lane * (tb ? 1 : g.ldb), sb, vb, 32 * q + lane < tk.n ? left : 0, x[3 * h + 2]);
}
template <int S>
__device__ __forceinline__ TcChunk tc_load(const KParams& p, const Task& tk, int s, int k0, int kacc, int q,
                                           double (&x)[6][8]) {
  const int warp = threadIdx.x >> 5;
  TcChunk c{0, 0, s, k0};
  Seg cur = load_seg(p, tk.seg0 + s);
  if constexpr (S == 8) {
    const int kc = min(64, cur.k - k0);
#pragma unroll
    for (int h = 0; h < 2; ++h) tc_octets(p, tk, cur, k0 + 8 * (warp + 4 * h), kc - 8 * (warp + 4 * h), q, h, x);
    c.nst = (kc + kPlaneK - 1) / kPlaneK;
    c.k0 += kc;
    if (c.k0 >= cur.k) {
      c.k0 = 0;
      ++c.s;
    }
    return c;
  }
  Seg g[2] = {cur, cur};  // of this warp's octets, their first K in it and what is left from there
  int k[2] = {0, 0}, left[2] = {0, 0};
  for (;;) {
    const int kc = min(min(16 * (4 - c.nst), cur.k - c.k0), PlaneFmt<S>::KMAX - kacc - c.kadd);
    const int n = (kc + kPlaneK - 1) / kPlaneK;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int st = (warp >> 1) + 2 * h - c.nst;  // of the octet, from the first of these
      if (st >= 0 && st < n) {
        g[h] = cur;
        k[h] = c.k0 + kPlaneK * st + 8 * (warp & 1);
        left[h] = kc - kPlaneK * st - 8 * (warp & 1);
      }
    }
    c.nst += n;
    c.kadd += (kc + 31) / 32 * 32;
    c.k0 += kc;
    if (c.k0 < cur.k) break;
    c.k0 = 0;
    if (++c.s >= tk.nseg || c.nst >= 4 || kacc + c.kadd + 32 > PlaneFmt<S>::KMAX) break;
    cur = load_seg(p, tk.seg0 + c.s);
    if (cur.k > 16 * (4 - c.nst)) break;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) tc_octets(p, tk, g[h], k[h], left[h], q, h, x);
  return c;
}

// The planes of 8 K-adjacent values, 16 bytes each: plane t at dst + (t % 4) s1 + (t / 4) s2.
template <int S, bool GLOBAL>
__device__ __forceinline__ void store_planes(const double (&x)[8], int emax, uint8_t* dst, int s1, int s2) {
  uint32_t w[4][S];
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    if constexpr (S == 8) digit_pairs(x[2 * y], x[2 * y + 1], emax, w[y]);
    else piece_pairs(x[2 * y], x[2 * y + 1], w[y]);
  }
#pragma unroll
  for (int t = 0; t < PlaneFmt<S>::NP; ++t) {
    uint4* d = reinterpret_cast<uint4*>(dst + (t % 4) * s1 + (t / 4) * s2);
    const uint4 v = make_uint4(w[0][t], w[1][t], w[2][t], w[3][t]);
    if constexpr (GLOBAL) __stcg(d, v);
    else *d = v;
  }
}
// s1, s2 of a stage's left- / right-hand planes (64 / 32 vectors)
template <int S>
struct PlaneStep {
  static constexpr int A1 = S == 8 ? 4096 : 2048, A2 = 2048, B1 = 1024, B2 = 4096;
};

// A 64 x 32 part (columns 32 q ..) that splits its own operands: 64 of K at a
// time. Thread (warp, lane) loads the K octets warp and warp + 4 of the vectors
// lane and lane + 32 of op(A) and lane of op(B) (48 values, the next 64 of K in
// flight while the MMAs of these run), takes the exponents from them (emulated
// FP64: one per vector and 64 of K) and writes the planes of four stages. What
// bounds it: the splits (about 35 instructions per operand value, 48 values per
// thread for 1664 cycles of MMAs) and, for the factor's updates with an inner
// length of 64, the fixed cost of a task. The 32 x 32 parts before split each
// operand twice as often and scanned the whole K for exponents first: factor +
// selected inversion of (28, 1024, 4, 64) in emulated FP64 464 ms then, 205 ms
// with these parts and phase 2 from planes (454 ms with phase 2 in these parts).
template <int S, bool WHOLE>
__device__ __noinline__ void run_tc(const KParams& p, const Task& tk, int q, double* smem, TcShared& ts) {
  using F = PlaneFmt<S>;
  static_assert(4 * F::STAGE <= PL_STAGE_BYTES, "64 of K in the staging region");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint8_t* stage = reinterpret_cast<uint8_t*>(smem);
  const uint32_t stage_a = tc::smem_addr(stage);
  // column exponents, partial exponents [4 warps][64 rows, then 32 columns]
  int* cexp = reinterpret_cast<int*>(stage + PL_EXP_OFF);
  int* pexp = cexp + 32;
  if (tk.op == OP_UPD) {  // the input block into L2, one line per thread
    const int col = 32 * q + (tid >> 2), r = 16 * (tid & 3);
    if (col < tk.n && r < tk.m)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(resolve(p, tk.cin) + r + (int64_t)col * tk.ldc));
  }
  double r16[16];
#pragma unroll
  for (int x = 0; x < 16; ++x) r16[x] = 0.0;
  uint32_t ndone = ts.pdone_n;
  int kacc = 0;
  double x[6][8];
  TcChunk next = tc_load<S>(p, tk, 0, 0, 0, q, x);
  for (bool last = false; !last;) {
    int er = 0, ea[2] = {0, 0}, eb = 0;
    if constexpr (S == 8) {
#pragma unroll
      for (int h = 0; h < 6; h += 3)
#pragma unroll
        for (int y = 0; y < 8; ++y) {
          ea[0] = max(ea[0], biased_exp(x[h][y]));
          ea[1] = max(ea[1], biased_exp(x[h + 1][y]));
          eb = max(eb, biased_exp(x[h + 2][y]));
        }
      int* mine = pexp + 96 * warp;
      mine[lane] = ea[0];
      mine[32 + lane] = ea[1];
      mine[64 + lane] = eb;
      __syncthreads();
      ea[0] = ea[1] = eb = 0;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        ea[0] = max(ea[0], pexp[96 * w + lane]);
        ea[1] = max(ea[1], pexp[96 * w + 32 + lane]);
        eb = max(eb, pexp[96 * w + 64 + lane]);
      }
      er = warp & 1 ? ea[1] : ea[0];
      if (warp == 0) cexp[lane] = eb;
    }
    // octet o of the chunk: stage o / 2, half o % 2 (a loop over the six octets, their
    // values rotated through x[0], for the instruction cache). A part that is not whole
    // leaves out the second three where K has no more of them, and rows 32-63 where the
    // block has none: those keep what was there, and their outputs are not read.
    const int nst = next.nst, nu = !WHOLE && nst <= 2 ? 3 : 6;
#pragma unroll 1
    for (int u = 0; u < nu; ++u) {
      const int o = warp + (u < 3 ? 0 : 4), t = u < 3 ? u : u - 3;
      const bool isa = t < 2;
      const int v = t == 1 ? lane + 32 : lane;
      if (o < 2 * nst && (WHOLE || t != 1 || tk.m > 32))
        store_planes<S, false>(x[0], t == 0 ? ea[0] : t == 1 ? ea[1] : eb,
                               stage + (o >> 1) * F::STAGE + (isa ? 0 : F::A_BYTES) + (o & 1) * 128 + (v >> 3) * 256 + (v & 7) * 16,
                               isa ? PlaneStep<S>::A1 : PlaneStep<S>::B1, isa ? PlaneStep<S>::A2 : PlaneStep<S>::B2);
#pragma unroll
      for (int w = 0; w < 5; ++w)
#pragma unroll
        for (int y = 0; y < 8; ++y) x[w][y] = x[w + 1][y];
    }
    const bool fresh = S == 8 || kacc == 0;
    kacc += next.kadd;
    last = next.s >= tk.nseg;
    const bool drain = S == 8 || last || kacc + 32 > F::KMAX;
    tc::fence_smem_to_async();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      for (int st = 0; st < nst; ++st) stage_mmas<S>(ts.tmem, stage_a + st * F::STAGE, !(fresh && st == 0));
      tc::commit(tc::smem_addr(&ts.pdone));
    }
    __syncwarp();
    if (drain) kacc = 0;
    if (!last) next = tc_load<S>(p, tk, next.s, next.k0, kacc, q, x);
    bool ok = tc_wait(p, tc::smem_addr(&ts.pdone), ndone & 1);
    ++ndone;
    ok = !__syncthreads_or(!ok);
    if (!ok) return;
    if (!drain) continue;
    tc::fence_after_sync();
    drain_cells<S, true, WHOLE>(ts.tmem, stage + PL_XCH_OFF, er, cexp, tk.m, tk.n - 32 * q, r16);
    tc::fence_before_sync();
    __syncthreads();  // TMEM and exchange reads done before the next MMAs
  }
  if (tid == 0) ts.pdone_n = ndone;  // (read again only after the next part's first barrier)
  store_part(p, tk, q, smem, r16);
}

// OP_SPLIT, part (vectors 16 (q & 3) .., K chunk q >> 2): the chunk's planes of
// 16 vectors, and their exponents (emulated FP64). Lane l of warp w holds vector
// l % 16 and the K octets 2 w + l / 16 + 8 u (u < 8) of the chunk in registers,
// read once: exponents first, then the digits, stored 16 bytes (one core-matrix
// row) at a time. Vectors beyond the tile and the padding of K are zeros. Bound by
// the latency of one round of loads and one of stores; a tile is split once for the
// 2 (w + 1) products and more per 64 rows that read it.
template <int S>
__device__ __noinline__ void run_split(const KParams& p, const Task& tk, int q, double* smem) {
  using F = PlaneFmt<S>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int v = 16 * (q & 3) + (lane & 15), oct0 = 2 * warp + (lane >> 4);
  const int k0 = tk.gcol + kPlaneChunk * (q >> 2), kc = min(kPlaneChunk, tk.zrows - k0);
  const int noct = (kc + kPlaneK - 1) / kPlaneK * 2;
  const bool kcont = tk.flags & TF_KCONT, bside = tk.flags & TF_BSIDE;
  const double* A = resolve(p, tk.cin);
  A += kcont ? (int64_t)v * tk.ldc + (k0 - tk.gcol) : v + (int64_t)(k0 - tk.gcol) * tk.ldc;
  const int64_t step = kcont ? 1 : tk.ldc;
  const bool pairs = kcont && pairs_ok(A, tk.ldc);
  double x[8][8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int k = 8 * (oct0 + 8 * u);
    load_octet(A + (int64_t)k * step, step, pairs, v < tk.m ? kc - k : 0, x[u]);
  }
  int emax = 0;
  const int nch = (tk.zrows + kPlaneChunk - 1) / kPlaneChunk;
  uint8_t* out = p.planes + 16 * (tk.out & OFF_MASK);
  if constexpr (S == 8) {
    int* part = reinterpret_cast<int*>(smem);
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int y = 0; y < 8; ++y) emax = max(emax, biased_exp(x[u][y]));
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 16));
    part[warp * 16 + (lane & 15)] = emax;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 4; ++w) emax = max(emax, part[16 * w + (lane & 15)]);
    if (tid < 16) __stcg(reinterpret_cast<int*>(out) + 64 * (k0 / kPlaneChunk) + v, emax);
    out += 256 * (int64_t)nch;
  }
  out += (int64_t)(k0 / kPlaneK) * F::A_BYTES;
  const int vg = bside ? (v & 31) : v;  // vector inside its plane
  out += (bside ? (v >> 5) * F::B_BYTES : 0) + (vg >> 3) * 256 + (vg & 7) * 16;
#pragma unroll 1
  for (int u = 0; u < 8; ++u) {  // (rotated through x[0], as in run_tc)
    const int o = oct0 + 8 * u;
    if (o < noct)
      store_planes<S, true>(x[0], emax, out + (int64_t)(o >> 1) * F::A_BYTES + (o & 1) * 128,
                            bside ? PlaneStep<S>::B1 : PlaneStep<S>::A1, bside ? PlaneStep<S>::B2 : PlaneStep<S>::A2);
#pragma unroll
    for (int w = 0; w < 7; ++w)
#pragma unroll
      for (int y = 0; y < 8; ++y) x[w][y] = x[w + 1][y];
  }
  tc::fence_global_async();
}

// X[rl][cl] = sign * acc (or cin - acc) over the whole (16 TM) x (8 TN) sub-tile
// (rows / columns beyond the sub-tile get -acc = 0 or are ignored later).
template <int TM, int TN>
__device__ __forceinline__ void acc_to_smem(const KParams& p, const Task& tk, const Sub& sb, const double (&acc)[TM][TN],
                                            double* X, bool sub_cin, double sign) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const double* C = sub_cin ? resolve(p, tk.cin) + sb.r0 + (int64_t)sb.c0 * tk.ldc : nullptr;
  // every load is issued before the first shared-memory store (a store
  // through a generic pointer would otherwise order the loads one by one)
  double v[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int r = tx + 16 * i, c = ty + 8 * j;
      v[i][j] = (sub_cin && r < sb.rm && c < sb.cn) ? __ldcg(C + r + (int64_t)c * tk.ldc) : 0.0;
    }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int r = tx + 16 * i, c = ty + 8 * j;
      const bool in = sub_cin && r < sb.rm && c < sb.cn;
      if (tk.nseg == 0) X[r * LDS + c] = v[i][j];  // no product to subtract (an FP64 instruction saved)
      else X[r * LDS + c] = in ? v[i][j] - acc[i][j] : sign * acc[i][j];
    }
}

// T[r][c] = lower triangle of the dim x dim block at tk.aux (zero above): thread
// t reads rows t % 64 of columns t / 64, +2, +4, ..., every load in flight before
// the first shared-memory store (one round trip to L2).
__device__ __forceinline__ void load_tri(const KParams& p, const Task& tk, int dim, double* T) {
  const double* S = resolve(p, tk.aux);
  const int r = threadIdx.x & (FB - 1), c0 = threadIdx.x / FB;
  constexpr int kStep = NTHREADS / FB, kBatch = FB / kStep;
  double v[kBatch];
#pragma unroll
  for (int u = 0; u < kBatch; ++u) {
    const int c = c0 + u * kStep;
    v[u] = (r < dim && c < dim && r >= c) ? __ldcg(S + r + (int64_t)c * tk.ldx) : 0.0;
  }
#pragma unroll
  for (int u = 0; u < kBatch; ++u) {
    const int c = c0 + u * kStep;
    if (r < dim && c < dim) T[r * LDS + c] = v[u];
  }
}

// out[r0 + r][c0 + c] = X[r][c] for the sub-tile (zero above the diagonal if lower_only)
__device__ __forceinline__ void store_sub(const KParams& p, const Task& tk, const Sub& sb, const double* X,
                                          bool lower_only) {
  double* O = resolve(p, tk.out) + sb.r0 + (int64_t)sb.c0 * tk.ldo;
  for (int e = threadIdx.x; e < sb.rm * sb.cn; e += NTHREADS) {
    const int r = e % sb.rm, c = e / sb.rm;
    O[r + (int64_t)c * tk.ldo] = (lower_only && r + sb.r0 < c + sb.c0) ? 0.0 : X[r * LDS + c];
  }
}

// ---- triangular sweeps on blocks in shared memory (row length LDS) -------
// FP64 runs at 1/64 of the FP32 rate on GB300, so these avoid block-wide
// barriers in their inner loops: independent rows (or columns) are owned by
// one warp and stepped with __syncwarp only.

// X (m x n, m <= 128 / LANES) <- X T^{-T} with the row values in registers. Tn: the
// block POTRF's multipliers T[c][j] / T[j][j] below the diagonal, 1 / T[j][j] on
// it. The LANES lanes of a row hold its columns ph, ph + LANES, ...; step j takes
// the finished (not yet scaled) value y_j of each row from the lane that holds it
// (a shuffle) and subtracts y_j Tn[c][j] from the columns c > j; x = y / diag(T)
// at the end. No shared-memory round trip, division or scaling between two steps.
// LANES = 8, 16, 32 for parts of 16, 8, 4 rows: at most 64 / LANES multiply-adds
// per step and lane (10k and 6k cycles of the FP64 pipe for 8 and 4 rows). A part of
// the block below the diagonal 13.7 -> 9.7 us, against a triangle loaded in four
// round trips, scaled by the pivots in every part and 8-row parts.
template <int LANES>
__device__ __forceinline__ void trsm_rows(double* X, const double* Tn, int m, int n) {
  constexpr int R = 32 / LANES, Q = FB / LANES;  // rows per warp, columns per lane
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = warp * R + lane % R, ph = lane / R;
  const bool own = r < m;
  double y[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int c = ph + LANES * q;
    y[q] = own && c < n ? X[r * LDS + c] : 0.0;
  }
#pragma unroll
  for (int j = 0; j < FB; ++j) {
    if (j >= n) break;
    const double yj = __shfl_sync(0xffffffffu, y[j / LANES], lane % R + R * (j % LANES));
#pragma unroll
    for (int q = j / LANES; q < Q; ++q) {
      const int c = ph + LANES * q;
      if (c > j) y[q] = fma(-yj, Tn[c * LDS + j], y[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int c = ph + LANES * q;
    if (own && c < n) X[r * LDS + c] = y[q] * Tn[c * LDS + c];
  }
}

// X (m x m) <- T^{-1} X for X the identity, T lower m x m, rcp[j*LDS] = 1 / T[j][j].
// Columns are independent; warp w owns columns 4q + w (interleaved, so that the
// triangular work is balanced), and the columns c > j, still zero in row j, are skipped.
__device__ __forceinline__ void invert_cols(double* X, const double* T, const double* rcp, int m) {
  const int lane = threadIdx.x & 31, c = 4 * (lane & 15) + (threadIdx.x >> 5), half = lane >> 4;
  for (int j = 0; j < m; ++j) {
    const bool act = c <= j;
    if (act && half == 0) X[j * LDS + c] *= rcp[j * LDS];
    __syncwarp();
    if (act) {
      const double xj = X[j * LDS + c];
      for (int r = j + 1 + half; r < m; r += 2) X[r * LDS + c] -= T[r * LDS + j] * xj;
    }
    __syncwarp();
  }
}

// After a block POTRF has released its successors: its log-diagonal partial
// sum (in a fixed tree order) and its first pivot that is not positive.
__device__ void finish_potrf(const KParams& p, const Task& tk, const double* S) {
  const int tid = threadIdx.x;
  __shared__ double s_lg[2];
  __shared__ int s_bad;
  if (tid == 0) s_bad = FB;
  __syncthreads();
  if (tid < FB) {
    double lg = tid < tk.n ? log(S[PT_DIAG + tid]) : 0.0;
    if (tid < tk.n && !(S[PT_PIV + tid] > 0.0)) atomicMin(&s_bad, tid);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lg += __shfl_down_sync(0xffffffffu, lg, o);
    if ((tid & 31) == 0) s_lg[tid >> 5] = lg;
  }
  __syncthreads();
  if (tid == 0) {
    p.logdet_part[tk.diag] = s_lg[0] + s_lg[1];
    if (s_bad < FB) {
      atomicCAS(&p.st->code, 0, STILES_DEV_NOT_SPD);
      atomicMin(&p.st->spd_col, (unsigned long long)tk.gcol + (unsigned long long)s_bad);
      if (p.badpiv) p.badpiv[tk.diag] = s_bad;
    }
  }
}

template <int TM, int TN>
__device__ void run_sub(const KParams& p, const Task& tk, const Sub& sb, double* smem) {
  double* As = smem;             // KC x LDS
  double* Bs = smem + KC * LDS;  // KC x LDS
  double* T = smem;              // FB x LDS, reuses As/Bs after the K-loop
  double* X = smem + 2 * KC * LDS;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m = tk.m, n = tk.n;
  double acc[TM][TN];
  // the small parts of critical paths have their input block in flight meanwhile
  constexpr bool EARLY = TM == 1 && TN == 2;
  double cin[TM][TN];
  if constexpr (EARLY) {
    const double* C = tk.op == OP_UPD ? resolve(p, tk.cin) + sb.r0 + (int64_t)sb.c0 * tk.ldc : nullptr;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int r = tx + 16 * i, c = ty + 8 * j;
        cin[i][j] = C && r < sb.rm && c < sb.cn ? __ldcg(C + r + (int64_t)c * tk.ldc) : 0.0;
      }
  }
  if (tk.op != OP_TRTRI) accumulate<TM, TN>(p, tk, sb, acc, As, Bs);

  switch (tk.op) {
    case OP_UPD:
    case OP_STORE:
    case OP_NEG: {
      double* O = resolve(p, tk.out) + sb.r0 + (int64_t)sb.c0 * tk.ldo;
      const double* C = tk.op == OP_UPD ? resolve(p, tk.cin) + sb.r0 + (int64_t)sb.c0 * tk.ldc : nullptr;
      // an off-diagonal Sigma block is final when its NEG task writes it (the
      // planner emits NEG and SYMUPD tasks only with outputs, and SYMUPD
      // mirror blocks, in the Sigma buffer, so the offsets below stay inside it)
      double* Om = tk.op == OP_NEG && p.smirror ? p.smirror + (O - p.buf[BUF_S]) : nullptr;
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int r = tx + 16 * i, c = ty + 8 * j;
          if (r < sb.rm && c < sb.cn) {
            double v = acc[i][j];
            if (tk.op == OP_UPD) v = (EARLY ? cin[i][j] : __ldcg(C + r + (int64_t)c * tk.ldc)) - v;
            else if (tk.op == OP_NEG || (tk.flags & TF_NEG)) v = -v;
            O[r + (int64_t)c * tk.ldo] = v;
            if (Om) Om[r + (int64_t)c * tk.ldo] = v;
          }
        }
      break;
    }
    case OP_SYMUPD: {
      acc_to_smem<TM, TN>(p, tk, sb, acc, X, true, 1.0);
      __syncthreads();
      double* O = resolve(p, tk.out);
      // the diagonal tile's Sigma blocks are final when their SYMUPD writes them
      if ((tk.flags & TF_SYM_DIAG) && sb.r0 == sb.c0) {  // diagonal sub-block: keep its lower triangle, mirror it
        double* D = O + sb.r0 + (int64_t)sb.c0 * tk.ldo;
        double* Dm = p.smirror ? p.smirror + (D - p.buf[BUF_S]) : nullptr;
        for (int e = tid; e < sb.rm * sb.cn; e += NTHREADS) {
          const int r = e % sb.rm, c = e / sb.rm;
          const double v = r >= c ? X[r * LDS + c] : X[c * LDS + r];
          D[r + (int64_t)c * tk.ldo] = v;
          if (Dm) Dm[r + (int64_t)c * tk.ldo] = v;
        }
      } else {
        // this sub-block, and its transpose into the mirror position: inside the
        // same block for a diagonal block, else the mirror block (aux)
        double* D = O + sb.r0 + (int64_t)sb.c0 * tk.ldo;
        const bool dblk = tk.flags & TF_SYM_DIAG;
        double* M = dblk ? O + sb.c0 + (int64_t)sb.r0 * tk.ldo : resolve(p, tk.aux) + sb.c0 + (int64_t)sb.r0 * tk.ldx;
        const int ldm = dblk ? tk.ldo : tk.ldx;
        double* Dm = p.smirror ? p.smirror + (D - p.buf[BUF_S]) : nullptr;
        double* Mm = p.smirror ? p.smirror + (M - p.buf[BUF_S]) : nullptr;
        for (int e = tid; e < sb.rm * sb.cn; e += NTHREADS) {
          const int r = e % sb.rm, c = e / sb.rm;
          D[r + (int64_t)c * tk.ldo] = X[r * LDS + c];
          if (Dm) Dm[r + (int64_t)c * tk.ldo] = X[r * LDS + c];
        }
        for (int e = tid; e < sb.rm * sb.cn; e += NTHREADS) {
          const int c = e % sb.cn, r = e / sb.cn;
          M[c + (int64_t)r * ldm] = X[r * LDS + c];
          if (Mm) Mm[c + (int64_t)r * ldm] = X[r * LDS + c];
        }
      }
      break;
    }
    case OP_TRSM_RLT: {  // X = (C - acc) T^{-T}, T lower n x n: rows are independent
      load_tri(p, tk, n, T);
      acc_to_smem<TM, TN>(p, tk, sb, acc, X, true, 1.0);
      __syncthreads();
      if (sb.rm <= 4) trsm_rows<32>(X, T, sb.rm, n);
      else if (sb.rm <= 8) trsm_rows<16>(X, T, sb.rm, n);
      else trsm_rows<8>(X, T, sb.rm, n);  // parts have at most 16 rows
      __syncthreads();
      store_sub(p, tk, sb, X, false);
      break;
    }
    default:
      if constexpr (TM == 4 && TN == 8) {
        switch (tk.op) {
          case OP_POTRF: {
            // (finish_potrf does the rest, once the successors are released)
            acc_to_smem<TM, TN>(p, tk, sb, acc, X, true, 1.0);
            __syncthreads();
            potrf_smem(X, smem, n);
            double* O = resolve(p, tk.out);
            double* Mo = resolve(p, tk.aux);  // multipliers and 1 / L_jj for the solves with this block
            for (int c = tid >> 5; c < n; c += NTHREADS / 32) {  // a warp per column
              const double rs = smem[PT_RS + c], rcp = smem[PT_RCP + c];
#pragma unroll
              for (int h = 0; h < FB / 32; ++h) {
                const int r = 32 * h + (tid & 31);
                double l = 0.0;
                if (32 * h + 31 >= c) {  // not all above the diagonal: no FP64 instruction for those
                  if (r >= c) l = r == c ? smem[PT_DIAG + c] : X[r * LDS + c] * rs;
                  if (r >= c && r < n) Mo[r + (int64_t)c * tk.ldx] = r == c ? rcp : l * rcp;
                }
                if (r < n) O[r + (int64_t)c * tk.ldo] = l;
              }
            }
            break;
          }
          case OP_TRTRI: {  // X = T^{-1}, T lower m x m: solve T X = I column by column
            load_tri(p, tk, m, T);
            for (int e = tid; e < FB * FB; e += NTHREADS) {
              const int r = e % FB, c = e / FB;
              X[r * LDS + c] = r == c ? 1.0 : 0.0;
            }
            __syncthreads();
            double* rcp = T + FB;
            if (tid < m) rcp[tid * LDS] = 1.0 / T[tid * LDS + tid];
            __syncthreads();
            invert_cols(X, T, rcp, m);
            __syncthreads();
            store_sub(p, tk, sb, X, true);
            break;
          }
          default:
            break;
        }
      }
      break;
  }
}

// OP_ZERO: the zrows x n block above the task's output block (column-major,
// leading dimension ldo) set to zero.
__device__ void run_zero(const KParams& p, const Task& tk) {
  double* Z = resolve(p, tk.out) - tk.zrows;
  for (int e = threadIdx.x; e < tk.zrows * tk.n; e += NTHREADS) Z[e % tk.zrows + (int64_t)(e / tk.zrows) * tk.ldo] = 0.0;
}

// Run part q of task tk (the planner only splits operations whose parts are
// independent: products, the row-wise TRSM and the mirrored Sigma_ii store).
template <bool TC>
__device__ void run_task(const KParams& p, const Task& tk, int t, int q, double* smem, TcShared* ts) {
#ifdef STILES_CHECKED
  // every part's accesses inside the launch's buffers (OP_PREP's bases have a layout of their own)
  unsigned present = 0;
  for (int x = 0; x < 4; ++x) present |= (p.buf[x] != nullptr) << x;
  const Bounds all{p.buf_len, present, p.planes ? p.plane_units : 0, INT32_MAX};
  if (tk.op != OP_PREP && part_fault(tk, q, p.segs, all)) {
    if (threadIdx.x == 0) check_fail(p, 7, t, q);
    return;
  }
#endif
  if (tk.op == OP_PREP) {
    run_prep(p, tk, t);
    return;
  }
  if (tk.op == OP_ZERO) {
    run_zero(p, tk);
    return;
  }
  if (tk.op == OP_JOIN) return;  // a dependency point only
  if constexpr (TC) {
    if (tk.op == OP_SPLIT) {
      if (tk.prec == PREC_EMU64) run_split<8>(p, tk, q, smem);
      else run_split<4>(p, tk, q, smem);
      return;
    }
    if (tk.flags & TF_PLANES) {
      if (tk.prec == PREC_EMU64) run_planes<8>(p, tk, q, smem, *ts);
      else run_planes<4>(p, tk, q, smem, *ts);
      return;
    }
    if (tk.prec != PREC_FP64) {
      const bool whole = !(tk.flags & TF_SMALL);
      if (tk.prec == PREC_EMU64) whole ? run_tc<8, true>(p, tk, q, smem, *ts) : run_tc<8, false>(p, tk, q, smem, *ts);
      else whole ? run_tc<4, true>(p, tk, q, smem, *ts) : run_tc<4, false>(p, tk, q, smem, *ts);
      return;
    }
  }
  const Sub sb = part_sub(tk.pmode, tk.m, tk.n, q);
  if (sb.rm <= 0 || sb.cn <= 0) return;
  switch (tk.pmode) {
    case PM_ROWS2: run_sub<2, 8>(p, tk, sb, smem); break;
    case PM_ROWS4:
    case PM_ROWS8:
    case PM_ROWS4F: run_sub<1, 8>(p, tk, sb, smem); break;
    case PM_TRI16:
    case PM_GRID16: run_sub<1, 2>(p, tk, sb, smem); break;
    case PM_QUAD4:
    case PM_TRI3: run_sub<2, 4>(p, tk, sb, smem); break;
    default: run_sub<4, 8>(p, tk, sb, smem); break;
  }
}

__device__ __forceinline__ unsigned smid() {
  unsigned r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return r;
}

// Per-CTA state of the tensor path, in static shared memory of the kernel
// instance that has one.
template <bool TC>
__device__ __forceinline__ TcShared* tc_shared() {
  if constexpr (TC) {
    __shared__ TcShared ts;
    return &ts;
  } else {
    return nullptr;
  }
}

// Two instances: TC = false for plans whose products are all FP64 (no
// tensor-core code at all), TC = true for plans with reduced-precision parts.
template <bool TC>
__global__ void __launch_bounds__(NTHREADS, 2) persistent_kernel(const __grid_constant__ KParams p) {
  extern __shared__ __align__(16) double smem[];
  __shared__ int s_item;
  TcShared* ts = tc_shared<TC>();
  // plans with reduced-precision products hold TC_COLS TMEM columns and two
  // completion barriers for the kernel's lifetime (two CTAs per SM: 512)
  if constexpr (TC) {
    if (threadIdx.x < 32) tc::tmem_alloc<TC_COLS>(&ts->tmem);
    if (threadIdx.x == 0) {
      for (int x = 0; x < PL_SLOTS; ++x) {
        tc::mbar_init(tc::smem_addr(&ts->pfull[x]), 1);
        tc::mbar_init(tc::smem_addr(&ts->pempty[x]), 1);
      }
      tc::mbar_init(tc::smem_addr(&ts->pdone), 1);
      ts->pdone_n = ts->pstage = 0;
      tc::fence_mbar_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  }
  // request server: idle workers give up this long after the kernel started
  const unsigned long long deadline = p.serve ? gtimer() + p.sv.deadline : 0ull;
  int kept = -1;  // warp 0: a part released to this worker by its last task
  for (;;) {
    unsigned long long t_claim = 0;
    if (threadIdx.x < 32) {
      if (p.trace && threadIdx.x == 0) t_claim = gtimer();
      const int v = kept >= 0 ? kept : pop_task(p, deadline);
      if (threadIdx.x == 0) s_item = v;
    }
    __syncthreads();
    const int v = s_item;
    if (v < 0) break;
    const int t = v / kMaxParts, q = v % kMaxParts;
#ifdef STILES_CHECKED
    if (t >= p.ntasks || q >= load_task(p, t).parts) {
      if (threadIdx.x == 0) check_fail(p, 8, t, q);
      break;
    }
#endif
    unsigned long long t_ready = 0;
    if (p.trace && threadIdx.x == 0) t_ready = gtimer();
    const Task tk = load_task(p, t);
    // the first 32 successors, read ahead (in flight while the part runs)
    int succ = -1;
    if (threadIdx.x < 32 && (int)threadIdx.x < tk.nsucc) succ = __ldcg(p.succ + tk.succ0 + threadIdx.x);
    run_task<TC>(p, tk, t, q, smem, ts);
    TaskWord word{0u};
    if (threadIdx.x < 32 && succ >= 0) word = load_task_word(p, succ);
    __syncthreads();
    int last = tk.parts <= 1;
    if (threadIdx.x < 32) {
      fence_dev();
      const bool by_part = counts_parts(tk);
      if (!by_part && !last) {
        if (threadIdx.x == 0) last = add_relaxed_i(p.q.pdone + t, 1) == tk.parts - 1;
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) fence_dev();
      }
      kept = -1;
      if (by_part || last) kept = release_successors(p, tk, succ, word);
      if (by_part && !last && threadIdx.x == 0) {
        last = add_relaxed_i(p.q.pdone + t, 1) == tk.parts - 1;
        if (last) fence_dev();
      }
    }
    if (tk.op == OP_POTRF) finish_potrf(p, tk, smem);  // what no successor waits for
    if (threadIdx.x == 0) {
      if (tk.op == OP_POTRF) fence_dev();
      if (last) account_task(p, t);
      if (p.trace) {  // one record per task part
        unsigned long long* tr = p.trace + kTraceWords * (kMaxParts * (size_t)t + q);
        tr[0] = t_claim;
        tr[1] = t_ready;
        tr[2] = gtimer();
        tr[3] = ((unsigned long long)smid() << 32) | ((unsigned long long)blockIdx.x << 12) |
                ((unsigned long long)tk.prec << 10) | ((unsigned long long)last << 9) |
                ((unsigned long long)(tk.flags & TF_URGENT) << 7) | tk.op;
      }
    }
  }
  // every part waited for its MMAs before it returned; after a timeout those of the
  // part that raised it have had a whole wait budget
  if constexpr (TC) {
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) {
      tc::fence_after_sync();
      tc::tmem_dealloc<TC_COLS>(ts->tmem);
    }
    if (threadIdx.x == 0) {
      for (int x = 0; x < PL_SLOTS; ++x) {
        tc::mbar_inval(tc::smem_addr(&ts->pfull[x]));
        tc::mbar_inval(tc::smem_addr(&ts->pempty[x]));
      }
      tc::mbar_inval(tc::smem_addr(&ts->pdone));
    }
  }
}

// Dynamic shared memory of a launch: the FP64 tasks' staging and block
// regions, or more when the plan has tensor-core parts.
size_t kernel_smem_bytes(bool use_tc) {
  const size_t fp64 = sizeof(double) * (size_t)(2 * KC * LDS + FB * LDS);
  return use_tc && (size_t)PL_SMEM_BYTES > fp64 ? (size_t)PL_SMEM_BYTES : fp64;
}

int kernel_threads() { return NTHREADS; }

const void* persistent_kernel_ptr(bool use_tc) {
  return use_tc ? (const void*)persistent_kernel<true> : (const void*)persistent_kernel<false>;
}

// The shared-memory limit is a per-device attribute of each kernel instance:
// it is set once for every device the process launches on (the current one).
cudaError_t configure_persistent() {
  constexpr int kMaxDevices = 64;
  static std::atomic<bool> configured[kMaxDevices];
  static std::mutex mu;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool cached = dev >= 0 && dev < kMaxDevices;
  if (cached && configured[dev].load(std::memory_order_acquire)) return cudaSuccess;
  std::lock_guard<std::mutex> lock(mu);
  if (cached && configured[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  e = cudaFuncSetAttribute(persistent_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kernel_smem_bytes(false));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(persistent_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kernel_smem_bytes(true));
  if (e == cudaSuccess && cached) configured[dev].store(true, std::memory_order_release);
  return e;
}

cudaError_t kernel_occupancy(bool use_tc, int* blocks_per_sm) {
  cudaError_t e = configure_persistent();
  if (e != cudaSuccess) return e;
  return use_tc ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, persistent_kernel<true>, NTHREADS,
                                                                kernel_smem_bytes(true))
                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, persistent_kernel<false>, NTHREADS,
                                                                kernel_smem_bytes(false));
}

cudaError_t launch_persistent(const KParams& p, int grid, cudaStream_t stream) {
  cudaError_t e = configure_persistent();
  if (e != cudaSuccess) return e;
  if (p.use_tc)
    persistent_kernel<true><<<grid, NTHREADS, kernel_smem_bytes(true), stream>>>(p);
  else
    persistent_kernel<false><<<grid, NTHREADS, kernel_smem_bytes(false), stream>>>(p);
  return cudaGetLastError();
}

}  // namespace stiles
