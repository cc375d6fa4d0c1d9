// The persistent step kernel: one launch runs one coarse step (Algorithm 1 of
// arXiv 2402.04606, unrolled over every level of every live instance) as a
// list of phases built by the host (api.cpp, build_step_phases):
//   PH_POSE   the poses of the coarse step of the moving bodies (Sec. 3.4-3.6)
//   PH_GEOM   the IBM geometry of one finest step of the moving bodies
//   PH_C2F    coarse-to-fine copy into the two halo layers (Sec. 2.4 step 2) at
//             the start of the coarse step; later copies are done by the coarse
//             sweep that produces the values (its cells next to the finer region)
//   PH_FUSED  pull streaming + boundary rules + collision of a work list of
//             blocks (Eqs. 3-10; the fine-to-coarse merge of Sec. 2.4 step 6
//             inside the coarse pull)
//   PH_IBM    multi-direct forcing of the bodies on their finest level (Sec. 2.2)
//   PH_FSUM   the FP64 force and moment sums of the coarse step (Eq. 16)
//   PH_FORCED FP64: the forced collision of the bodies' stencil cells, after the
//             IBM and the sweep of its sub-step (ibm_run's LIST)
// Every phase is cut into tasks of one thread block.  A phase may start once
// every task of the phases it depends on has finished: each phase has a
// counter of finished tasks, raised by one reduction with release semantics
// after each task's writes; a block that wants to run a phase reads its
// dependencies' counters (relaxed loads, all at once) and, once every one is
// full, fences with acquire semantics before the task reads.  A phase with no
// work and no dependency is finished from the start; one with no work but
// with dependencies gets one empty task, so that it finishes after them.
//
// Scheduling.  Critical phases form one list in a topological order; bulk
// phases (level-0 blocks with no dependency inside the step, most of the
// cells of a large instance) form a queue of their own.  Warp 0 of a thread
// block looks at a window of critical phases after the first one that still
// has tasks to hand out and takes a task of one whose dependencies have
// finished; else it takes a bulk task; only when the bulk queue is empty does
// it take the first critical task not yet taken and wait for its
// dependencies.  Every phase depends only on earlier critical phases, a
// waiting block holds a task of the first phase with tasks left, and all
// thread blocks are resident at once (cooperative launch), so the earliest
// unfinished task can always run: the step completes.  Each wait is still
// bounded (spin_ns of device time): past it the thread block raises
// ERRB_TIMEOUT and the abort flag, and every block leaves at its next
// decision, so a broken schedule returns an error instead of hanging the
// device.  Two exceptions to this hand-out, explained where they begin below:
// the IBM servers (an IBM task waits once more, before its stores, for its
// sub-step's sweep, which comes before it in the order; where a thread block
// takes both kinds, an IBM task is handed out only after all of that sweep's),
// and the fixed owners of single-level launches.
//
// Reads of buffers that other thread blocks wrote earlier in the launch use
// plain loads (no read-only cache path): the acquire fence after the
// dependency counters orders them after those writes.
#pragma once
#include "lbm_device.cuh"

namespace {

// the sweeps' scalar path holds the solid links (without them the D = 40
// cylinder measured the same, 49.1 us per coarse step)
constexpr bool STEP_SOLID = true;

enum { STEP_EXIT = 0, STEP_RUN = 1 };

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

template <class S>
__device__ __forceinline__ S* step_buf(const StepArgs& A, int i) {
    return i < 0 ? nullptr : (S*)(i == 0 ? A.f0 : A.f1);
}

// list items per task of a fused phase: the vector mapping covers one block
// per B * B / CPT threads (CPT cells per thread), the scalar one B * B cells
// per item over the thread block
template <class S, int B>
__device__ __forceinline__ bool fused_vec(const StepArgs& A, const StepPhase& ph, int n, int coll) {
    return B >= 16 && !(coll & COLL_SOLID) && ph.arg == 0 && A.vec_min_cells >= 0 &&
           (long long)n * B * B >= A.vec_min_cells;
}

template <class S, int B>
__device__ __forceinline__ int fused_items(bool vec, int T) {
    constexpr int CPT = sizeof(S) == 2 ? 8 : 4;
    return vec ? T / (B * B / CPT) : (T >= B * B ? T / (B * B) : 1);
}

// the most list items whose blocks' data a task of a sweep reads ahead
#define STEP_META_MAX (STEP_MAX_THREADS / 64)

// How fused phase ph with n items is cut into tasks: `per` items per round and
// `rounds` rounds per task, or (parts > 1) every item into `parts` tasks of its
// own.  Handing out a task costs some microseconds of dependent L2 round
// trips, so a task holds as many items as fill the thread block, and a bulk
// task (or one of a list of more than 8 fillings of every thread block) up to
// bulk_rounds fillings: as many as give every thread block the same number of
// tasks.  crit_items caps a critical task's items (a short sweep other phases
// wait for).  In FP64 the pipe is the bound (a 16 x 16 item keeps one SM busy for
// 11 us), so there a short list is spread over every SM, in parts of an item
// when it has fewer items than half the thread blocks.
// Measured against bulk tasks of a fixed 8 rounds, us per step: 128^2 in FP64
// (64 items: 8 tasks on 152 SMs) 41.9 -> 13.1; 2960 x 1488 with the LES
// collision in FP32 (538 tasks for 456 thread blocks, two unequal waves) 92 ->
// 71; a 1120 x 640 level of 16-bit blocks (15 tasks of up to 145 us each) in a
// pitching section's step 117 -> 103.  Spreading short FP32 lists over every SM
// as well measured slower (a D = 40 cylinder's step 64 -> 86): there the hand-out
// is the cost.
struct TaskShape {
    int per, rounds, parts;
    __device__ __forceinline__ int tasks(int n) const {
        return parts > 1 ? n * parts : (n + per * rounds - 1) / (per * rounds);
    }
};
// A launch of fixed owners (StepArgs::fixed) cuts a sweep into at most one task
// per thread block: handing out costs nothing there, so a short list is spread
// over all of them.
template <class S, int B>
__device__ __forceinline__ TaskShape task_shape(const StepArgs& A, const StepPhase& ph, int n, bool vec, int T,
                                                int grid) {
    TaskShape t{fused_items<S, B>(vec, T), 1, 1};
    const long long fill = (long long)t.per * grid;  // items of one filling of every thread block
    if (A.fixed) {
        t.rounds = (int)((n + fill - 1) / fill);
        if (n < fill) t.per = (n + grid - 1) / grid;
    } else if (ph.bulk || n > 8 * fill) {
        const long long waves = (n + fill * A.bulk_rounds - 1) / (fill * A.bulk_rounds);
        t.rounds = (int)((n + fill * waves - 1) / (fill * waves));
    } else if (A.crit_items > 0) {
        t.per = min(t.per, A.crit_items);
    } else if (!vec && n > fill) {
        // a critical sweep of more fillings than one: a single task per thread
        // block where its blocks' data fit (STEP_META_MAX)
        const int want = (int)((n + fill - 1) / fill) * t.per;
        t.per = min(want, min(STEP_META_MAX, T / 32) / t.per * t.per);
    }
    if (sizeof(S) == 8 && n < fill) t.per = (n + grid - 1) / grid;
    if (sizeof(S) == 8 && !vec && 2LL * n <= grid) t.parts = 4LL * n <= grid ? 4 : 2;
    return t;
}

// tasks of phase p at this launch (from the device list lengths)
template <class S, int B>
__device__ int step_ntasks(const DevPool& P, const StepArgs& A, const StepPhase& ph, int T, int grid) {
    const int n = A.counts[ph.count_idx];
    if (n <= 0) return 0;
    switch (ph.kind) {
    case PH_FUSED: {
        return task_shape<S, B>(A, ph, n, A.any_vec && fused_vec<S, B>(A, ph, n, P.coll), T, grid).tasks(n);
    }
    case PH_C2F: {
        const int per = T >= B * B ? T / (B * B) : 1;
        return (n + per - 1) / per;
    }
    case PH_FSUM:
    case PH_FORCED: return n * ph.arg;
    default: return n;  // one body per task
    }
}

// the scalar mapping of a fused or copy phase: items [i0, i0 + k) of the list,
// B * B cells each, spread over the thread block's threads
template <class F>
__device__ __forceinline__ void for_cells(int n, int i0, int k, int BB, F&& fn) {
    const int cells = k * BB;
    for (int c = threadIdx.x; c < cells; c += blockDim.x) {
        const int item = i0 + c / BB;
        if (item < n) fn(item, c % BB);
    }
}

// A fused phase's task.  gate(): see step_task.  A critical task on the
// scalar mapping first reads its blocks' data (slot tables, neighbours and
// their types, children) into shared memory, which it may do before the
// phases it depends on have finished: after the gate only the population
// and force loads remain on its path.
// key: which task's blocks' data the shared memory holds (a thread block of a
// launch of fixed owners runs the same task in every step, and reads them once;
// there a list is cut the same way in every phase, which elsewhere it is not: a
// level-0 list is bulk in the first step and critical in the others.  A key of the
// items themselves would hold them there too, and gained a D = 128 cylinder 0.7 %,
// but cost every launch registers: 4096^2 in FP32 200.6 -> 204.3 us per step).
template <class S, class C, int B, int COLL, bool VEC, class G>
__device__ void step_fused(const DevPool& P, const StepArgs& A, const StepPhase& ph, int local, int grid, int2& key,
                           G& gate) {
    __shared__ SlotMeta<C> meta[STEP_META_MAX];
    const int n = A.counts[ph.count_idx];
    const int* list = A.lists + ph.list_off;
    const S* fin = step_buf<S>(A, ph.fin);
    S* fout = step_buf<S>(A, ph.fout);
    const S* ffine = step_buf<S>(A, ph.ffine);
    S* fhalo = ph.fold ? step_buf<S>(A, ph.ffine) : nullptr;  // the coarse-to-fine copy rides on this sweep
    const int T = blockDim.x;
    const bool vec = VEC && fused_vec<S, B>(A, ph, n, P.coll);
    const TaskShape sh = task_shape<S, B>(A, ph, n, vec, T, grid);
    const int per = sh.per, rounds = sh.rounds;
    if (rounds == 1 && !vec && per <= STEP_META_MAX && per <= T / 32) {
        const int i0 = sh.parts > 1 ? local / sh.parts : local * per, ne = min(n, i0 + per), w = threadIdx.x >> 5;
        // its cells: those of its items, or a part of one item's
        const int len = sh.parts > 1 ? B * B / sh.parts : (ne - i0) * B * B;
        const int c0 = sh.parts > 1 ? (local - i0 * sh.parts) * len : 0;
        const bool held = A.fixed && key.x == ph.list_off && key.y == local;
        if (!held && i0 + w < ne) load_meta<C>(P, list[i0 + w], ph.level, meta[w]);
        if (!gate(true)) return;
        if (A.fixed && threadIdx.x == 0) key = make_int2(ph.list_off, local);
        for (int c = c0 + threadIdx.x; c < c0 + len; c += T) {
            const SlotMeta<C>& m = meta[c / (B * B)];
            const int cell = c % (B * B);
            fused_cell<S, C, COLL, STEP_SOLID, MetaS<C>>(P, MetaS<C>{&m}, fin, fout, ffine, m.type, P.inst[m.inst], ph.level,
                                                 cell % B, cell / B, fhalo);
        }
        return;
    }
    if (!gate(false)) return;
    if constexpr (B >= 16 && VEC) {
        if (vec) {
            const int i0 = local * rounds * per, end = min(n, i0 + rounds * per);
            if (sizeof(S) == 2 && (P.coll & COLL_SHIFT))
                fused_vec_run<S, C, B, COLL, false, true>(P, list, end, i0, per, fin, fout, ffine, ph.level, fhalo);
            else
                fused_vec_run<S, C, B, COLL, false, false>(P, list, end, i0, per, fin, fout, ffine, ph.level, fhalo);
            return;
        }
    }
    for (int r = 0; r < rounds; r++) {
        const int i0 = (local * rounds + r) * per;
        if (i0 >= n) break;
        const int ne = min(n, i0 + per);  // this round's items end here
        for_cells(ne, i0, per, B * B, [&](int item, int cell) {
            const int slot = list[item];
            fused_cell<S, C, COLL, STEP_SOLID>(P, fin, fout, ffine, slot, P.slot_type[slot], P.inst[P.slot_inst[slot]],
                                          ph.level, cell % B, cell / B, fhalo);
        });
    }
}

// One task of phase ph.  gate(prologue) is called exactly once by the whole
// thread block: it waits, when the task was taken before the phases it
// depends on had finished, for them; the task reads nothing they write
// before it.  prologue: the task wrote shared memory before it (a barrier
// is then due even when there is nothing to wait for).  It returns false
// when the launch is aborting (the task then stops).
// An IBM task waits before its stores for the sweep of its sub-step
// (ph.after): await() by one warp, swept() by all after a barrier (ibm_run).
template <class S, class C, int B, int COLL, bool VEC, class G, class G1, class G2>
__device__ void step_task(const DevPool& P, const StepArgs& A, const StepPhase& ph, int local, int grid, int2& key,
                          unsigned char* smraw, IbmShared& sh, G& gate, G1& await, G2& swept) {
    const int* list = A.lists + ph.list_off;
    if (A.counts[ph.count_idx] <= 0) {  // the empty task of a phase with no work
        gate(false);
        return;
    }
    switch (ph.kind) {
    case PH_FUSED: step_fused<S, C, B, COLL, VEC>(P, A, ph, local, grid, key, gate); break;
    case PH_IBM:
        ibm_run<S, C, COLL, sizeof(S) == STEP_LIST_BYTES, true>(P, list[local], step_buf<S>(A, ph.fin),
                                                                step_buf<S>(A, ph.fout), ph.level, 0, 1, ph.arg, smraw,
                                                                sh, gate, await, swept);
        break;
    default: {
        if (!gate(false)) return;
        switch (ph.kind) {
        case PH_C2F: {
            const int n = A.counts[ph.count_idx], k = blockDim.x >= B * B ? blockDim.x / (B * B) : 1;
            const S* fc = step_buf<S>(A, ph.fin);
            S* ff = step_buf<S>(A, ph.fout);
            for_cells(n, local * k, k, B * B, [&](int item, int cell) { c2f_cell<S>(P, list[item], cell, fc, ff); });
            break;
        }
        case PH_GEOM: ibm_geom_run<C>(P, list[local], ph.arg, smraw, sh); break;
        case PH_POSE: pose_run(P, list[local]); break;
        case PH_FORCED:
            if constexpr (sizeof(S) == STEP_LIST_BYTES)
                ibm_forced_run<S, C, COLL>(P, list[local / ph.arg], step_buf<S>(A, ph.fin), step_buf<S>(A, ph.fout),
                                           ph.level, local % ph.arg, ph.arg);
            break;
        case PH_FSUM: force_sum_run<C>(P, list[local / ph.arg], local % ph.arg, sh.red); break;
        default: break;
        }
    }
    }
}

// the last phase whose first task index (exclusive prefix `first`) is at most t
__device__ __forceinline__ int phase_of(const int* first, int nph, int t) {
    int lo = 0, hi = nph - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= t)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int ld_relaxed(const int* p) { return *(const volatile int*)p; }

__device__ __forceinline__ void step_abort(const DevPool& P, const StepArgs& A, int bit) {
    atomicOr(P.err, bit);
    atomicExch(&A.ctl->abort, 1);
}

__device__ __forceinline__ int ld_relaxed_gpu(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add(int* p, int v) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ int ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The dependencies of every phase, copied to shared memory at the start of
// the launch (the phase table does not change during it).
struct StepDeps {
    int n[STEP_MAX_PHASES];  // their number; from bit 8 on, 1 + the phase awaited before the stores (StepPhase::after)
    unsigned short d[STEP_MAX_PHASES][8];
};

// One thread: has every phase that q depends on finished all its tasks?
// Relaxed loads, issued together: a screen; a yes is confirmed by
// deps_acquire before the task runs.
__device__ __forceinline__ bool deps_screen(const StepArgs& A, const StepDeps& D, int q, const int* ntask) {
    const int nd = D.n[q] & 255;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (k < nd) {
            const int d = D.d[q][k];
            ok &= ld_relaxed_gpu(&A.ctl->done[d]) >= ntask[d];
        }
    }
    return ok;
}

// Warp 0, all lanes: the same question with acquire loads, lane k reading
// dependency k (one round trip); after a yes, the writes of those phases are
// visible to the warp and, through the barrier that follows, to the block.
__device__ __forceinline__ bool deps_acquire(const StepArgs& A, const StepDeps& D, int q, const int* ntask) {
    const int lane = threadIdx.x & 31;
    bool ok = true;
    if (lane < (D.n[q] & 255)) {
        const int d = D.d[q][lane];
        ok = ld_acquire(&A.ctl->done[d]) >= ntask[d];
    }
    return __all_sync(0xffffffffu, ok);
}

// Warp 0, all lanes: wait until ready() (acquire loads, the same answer in
// every lane), bounded by A.spin_ns of device time; false when the launch is
// aborting (by this wait or another)
template <class R>
__device__ bool wait_until(const DevPool& P, const StepArgs& A, R&& ready) {
    const unsigned long long t0 = global_ns();
    for (unsigned ns = 16;; ns = ns < 64 ? 2 * ns : ns) {  // short naps: each poll is an L2 round trip anyway
        if (ready()) return true;
        int stop = 0;
        if ((threadIdx.x & 31) == 0) {
            if (ld_relaxed(&A.ctl->abort)) {
                stop = 1;
            } else if ((long long)(global_ns() - t0) >= A.spin_ns) {
                step_abort(P, A, ERRB_TIMEOUT);
                stop = 1;
            }
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) return false;
        __nanosleep(ns);
    }
}

// VEC: some sweep of the launch takes the vector mapping (StepArgs::any_vec).  A
// kernel without it: the vector sweep's registers make the rest spill
// (immersed cylinder in a cavity 36.2 -> 32.4 us per step without it, D = 40
// cylinder 50.5 -> 49.8).
// FP64: the register count follows the thread blocks per SM asked for here.  One for
// blocks of 16 and 32 (198 to 212 registers with the vector sweep, no spills; left
// to the compiler it took 128 and spilled: 1024^2 220 -> 237 us per step, with the LES
// collision 362 -> 406), whose FP64 work fills the pipe from one; two for blocks of 8.
#define STEP_MIN_BLOCKS(S, B) (sizeof(S) == 8 ? ((B) == 8 ? 2 : 1) : 0)
template <class S, class C, int B, int COLL, bool VEC>
__global__ void __launch_bounds__(sizeof(S) == 8 ? 256 : STEP_MAX_THREADS, STEP_MIN_BLOCKS(S, B)) k_step(const __grid_constant__ DevPool P, const __grid_constant__ StepArgs A) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ IbmShared sh;
    __shared__ int ntask[STEP_MAX_PHASES];   // tasks of each phase at this launch
    __shared__ StepDeps deps;                // dependencies of each phase
    __shared__ int crit[STEP_MAX_PHASES];    // the critical phases with tasks, in list order
    __shared__ int cpos[STEP_MAX_PHASES];    // (scratch: their positions)
    __shared__ int bfirst[STEP_MAX_PHASES];  // first task of each phase in the bulk queue
    __shared__ int wtot[32];
    // the scheduler's state lives in shared memory, so that no register is
    // held across a task (the vector sweep needs all of them)
    __shared__ int s_cmd, s_phase, s_local, s_last, s_ncp, s_nbulk, s_bulk_left, s_turn, s_next;
    __shared__ int2 s_key;  // whose blocks' data are held (step_fused)
    __shared__ int s_wait, s_go;  // the claimed critical phase to wait for (-1: none), the wait's outcome
    __shared__ int s_body[SBOT_MAXLEV + 1];  // first server of each group's bodies, their number
    const int tid = threadIdx.x, nph = A.nph;
    StepCtl* ctl = A.ctl;
    constexpr unsigned FULL = 0xffffffffu;

    // IBM servers: where there are at most max_servers bodies (the rule stands
    // where the host sets it), the first thread blocks run one body's IBM each and
    // nothing else, so that the IBM's code and its data stay in that SM's caches, a
    // static body's geometry in its shared memory, and one step's IBM follows the
    // last without a hand-over between SMs (D = 40 cylinder 54.7 -> 50.2 us per
    // coarse step, the D = 128 one 361 against 453 with the IBM handed out after the
    // sweep's tasks)
    if (tid == 0) {
        int n = 0;
        for (int g = 0; g < SBOT_MAXLEV; g++) {
            s_body[g] = n;
            if (A.body_count[g] >= 0) n += max(A.counts[A.body_count[g]], 0);
        }
        s_body[SBOT_MAXLEV] = n <= A.max_servers ? n : 0;
        s_turn = 0;
        s_next = -1;
        s_key = make_int2(-1, -1);
        sh.geo_inst = -1;
    }
    __syncthreads();
    const int nsrv = s_body[SBOT_MAXLEV];
    const bool server = (int)blockIdx.x < nsrv;
    const int workers = gridDim.x - nsrv;
    // Fixed owners: where every instance has one level, the phases of a step
    // form one chain, and a task taken early only waits.  Each thread block then
    // walks the list in order and runs the tasks that are its own by number (a
    // sweep's from the first thread block on, the next sweep's after them, the
    // others' from the last one back): no hand-out, whose four dependent L2 round
    // trips were most of a short step, and a sweep's thread block keeps its blocks'
    // data.  (In order and all resident, so the earliest unfinished task always
    // runs.)
    auto served = [&](const StepPhase& ph) { return nsrv > 0 && ph.kind == PH_IBM && A.counts[ph.count_idx] > 0; };

    // task counts from this launch's list lengths (a critical phase with no
    // work but with dependencies gets one empty task, so that the phases after
    // it wait for its dependencies); the critical phases that have tasks,
    // compacted in order; the bulk queue's prefix sums
    for (int p = tid; p < nph; p += blockDim.x) {
        const StepPhase& ph = A.ph[p];
        int nt = step_ntasks<S, B>(P, A, ph, blockDim.x, workers);
        if (nt == 0 && (A.fixed || !ph.bulk) && ph.ndep > 0) nt = 1;
        ntask[p] = nt;
        deps.n[p] = ph.ndep | (ph.after + 1) << 8;
        for (int k = 0; k < ph.ndep; k++) deps.d[p][k] = (unsigned short)ph.dep[k];
        cpos[p] = ((A.fixed || !ph.bulk) && nt > 0 && served(ph) == server) ? 1 : 0;
        bfirst[p] = ph.bulk && !A.fixed ? nt : 0;
    }
    __syncthreads();
    {
        const int ncp = block_scan_inplace(cpos, nph, wtot);
        const int nbulk = block_scan_inplace(bfirst, nph, wtot);
        if (tid == 0) {
            s_ncp = ncp;
            s_nbulk = nbulk;
            s_bulk_left = nbulk > 0;
        }
    }
    for (int p = tid; p < nph; p += blockDim.x) {
        const StepPhase& ph = A.ph[p];
        if ((A.fixed || !ph.bulk) && ntask[p] > 0 && served(ph) == server) crit[cpos[p]] = p;
    }
    __syncthreads();
    if (A.tr_start && tid == 0) atomicMin(&A.tr_start[STEP_MAX_PHASES], global_ns());

    for (;;) {
        if (server) {
            if (threadIdx.x == 0) {  // the next IBM phase that its body has
                int i = s_turn, local = 0;
                for (; i < s_ncp; i++) {
                    local = (int)blockIdx.x - s_body[A.ph[crit[i]].level];  // (a body's group is its finest level)
                    if (local >= 0 && local < ntask[crit[i]]) break;
                }
                s_turn = i + 1;
                s_cmd = i < s_ncp ? STEP_RUN : STEP_EXIT;
                s_phase = s_wait = i < s_ncp ? crit[i] : -1;
                s_local = local;
                s_go = 1;
            }
        } else if (A.fixed) {
            if (threadIdx.x == 0) {
                const int w = (int)blockIdx.x - nsrv;
                int i = s_turn, t = s_next, q = -1;
                for (; i < s_ncp; i++, t = -1) {
                    q = crit[i];
                    if (t < 0) {  // its first task of this phase
                        const bool sweep = A.ph[q].kind == PH_FUSED;
                        const int off = sweep && i > 0 && A.ph[crit[i - 1]].kind == PH_FUSED ? ntask[crit[i - 1]] : 0;
                        t = sweep ? (w + workers - off % workers) % workers : workers - 1 - w;
                    }
                    if (t < ntask[q]) break;
                }
                s_turn = i;
                s_next = t + workers;
                s_cmd = i < s_ncp && !ld_relaxed(&ctl->abort) ? STEP_RUN : STEP_EXIT;
                s_phase = s_wait = i < s_ncp ? q : -1;
                s_local = t;
                s_go = 1;
            }
        } else if (threadIdx.x < 32) {  // warp 0 decides
            const int lane = threadIdx.x, ncp = s_ncp, nbulk = s_nbulk;
            int cmd = STEP_EXIT, p = -1, local = 0;
            int wq = -1;  // a claimed critical phase: its dependencies are read with acquire before it runs
            if (!ld_relaxed(&ctl->abort)) {
                bool got = false;
                // 1. a task of a critical phase whose dependencies have
                //    finished, in a window after the first one with tasks
                //    left to take
                const int h = ld_relaxed(&ctl->head);
                for (int base = h; !got && base < ncp && base < h + 64; base += 32) {
                    const int i = base + lane;
                    const int q = i < ncp ? crit[i] : -1;
                    // an IBM is ready only when every task of its sub-step's sweep
                    // has been taken too: the phases of a window are looked at one
                    // after the other, and the dependencies that both share may
                    // finish in between, so that the sweep is seen waiting and the
                    // IBM ready
                    const int sweep = q >= 0 ? (deps.n[q] >> 8) - 1 : -1;
                    const int taken = q >= 0 ? ld_relaxed(&ctl->taken[q]) : 0;
                    const int swept = sweep >= 0 ? ld_relaxed(&ctl->taken[sweep]) : 0;
                    const bool avail = q >= 0 && taken < ntask[q];
                    const bool rdy = avail && (sweep < 0 || swept >= ntask[sweep]) && deps_screen(A, deps, q, ntask);
                    if (base == h) {  // phases that have nothing left to take leave the window for good
                        const unsigned av = __ballot_sync(FULL, avail);
                        const int nh = av ? base + __ffs(av) - 1 : min(base + 32, ncp);
                        if (lane == 0 && nh > h) atomicMax(&ctl->head, nh);
                    }
                    unsigned m = __ballot_sync(FULL, rdy);
                    while (m && !got) {
                        const int qq = __shfl_sync(FULL, q, __ffs(m) - 1);
                        int t = 0;
                        if (lane == 0) t = atomicAdd(&ctl->taken[qq], 1);
                        t = __shfl_sync(FULL, t, 0);
                        if (t < ntask[qq]) {
                            got = true;
                            p = qq;
                            local = t;
                            wq = qq;
                        }
                        m &= m - 1;
                    }
                }
                // 2. else a bulk task (no dependency)
                if (!got && s_bulk_left) {
                    int b = 0;
                    if (lane == 0) b = atomicAdd(&ctl->bulk_next, 1);
                    b = __shfl_sync(FULL, b, 0);
                    if (b < nbulk) {
                        got = true;
                        p = phase_of(bfirst, nph, b);
                        local = b - bfirst[p];
                        cmd = STEP_RUN;
                    } else if (lane == 0) {
                        s_bulk_left = 0;
                    }
                }
                // 3. else the first critical task not yet taken, waiting for
                //    its dependencies (every phase before it in the order has
                //    all its tasks taken)
                if (!got) {
                    if (lane == 0) {
                        for (int i = ld_relaxed(&ctl->head); i < ncp; i++) {
                            const int q = crit[i];
                            if (ld_relaxed(&ctl->taken[q]) >= ntask[q]) continue;
                            const int t = atomicAdd(&ctl->taken[q], 1);
                            if (t < ntask[q]) {
                                p = q;
                                local = t;
                                break;
                            }
                        }
                    }
                    p = __shfl_sync(FULL, p, 0);
                    local = __shfl_sync(FULL, local, 0);
                    wq = p;
                }
                if (wq >= 0) cmd = STEP_RUN;
            }
            if (lane == 0) {
                s_cmd = cmd;
                s_phase = p;
                s_local = local;
                s_wait = wq;
                s_go = 1;
            }
        }
        __syncthreads();
        if (s_cmd != STEP_RUN) break;
        // the task's gate: a claimed critical task waits here (warp 0, with
        // acquire loads) for the phases it depends on, after whatever part
        // of the task may run before them
        auto gate = [&](bool prologue = true) -> bool {
            if (!prologue && s_wait < 0) {  // nothing to wait for, nothing to publish
                if (threadIdx.x == 0 && A.tr_start) {
                    const unsigned long long t = global_ns();
                    atomicMin(&A.tr_start[s_phase], t);
                    atomicMax(&A.tr_start2[s_phase], t);
                }
                return true;
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                const int q = s_wait;
                const bool ok = q < 0 || wait_until(P, A, [&] { return deps_acquire(A, deps, q, ntask); });
                if (threadIdx.x == 0) {
                    s_go = ok;
                    if (ok && A.tr_start) {
                        const unsigned long long t = global_ns();
                        atomicMin(&A.tr_start[s_phase], t);
                        atomicMax(&A.tr_start2[s_phase], t);
                    }
                }
            }
            __syncthreads();
            return s_go != 0;
        };
        // an IBM task before its stores: the sweep of its sub-step has
        // finished (no deadlock: all that sweep's tasks were taken before this
        // one -- the screen asks for it, a task taken before it is ready or by a
        // fixed owner comes later in the order, and where servers run the IBM the
        // others take every sweep -- and a sweep's task never waits after its gate)
        auto await = [&]() {
            const int d = A.ph[s_phase].after;
            const bool ok = d < 0 || wait_until(P, A, [&] { return ld_acquire(&A.ctl->done[d]) >= ntask[d]; });
            if ((threadIdx.x & 31) == 0 && !ok) s_go = 0;
        };
        auto swept = [&]() -> bool { return s_go != 0; };
        step_task<S, C, B, COLL, VEC>(P, A, A.ph[s_phase], s_local, workers, s_key, smraw, sh, gate, await, swept);
        __syncthreads();  // the task's writes, then its count (a release: the
                          // barrier orders every thread's writes before it)
        if (threadIdx.x == 0 && s_go) {
            const int p = s_phase;
            if (A.tr_start) {  // the task's end, before it is counted
                const unsigned long long t = global_ns();
                atomicMax(&A.tr_end[p], t);
                atomicMin(&A.tr_end1[p], t);
                atomicAdd(&A.tr_tasks[p], 1);
            }
            red_release_add(&ctl->done[p], 1);
        }
        if (server && !s_go) break;
    }
    // the last thread block to leave zeroes the control block for the next launch
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&ctl->exited, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        for (int p = threadIdx.x; p < nph; p += blockDim.x) {
            ctl->taken[p] = 0;
            ctl->done[p] = 0;
        }
        if (threadIdx.x == 0) {
            ctl->head = 0;
            ctl->bulk_next = 0;
            ctl->abort = 0;
            ctl->exited = 0;
        }
    }
}

template <class S, class C, int B, int COLL>
cudaError_t launch_step_k(const DevPool& P, const StepArgs& A, int grid, int threads, size_t smem, cudaStream_t s) {
    auto kern = B >= 16 && A.any_vec ? k_step<S, C, B, COLL, (B >= 16)> : k_step<S, C, B, COLL, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;  // every thread block resident at once
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P, A);
}

template <class K>
int occupancy_of(K kern, int threads, size_t smem, size_t* static_smem) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return 0;
    if (static_smem && *static_smem < fa.sharedSizeBytes) *static_smem = fa.sharedSizeBytes;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

// thread blocks per SM that either variant has room for: one grid serves both, and
// which one a launch takes (any_vec) may change from step to step
template <class S, class C, int B, int COLL>
int occupancy_k(int threads, size_t smem, size_t* static_smem) {
    if (static_smem) *static_smem = 0;
    const int plain = occupancy_of(k_step<S, C, B, COLL, false>, threads, smem, static_smem);
    if (B < 16) return plain;
    const int vec = occupancy_of(k_step<S, C, B, COLL, (B >= 16)>, threads, smem, static_smem);
    return plain < vec ? plain : vec;
}

// the kernel of the context's block size and collision kind, one storage type
template <class S, class C>
int launch_step_s(const DevPool& P, const StepArgs& A, int grid, int threads, size_t smem, cudaStream_t s) {
    const int k = P.coll & 15;
    cudaError_t e = cudaErrorInvalidValue;
    if (P.B == 8)
        e = k == 1 ? launch_step_k<S, C, 8, 1>(P, A, grid, threads, smem, s)
                   : (k == 2 ? launch_step_k<S, C, 8, 2>(P, A, grid, threads, smem, s)
                             : launch_step_k<S, C, 8, 0>(P, A, grid, threads, smem, s));
    else if (P.B == 16)
        e = k == 1 ? launch_step_k<S, C, 16, 1>(P, A, grid, threads, smem, s)
                   : (k == 2 ? launch_step_k<S, C, 16, 2>(P, A, grid, threads, smem, s)
                             : launch_step_k<S, C, 16, 0>(P, A, grid, threads, smem, s));
    else if (P.B == 32)
        e = k == 1 ? launch_step_k<S, C, 32, 1>(P, A, grid, threads, smem, s)
                   : (k == 2 ? launch_step_k<S, C, 32, 2>(P, A, grid, threads, smem, s)
                             : launch_step_k<S, C, 32, 0>(P, A, grid, threads, smem, s));
    return (int)e;
}

template <class S, class C>
int step_occupancy_s(int B, int coll, int threads, size_t smem, size_t* static_smem) {
    const int k = coll & 15;
    if (B == 8)
        return k == 1 ? occupancy_k<S, C, 8, 1>(threads, smem, static_smem)
                      : (k == 2 ? occupancy_k<S, C, 8, 2>(threads, smem, static_smem)
                                : occupancy_k<S, C, 8, 0>(threads, smem, static_smem));
    if (B == 16)
        return k == 1 ? occupancy_k<S, C, 16, 1>(threads, smem, static_smem)
                      : (k == 2 ? occupancy_k<S, C, 16, 2>(threads, smem, static_smem)
                                : occupancy_k<S, C, 16, 0>(threads, smem, static_smem));
    if (B == 32)
        return k == 1 ? occupancy_k<S, C, 32, 1>(threads, smem, static_smem)
                      : (k == 2 ? occupancy_k<S, C, 32, 2>(threads, smem, static_smem)
                                : occupancy_k<S, C, 32, 0>(threads, smem, static_smem));
    return 0;
}

}  // namespace
