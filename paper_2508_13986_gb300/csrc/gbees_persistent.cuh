// The whole step loop of a propagate call in one launch.
//
// k_persistent: for the grids of 10^4-10^5 cells of the Lorenz '63 workloads a
// time step is a few microseconds of work split into dependent phases; kernel
// launches and their drain would dominate. This cooperative kernel keeps one
// block per SM resident and separates the phases by a bounded grid barrier
// (the cooperative-kernel structure of Sec. 4, with GB300's block count). 512
// threads: a pool of 7.8 * 10^4 entries has one entry per thread.
// What bounds a step is the longest chain of its phases and the instruction
// fetch (L1 instruction cache 32 KB, beyond it straight code runs at a third of
// the rate): the phases' code is kept small, rare work out of line. Lorenz '63,
// h = 0.25, 5 * 10^3 to 5 * 10^4 pool entries: 24.0 us per step in both precisions
// (38.2 us in FP64 and 35.4 us in FP32 with five phases, each work item's chain in one
// thread, in 214 KB of code); h = 0.5, 7 * 10^3 entries: 24 us (35.3 us).
//
// k_batch: many independent grids in one launch. With a team of blocks per grid
// (all grids resident, a cooperative launch), or as a queue: each block takes a
// grid and runs its whole step loop alone, the phases separated by block
// barriers; blocks never wait on each other then, so the launch needs no
// co-residency and ragged grids balance over the SMs.
//
// Every block computes the step's scalars (dt, normalisation, maximum) itself
// from the same sums, so the scalars need no extra barrier; block 0 of the grid
// writes them back at the end.
//
// Barriers per step: waves + grow | new halo cells + fluxes | update; a prune
// adds mark | scatter | status | compact | relink. The normalisation of a step
// and the next dt are formed by one warp beside the grow of the next step.
#pragma once

#include "gbees_kernels.cuh"

namespace gbees {

// What one thread of each block reads or computes for the others.
struct StepShared {
    double dt, t_new, scale, maxq, w;
    double dth[MAXN];
    unsigned long long maxrate;           // largest CFL rate of the active cells
    long long n_ins, n_act, n_halo;  // counts after the grow, after the halo
    int last, bad;
};

// w = (prod h) sum, 1 / w and the maximum from combined sums (one thread).
static __device__ __noinline__ void normalisation(const Model& m, const long long* acc, unsigned long long maxq_ord,
                                              StepShared& ss) {
    const double w = m.prod_h * acc_to_double(acc);
    ss.w = w;
    ss.bad = !(w > 0.0) || !isfinite(w);
    ss.scale = ss.bad ? 0.0 : 1.0 / w;
    ss.maxq = maxq_ord ? ord_val(maxq_ord) : 0.0;
}

// Up to max_steps steps of the grid (m, b) by the nb blocks of index bi that
// share it (the whole launch, a team of a batched launch, or one block): grid
// barriers between the phases, block barriers when the block is alone.
// max_pool: the loop also stops after a step that leaves more pool entries
// than that (the persistent kernel hands a grown grid to the graph path; every
// block sees the same count, so all leave together).
// sc->bar_seq was zero when the launch began.
template <int N, typename T>
__device__ __forceinline__ void step_loop(const Model& m, const Bufs& b, long long max_steps, int nb, int bi,
                                          long long max_pool = 0x7fffffffffffffffll) {
    __shared__ StepShared ss;
    __shared__ GrowQueue gq;
    DevScalars* sc = b.sc;
    // The result is the same for every thread of the block: a warp that read
    // the error flag after another warp of the block had already raised it in
    // the next phase must not return while the others go on (their block
    // barriers would then pair with the wrong ones).
    unsigned long long n_bar = 0;
    auto barrier = [&](auto&& fetch) -> bool {
        if (nb == 1) return block_barrier(sc, fetch);
        return grid_barrier_seq(sc, nb + m.bar_extra, n_bar, m.spin_limit, fetch);
    };
    auto nothing = [] {};
    StepView v = view_of(m, sc);
    v.nb = nb;
    v.bi = bi;
    double t = *(volatile double*)&sc->t;
    const double tt = *(volatile double*)&sc->t_target;
    int done = *(volatile int*)&sc->done;
    long long step = *(volatile long long*)&sc->step;
    unsigned long long maxrate = *(volatile unsigned long long*)&sc->maxrate_bits;
    double w = *(volatile double*)&sc->w;
    double last_dt = *(volatile double*)&sc->dt;
    long long n_active = *(volatile long long*)&sc->NA;
    long long nsteps = 0, nupd = 0;
    const bool lead = bi == 0 && threadIdx.x == 0;
    // the running reductions start from the state (before the first barrier,
    // which orders these writes before every use)
    int ep = 0;  // parity of the prune epoch in loop_rate
    if (lead && !done) {
        sc->loop_rate[0] = maxrate;
        for (int e = 0; e < 2; ++e) {
            sc->loop_maxq[e] = 0;
            for (int q = 0; q < NDIG; ++q) sc->loop_acc[e][q] = 0;
        }
    }
    if (threadIdx.x == 0) {
        ss.maxrate = maxrate;
        ss.bad = 0;
    }
    // every block has read the state before anyone changes it
    if (done || *(volatile int*)&sc->error || !barrier(nothing)) return;
    // phase timing by block 0 (cycles between the barriers it passes)
    long long pc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    long long t_mark = clock64();
    auto mark = [&](int ph) {
        if (lead) {
            const long long now = clock64();
            pc[ph] += now - t_mark;
            t_mark = now;
        }
    };
    // The normalisation of the step before is still to be formed from its sums
    // (slot `from` of loop_acc), by one thread: beside the grow of the next step
    // in the block's last warp (the grow needs the maximum alone), or at once
    // before a prune and at the end.
    bool pending = false;
    auto normalise = [&](int from) {
        long long acc[NDIG];
#pragma unroll
        for (int q = 0; q < NDIG; ++q) acc[q] = *(volatile long long*)&sc->loop_acc[from][q];
        normalisation(m, acc, *(volatile unsigned long long*)&sc->loop_maxq[from], ss);
    };
    auto take = [&] {  // every thread, after a block barrier
        w = ss.w;
        v.scale = ss.scale;
        v.maxq = ss.maxq;
        pending = false;
    };
    bool marks = false;      // the last step's activated cells still carry their marks
    double free_dt = 0.0;    // thread 0: cfl / rate of free_rate
    unsigned long long free_rate = 0;

    for (long long it = 0; it < max_steps && !done; ++it) {
        // 1: waves of the existing entries; the grow
        v.fresh = (it & 1) ? 2u * OM_NEW : 1u * OM_NEW;
        if (threadIdx.x == 0) gq.n = 0;
        if (pending && threadIdx.x == blockDim.x - 64) {
            const unsigned long long o = *(volatile unsigned long long*)&sc->loop_maxq[(it - 1) & 1];
            ss.maxq = o ? ord_val(o) : 0.0;
        }
        waves_small_body<N, T>(m, b, v);
        __syncthreads();
        if (pending) v.maxq = ss.maxq;
        // dt of Eq. 8 needs the new active cells' rates. They rarely exceed the
        // largest one known: the step's time is formed for that before the
        // barrier and again only if it does
        auto set_time = [&](unsigned long long r) {
            if (r != free_rate || free_dt == 0.0) {
                free_rate = r;
                const double rate = __longlong_as_double((long long)r);
                free_dt = rate > 0.0 ? __ddiv_rn(m.cfl, rate) : (double)INFINITY;
            }
            const StepTime st = step_time_of(m, free_dt, t, tt, ss.dth);
            ss.dt = st.dt;
            ss.t_new = st.t_new;
            ss.last = st.last;
            if (r != ss.maxrate) ss.maxrate = r;
        };
        if (threadIdx.x == blockDim.x - 32) {
            if (pending) normalise((int)((it - 1) & 1));
            set_time(ss.maxrate);
        }
        grow_detect<N, T>(m, b, v, gq, ss.maxrate, &sc->loop_rate[ep]);
        __syncthreads();
        grow_drain<N, T>(m, b, v, gq, ss.maxrate, &sc->loop_rate[ep]);
        if (!barrier([&] {
                const long long n_ins = *(volatile long long*)&sc->N;
                ss.n_act = *(volatile long long*)&sc->n_act;
                const unsigned long long r =
                    max(ss.maxrate, *(volatile unsigned long long*)&sc->loop_rate[ep]);
                ss.n_ins = min(n_ins, m.cap);
                if (r != ss.maxrate) set_time(r);
            }))
            return;
        if (pending) {
            take();
            if (ss.bad) {
                set_error(sc, ST_EDEGENERATE);
                return;
            }
        }
        const long long n_ins = ss.n_ins, n_act = ss.n_act;
        n_active += n_ins - v.N_prev + n_act;
        const double t_new = ss.t_new;
        const int last = ss.last;
        maxrate = ss.maxrate;
        v.dt = ss.dt;
#pragma unroll
        for (int k = 0; k < N; ++k) v.dth[k] = ss.dth[k];
        if (!(v.dt > 0.0)) {
            set_error(sc, ST_EDEGENERATE);
            return;
        }
        mark(0);
        // every block has read the other slot of the sums: clear it for the next step
        if (lead) {
            sc->loop_maxq[(it + 1) & 1] = 0;
            for (int q = 0; q < NDIG; ++q) sc->loop_acc[(it + 1) & 1][q] = 0;
        }
        // 2: new halo cells; fluxes between existing entries
        halo_claim_body<N, T>(m, b, v, n_ins, n_act);
        faces_old_body<N, T>(m, b, v);
        if (!barrier([&] { ss.n_halo = *(volatile long long*)&sc->n_halo; })) return;
        v.N = min(n_ins + ss.n_halo, m.cap);
        mark(3);
        // the counts have been read by all: the next grow starts from them
        if (lead) {
            sc->N = v.N;
            sc->n_act = 0;
        }
        // 3: the update; the new halo cells
        halo_complete_body<N, T>(m, b, v, n_ins);
        {
            long long d[NDIG] = {0, 0, 0, 0, 0, 0};
            T mx = -INFINITY;
            int err = 0;
            apply_small_body<N, T>(m, b, v, n_ins, n_act, d, mx, err);
            if (err) set_error(sc, ST_EDEGENERATE);
            block_atomics(sc->loop_acc[it & 1], &sc->loop_maxq[it & 1], d, (double)mx);
        }
        if (!barrier(nothing)) return;
        mark(4);
        if (lead) sc->n_halo = 0;  // read by all before this barrier, added to after the next
        pending = true;
        marks = n_act > 0;
        t = t_new;
        last_dt = v.dt;
        done = last;
        step += 1;
        nsteps += 1;
        nupd += n_active;
        v.pb ^= 1;
        const bool prune = m.prune_interval > 0 && step % m.prune_interval == 0;
        const bool leave = done || it + 1 == max_steps || v.N > max_pool;
        if (prune || leave) {
            if (threadIdx.x == 0) normalise((int)(it & 1));
            __syncthreads();
            take();
            if (ss.bad) {
                set_error(sc, ST_EDEGENERATE);
                return;
            }
            mark(6);
        }
        if (leave && !prune && marks) clear_marks(b, v, n_act);
        v.N_prev = v.N;
        // prune (Algorithm 3) every prune_interval steps
        if (prune) {
            prune_mark_body<T>(m, b, v);
            if (!barrier(nothing)) return;
            prune_scatter_body<N, T>(m, b, v);
            if (!barrier(nothing)) return;
            prune_count_body<N>(m, b, v);
            if (!barrier(nothing)) return;
            const Survivors sv = block_offsets(b, v.nb, v.bi);
            const long long total = sv.total_a + sv.total_g;
            n_active = sv.total_a;
            if (lead) {  // before the next grow appends
                sc->N = total;
                // a new epoch of the running rate: the new cells' largest, beside
                // the survivors' (in ss.maxrate)
                sc->loop_rate[ep ^ 1] = 0;
            }
            {
                long long dp[NDIG] = {0, 0, 0, 0, 0, 0};
                double mxp = -INFINITY, rmax = 0.0;
                int errp = 0;
                prune_compact_body<N, T>(m, b, v, sv, dp, mxp, rmax, errp);
                if (errp) set_error(sc, ST_EDEGENERATE);
                block_partial(b.part, dp, mxp, rmax, bi);
            }
            if (!barrier(nothing)) return;
            prune_relink_body<N>(m, b, v);
            if (!barrier(nothing)) return;
            const Combined cp = combine_partials(b.part, nb);
            if (threadIdx.x == 0) {
                normalisation(m, cp.acc, cp.maxq_ord, ss);
                ss.maxrate = cp.rate_bits;
            }
            __syncthreads();
            take();
            if (ss.bad || sv.total_a == 0) {
                set_error(sc, ST_EDEGENERATE);
                return;
            }
            maxrate = cp.rate_bits;
            ep ^= 1;
            mark(5);
            v.N = total;
            v.N_prev = total;
            v.g ^= 1;
            v.pb ^= 1;
        }
        if (v.N > max_pool) break;
    }
    if (lead) {
        sc->N = v.N;
        sc->NA = n_active;
        sc->N_prev = v.N_prev;
        sc->pbuf = v.pb;
        sc->gen = v.g;
        sc->maxq = v.maxq;
        sc->scale = v.scale;
        sc->w = w;
        sc->t = t;
        sc->dt = last_dt;
        sc->step = step;
        sc->done = done;
        sc->maxrate_bits = maxrate;
        sc->steps_call += nsteps;
        sc->updates_call += nupd;
        sc->prune_now = 0;
        for (int q = 0; q < 8; ++q) sc->phase_cycles[q] += pc[q];
        sc->phase_steps += nsteps;
    }
}


template <int N, typename T>
__global__ void __launch_bounds__(PERSIST_THREADS, 1) k_persistent(const __grid_constant__ Model m,
                                                                   const __grid_constant__ Bufs b, long long max_steps,
                                                                   long long max_pool) {
    step_loop<N, T>(m, b, max_steps, gridDim.x, blockIdx.x, max_pool);
}

// Resident blocks per SM of the batch kernels: the register cap (64) spills a
// little, but four blocks keep four times the loads of one in flight, and the
// phases are bound by dependent global loads (measured: 2.1x the throughput of
// two blocks per SM on 256 Lorenz '63 grids).
constexpr int BATCH_BLOCKS_PER_SM = 4;

// Many grids in one launch, in one of two forms.
// slots null (queue): block after block takes the next grid of the queue (next
// counts the grids handed out) and runs up to max_steps of its steps. A grid
// that is done or in error returns at once, so a launch can be repeated until
// all are done.
// slots given (teams): a cooperative launch in which every grid has a team of
// blocks (slots[blockIdx.x]) sized to its work, the team's phases separated by
// a barrier on the grid's own scalars.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS, BATCH_BLOCKS_PER_SM) k_batch(const BatchItem* items, int count,
                                                                        unsigned int* next, const TeamSlot* slots,
                                                                        long long max_steps) {
    __shared__ int s_item;
    for (;;) {
        int i, nb = 1, bi = 0;
        if (slots) {
            const TeamSlot ts = slots[blockIdx.x];
            i = ts.item;
            nb = ts.nb;
            bi = ts.bi;
            if (i < 0) return;
        } else {
            if (threadIdx.x == 0) s_item = (int)atomicAdd(next, 1u);
            __syncthreads();
            i = s_item;
            __syncthreads();
            if (i >= count) return;
        }
        step_loop<N, T>(items[i].m, items[i].b, max_steps, nb, bi);
        if (slots) return;
        __syncthreads();
    }
}

}  // namespace gbees
