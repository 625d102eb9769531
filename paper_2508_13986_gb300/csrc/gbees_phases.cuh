// The phases of one GBEES time step as device functions over "all threads of
// the grid", shared by the one-kernel-per-phase path (gbees_kernels.cuh, run as
// a CUDA graph) and the persistent cooperative kernel (gbees_persistent.cuh).
// Data that a phase writes is read by later phases of the same persistent
// launch, so no pointer here is marked read-only (no non-coherent loads): the
// grid barrier's fences make plain loads see the other blocks' writes.
//
// A large grid runs them one kernel each; the step loop of a small grid (one
// resident launch, gbees_persistent.cuh) has forms of its own for grow, halo,
// link, faces and apply (below, "step loop of a small grid").
//
//   grow       directional grow of the significant cells (Sec. 3.3, Algorithm 2)
//   halo       the missing face neighbours of the newly active cells, as halo cells
//   link       neighbour links, outward mask and CFL rate of the new entries (Sec. 4.1)
//   waves      per-entry jumps and transverse terms
//   faces      one flux per face (Eq. 7 + Algorithm 1 gathered + HR term)
//   apply      P -= sum_j dt/h_j (F_hi - F_lo), normalised, reduced
//              (faces and apply in one pass on large FP32 grids)
//   prune      mark S, mark D(S), status, compact, relink and rehash (Algorithm 3)
//
// The pool holds the active cells and, as halo cells with p = 0, every face
// neighbour of an active cell that is not active (a missing cell of the method:
// p = 0, not updated). With links between all pool entries, every cell of the
// update stencil is reached through links and the update needs no hashtable.
#pragma once

#include "gbees_device.cuh"

namespace gbees {

// What a phase needs to know about the step in progress.
struct StepView {
    long long N;       // pool entries (clamped to the capacity)
    long long N_prev;  // pool entries before this step's grow
    int pb, g;         // current value buffer and key/link buffer
    double maxq;       // max stored value (threshold p* = thr_rel * maxq)
    double scale;      // 1 / w of the previous normalisation
    double dth[MAXN];  // dt / h_j of this step
    double dt;         // dt of this step
    int nb, bi;        // the blocks that share this grid's work, and this block's index among them
    unsigned fresh;    // flag of the halo cells that this step makes active (step loop of a small grid)
};

// (volatile: the step loop reads the state itself, which other blocks change)
__device__ __forceinline__ StepView view_of(const Model& m, const volatile StepHead* h) {
    StepView v;
    v.N = min((long long)h->N, m.cap);
    v.N_prev = min((long long)h->N_prev, m.cap);
    v.pb = h->pbuf;
    v.g = h->gen;
    v.maxq = h->maxq;
    v.scale = h->scale;
    for (int j = 0; j < MAXN; ++j) v.dth[j] = h->coef_dth[j];
    v.dt = h->step_dt;
    v.nb = gridDim.x;
    v.bi = blockIdx.x;
    v.fresh = OM_NEW;
    return v;
}

// dt of Eq. 8 (CFL over the maximum rate, clipped to land on the target) and
// its coefficients dt / h_j; the same IEEE operations wherever it is evaluated.
struct StepTime {
    double dt, t_new;
    int last;
};
// free_dt: cfl over the maximum rate (infinite when every rate is zero).
__device__ __forceinline__ StepTime step_time_of(const Model& m, double free_dt, double t, double tt, double* dth) {
    double dt = free_dt;
    const double rem = __dsub_rn(tt, t);
    const bool last = dt >= rem;
    if (last) dt = rem;
#pragma unroll
    for (int j = 0; j < MAXN; ++j) dth[j] = j < m.n ? dt * m.inv_h[j] : 0.0;
    StepTime s;
    s.dt = dt;
    s.last = last;
    s.t_new = last ? tt : __dadd_rn(t, dt);
    // t + dt can round onto the target although dt < tt - t: that step ends
    // the call too (as the loop 'while t < t_target' of the method does)
    if (!last && !(s.t_new < tt)) {
        s.last = 1;
        s.t_new = tt;
    }
    return s;
}
__device__ __forceinline__ StepTime step_time(const Model& m, double rate, double t, double tt, double* dth) {
    return step_time_of(m, rate > 0.0 ? __ddiv_rn(m.cfl, rate) : (double)INFINITY, t, tt, dth);
}

// Index of cell c + s1 e_j + s2 e_d (j != d) through the links (L: the links
// of c), -1 when it is not in the pool. For an active cell c the face
// neighbour c + s1 e_j is in the pool, so its link decides; -2 only when both
// intermediate cells are missing.
template <int N>
__device__ __forceinline__ int edge_by_links(const int* link, long long cap, const int* L, int j, int s1, int d,
                                             int s2) {
    int a = L[2 * j + s1];
    if (a >= 0) return __ldcg(link + (long long)(2 * d + s2) * cap + a);
    int b = L[2 * d + s2];
    if (b >= 0) return __ldcg(link + (long long)(2 * j + s1) * cap + b);
    return -2;
}

// The 2n links of entry c (direction-major arrays: one coalesced load per
// direction across a warp of consecutive entries).
template <int N>
__device__ __forceinline__ void load_links(const int* link, long long cap, long long c, int* L) {
#pragma unroll
    for (int d = 0; d < 2 * N; ++d) L[d] = link[(long long)d * cap + c];
}

// Insert cell c (key k) into the table; the key must be new. slots[c]
// records the table slot, so that a prune can empty exactly the used slots.
__device__ __forceinline__ void table_insert_new(const Model& m, const Bufs& b, unsigned long long k, long long c,
                                                 unsigned int* slots) {
    unsigned long long slot;
    int r = table_claim(m, b.table, b.sc, k, &slot);
    if (r == 1) {
        b.table[slot].val = c;
        slots[c] = (unsigned int)slot;
    } else if (r == 0) {
        set_error(b.sc, ST_EINVAL);  // duplicate cell
    } else {
        set_error(b.sc, ST_ETABLE);
    }
}

// ------------------------------------------------------------------ grow

// Entry e is a halo cell: make it active (mark: flags to set with it). True for
// the one thread that does.
__device__ __forceinline__ bool activate(unsigned short* om, long long e, unsigned short mark = 0) {
    unsigned short old = *(volatile unsigned short*)&om[e];
    while (old & OM_GHOST) {
        const unsigned short prev = atomicCAS(&om[e], old, (unsigned short)((old & ~OM_GHOST) | mark));
        if (prev == old) return true;
        old = prev;
    }
    return false;
}

// Active cells keep one layer away from the edge of the key range, so that
// their face neighbours (halo cells) have keys.
template <int N>
__device__ __forceinline__ bool interior(const Model& m, const int* I) {
    const long long bias = 1ll << (m.key_bits - 1);
    const long long top = (1ll << m.key_bits) - 2;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const long long u = (long long)I[k] + bias;
        if (u < 1 || u > top) return false;
    }
    return true;
}

// Claim the key of cell I and append it to the pool at base + (*counter)++
// with p = 0 and the given flags. Returns the new index, or -1 when the key is
// present already (or on an error, which is recorded).
template <int N, typename T>
__device__ __forceinline__ long long insert_cell(const Model& m, const Bufs& b, const StepView& v, const int* I,
                                                 unsigned short flags, long long* counter, long long base) {
    DevScalars* sc = b.sc;
    unsigned long long k;
    if (!pack_key<N>(m, I, k)) {
        set_error(sc, ST_EKEYRANGE);
        return -1;
    }
    unsigned long long slot;
    const int r = table_claim(m, b.table, b.sc, k, &slot);
    if (r < 0) {
        set_error(sc, ST_ETABLE);
        return -1;
    }
    if (r == 0) return -1;
    const long long c = base + warp_aggregated_add(counter);
    if (c >= m.cap) {
        set_error(sc, ST_ECAPACITY);
        return -1;
    }
    b.table[slot].val = c;
    b.slot[v.g][c] = (unsigned int)slot;
    b.key[v.g][c] = k;
    static_cast<T*>(b.q[v.pb])[c] = (T)0;
    b.om[v.g][c] = flags;
    return c;
}

// Directional grow (Sec. 3.3): every significant cell makes its downwind set
// active. A face neighbour of an active cell is always in the pool; an edge
// neighbour c + s1 e_j + s2 e_l is found through the link of the face
// neighbour c + s1 e_j. A halo cell found there becomes active (listed in map
// for the halo phase); a missing one is inserted as active. A cell whose
// downwind set was made active since the last prune is skipped.
//
// The candidates of a cell (2n faces, 4 C(n,2) edges, those that are not
// downwind skipped at once) are independent chains of dependent loads and
// atomics, spread over many threads: for large grids a sweep lists the
// growing cells (grow_list_mark) and a second kernel spreads every (cell,
// candidate) pair of the list over the grid (grow_list_body); the step loop of
// a small grid has grow_detect and grow_act.
struct GrowWork {
    double rmax = 0.0;  // largest CFL rate of the halo cells this thread activated
};

// Candidate of cell cc in direction d1 of its downwind directions, and d2 of a later
// dimension (-1: none).
template <int N, typename T>
__device__ __forceinline__ void grow_candidate(const Model& m, const Bufs& b, const StepView& v, long long cc, int d1,
                                               int d2, GrowWork& gw) {
    DevScalars* sc = b.sc;
    const long long cap = m.cap;
    const int* link = b.link[v.g];
    unsigned short* om = b.om[v.g];
    const int a = link[(long long)d1 * cap + cc];
    long long e;
    if (d2 < 0) {
        e = a;
    } else if (a >= 0) {
        e = link[(long long)d2 * cap + a];
    } else {
        const int a2 = link[(long long)d2 * cap + cc];
        e = a2 >= 0 ? link[(long long)d1 * cap + a2] : -1;
    }
    if (e >= 0) {  // in the pool: a halo cell becomes active
        if (!(om[e] & OM_GHOST) || !activate(om, e)) return;
        warp_aggregated_add(&sc->NA);
        b.map[warp_aggregated_add(&sc->n_act)] = (int)e;
        gw.rmax = fmax(gw.rmax, b.rate[v.g][e]);  // fixed when the halo cell was linked
        return;
    }
    int J[N];
    unpack_key<N>(m, b.key[v.g][cc], J);
    J[d1 >> 1] += (d1 & 1) ? 1 : -1;
    if (d2 >= 0) J[d2 >> 1] += (d2 & 1) ? 1 : -1;
    if (!interior<N>(m, J)) {
        set_error(sc, ST_EKEYRANGE);
        return;
    }
    if (insert_cell<N, T>(m, b, v, J, 0, &sc->N, 0) >= 0) warp_aggregated_add(&sc->NA);
}

// Whether cell c takes part in this step's grow: significant, active, with
// outward directions, its downwind set not yet known to be active.
template <typename T>
__device__ __forceinline__ bool grows(const unsigned short* om, const T* Q, const Above<T>& above, long long c,
                                      unsigned& out) {
    if (!above(Q[c])) return false;
    const unsigned f = om[c];
    out = f & 0xfffu;
    return !(f & (OM_COMPLETE | OM_GHOST)) && out;
}

// First half: cell c joins the step's grow list (in the flux scratch, free until
// the flux pass) when it grows.
template <typename T>
__device__ __forceinline__ void grow_list_mark(const Bufs& b, const StepView& v, const Above<T>& above, long long c) {
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    unsigned out;
    if (grows<T>(b.om[v.g], Q, above, c, out)) {
        int* glist = static_cast<int*>(b.fl);
        glist[warp_aggregated_add(&b.sc->n_glist)] = (int)c;
    }
}

// Second half: every (listed cell, dimension or pair of dimensions), over all threads
// of the grid, and its candidates: mostly one, because the flow leaves a cell through
// one face of a dimension (items by direction, 84 of them in six dimensions in place
// of 21, left three lanes of four idle: 2.0e6 listed cells 2.55 ms, now 1.11). The thread of a cell's first item marks
// it complete (only its own flag bit, and nothing else writes that word now).
template <int N, typename T>
__device__ __forceinline__ double grow_list_body(const Model& m, const Bufs& b, const StepView& v, long long nl) {
    constexpr int K = N + N * (N - 1) / 2;
    const int* glist = static_cast<const int*>(b.fl);
    unsigned short* om = b.om[v.g];
    GrowWork gw;
    const long long items = nl * K;
    const long long tid = (long long)v.bi * blockDim.x + threadIdx.x;
    const long long nth = (long long)v.nb * blockDim.x;
    for (long long it = tid; it < items; it += nth) {
        const long long rank = it / K;
        const int k = (int)(it - rank * K);
        const long long c = glist[rank];
        const unsigned out = om[c] & 0xfffu;
        // dimension j1, or the pair j1 < j2
        int j1 = k, j2 = -1;
        if (k >= N) {
            int rem = k - N;
            j1 = 0;
            while (rem >= N - 1 - j1) {
                rem -= N - 1 - j1;
                ++j1;
            }
            j2 = j1 + 1 + rem;
        }
        const unsigned s1 = (out >> (2 * j1)) & 3u, s2 = j2 < 0 ? 1u : (out >> (2 * j2)) & 3u;
        // bit 2 a + c: side a of j1 with side c of j2
        unsigned sides = (s1 & 1u ? s2 : 0u) | (s1 & 2u ? s2 << 2 : 0u);
#pragma unroll 1
        for (; sides; sides &= sides - 1) {
            const int i = __ffs(sides) - 1;
            grow_candidate<N, T>(m, b, v, c, 2 * j1 + (i >> 1), j2 < 0 ? -1 : 2 * j2 + (i & 1), gw);
        }
        if (k == 0) om[c] = (unsigned short)(om[c] | OM_COMPLETE);
    }
    return gw.rmax;
}

// ------------------------------------------------------------------ halo

// The face neighbours of the cells made active by this step's grow that are
// not in the pool are appended as halo cells at base + n_halo. Work items
// (cell, face) over the inserted cells [lo, hi), which have no links yet (each
// neighbour is claimed, the claim finds the present ones), and over the nact
// activated halo cells listed in map (only their neighbours without a link).
template <int N, typename T>
__device__ __forceinline__ void halo_body(const Model& m, const Bufs& b, const StepView& v, long long lo, long long hi,
                                          long long nact) {
    const unsigned long long* key = b.key[v.g];
    const int* link = b.link[v.g];
    const long long cap = m.cap;
    const long long ni = hi - lo;
    const long long items = (ni + nact) * 2 * N;
    // runs of 32 items, one per warp, the warps of consecutive runs on
    // different SMs: a few hundred items of a small grid spread over the GPU
#pragma unroll 1
    for (WarpRuns wr(items, v.nb, v.bi); wr.next();) {
        const long long it = wr.c;
        if (it >= items) continue;
        const long long q = it / (2 * N);
        const int d = (int)(it - q * 2 * N);
        long long x;
        if (q < ni) {
            x = lo + q;
        } else {
            x = b.map[q - ni];
            if (link[(long long)d * cap + x] >= 0) continue;
        }
        int I[N];
        unpack_key<N>(m, key[x], I);
        if (!step_index<N>(I, d >> 1, d & 1)) {
            set_error(b.sc, ST_EKEYRANGE);
            continue;
        }
        insert_cell<N, T>(m, b, v, I, OM_GHOST, &b.sc->n_halo, hi);
    }
}

// ------------------------------------------------------------------ link

// f_j with component j of the state replaced by yj (y: the cell's centre): the
// operations of drift, in its order.
template <int N, int DYN>
__device__ __forceinline__ double drift_at(const Model& m, const double* y, int j, double yj) {
    using A = Ar;
    auto at = [&](int k) { return k == j ? yj : y[k]; };
    if constexpr (DYN == DYN_CONSTANT) {
        return m.a[j];
    } else if constexpr (DYN == DYN_LINEAR) {
        double s = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) s = A::add(s, A::mul(m.a[j * N + k], at(k)));
        return A::add(s, m.a[N * N + j]);
    } else if constexpr (DYN == DYN_LORENZ63 && N == 3) {
        if (j == 0) return A::mul(m.a[0], A::sub(at(1), at(0)));
        if (j == 1) return A::sub(A::mul(at(0), A::sub(m.a[1], at(2))), at(1));
        return A::sub(A::mul(at(0), at(1)), A::mul(m.a[2], at(2)));
    } else if constexpr (DYN == DYN_LORENZ63_SHIFTED && N == 3) {
        if (j == 0) return A::mul(m.a[0], A::sub(at(1), at(0)));
        if (j == 1) return A::sub(-at(1), A::mul(at(0), at(2)));
        return A::sub(A::add(A::mul(-m.a[1], at(2)), A::mul(at(0), at(1))), A::mul(m.a[1], m.a[2]));
    } else if constexpr (DYN == DYN_LORENZ96 && N >= 4) {
        return A::add(A::sub(A::mul(A::sub(at((j + 1) % N), at((j + N - 2) % N)), at((j + N - 1) % N)), at(j)), m.a[0]);
    } else {
        return 0.0;
    }
}

// x > 0 and x < 0 without the FP64 pipe (false for NaN, as the comparisons).
__device__ __forceinline__ bool is_number(double x) {
    const int a = __double2hiint(x) & 0x7fffffff;
    return a < 0x7ff00000 || (a == 0x7ff00000 && __double2loint(x) == 0);
}
__device__ __forceinline__ bool above0(double x) { return gt0(x) && is_number(x); }
__device__ __forceinline__ bool below0(double x) { return lt0(x) && is_number(x); }

// Face velocities, outward mask and CFL rate of entry c of generation g (cell
// I; Eq. 7, Eq. 8 with |f|): bit 2j+1 of the mask when the flow leaves through the
// upper j-face (f_j at the upper face > 0), bit 2j when it leaves through the lower
// one (f_j < 0). The velocities and the rate are stored, the mask and the rate
// returned. The FP64 pipe bounds the pass over many new entries, so each model has
// its own straight code (one branch for all faces), the faces of a cell share its
// index in double and what the drift has in common, and the signs are read from
// the bits: 110 to 130 FP64 instructions per entry of Lorenz '96 6-D (493 with the
// models selected face by face and divisions).
template <int N, int DYN, typename T>
__device__ __forceinline__ double entry_velocities_of(const Model& m, const Bufs& b, int g, long long c, const int* I,
                                                      unsigned& msk) {
    double di[N], y[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        di[k] = (double)I[k];
        y[k] = __dadd_rn(m.x0[k], __dmul_rn(di[k], m.h[k]));
    }
    double r = 0.0;
    msk = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        // x0 + (i -+ 1/2) h (i + 1/2 is exact, as (i + 1) - 1/2)
        const double lo = __dadd_rn(m.x0[j], __dmul_rn(__dsub_rn(di[j], 0.5), m.h[j]));
        const double hi = __dadd_rn(m.x0[j], __dmul_rn(__dadd_rn(di[j], 0.5), m.h[j]));
        const double ul = drift_at<N, DYN>(m, y, j, lo);
        if (above0(drift_at<N, DYN>(m, y, j, hi))) msk |= 1u << (2 * j + 1);
        if (below0(ul)) msk |= 1u << (2 * j);
        static_cast<T*>(b.u[g])[j * m.cap + c] = (T)ul;
        r = __dadd_rn(r, div_h(m, abs_bits(ul), j));
    }
    b.rate[g][c] = r;
    return r;
}
template <int N, typename T>
__device__ __forceinline__ double entry_velocities(const Model& m, const Bufs& b, int g, long long c, const int* I,
                                                   unsigned& msk) {
    switch (m.dyn) {
        case DYN_CONSTANT: return entry_velocities_of<N, DYN_CONSTANT, T>(m, b, g, c, I, msk);
        case DYN_LINEAR: return entry_velocities_of<N, DYN_LINEAR, T>(m, b, g, c, I, msk);
        case DYN_LORENZ63:
            if constexpr (N == 3) return entry_velocities_of<N, DYN_LORENZ63, T>(m, b, g, c, I, msk);
            break;
        case DYN_LORENZ63_SHIFTED:
            if constexpr (N == 3) return entry_velocities_of<N, DYN_LORENZ63_SHIFTED, T>(m, b, g, c, I, msk);
            break;
        case DYN_LORENZ96:
            if constexpr (N >= 4) return entry_velocities_of<N, DYN_LORENZ96, T>(m, b, g, c, I, msk);
            break;
    }
    msk = 0;
    return 0.0;
}

// Face velocities and outward masks of the new entries [lo, hi) (the mask is
// added to the flags their inserter wrote), and the largest CFL rate among the
// active ones.
template <int N, typename T>
__device__ __forceinline__ double link_masks(const Model& m, const Bufs& b, long long lo, long long hi, int g,
                                              int nb, int bi) {
    const unsigned long long* key = b.key[g];
    double rmax = 0.0;
    // runs of 32 entries, one per warp, consecutive runs on different SMs (the
    // FP64 drift evaluations of a few hundred new entries spread over the GPU)
#pragma unroll 1
    for (WarpRuns wr(hi - lo, nb, bi); wr.next();) {
        const long long c = lo + wr.c;
        if (c >= hi) continue;
        int I[N];
        unpack_key<N>(m, key[c], I);
        const unsigned short f = b.om[g][c];
        unsigned msk;
        const double r = entry_velocities<N, T>(m, b, g, c, I, msk);
        b.om[g][c] = (unsigned short)(f | msk);
        if (!(f & OM_GHOST)) rmax = fmax(rmax, r);
    }
    return rmax;
}

// f_j at the lower (up = 0) or upper (up = 1) j-face of the cell with packed
// key k: drift_at with j known at run time, out of line (the code of a
// small grid's step loop runs once per step from the instruction caches, so what
// is not a matter of a few instructions is kept in one place).
template <int N>
__device__ __noinline__ double face_velocity_key(const Model& m, unsigned long long k, int j, int up) {
    using A = Ar;
    const int bits = m.key_bits;
    const long long bias = 1ll << (bits - 1);
    const unsigned long long mask = (1ull << bits) - 1;
    auto y = [&](int a) -> double {
        const int i = (int)((long long)((k >> (bits * (N - 1 - a))) & mask) - bias);
        const double s = a == j ? __dadd_rn((double)i, up ? 0.5 : -0.5) : (double)i;
        return __dadd_rn(m.x0[a], __dmul_rn(s, m.h[a]));
    };
    if (m.dyn == DYN_CONSTANT) return m.a[j];
    if (m.dyn == DYN_LINEAR) {
        double s = 0;
#pragma unroll 1
        for (int a = 0; a < N; ++a) s = A::add(s, A::mul(m.a[j * N + a], y(a)));
        return A::add(s, m.a[N * N + j]);
    }
    if (m.dyn == DYN_LORENZ96) {
        const int jp = j + 1 < N ? j + 1 : j + 1 - N, jm1 = j >= 1 ? j - 1 : j + N - 1, jm2 = j >= 2 ? j - 2 : j + N - 2;
        return A::add(A::sub(A::mul(A::sub(y(jp % N), y(jm2 % N)), y(jm1 % N)), y(j)), m.a[0]);
    }
    if constexpr (N == 3) {
        const double y0 = y(0), y1 = y(1), y2 = y(2);
        if (m.dyn == DYN_LORENZ63) {
            if (j == 0) return A::mul(m.a[0], A::sub(y1, y0));
            if (j == 1) return A::sub(A::mul(y0, A::sub(m.a[1], y2)), y1);
            return A::sub(A::mul(y0, y1), A::mul(m.a[2], y2));
        }
        if (j == 0) return A::mul(m.a[0], A::sub(y1, y0));
        if (j == 1) return A::sub(-y1, A::mul(y0, y2));
        return A::sub(A::add(A::mul(-m.a[1], y2), A::mul(y0, y1)), A::mul(m.a[1], m.a[2]));
    }
    return 0.0;
}

// New entries of a warp, 2N lanes per entry (on: this lane has one; index c, key
// k and flags the same in its lanes), one face each: face velocities, outward
// mask, CFL rate (an FP64 instruction holds a warp scheduler for 64 cycles
// whatever its active lanes, so one lane with all faces of its entry takes 2N
// times as long), and with look the links to the neighbours in the table, both
// ways. All lanes must call it. Returns the entry's rate.
template <int N, typename T>
__device__ __noinline__ double complete_group(const Model& m, const Bufs& b, int g, bool on, int c,
                                              unsigned long long k, unsigned flags, bool look) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int F = 2 * N;
    const long long cap = m.cap;
    const int lane = threadIdx.x & 31;
    const int s = lane / F, e = lane - s * F;
    double u = 0.0, term = 0.0;
    if (on) {
        // the neighbour in direction e: one field of the key up or down, unless
        // at its end; its first probe is in flight beside the velocity
        const int shift = m.key_bits * (N - 1 - (e >> 1));
        const unsigned long long last = (1ull << m.key_bits) - 1, field = (k >> shift) & last;
        const bool end = field == ((e & 1) ? last : 0ull);
        const unsigned long long nk = (e & 1) ? k + (1ull << shift) : k - (1ull << shift);
        ulonglong2 first = make_ulonglong2(EMPTY_KEY, ~0ull);
        if (look && !end) first = __ldcg(reinterpret_cast<const ulonglong2*>(b.table + table_home(nk, m.tmask)));
        u = face_velocity_key<N>(m, k, e >> 1, e & 1);
        if (!(e & 1)) {
            (static_cast<T*>(b.u[g]) + (e >> 1) * cap)[c] = (T)u;
            term = div_h(m, abs_bits(u), e >> 1);
        }
        if (look) {
            int nbr = -1;
            if (first.x == nk) nbr = (int)(long long)first.y;
            else if (first.x != EMPTY_KEY) nbr = table_find(m, b.table, nk);
            (b.link[g] + e * cap)[c] = nbr;
            if (nbr >= 0) (b.link[g] + (e ^ 1) * cap)[nbr] = c;
        }
    }
    // outward: upper face and u > 0, lower face and u < 0
    const unsigned out = __ballot_sync(full, on && ((e & 1) ? above0(u) : below0(u)));
    double r = 0.0;
#pragma unroll
    for (int j = 0; j < N; ++j) r = __dadd_rn(r, __shfl_sync(full, term, (s * F + 2 * j) & 31));
    if (on && e == 0) {
        b.om[g][c] = (unsigned short)(flags | ((out >> lane) & ((1u << F) - 1u)));
        b.rate[g][c] = r;
    }
    return r;
}

// link_body for few new entries: 2N lanes per entry (complete_group). One thread's
// chain of 2N lookups and FP64 drift evaluations takes about 10 us however few the
// entries are; this takes 1.6 times the FP64 issue slots of link_body, which
// counts only when there are many.
template <int N, typename T>
__device__ __forceinline__ double link_few_body(const Model& m, const Bufs& b, long long lo, long long hi, int g,
                                                int nb, int bi) {
    constexpr int F = 2 * N, G = 32 / F;  // entries per warp
    const int total = (int)(hi - lo);
    const int lane = threadIdx.x & 31, s = lane / F;
    double rmax = 0.0;
    for (Runs r((total + G - 1) / G, nb, bi); r.next();) {
        const int q = r.k * G + s;
        const bool on = s < G && q < total;
        const int c = on ? (int)lo + q : 0;
        const unsigned long long k = on ? b.key[g][c] : 0ull;
        const unsigned f = on ? b.om[g][c] : OM_GHOST;
        const double rate = complete_group<N, T>(m, b, g, on, c, k, f, true);
        if (on && !(f & OM_GHOST)) rmax = fmax(rmax, rate);
    }
    return rmax;
}

// Entries [lo, hi) are new: their 2n links by hashtable lookups, the reverse
// links of the entries below lo (two new entries find one another by their own
// lookups), velocities, masks and rates. Returns this thread's largest CFL rate
// among the active ones. One thread per entry, the first probes of N directions
// in flight together: a probe of a table larger than L2 takes a microsecond, and
// one per thread left the memory idle. Paper's 6-D case, 3.1e6 entries at init:
// 1.01 ms (5.7 ms with one thread per (entry, direction), the models selected face
// by face and single slots hashed); 2.1e6 entries in its first step: 0.78 ms.
template <int N, typename T>
__device__ __forceinline__ double link_body(const Model& m, const Bufs& b, long long lo, long long hi, int g, int nb,
                                             int bi) {
    const long long cap = m.cap;
    const unsigned long long last = (1ull << m.key_bits) - 1;
    double rmax = 0.0;
    for (WarpRuns wr(hi - lo, nb, bi); wr.next();) {
        const long long c = lo + wr.c;
        const bool on = c < hi;
        const unsigned long long k = on ? b.key[g][c] : 0ull;
#pragma unroll 1
        for (int up = 0; up < 2; ++up) {
            unsigned long long nk[N];
            ulonglong2 first[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                // one field of the key up or down, unless it is at its end
                const int shift = m.key_bits * (N - 1 - j);
                const unsigned long long field = (k >> shift) & last;
                nk[j] = field == (up ? last : 0ull) ? EMPTY_KEY : up ? k + (1ull << shift) : k - (1ull << shift);
                first[j] = __ldcg(reinterpret_cast<const ulonglong2*>(b.table + table_home(nk[j], m.tmask)));
            }
#pragma unroll
            for (int j = 0; j < N; ++j) {
                int nbr = -1;
                if (on && nk[j] != EMPTY_KEY && first[j].x != EMPTY_KEY)
                    nbr = first[j].x == nk[j] ? (int)(long long)first[j].y : table_find(m, b.table, nk[j]);
                if (on) b.link[g][(2 * j + up) * cap + c] = nbr;
                if (nbr >= 0 && nbr < lo) b.link[g][(2 * j + 1 - up) * cap + nbr] = (int)c;
            }
            // the look-ups leave the warp in pieces, and it would stay so through the
            // FP64 part (four times its instructions)
            __syncwarp();
        }
        if (on) {
            int I[N];
            unpack_key<N>(m, k, I);
            unsigned msk;
            const double r = entry_velocities<N, T>(m, b, g, c, I, msk);
            const unsigned short f = b.om[g][c];
            b.om[g][c] = (unsigned short)(f | msk);
            if (!(f & OM_GHOST)) rmax = fmax(rmax, r);
        }
        __syncwarp();
    }
    return rmax;
}

// Cooperative variant: W lanes probe W consecutive slots together.
template <int N, int W, typename T>
__device__ __forceinline__ double link_body_tile(const Model& m, const Bufs& b, long long lo, long long hi, int g,
                                                  int nb, int bi) {
    const unsigned long long* key = b.key[g];
    int* link = b.link[g];
    const long long cap = m.cap;
    auto tile = cg::tiled_partition<W>(cg::this_thread_block());
    const long long tiles = (long long)nb * (blockDim.x / W);
    const long long tile_id = (long long)bi * (blockDim.x / W) + threadIdx.x / W;
    const long long work = (hi - lo) * 2 * N;
    for (long long wi = tile_id; wi < work; wi += tiles) {
        const long long c = lo + wi / (2 * N);
        const int dir = (int)(wi % (2 * N));
        const int j = dir >> 1, s = dir & 1;
        int I[N];
        unpack_key<N>(m, key[c], I);
        unsigned long long k;
        const int nbr =
            step_index<N>(I, j, s) && pack_key<N>(m, I, k) ? table_find_tile<W>(m, b.table, k, tile) : -1;
        if (tile.thread_rank() == 0) {
            link[(long long)dir * cap + c] = nbr;
            if (nbr >= 0) link[(long long)(2 * j + (1 - s)) * cap + nbr] = (int)c;
        }
    }
    return link_masks<N, T>(m, b, lo, hi, g, nb, bi);
}

// ------------------------------------------------------------------ update

template <typename T>
__device__ __forceinline__ T q_or_zero(const T* Q, int i) {
    return i >= 0 ? Q[i] : (T)0;
}

__device__ __forceinline__ bool is_halo(const unsigned short* om, long long i) { return (om[i] & OM_GHOST) != 0; }

// 0 - x as IEEE subtraction gives it, without FP64 arithmetic for doubles:
// the sign flips, except that both zeros give +0.
__device__ __forceinline__ double zero_minus(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    return __hiloint2double(((hi & 0x7fffffff) | lo) == 0 ? 0 : hi ^ (int)0x80000000, lo);
}
__device__ __forceinline__ float zero_minus(float x) { return 0.0f - x; }

// Per entry y and dimension d the update works with the jump across the lower face,
//   wl_d(y) = P_y - P_{y-e_d},
// and the entering wave
//   G_d(y) = max(u_lo, 0) (P_y - P_{y-e_d}) + min(u_hi, 0) (P_{y+e_d} - P_y),
// u_lo, u_hi the velocities at its lower and upper d-face (the upper one is the
// lower one of the neighbour above; a missing neighbour above of a halo cell
// leaves both P at 0). The corrections that Algorithm 1 scatters onto the lower
// j-face of X add up to -u_j(X) dt sum_{d != j} G_d(Y) / (2 h_d), Y the cell upwind
// of the face, so that donor cell and corrections together are u_j(X) base_j(Y),
//   base_j(y) = P_y - dt sum_{d != j} G_d(y) / (2 h_d).
//
// Large grids, pass 1, one thread per entry (active and halo, the step's new ones
// too: their neighbours have no density, so theirs come out as 0): (wl_j, base_j)
// as a pair per dimension. The pass runs when dt is known, after the links, so
// that a face needs one pair of its own cell and one of a neighbour (four gathers
// with the waves and their sum in separate arrays, formed before dt). Six
// dimensions, 5.0e6 entries in storage order: 0.42 ms in FP64, 81 % of the FP64
// pipe; 0.14 ms in FP32, bound by the gathers' sectors.
template <typename T>
struct alignas(2 * sizeof(T)) Wave {
    T wl, base;
};

template <int N, typename T>
__device__ __forceinline__ void waves_body(const Model& m, const Bufs& b, const StepView& v) {
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    const int* link = b.link[v.g];
    const T* U = static_cast<const T*>(b.u[v.g]);
    // the output aliases no input (restrict: loads may be scheduled ahead of the
    // stores; no read-only cache path is implied)
    Wave<T>* __restrict__ wave = static_cast<Wave<T>*>(b.wl);
    const long long cap = m.cap;
    const T ndt = -(T)v.dt;
    T i2h[N];  // 1 / (2 h_d) in the arithmetic type, converted once
#pragma unroll
    for (int d = 0; d < N; ++d) i2h[d] = (T)m.inv_2h[d];
    for (WarpRuns wr(v.N, v.nb, v.bi); wr.next();) {
        const long long c = wr.c;
        if (c >= v.N) continue;
        const unsigned act = __activemask();
        int L[2 * N];
        load_links<N>(link, cap, c, L);
        const T P0 = Q[c];
        // the gathers of all dimensions in flight together, in two steps (the jump
        // across the upper face is needed only where the flow comes in through it)
        T ul[N], uh[N], Pm[N], Pp[N];
#pragma unroll
        for (int d = 0; d < N; ++d) {
            ul[d] = U[d * cap + c];
            Pm[d] = q_or_zero<T>(Q, L[2 * d]);
            uh[d] = L[2 * d + 1] >= 0 ? U[d * cap + L[2 * d + 1]] : (T)0;
        }
#pragma unroll
        for (int d = 0; d < N; ++d) Pp[d] = lt0(uh[d]) ? Q[L[2 * d + 1]] : (T)0;
        // a warp of halo entries (P = 0; the pool keeps them together after a
        // prune) needs no subtraction: 0 - P_m and P_p - 0 are exact
        const bool zeros = __all_sync(act, !nonzero(P0));
        T G[N], wl[N], t = (T)0;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const bool in_lo = gt0(ul[d]), in_hi = lt0(uh[d]);
            wl[d] = zeros ? zero_minus(Pm[d]) : P0 - Pm[d];
            // one product in the usual case (flow through the cell, or out of it on
            // one side only); the flow direction varies slowly: when no lane of the
            // warp takes flow in through a face, that face's term is skipped
            G[d] = (T)0;
            if (__any_sync(act, in_lo)) G[d] = (in_lo ? ul[d] : (T)0) * wl[d];
            if (__any_sync(act, in_hi)) {
                const T wh = zeros ? Pp[d] : Pp[d] - P0;
                if (in_hi) G[d] = in_lo ? fmadd(uh[d], wh, G[d]) : uh[d] * wh;
            }
            t = fmadd(G[d], i2h[d], t);
        }
#pragma unroll
        for (int d = 0; d < N; ++d) {
            Wave<T> w;
            w.wl = wl[d];
            w.base = fmadd(ndt, fmadd(-i2h[d], G[d], t), P0);
            wave[d * cap + c] = w;
        }
    }
}

// The waves of the step loop of a small grid, formed beside the grow (before dt),
// in little code: wl, G and tg = sum_d G_d / (2 h_d) of the existing entries.
template <int N, typename T>
__device__ __forceinline__ void waves_small_body(const Model& m, const Bufs& b, const StepView& v) {
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    const long long cap = m.cap;
    const int ncell = (int)v.N_prev;
#pragma unroll 1
    for (Runs r(runs_of(ncell), v.nb, v.bi); r.next();) {
        const int c = r.cell();
        if (c >= ncell) continue;
        const unsigned act = __activemask();
        const T P0 = Q[c];
        int dn[N], up[N];
        T ul[N], Pm[N], Pp[N], uh[N];
#pragma unroll
        for (int d = 0; d < N; ++d) {
            dn[d] = (b.link[v.g] + (2 * d) * cap)[c];
            up[d] = (b.link[v.g] + (2 * d + 1) * cap)[c];
            ul[d] = (static_cast<const T*>(b.u[v.g]) + d * cap)[c];
        }
#pragma unroll
        for (int d = 0; d < N; ++d) {
            Pm[d] = dn[d] >= 0 ? Q[dn[d]] : (T)0;
            Pp[d] = (T)0;
            uh[d] = (T)0;
            if (up[d] >= 0) {
                Pp[d] = Q[up[d]];
                uh[d] = (static_cast<const T*>(b.u[v.g]) + d * cap)[up[d]];
            }
        }
        T t = (T)0;
#pragma unroll
        for (int d = 0; d < N; ++d) {
            const T wlo = P0 - Pm[d];
            const bool in_lo = gt0(ul[d]), in_hi = lt0(uh[d]);
            T G = (in_lo ? ul[d] : (T)0) * wlo;
            if (__any_sync(act, in_hi)) {
                const T whi = Pp[d] - P0;
                if (in_hi) G = in_lo ? fmadd(uh[d], whi, G) : uh[d] * whi;
            }
            (static_cast<T*>(b.wl) + d * cap)[c] = wlo;
            (static_cast<T*>(b.wg) + d * cap)[c] = G;
            t = fmadd(G, (T)m.inv_2h[d], t);
        }
        static_cast<T*>(b.tg)[c] = t;
    }
}

// a[j] of a short array in registers, j known at run time only.
template <int N, typename T, int M>
__device__ __forceinline__ T pick_of(const T (&a)[M], int j) {
    T x = a[0];
#pragma unroll
    for (int k = 1; k < N; ++k) x = j == k ? a[k] : x;
    return x;
}

// The flux through a face with velocity u != 0: Eq. 7 and the corrections of
// Algorithm 1 (u times the upwind cell's base), and the limited high-resolution
// term 1/2 |u| (1 - dt |u| / h_j) phi W of the jump W across the face, Wup the jump
// across the face beyond the upwind cell.
template <typename T>
__device__ __forceinline__ T flux_of(int lim, T u, T base, T W, T Wup, T dth) {
    if (!flows(u)) return (T)0;
    const T f = u * base;
    if (lim == LIM_NONE || !nonzero(W)) return f;
    const T au = abs_bits(u);
    return fmadd(half_nonneg(au) * fmadd(-dth, au, (T)1), limited_wave<T>(lim, W, Wup), f);
}

// Large FP64 grids, pass 2: the flux through every face with an active cell on at
// least one side, stored as the lower face of the entry above it: all n lower faces
// of an active cell, and the lower faces of a halo cell whose neighbour below is
// active. Each warp takes runs of 32 consecutive entries, queues their needed
// faces (entry, j) in shared memory, dimension by dimension, and evaluates
// them 64 at a time, two per lane with their loads in flight together, so that the
// lanes of a warp all work although a halo cell needs only the few faces it shares
// with active cells. The upper face of an active cell is the lower face of its upper
// neighbour, which is in the pool (active or halo). Five FP64 instructions per face
// (13 with the compiler's, see gt0); 5.0e6 entries in six dimensions: 0.34 ms (0.58
// ms), 50 % of the FP64 pipe. One active cell per lane with all its faces unrolled
// was slower (0.35 ms: fewer warps fit).
template <int N, typename T>
__device__ __forceinline__ void faces_body(const Model& m, const Bufs& b, const StepView& v) {
    constexpr int E = 2;  // faces per lane and evaluation
    const long long ncell = v.N;
    const long long cap = m.cap;
    const unsigned short* om = b.om[v.g];
    const int* link = b.link[v.g];
    const T* U = static_cast<const T*>(b.u[v.g]);
    const Wave<T>* wave = static_cast<const Wave<T>*>(b.wl);
    T* __restrict__ fl = static_cast<T*>(b.fl);  // aliases no input
    const int lim = m.limiter;
    constexpr int QCAP = 32 * N + 32 * E;
    __shared__ int s_qx[WARPS][QCAP];
    __shared__ unsigned char s_qj[WARPS][QCAP];
    __shared__ T s_dth[N];  // dt / h_j, read with a face's j
    if (threadIdx.x < N) s_dth[threadIdx.x] = (T)v.dth[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int n_q = 0;  // the same in every lane
    auto eval = [&](int k) {  // the top k queued faces
        n_q -= k;
        long long X[E];
        int j[E], lo[E], up[E];
        T u[E];
        Wave<T> own[E], other[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int at = lane + 32 * e;
            X[e] = at < k ? s_qx[wid][n_q + at] : -1;
            j[e] = at < k ? s_qj[wid][n_q + at] : 0;
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (X[e] < 0) continue;
            u[e] = U[j[e] * cap + X[e]];
            lo[e] = link[(long long)(2 * j[e]) * cap + X[e]];
            up[e] = link[(long long)(2 * j[e] + 1) * cap + X[e]];
            own[e] = wave[j[e] * cap + X[e]];
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (X[e] < 0) continue;
            // the cell below (upwind when the flow crosses upwards), else the one above,
            // whose lower face is the one beyond (missing only above a halo cell: no jump)
            const int z = gt0(u[e]) ? lo[e] : up[e];
            other[e].wl = other[e].base = (T)0;
            if (z >= 0) other[e] = wave[j[e] * cap + z];
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (X[e] < 0) continue;
            fl[j[e] * cap + X[e]] =
                flux_of<T>(lim, u[e], gt0(u[e]) ? other[e].base : own[e].base, own[e].wl, other[e].wl, s_dth[j[e]]);
        }
        __syncwarp();
    };
    for (WarpRuns wr(ncell, v.nb, v.bi); wr.next();) {
        const long long c = wr.c;
        unsigned need = 0;
        if (c < ncell) {
            if (!is_halo(om, c)) {
                need = (1u << N) - 1u;
            } else {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    const int Llo = link[(long long)(2 * j) * cap + c];
                    if (Llo >= 0 && !is_halo(om, Llo)) need |= 1u << j;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const unsigned bal = __ballot_sync(0xffffffffu, (need >> j) & 1u);
            if ((need >> j) & 1u) {
                const int at = n_q + __popc(bal & lt);
                s_qx[wid][at] = (int)c;
                s_qj[wid][at] = (unsigned char)j;
            }
            n_q += __popc(bal);
        }
        __syncwarp();
        while (n_q >= 32 * E) eval(32 * E);
    }
    if (n_q > 0) eval(n_q);
}

// Large FP64 grids, pass 3: the conservative update of the active cells with the
// previous normalisation applied (halo cells stay 0); adds this thread's new values
// to its digits and maximum. Each warp queues the active cells of its runs in
// shared memory and updates them 32 at a time, so the FP64 lanes all work where
// halo and active entries mix (after growth).
template <int N, typename T>
__device__ __forceinline__ void apply_body(const Model& m, const Bufs& b, const StepView& v, long long (&dacc)[NDIG],
                                           double& mx, int& err) {
    const long long ncell = v.N;
    const long long cap = m.cap;
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    T* __restrict__ Qn = static_cast<T*>(b.q[v.pb ^ 1]);  // aliases no input
    const int* link = b.link[v.g];
    const unsigned short* om = b.om[v.g];
    const T* fl = static_cast<const T*>(b.fl);
    const T scale = (T)v.scale;
    T dth[N];
#pragma unroll
    for (int k = 0; k < N; ++k) dth[k] = (T)v.dth[k];
    T tmax = -INFINITY;
    auto update = [&](long long c) {
        int up[N];
        T lo[N], hi[N];
#pragma unroll
        for (int j = 0; j < N; ++j) up[j] = link[(long long)(2 * j + 1) * cap + c];
#pragma unroll
        for (int j = 0; j < N; ++j) lo[j] = fl[j * cap + c];
#pragma unroll
        for (int j = 0; j < N; ++j) hi[j] = up[j] >= 0 ? fl[j * cap + up[j]] : (T)0;
        T upd = (T)0;
#pragma unroll
        for (int j = 0; j < N; ++j) upd = fmadd(dth[j], hi[j] - lo[j], upd);
        const T qn = (Q[c] - upd) * scale;
        Qn[c] = qn;
        acc_add(dacc, qn, err);
        tmax = vmax(tmax, qn);
    };
    __shared__ int s_ac[WARPS][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int n_a = 0;  // the same in every lane
    for (WarpRuns wr(ncell, v.nb, v.bi); wr.next();) {
        const long long c = wr.c;
        bool act = false;
        if (c < ncell) {
            if (is_halo(om, c)) Qn[c] = (T)0;
            else act = true;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, act);
        if (act) s_ac[wid][n_a + __popc(bal & lt)] = (int)c;
        n_a += __popc(bal);
        __syncwarp();
        if (n_a >= 32) {
            n_a -= 32;
            update(s_ac[wid][n_a + lane]);
            __syncwarp();
        }
    }
    if (lane < n_a) update(s_ac[wid][lane]);
    if (tmax > -INFINITY) mx = fmax(mx, (double)tmax);
}

// Large FP32 grids, passes 2 and 3 in one: every active cell forms the fluxes of
// all its 2n faces itself (those of its upper faces as the lower faces of the
// neighbours above: the same operations on the same values on both sides of a
// face) and is updated at once. Each flux is formed twice, which single precision
// has room for, while the fluxes' way through memory, the faces of the halo and a
// sweep over the pool go; the loads of a cell's dimensions are all independent. Six
// dimensions, 3.2e6 active cells: 0.28 ms in storage order (two kernels, flux and
// update: 0.64 ms with the pool partly out of order, where this takes 0.50 ms).
template <int N, typename T>
__device__ __forceinline__ void update_body(const Model& m, const Bufs& b, const StepView& v, long long (&dacc)[NDIG],
                                            double& mx, int& err) {
    const long long cap = m.cap;
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    T* __restrict__ Qn = static_cast<T*>(b.q[v.pb ^ 1]);  // aliases no input
    const int* link = b.link[v.g];
    const unsigned short* om = b.om[v.g];
    const T* U = static_cast<const T*>(b.u[v.g]);
    const Wave<T>* wave = static_cast<const Wave<T>*>(b.wl);
    const T scale = (T)v.scale;
    const int lim = m.limiter;
    T tmax = -INFINITY;
    for (WarpRuns wr(v.N, v.nb, v.bi); wr.next();) {
        const long long c = wr.c;
        if (c >= v.N) continue;
        if (is_halo(om, c)) {
            Qn[c] = (T)0;
            continue;
        }
        int L[2 * N];
        load_links<N>(link, cap, c, L);  // (an active cell has all its face neighbours)
        T ul[N], uh[N];
        Wave<T> own[N], above[N], other[N];
        T beyond[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            ul[j] = U[j * cap + c];
            own[j] = wave[j * cap + c];
            above[j] = wave[j * cap + L[2 * j + 1]];
            uh[j] = U[j * cap + L[2 * j + 1]];
        }
#pragma unroll
        for (int j = 0; j < N; ++j) {
            // lower face: the cell below when the flow crosses upwards
            other[j].wl = other[j].base = (T)0;
            if (gt0(ul[j])) other[j] = wave[j * cap + L[2 * j]];
            // upper face, flow downwards: the jump beyond the cell above
            beyond[j] = (T)0;
            if (lt0(uh[j])) {
                const int z = link[(long long)(2 * j + 1) * cap + L[2 * j + 1]];
                if (z >= 0) beyond[j] = wave[j * cap + z].wl;
            }
        }
        T upd = (T)0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const T dth = (T)v.dth[j];
            const T lo = flux_of<T>(lim, ul[j], gt0(ul[j]) ? other[j].base : own[j].base, own[j].wl,
                                    gt0(ul[j]) ? other[j].wl : above[j].wl, dth);
            const T hi = flux_of<T>(lim, uh[j], gt0(uh[j]) ? own[j].base : above[j].base, above[j].wl,
                                    gt0(uh[j]) ? own[j].wl : beyond[j], dth);
            upd = fmadd(dth, hi - lo, upd);
        }
        const T qn = (Q[c] - upd) * scale;
        Qn[c] = qn;
        acc_add(dacc, qn, err);
        tmax = vmax(tmax, qn);
    }
    if (tmax > -INFINITY) mx = fmax(mx, (double)tmax);
}

// ------------------------------------------------------------------ step loop of a small grid
// A grid of 10^3 to 10^5 cells in one resident launch is bound by chains of
// dependent operations and by its grid barriers, not by any pipe's throughput.
// Measured on GB300 in SM cycles: a load from L2 290, an atomic that returns 690
// (a 16-bit compare-and-swap 1380), a fence after a store 620, an FP64
// instruction 64 per warp, a grid barrier of 152 blocks 2360; code that does not
// stay in the instruction caches costs more than any of these. So these forms of
// the phases keep one entry, face or neighbour per lane, leave no chain to a
// single thread where lanes can share it, keep rare work out of line, and need
// three barriers per step:
//   1  waves of the existing entries; grow. A new active cell gets its
//      velocities and rate from the warp that inserts it, so dt is known
//      after this phase
//   2  the keys of the missing face neighbours of the newly active cells are
//      claimed (new halo cells); the fluxes of the faces between existing entries
//   3  the update; velocities and links of the new halo cells
// Only newly active cells have faces that touch a new entry (every face neighbour
// of an active cell is in the pool), and few of those fluxes differ from zero
// (apply_small_body).

// The requests of the block's growing cells, in shared memory: the neighbour of
// cell c in direction d1, or the edge neighbour in d1 and d2 (code d1 | d2 << 4;
// d2 = 15: none), is to be made active.
constexpr int GROW_QUEUE = 1024;
struct GrowQueue {
    int n;
    int cell[GROW_QUEUE];
    unsigned char code[GROW_QUEUE];
};

// A rate (as the word of a non-negative double) above the largest known; one that is no
// number is none, as in the maxima of the other phases.
__device__ __forceinline__ bool larger_rate(unsigned long long rb, unsigned long long known) {
    return rb > known && rb <= 0x7ff0000000000000ull;
}

// A warp's grow requests: neighbour `code` of cell cc (made active as
// grow_candidate does it, with the marks of the step loop, and the inserted
// cells' velocities formed at once). rate_now: the largest CFL rate known; only a larger one is written (it
// rarely is). All lanes must call it.
template <int N, typename T>
__device__ __noinline__ void grow_act(const Model& m, const Bufs& b, int g, int pb, unsigned fresh, bool has, int cc,
                                      unsigned code, unsigned long long rate_now, unsigned long long* rate) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int F = 2 * N, G = 32 / F;
    DevScalars* sc = b.sc;
    const long long cap = m.cap;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int d1 = code & 15, d2 = code >> 4;
    int e = -2;
    if (has) {
        e = (b.link[g] + d1 * cap)[cc];
        if (d2 < F && e >= 0) e = (b.link[g] + d2 * cap)[e];
    }
    // a halo cell: the one lane that clears its flag activates it (32-bit
    // atomics: a 16-bit compare-and-swap is a loop around a 32-bit one)
    bool act = false;
    if (e >= 0) {
        unsigned* word = reinterpret_cast<unsigned*>(b.om[g]) + (e >> 1);
        const int sh = (e & 1) * 16;
        act = (atomicAnd(word, ~((unsigned)OM_GHOST << sh)) >> sh) & OM_GHOST;
        if (act) {
            atomicOr(word, fresh << sh);
            const unsigned long long rb = (unsigned long long)__double_as_longlong(b.rate[g][e]);
            if (larger_rate(rb, rate_now)) atomicMax(rate, rb);
        }
    }
    const unsigned acts = __ballot_sync(full, act);
    if (acts) {
        long long base = 0;
        if (lane == 0) base = (long long)atomicAdd((unsigned long long*)&sc->n_act, (unsigned long long)__popc(acts));
        base = __shfl_sync(full, base, 0);
        if (act) b.map[base + __popc(acts & lt)] = e;
    }
    if (!__any_sync(full, e == -1)) return;
    // missing cells (rare): inserted as active
    bool inserted = false;
    long long c = 0;
    unsigned long long key = 0;
    if (e == -1) {
        int J[N];
        unpack_key<N>(m, b.key[g][cc], J);
#pragma unroll
        for (int x = 0; x < N; ++x) {
            if ((d1 >> 1) == x) J[x] += (d1 & 1) ? 1 : -1;
            if ((d2 >> 1) == x) J[x] += (d2 & 1) ? 1 : -1;  // (15: no dimension)
        }
        if (!interior<N>(m, J)) {
            set_error(sc, ST_EKEYRANGE);
        } else {
            pack_key<N>(m, J, key);
            unsigned long long slot;
            const int claim = table_claim(m, b.table, sc, key, &slot);
            if (claim < 0) set_error(sc, ST_ETABLE);
            if (claim > 0) {
                c = (long long)atomicAdd((unsigned long long*)&sc->N, 1ull);
                if (c >= cap) {
                    set_error(sc, ST_ECAPACITY);
                } else {
                    inserted = true;
                    b.table[slot].val = c;
                    b.slot[g][c] = (unsigned int)slot;
                    b.key[g][c] = key;
                    static_cast<T*>(b.q[pb])[c] = (T)0;
#pragma unroll 1
                    for (int d = 0; d < F; ++d) b.link[g][(long long)d * cap + c] = -1;
                }
            }
        }
    }
    const int s = lane / F;
#pragma unroll 1
    for (unsigned todo = __ballot_sync(full, inserted); todo;) {
        unsigned rest = todo;  // lanes of slot s work on the s-th entry still to do
#pragma unroll 1
        for (int i = 0; i < s && rest; ++i) rest &= rest - 1;
        const bool on = s < G && rest;
        const int owner = on ? __ffs(rest) - 1 : 0;
        const unsigned long long ko = __shfl_sync(full, key, owner);
        const int co = __shfl_sync(full, (int)c, owner);
        const double r = complete_group<N, T>(m, b, g, on, co, ko, 0u, false);
        const unsigned long long rb = (unsigned long long)__double_as_longlong(r);
        if (on && lane == s * F && larger_rate(rb, rate_now)) atomicMax(rate, rb);
#pragma unroll 1
        for (int i = 0; i < G; ++i) todo &= todo - 1;
    }
}

// Every growing cell of the existing entries looks at its downwind set: face
// neighbours (in the pool, perhaps as halo cells) and edge neighbours (through
// the link of the first face), four neighbours at a time with their loads in
// flight together (links do not change in this phase). A cell's outward
// directions are mostly one per dimension, so its list is short: N faces and
// N (N - 1) / 2 edges. What is still to be made active goes to the block's list,
// and from there to all its warps; a warp that finds the list full acts on its
// own requests at once.
template <int N, typename T>
__device__ __forceinline__ void grow_detect(const Model& m, const Bufs& b, const StepView& v, GrowQueue& gq,
                                            unsigned long long rate_now, unsigned long long* rate) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int C = 4;
    const int ncell = (int)v.N_prev;
    const long long cap = m.cap;
    const Above<T> above(m.thr_rel * v.maxq);
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    const int* link = b.link[v.g];
    unsigned short* om = b.om[v.g];
    const unsigned stale = v.fresh ^ (3u * OM_NEW);  // the mark of the step before
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (Runs r(runs_of(ncell), v.nb, v.bi); r.next();) {
        const int c = r.cell();
        unsigned out = 0;
        if (c < ncell) {
            const unsigned f = *(volatile unsigned short*)&om[c];
            out = f & 0xfffu;
            const bool grow = !(f & (OM_COMPLETE | OM_GHOST)) && out && above(Q[c]);
            if (grow || (f & stale)) om[c] = (unsigned short)((f & ~stale) | (grow ? OM_COMPLETE : 0));
            if (!grow) out = 0;
        }
        // (d1, d2) runs over the outward directions d1, alone and with each later d2
        unsigned rem1 = out, rem2 = 0;
        int d1 = 0;
        bool face = false;  // d1 alone is next
        auto next = [&]() -> unsigned {  // the next code, or 0xff
            if (!face && !rem2) {
                if (!rem1) return 0xffu;
                d1 = __ffs(rem1) - 1;
                rem1 &= rem1 - 1;
                face = true;
            }
            if (face) {
                face = false;
                rem2 = out & (~0u << ((d1 | 1) + 1));
                return (unsigned)d1 | 0xf0u;
            }
            const int d2 = __ffs(rem2) - 1;
            rem2 &= rem2 - 1;
            return (unsigned)(d1 | (d2 << 4));
        };
#pragma unroll 1
        while (__any_sync(full, (rem1 | rem2) != 0 || face)) {
            unsigned code[C];
            int e[C];
#pragma unroll
            for (int i = 0; i < C; ++i) {
                code[i] = next();
                e[i] = code[i] != 0xffu ? (link + (code[i] & 15) * cap)[c] : -2;
            }
#pragma unroll
            for (int i = 0; i < C; ++i)
                if (e[i] >= 0 && (code[i] >> 4) != 15) e[i] = (link + (code[i] >> 4) * cap)[e[i]];
            unsigned need = 0;  // four codes of eight bits
            int n_need = 0;
            unsigned f[C];
#pragma unroll
            for (int i = 0; i < C; ++i) f[i] = e[i] >= 0 ? *(volatile unsigned short*)&om[e[i]] : 0u;
#pragma unroll
            for (int i = 0; i < C; ++i)
                if (e[i] == -1 || (f[i] & OM_GHOST)) {
                    need = (need << 8) | code[i];
                    ++n_need;
                }
#pragma unroll 1
            for (unsigned bal; (bal = __ballot_sync(full, n_need > 0)) != 0; --n_need, need >>= 8) {
                const bool want = n_need > 0;
                int at = 0;
                if (lane == 0) at = atomicAdd(&gq.n, __popc(bal));
                at = __shfl_sync(full, at, 0) + __popc(bal & ((1u << lane) - 1u));
                if (want && at < GROW_QUEUE) {
                    gq.cell[at] = c;
                    gq.code[at] = (unsigned char)need;
                }
                const bool over = want && at >= GROW_QUEUE;
                if (__any_sync(full, over))
                    grow_act<N, T>(m, b, v.g, v.pb, v.fresh, over, c, need & 0xffu, rate_now, rate);
            }
        }
    }
}

// The listed requests, 32 per warp and round (after a block barrier).
template <int N, typename T>
__device__ __forceinline__ void grow_drain(const Model& m, const Bufs& b, const StepView& v, const GrowQueue& gq,
                                           unsigned long long rate_now, unsigned long long* rate) {
    const int n = min(gq.n, GROW_QUEUE);
#pragma unroll 1
    for (int q0 = threadIdx.x & ~31; q0 < n; q0 += blockDim.x) {
        const int q = q0 + (threadIdx.x & 31);
        const bool has = q < n;
        grow_act<N, T>(m, b, v.g, v.pb, v.fresh, has, has ? gq.cell[q] : 0, has ? gq.code[q] : 0u, rate_now, rate);
    }
}

// The slot of key: claimed (1, was free), found (0) or the table is full (-1).
// Compare-and-swap at once: most keys asked for here are new.
__device__ __forceinline__ int table_claim_or_find(const Model& m, Slot* T, const DevScalars* sc,
                                                   unsigned long long key, unsigned long long* slot) {
    unsigned long long h = table_home(key, m.tmask);
#pragma unroll 1
    for (unsigned long long probe = 0; probe <= m.tmask; ++probe) {
        const unsigned long long k = atomicCAS(&T[h].key, EMPTY_KEY, key);
        *slot = h;
        if (k == EMPTY_KEY) return 1;
        if (k == key) return 0;
        if (claim_hopeless(sc, probe)) return -1;
        h = table_next(h, probe, m.tmask);
    }
    return -1;
}

// The face neighbours of the newly active cells, one (cell, face) per lane: the
// inserted cells [N_prev, n_ins) and the nact activated halo cells listed in map
// (only their missing neighbours). A neighbour that was in the pool before this
// phase is linked with the cell; a key that is not in the table is claimed for a
// new halo cell, appended at n_ins + n_halo, whose links and velocities phase 3
// makes (halo_complete_body), when all new cells have their indices in the table.
template <int N, typename T>
__device__ __forceinline__ void halo_claim_body(const Model& m, const Bufs& b, const StepView& v, long long n_ins,
                                                long long nact) {
    constexpr int F = 2 * N, G = 32 / F;  // cells per warp
    DevScalars* sc = b.sc;
    const long long cap = m.cap;
    const int lo = (int)v.N_prev, ni = (int)(n_ins - lo), total = ni + (int)nact;
    const int lane = threadIdx.x & 31;
    const int s = lane / F, d = lane - s * F;
#pragma unroll 1
    for (Runs r((total + G - 1) / G, v.nb, v.bi, LAST); r.next();) {
        const int q = r.k * G + s;
        if (s >= G || q >= total) continue;
        const int x = q < ni ? lo + q : b.map[q - ni];
        unsigned long long k = b.key[v.g][x];
        if (*(volatile int*)&(b.link[v.g] + d * cap)[x] >= 0) continue;
        const int shift = m.key_bits * (N - 1 - (d >> 1));
        const unsigned long long last = (1ull << m.key_bits) - 1, field = (k >> shift) & last;
        // an activated halo cell at the end of the key range has a neighbour without a key
        if (field == ((d & 1) ? last : 0ull)) {
            set_error(sc, ST_EKEYRANGE);
            continue;
        }
        k = (d & 1) ? k + (1ull << shift) : k - (1ull << shift);
        unsigned long long slot;
        const int claim = table_claim_or_find(m, b.table, sc, k, &slot);
        if (claim < 0) {
            set_error(sc, ST_ETABLE);
        } else if (claim == 0) {
            const long long nbr = *(volatile long long*)&b.table[slot].val;
            if (nbr >= 0 && nbr < n_ins) {
                (b.link[v.g] + d * cap)[x] = (int)nbr;
                (b.link[v.g] + (d ^ 1) * cap)[nbr] = x;
            }
        } else {
            const long long c = n_ins + warp_aggregated_add(&sc->n_halo);
            if (c >= cap) {
                set_error(sc, ST_ECAPACITY);
                continue;
            }
            *(volatile long long*)&b.table[slot].val = c;
            b.slot[v.g][c] = (unsigned int)slot;
            b.key[v.g][c] = k;
        }
    }
}

// Phase 3 of the new halo cells [n_ins, N): velocities, mask, rate, links, value 0.
template <int N, typename T>
__device__ __forceinline__ void halo_complete_body(const Model& m, const Bufs& b, const StepView& v,
                                                   long long n_ins) {
    constexpr int F = 2 * N, G = 32 / F;  // entries per warp
    const int lo = (int)n_ins, total = (int)(v.N - n_ins);
    const int lane = threadIdx.x & 31, s = lane / F;
#pragma unroll 1
    for (Runs r((total + G - 1) / G, v.nb, v.bi, LAST); r.next();) {
        const int q = r.k * G + s;
        const bool on = s < G && q < total;
        const int c = on ? lo + q : 0;
        const unsigned long long k = on ? b.key[v.g][c] : 0ull;
        complete_group<N, T>(m, b, v.g, on, c, k, OM_GHOST, true);
        if (on && lane == s * F) static_cast<T*>(b.q[v.pb ^ 1])[c] = (T)0;
    }
}

// The fluxes of the faces between existing entries that touch an active cell
// (both sides below nold: halo_claim_body meanwhile writes links to or from
// entries beyond it only, so what it changes is not read here). One face per thread,
// the runs of 32 entries of dimension after dimension.
template <int N, typename T>
__device__ __forceinline__ void faces_old_body(const Model& m, const Bufs& b, const StepView& v) {
    const unsigned short* om = b.om[v.g];
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    const T* tg = static_cast<const T*>(b.tg);
    const long long cap = m.cap;
    const int nold = (int)v.N_prev, runs = runs_of(nold);
    const int lim = m.limiter;
    const T dt = (T)v.dt;
#pragma unroll 1
    for (Runs r(runs * N, v.nb, v.bi); r.next();) {
        int j = 0, k = r.k;
#pragma unroll 1
        while (k >= runs) {
            k -= runs;
            ++j;
        }
        const int X = k * 32 + (int)(threadIdx.x & 31);
        if (X >= nold) continue;
        const int* lo = b.link[v.g] + 2 * j * cap;
        const T* wl = static_cast<const T*>(b.wl) + j * cap;
        const int Llo = lo[X], Lup = (lo + cap)[X];
        const T u = (static_cast<const T*>(b.u[v.g]) + j * cap)[X];
        const unsigned short fX = om[X];
        const T P0 = Q[X], W = wl[X];
        if (Llo < 0 || Llo >= nold) continue;
        if ((fX & OM_GHOST) && is_halo(om, Llo)) continue;
        T f = (T)0;
        if (flows(u)) {
            const bool up = gt0(u);  // the upwind cell is Llo, else X
            const int y = up ? Llo : X;
            // the jump across the face beyond the upwind cell
            const int z = up ? Llo : (Lup < nold ? Lup : -1);
            const T Wb = z >= 0 ? wl[z] : zero_minus(P0);
            const T Py = up ? Q[Llo] : P0;
            const T S = fmadd(-(T)m.inv_2h[j], (static_cast<const T*>(b.wg) + j * cap)[y], tg[y]);
            f = u * fmadd(-dt, S, Py);
            if (lim != LIM_NONE && nonzero(W)) {
                const T au = abs_bits(u);
                f = fmadd(half_nonneg(au) * fmadd(-(T)pick_of<N>(v.dth, j), au, (T)1), limited_wave<T>(lim, W, Wb), f);
            }
        }
        (static_cast<T*>(b.fl) + j * cap)[X] = f;
    }
}

// Phase 3: the update.
// Newly active cells (density 0; the inserted ones and the nact listed in map):
// 2N lanes of a warp per cell, one face each, and the update in the first of
// them. Let x be the cell and z its neighbour across a face.
//   both existing entries: the flux is there (faces_old_body);
//   both new: nothing nearby has a density (a new entry is no face neighbour of
//     a cell that was active before), the flux is 0;
//   one of them new: both densities are 0, so neither the donor term nor the
//     limited term contributes, and only the transverse sum of the existing one
//     does, when it is upwind of the face.
// (Zeros enter the update as +0 here where the general form may give -0; a sum
// that starts from +0 is the same with either.)
// The existing entries that were active before this step: one lane per cell, all
// its faces lie between existing entries; existing halo entries get 0.
// The new values add to the thread's digits and maximum.
template <int N, typename T>
__device__ __forceinline__ void apply_small_body(const Model& m, const Bufs& b, const StepView& v, long long n_ins,
                                                 long long nact, long long (&dacc)[NDIG], T& mx, int& err) {
    constexpr unsigned full = 0xffffffffu;
    constexpr int F = 2 * N, G = 32 / F;  // new cells per warp
    const long long cap = m.cap;
    const int nold = (int)v.N_prev, ni = (int)(n_ins - v.N_prev), total = ni + (int)nact;
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    T* Qn = static_cast<T*>(b.q[v.pb ^ 1]);
    const int* link = b.link[v.g];
    const unsigned short* om = b.om[v.g];
    const T* U = static_cast<const T*>(b.u[v.g]);
    const T* fl = static_cast<const T*>(b.fl);
    const T* wg = static_cast<const T*>(b.wg);
    const T* tg = static_cast<const T*>(b.tg);
    const T scale = (T)v.scale;
    const int lane = threadIdx.x & 31;
    const int s = lane / F, d = lane - s * F;
    Runs fresh((total + G - 1) / G, v.nb, v.bi, MIDDLE);
    Runs old(runs_of(nold), v.nb, v.bi);
#pragma unroll 1
    for (;;) {
        int c = 0;
        bool active = false;
        T upd = (T)0;
        if (fresh.next()) {
            const int q = fresh.k * G + s;
            const bool mine = s < G && q < total;
            const int j = d >> 1;
            T f = (T)0;
            if (mine) {
                c = q < ni ? nold + q : b.map[q - ni];
                // (links to new halo cells appear while this runs: missing or new, it is the same)
                const int z = (link + d * cap)[c];
                const bool oldx = c < nold, oldz = z >= 0 && z < nold;
                if (oldx && oldz) {
                    f = (fl + j * cap)[(d & 1) ? z : c];
                } else if (oldx || oldz) {
                    const int y = oldx ? c : z;
                    const T S = fmadd(-(T)m.inv_2h[j], (wg + j * cap)[y], tg[y]);
                    T u;
                    if (!(d & 1)) u = (U + j * cap)[c];
                    else if (z >= 0 && z < n_ins) u = (U + j * cap)[z];
                    else u = (T)face_velocity_key<N>(m, b.key[v.g][c], j, 1);
                    // the existing one upwind: z below and the flow up, or z above and it down; c the other way round
                    if ((oldz == !(d & 1)) ? gt0(u) : lt0(u)) f = u * fmadd(-(T)v.dt, S, (T)0);
                }
            }
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const T lo = __shfl_sync(full, f, (lane + 2 * i) & 31);
                const T hi = __shfl_sync(full, f, (lane + 2 * i + 1) & 31);
                upd = fmadd((T)v.dth[i], hi - lo, upd);
            }
            active = mine && d == 0;
        } else if (old.next()) {
            c = old.cell();
            const unsigned f = c < nold ? om[c] : v.fresh;
            if (f & OM_GHOST) Qn[c] = (T)0;
            active = !(f & (OM_GHOST | v.fresh));
            if (active) {
                T hi[N], lo[N];
                int up[N];
#pragma unroll
                for (int j = 0; j < N; ++j) up[j] = (link + (2 * j + 1) * cap)[c];
#pragma unroll
                for (int j = 0; j < N; ++j) lo[j] = (fl + j * cap)[c];
#pragma unroll
                for (int j = 0; j < N; ++j) hi[j] = up[j] >= 0 ? (fl + j * cap)[up[j]] : (T)0;
#pragma unroll
                for (int j = 0; j < N; ++j) upd = fmadd((T)v.dth[j], hi[j] - lo[j], upd);
            }
        } else {
            break;
        }
        if (active) {
            const T qn = (Q[c] - upd) * scale;
            Qn[c] = qn;
            acc_add(dacc, qn, err);
            mx = vmax(mx, qn);
        }
    }
}

// The end of a launch: the marks of its last step's activated cells.
__device__ __forceinline__ void clear_marks(const Bufs& b, const StepView& v, long long nact) {
    unsigned short* om = b.om[v.g];
#pragma unroll 1
    for (WarpRuns wr(nact, v.nb, v.bi); wr.next();) {
        if (wr.c >= nact) continue;
        const int x = b.map[wr.c];
        om[x] = (unsigned short)(om[x] & ~(3u * OM_NEW));
    }
}

// ------------------------------------------------------------------ prune

// keep[c] = (p_c > p*) for the active cells: the significant cells S. (all: a
// re-sort, which keeps every active cell and, with them, every halo cell.)
template <typename T>
__device__ __forceinline__ void prune_mark_body(const Model& m, const Bufs& b, const StepView& v, bool all = false) {
    const double pstar = m.thr_rel * v.maxq;
    const Above<T> above(pstar);
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    const unsigned short* om = b.om[v.g];
#pragma unroll 1
    for (WarpRuns r(v.N, v.nb, v.bi); r.next();) {
        const long long c = r.c;
        if (c < v.N) b.keep[c] = !is_halo(om, c) && (all || above(Q[c]));
    }
}

// keep[D(S)] = 1: each significant cell marks the pool entries of its
// downwind set (Sec. 3.3, Fig. 3); only the active ones among them are kept.
template <int N, typename T>
__device__ __forceinline__ void prune_scatter_body(const Model& m, const Bufs& b, const StepView& v) {
    const double pstar = m.thr_rel * v.maxq;
    const Above<T> above(pstar);
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    const int* link = b.link[v.g];
    const unsigned short* om = b.om[v.g];
    const long long cap = m.cap;
#pragma unroll 1
    for (WarpRuns r(v.N, v.nb, v.bi); r.next();) {
        const long long c = r.c;
        if (c >= v.N) continue;
        const unsigned f = om[c];
        if ((f & OM_GHOST) || !above(Q[c])) continue;
        const unsigned out = f & 0xfffu;
        if (!out) continue;
        int L[2 * N];
        load_links<N>(link, cap, c, L);
#pragma unroll
        for (int d = 0; d < 2 * N; ++d)
            if (((out >> d) & 1u) && L[d] >= 0) b.keep[L[d]] = 1;
#pragma unroll
        for (int d1 = 0; d1 < 2 * N; ++d1) {
            if (!((out >> d1) & 1u)) continue;
            int e[2 * N];  // (loaded together: the marks may alias the links, for the compiler)
#pragma unroll
            for (int d2 = 0; d2 < 2 * N; ++d2)
                e[d2] = (d2 >> 1) > (d1 >> 1) && ((out >> d2) & 1u)
                            ? edge_by_links<N>(link, cap, L, d1 >> 1, d1 & 1, d2 >> 1, d2 & 1)
                            : -1;
#pragma unroll
            for (int d2 = 0; d2 < 2 * N; ++d2)
                if (e[d2] >= 0) b.keep[e[d2]] = 1;
        }
    }
}

// chunk [c0, c1) of a range of `total` items handled by block bi of nb
__device__ __forceinline__ void block_chunk(long long total, long long& c0, long long& c1, int nb, int bi) {
    long long per = (total + nb - 1) / nb;
    per = (per + THREADS - 1) / THREADS * THREADS;
    c0 = min(total, per * bi);
    c1 = min(total, c0 + per);
}
__device__ __forceinline__ void block_chunk(long long total, long long& c0, long long& c1) {
    block_chunk(total, c0, c1, gridDim.x, blockIdx.x);
}

// Sum of a per-thread count over the block (every thread gets it).
__device__ __forceinline__ long long block_count(int cnt) {
    __shared__ long long s[MAX_WARPS];
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, off);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = cnt;
    __syncthreads();
    long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s[w];
    __syncthreads();
    return t;
}

// Range of the key fields of the entries a thread has seen, folded into the
// scalars (for the sort's codes). All threads of the block must call fold.
template <int N>
struct FieldRange {
    unsigned lo[N], hi[N];
    __device__ __forceinline__ FieldRange() {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            lo[j] = ~0u;
            hi[j] = 0u;
        }
    }
    __device__ __forceinline__ void see(const Model& m, unsigned long long k) {
        const unsigned long long mask = (1ull << m.key_bits) - 1;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const unsigned f = (unsigned)((k >> (m.key_bits * (N - 1 - j))) & mask);
            lo[j] = min(lo[j], f);
            hi[j] = max(hi[j], f);
        }
    }
    __device__ __forceinline__ void fold(DevScalars* sc) {
        __shared__ unsigned s_lo[N], s_hi[N];
        if (threadIdx.x < N) {
            s_lo[threadIdx.x] = ~0u;
            s_hi[threadIdx.x] = 0u;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const unsigned l = __reduce_min_sync(0xffffffffu, lo[j]), h = __reduce_max_sync(0xffffffffu, hi[j]);
            if ((threadIdx.x & 31) == 0 && l <= h) {
                atomicMin(&s_lo[j], l);
                atomicMax(&s_hi[j], h);
            }
        }
        __syncthreads();
        if (threadIdx.x < N && s_lo[threadIdx.x] <= s_hi[threadIdx.x]) {
            atomicMin(&sc->sort_lo[threadIdx.x], s_lo[threadIdx.x]);
            atomicMax(&sc->sort_hi[threadIdx.x], s_hi[threadIdx.x]);
        }
    }
};

// Status of every entry into map: 1 active and kept, 2 halo of a kept cell
// (not kept, with a kept face neighbour), 0 dropped. The block's counts of
// both go to blk and blk2; the table slots of the current entries are emptied
// for the rehash (the table holds nothing else). SORTED: a sort follows, which
// needs the range of the survivors' key fields and, of the counts, only their totals:
// the blocks take their entries in turn then, not chunk by chunk (the halo cells,
// together in the pool, are nearly all the work: 4.9e6 entries in six dimensions 0.31
// ms, now 0.19; 6.5e5 77 us, now 45).
template <int N, bool SORTED = false>
__device__ __forceinline__ void prune_count_body(const Model& m, const Bufs& b, const StepView& v) {
    FieldRange<N> range;
    const int* link = b.link[v.g];
    const unsigned short* om = b.om[v.g];
    const unsigned int* slots = b.slot[v.g];
    const long long cap = m.cap;
    int na = 0, ng = 0;
    auto status = [&](long long c) {
        int st = 0;
        if (b.keep[c] && !is_halo(om, c)) {
            st = 1;
        } else {
            int L[2 * N];
            load_links<N>(link, cap, c, L);
            // (the flags of all neighbours in flight together; few are kept)
            unsigned kept[2 * N];
#pragma unroll
            for (int d = 0; d < 2 * N; ++d) kept[d] = L[d] >= 0 ? b.keep[L[d]] : 0u;
#pragma unroll
            for (int d = 0; d < 2 * N; ++d)
                if (kept[d] && !st && !is_halo(om, L[d])) st = 2;
        }
        b.map[c] = st;
        na += st == 1;
        ng += st == 2;
        reinterpret_cast<ulonglong2*>(b.table)[slots[c]] = make_ulonglong2(EMPTY_KEY, ~0ull);
        if (SORTED && st) range.see(m, b.key[v.g][c]);
    };
    if constexpr (SORTED) {
#pragma unroll 1
        for (WarpRuns r(v.N, v.nb, v.bi); r.next();)
            if (r.c < v.N) status(r.c);
        range.fold(b.sc);
    } else {
        long long c0, c1;
        block_chunk(v.N, c0, c1, v.nb, v.bi);
#pragma unroll 1
        for (long long c = c0 + threadIdx.x; c < c1; c += blockDim.x) status(c);
    }
    const long long ta = block_count(na);
    const long long tg = block_count(ng);
    if (threadIdx.x == 0) {
        b.blk[v.bi] = ta;
        b.blk2[v.bi] = tg;
    }
}

// The survivors of a sorting prune in their new order (the flux scratch, free until
// the next step).
__device__ __forceinline__ int* sorted_order(const Bufs& b) { return static_cast<int*>(b.fl); }

// Offsets of this block's survivors in the new pool (active cells first, then
// halo cells) and the totals, read by every block from blk and blk2.
struct Survivors {
    long long base_a, base_g, total_a, total_g;
};
__device__ __forceinline__ Survivors block_offsets(const Bufs& b, int nb, int bi) {
    __shared__ long long s[4][MAX_WARPS];
    long long v[4] = {0, 0, 0, 0};  // offset a, total a, offset g, total g
#pragma unroll 1
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const long long a = __ldcg(&b.blk[i]);
        const long long g = __ldcg(&b.blk2[i]);
        v[1] += a;
        v[3] += g;
        if (i < bi) {
            v[0] += a;
            v[2] += g;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        for (int off = 16; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
        if ((threadIdx.x & 31) == 0) s[k][threadIdx.x >> 5] = v[k];
    }
    __syncthreads();
    long long t[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll 1
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t[k] += s[k][w];
    __syncthreads();
    Survivors r;
    r.base_a = t[0];
    r.total_a = t[1];
    r.base_g = t[1] + t[2];
    r.total_g = t[3];
    return r;
}

// The face velocities and the CFL rate of entry c (generation g) move to nc of
// the other generation.
template <int N, typename T>
__device__ __forceinline__ void copy_velocities(const Model& m, const Bufs& b, int g, long long c, long long nc) {
    const T* U = static_cast<const T*>(b.u[g]);
    T* Uo = static_cast<T*>(b.u[g ^ 1]);
#pragma unroll
    for (int j = 0; j < N; ++j) Uo[j * m.cap + nc] = U[j * m.cap + c];
    b.rate[g ^ 1][nc] = b.rate[g][c];
}

// Stream compaction of the survivors in storage order into the other buffer
// set: the kept active cells at [0, total_a), the halo cells after them;
// map[c] = new index or -1. Values of active cells are rescaled by an exact
// power of two that brings the maximum into [1, 2) (their ratios do not
// change, and the exact sum stays in its window even after a very unlikely
// measurement); halo cells hold 0. Adds the active cells' digits, maximum and
// CFL rates. (resort: the order alone changes, not the values, nor what is known to
// be complete.)
template <int N, typename T>
__device__ __forceinline__ void prune_compact_body(const Model& m, const Bufs& b, const StepView& v, Survivors sv,
                                                   long long (&d)[NDIG], double& mx, double& rmax, int& err,
                                                   bool resort = false) {
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    T* Qo = static_cast<T*>(b.q[v.pb ^ 1]);
    const unsigned long long* key = b.key[v.g];
    unsigned long long* keyo = b.key[v.g ^ 1];
    const unsigned short* om = b.om[v.g];
    unsigned short* omo = b.om[v.g ^ 1];
    const double mq = v.maxq;
    const double s2 = (mq > 0.0 && isfinite(mq) && !resort) ? ldexp(1.0, -ilogb(mq)) : 1.0;
    const unsigned kept_flags = resort ? 0xfffu | OM_COMPLETE : 0xfffu;
    long long ba = sv.base_a, bg = sv.base_g;
    long long c0, c1;
    block_chunk(v.N, c0, c1, v.nb, v.bi);
#pragma unroll 1
    for (long long t0 = c0; t0 < c1; t0 += blockDim.x) {
        const long long c = t0 + threadIdx.x;
        const int st = (c < c1) ? b.map[c] : 0;
        int na, ng;
        const int pa = block_exclusive_scan(st == 1, na);
        const int pg = block_exclusive_scan(st == 2, ng);
        if (c < c1) {
            const unsigned long long k = key[c];
            if (st == 1) {
                const long long nc = ba + pa;
                const T val = (T)((double)Q[c] * s2);
                keyo[nc] = k;
                Qo[nc] = val;
                omo[nc] = (unsigned short)(om[c] & kept_flags);
                copy_velocities<N, T>(m, b, v.g, c, nc);
                b.map[c] = (int)nc;
                acc_add(d, (double)val, err);
                mx = fmax(mx, (double)val);
                rmax = fmax(rmax, b.rate[v.g][c]);
            } else if (st == 2) {
                const long long nc = bg + pg;
                keyo[nc] = k;
                Qo[nc] = (T)0;
                omo[nc] = (unsigned short)((om[c] & 0xfffu) | OM_GHOST);
                copy_velocities<N, T>(m, b, v.g, c, nc);
                b.map[c] = (int)nc;
            } else {
                b.map[c] = -1;
            }
        }
        ba += na;
        bg += ng;
    }
}

// The compaction of the graph and direct paths with a sort: the survivor at place nc
// of the new order is entry order[nc] (status in keep, new index of any entry in
// map); the same values, rescaling and partials as prune_compact_body, its links
// through the map and its place in the hashtable too. One thread per new place, so
// that what is scattered are reads, whole sectors of them: written from the old order
// (a kernel for the state and one for the links) partial sectors went to memory and
// back. 4.9e6 entries in six dimensions, wholly out of order: 1.18 ms (1.69 ms), 4.7
// GB to and from memory; nearly in order, 1.4e6: 0.14 ms either way.
template <int N, typename T>
__device__ __forceinline__ void prune_move_body(const Model& m, const Bufs& b, const StepView& v, long long n_new,
                                                long long (&d)[NDIG], double& mx, double& rmax, int& err,
                                                bool resort) {
    const T* Q = static_cast<const T*>(b.q[v.pb]);
    T* Qo = static_cast<T*>(b.q[v.pb ^ 1]);
    const int* link = b.link[v.g];
    int* linko = b.link[v.g ^ 1];
    const unsigned short* om = b.om[v.g];
    unsigned short* omo = b.om[v.g ^ 1];
    const int* order = sorted_order(b);
    const long long cap = m.cap;
    const double mq = v.maxq;
    const double s2 = (mq > 0.0 && isfinite(mq) && !resort) ? ldexp(1.0, -ilogb(mq)) : 1.0;
    const unsigned kept_flags = resort ? 0xfffu | OM_COMPLETE : 0xfffu;
#pragma unroll 1
    for (WarpRuns r(n_new, v.nb, v.bi); r.next();) {
        const long long nc = r.c;
        if (nc < n_new) {
            const long long c = order[nc];
            int L[2 * N];
            load_links<N>(link, cap, c, L);
            const unsigned long long k = b.key[v.g][c];
            const bool halo = b.keep[c] == 2;
            const unsigned short f = om[c];
            const T q = Q[c];
            const double rate = b.rate[v.g][c];
            copy_velocities<N, T>(m, b, v.g, c, nc);
            b.key[v.g ^ 1][nc] = k;
#pragma unroll
            for (int e = 0; e < 2 * N; ++e) linko[(long long)e * cap + nc] = L[e] >= 0 ? b.map[L[e]] : -1;
            if (halo) {
                Qo[nc] = (T)0;
                omo[nc] = (unsigned short)((f & 0xfffu) | OM_GHOST);
            } else {
                const T val = (T)((double)q * s2);
                Qo[nc] = val;
                omo[nc] = (unsigned short)(f & kept_flags);
                acc_add(d, (double)val, err);
                mx = fmax(mx, (double)val);
                rmax = fmax(rmax, rate);
            }
            table_insert_new(m, b, k, nc, b.slot[v.g ^ 1]);
        }
        __syncwarp();
    }
}

// New links through the map, and the rehash of the survivors.
template <int N>
__device__ __forceinline__ void prune_relink_body(const Model& m, const Bufs& b, const StepView& v) {
    const int* link = b.link[v.g];
    int* linko = b.link[v.g ^ 1];
    const unsigned long long* keyo = b.key[v.g ^ 1];
    const long long cap = m.cap;
#pragma unroll 1
    for (WarpRuns r(v.N, v.nb, v.bi); r.next();) {
        const long long c = r.c;
        if (c >= v.N) continue;
        const int nc = b.map[c];
        if (nc < 0) continue;
        int L[2 * N];
        load_links<N>(link, cap, c, L);
#pragma unroll
        for (int d = 0; d < 2 * N; ++d) linko[(long long)d * cap + nc] = L[d] >= 0 ? b.map[L[d]] : -1;
        table_insert_new(m, b, keyo[nc], nc, b.slot[v.g ^ 1]);
    }
}

}  // namespace gbees
