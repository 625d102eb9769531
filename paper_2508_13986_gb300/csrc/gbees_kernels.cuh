// Kernels of the GBEES step other than the flux update: initial grid, directional
// grow (Sec. 3.3, Algorithm 2), neighbour links (Sec. 4.1), Bayesian update
// (Eq. 4), directional prune with stream compaction and rehash (Algorithm 3),
// read-out and moments. All kernels use a fixed grid and loop over the cells,
// whose count they read from device memory, so that no step needs the host.
#pragma once

#include "gbees_phases.cuh"
#include "gbees_rows.cuh"

namespace gbees {

// ------------------------------------------------------------------ links

// The CFL rates of the cells that a kernel made active join the running maximum
// (known: the maximum when the kernel began; rates are compared as the words of
// non-negative doubles, off the FP64 pipe). All threads of the block.
__device__ __forceinline__ void join_rates(DevScalars* sc, double rate, unsigned long long known) {
    __shared__ unsigned long long s_r[MAX_WARPS];
    long long x = __double_as_longlong(rate);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x = max(x, __shfl_down_sync(0xffffffffu, x, off));
    if ((threadIdx.x & 31) == 0) s_r[threadIdx.x >> 5] = x > 0 ? (unsigned long long)x : 0ull;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long r = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = max(r, s_r[w]);
        if (r > known) atomicMax(&sc->maxrate_bits, r);
    }
}

// Finish a step's time after the link phase: dt from the maximum CFL rate over all
// cells, with its coefficients.
// step: 1 of a time step; 0 and -1 of a new grid, whose normalisation follows
// (-1: cells taken as given).
__device__ __forceinline__ void finish_link(const Model& m, DevScalars* sc, int step) {
    const unsigned long long r = *(volatile unsigned long long*)&sc->maxrate_bits;
    if (step <= 0) {
        finalise_norm(m, sc, step < 0 ? 2 : 0);
        sc->N_sorted = step < 0 ? 0 : sc->NA;  // a Gaussian's cells are written in key order
    }
    if (step > 0) {
        StepTime st = step_time(m, __longlong_as_double((long long)r), sc->t, sc->t_target, sc->coef_dth);
        if (!(st.dt > 0.0)) set_error(sc, ST_EDEGENERATE);  // no progress possible
        sc->step_dt = st.dt;
        sc->step_t_new = st.t_new;
        sc->step_last = st.last;
    }
    sc->ticket = 0;
}

// Link entries [N_prev, N) (neighbour references of Sec. 4.1), set their outward
// masks and rates; with step > 0 the last block also fixes dt (Eq. 8), else it ends the new grid.
// W lanes probe the hashtable together (warp-cooperative probing).
template <int N, int W, typename T>
__global__ void __launch_bounds__(THREADS, 4) k_link(const __grid_constant__ Model m, const __grid_constant__ Bufs b,
                                                     int step) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.error || (step > 0 && h.done)) return;
    const StepView v = view_of(m, &h);
    double r;
    if constexpr (W == 1) {
        // few: at most four rounds of all warps with one or a few entries each
        const long long few = 4ll * v.nb * (blockDim.x >> 5) * (32 / (2 * N));
        r = v.N - v.N_prev <= few ? link_few_body<N, T>(m, b, v.N_prev, v.N, v.g, v.nb, v.bi)
                                  : link_body<N, T>(m, b, v.N_prev, v.N, v.g, v.nb, v.bi);
    } else {
        r = link_body_tile<N, W, T>(m, b, v.N_prev, v.N, v.g, v.nb, v.bi);
    }
    // (the rate alone, by an atomic: as one of the sums and maxima that the last block
    // folds from every block's partials it took 5 us more, 31 of a step of 6.5e5 entries
    // that links a few thousand, now 26)
    join_rates(sc, r, h.maxrate_bits);
    if (last_block(sc) && threadIdx.x == 0) finish_link(m, sc, step);
}

// ------------------------------------------------------------------ initial Gaussian

struct InitBox {
    int lo[MAXN];
    long long dims[MAXN];
    long long total;
    double mean[MAXN];
    double icov[MAXN * MAXN];
    double pstar;
    float qlim;              // pass 1: q of the cell nearest the mean, from above; then: -2 ln pstar (inf: FP64 decides)
    float slack;             // centre_slack of the last dimension
    float icovc[MAXN * MAXN];  // icov in cells: icov[a][c] h_a h_c
    unsigned long long nonzero;  // bit a N + c: icov[a][c] != 0 (a comparison would take the FP64 pipe)
};

// Distance of the cells' centres from the mean, per dimension and index of the
// box, and in cells, formed once per block (five FP64 instructions per look otherwise).
constexpr int AXIS_MAX = 1024;  // entries; a box with longer axes forms them where they are used
struct AxisTable {
    double dx[AXIS_MAX];
    float cells[AXIS_MAX];
};
template <int N>
struct Axes {
    const AxisTable* tab;  // null: not tabulated
    int at[N];             // place of index lo_k of axis k, less lo_k
    static __device__ __forceinline__ double form(const Model& m, const InitBox& bx, int k, int i) {
        return __dsub_rn(centre64(m, k, i), bx.mean[k]);
    }
    // (out of line: in line, its FP64 instructions were executed and dropped)
    static __device__ __noinline__ float form_cells(const Model& m, const InitBox& bx, int k, int i) {
        return (float)__dmul_rn(form(m, bx, k, i), m.inv_h[k]);
    }
    __device__ __forceinline__ double dx(const Model& m, const InitBox& bx, int k, int i) const {
        return tab ? tab->dx[at[k] + i] : form(m, bx, k, i);
    }
    __device__ __forceinline__ float cells(const Model& m, const InitBox& bx, int k, int i) const {
        return tab ? tab->cells[at[k] + i] : form_cells(m, bx, k, i);
    }
};
// (all threads of the block)
template <int N>
__device__ __forceinline__ Axes<N> make_axes(const Model& m, const InitBox& bx, AxisTable& s_tab) {
    Axes<N> ax;
    long long n = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) n += bx.dims[k];
    ax.tab = n <= AXIS_MAX ? &s_tab : nullptr;
    int off = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        ax.at[k] = off - bx.lo[k];
        if (ax.tab) {
            for (int i = threadIdx.x; i < (int)bx.dims[k]; i += blockDim.x) {
                const double d = Axes<N>::form(m, bx, k, bx.lo[k] + i);
                s_tab.dx[off + i] = d;
                s_tab.cells[off + i] = (float)__dmul_rn(d, m.inv_h[k]);
            }
            off += (int)bx.dims[k];
        }
    }
    __syncthreads();
    return ax;
}

template <int N>
__device__ __forceinline__ void box_index(const InitBox& bx, long long lin, int* I) {
#pragma unroll
    for (int k = N - 1; k >= 0; --k) {
        I[k] = bx.lo[k] + (int)(lin % bx.dims[k]);
        lin /= bx.dims[k];
    }
}

// exp(-1/2 (x - mean)^T icov (x - mean)) at the centre of cell I. (A zero of icov
// adds a zero to the sum: left out, a diagonal covariance takes N terms.)
template <int N>
__device__ __noinline__ double gauss_at(const Model& m, const InitBox& bx, const Axes<N>& ax, const int* I) {
    double dx[N];
#pragma unroll
    for (int k = 0; k < N; ++k) dx[k] = ax.dx(m, bx, k, I[k]);
    double q = 0.0;
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int c = 0; c < N; ++c)
            if ((bx.nonzero >> (a * N + c)) & 1ull)
                q = __dadd_rn(q, __dmul_rn(__dmul_rn(dx[a], bx.icov[a * N + c]), dx[c]));
    return exp(__dmul_rn(-0.5, q));
}

// From three dimensions on, most of the box lies outside the ellipsoid of the
// initial set (97 % of it in six), and FP64 is scarce: the box is swept by rows
// along the last dimension, one thread per row, with the quadratic form q of each
// cell in single precision and a bound of its error (gbees_rows.cuh). Only a cell whose q lies
// within that bound of the limit is decided in FP64, so the set is the one that
// FP64 gives everywhere; the densities of the cells in the set are FP64. The
// paper's 6-D case (2.0e6 cells in the set, a box of 6.4e7): 0.11 + 0.13 + 0.6 ms
// for the three passes (81 ms with the FP64 density at every cell of the box in
// each of them); the whole call 87.5 -> 3.0 ms, Lorenz '96 6-D with h = 0.25
// 286 -> 8.0 ms.
// Longer rows than INIT_ROW_MAX (a chain of that many steps per thread) and
// fewer dimensions (the set fills most of the box) are swept cell by cell.
constexpr int INIT_ROW_MAX = 1024;
template <int N>
__device__ __forceinline__ bool by_rows(const InitBox& bx) {
    return N >= 3 && bx.dims[N - 1] <= INIT_ROW_MAX;
}
// Rows [c0, c1) of this block, as even as possible: a small box spreads over all blocks.
__device__ __forceinline__ void row_chunk(long long rows, long long& c0, long long& c1) {
    const long long per = (rows + gridDim.x - 1) / gridDim.x;
    c0 = min(rows, per * blockIdx.x);
    c1 = min(rows, c0 + per);
}

template <int N>
__device__ __forceinline__ void row_index(const InitBox& bx, long long row, int* I) {
    I[N - 1] = bx.lo[N - 1];
    if (bx.total <= 0x7fffffffll) {
        unsigned r = (unsigned)row;
#pragma unroll
        for (int k = N - 2; k >= 0; --k) {
            const unsigned d = (unsigned)bx.dims[k];
            I[k] = bx.lo[k] + (int)(r % d);
            r /= d;
        }
    } else {
#pragma unroll
        for (int k = N - 2; k >= 0; --k) {
            I[k] = bx.lo[k] + (int)(row % bx.dims[k]);
            row /= bx.dims[k];
        }
    }
}

template <int N>
__device__ __forceinline__ InitRow row_at(const Model& m, const InitBox& bx, const Axes<N>& ax, const int* I) {
    float dx[N];
#pragma unroll
    for (int k = 0; k < N; ++k) dx[k] = ax.cells(m, bx, k, I[k]);
    return row_form<N>(dx, bx.icovc, (float)bx.dims[N - 1], bx.slack);
}

// Whether cell i of the row at I is in the set p > pstar (qlim: -2 ln pstar).
template <int N>
__device__ __forceinline__ bool row_in(const Model& m, const InitBox& bx, const Axes<N>& ax, const InitRow& r, int* I,
                                       int i) {
    float e;
    const float d = row_gap(r, i, bx.qlim, e);
    if (d > e) return false;
    if (d < -e) return true;
    I[N - 1] = bx.lo[N - 1] + i;  // too near the limit (or not a number)
    return gauss_at<N>(m, bx, ax, I) > bx.pstar;
}

// Initial Gaussian (Sec. 5.1), pass 1: the largest density over the box of
// candidate cells, which fixes the threshold p* = thr_rel * max p. By rows: the
// cells whose q may be as small as that of the cell nearest the mean (bx.qlim).
template <int N>
__global__ void __launch_bounds__(THREADS) k_init_max(const __grid_constant__ Model m, Bufs b,
                                                        const __grid_constant__ InitBox bx) {
    __shared__ AxisTable s_tab;
    const Axes<N> ax = make_axes<N>(m, bx, s_tab);
    double mx = 0.0;
    const long long first = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (by_rows<N>(bx)) {
        const int len = (int)bx.dims[N - 1];
        const long long rows = bx.total / len;
        for (long long row = first; row < rows; row += stride) {
            int I[N];
            row_index<N>(bx, row, I);
            const InitRow r = row_at<N>(m, bx, ax, I);
            for (int i = 0; i < len; ++i) {
                float e;
                const float d = row_gap(r, i, bx.qlim, e);
                if (d > e) continue;
                I[N - 1] = bx.lo[N - 1] + i;
                mx = fmax(mx, gauss_at<N>(m, bx, ax, I));
            }
        }
    } else {
        for (long long lin = first; lin < bx.total; lin += stride) {
            int I[N];
            box_index<N>(bx, lin, I);
            mx = fmax(mx, gauss_at<N>(m, bx, ax, I));
        }
    }
    mx = block_max(mx);
    if (threadIdx.x == 0 && mx > 0.0) atomicMax(&b.sc->tmp_ord, ord_key(mx));
}

// Initial Gaussian, pass 2: per-block counts of the box cells above p*, the
// offsets of the write pass.
template <int N>
__global__ void __launch_bounds__(THREADS) k_init_count(const __grid_constant__ Model m, Bufs b,
                                                        const __grid_constant__ InitBox bx) {
    __shared__ AxisTable s_tab;
    const Axes<N> ax = make_axes<N>(m, bx, s_tab);
    long long c0, c1;
    long long cnt = 0;
    if (by_rows<N>(bx)) {
        const int len = (int)bx.dims[N - 1];
        row_chunk(bx.total / len, c0, c1);
        for (long long row = c0 + threadIdx.x; row < c1; row += blockDim.x) {
            int I[N];
            row_index<N>(bx, row, I);
            const InitRow r = row_at<N>(m, bx, ax, I);
            for (int i = 0; i < len; ++i) cnt += row_in<N>(m, bx, ax, r, I, i);
        }
    } else {
        block_chunk(bx.total, c0, c1);
        for (long long lin = c0 + threadIdx.x; lin < c1; lin += blockDim.x) {
            int I[N];
            box_index<N>(bx, lin, I);
            cnt += gauss_at<N>(m, bx, ax, I) > bx.pstar;
        }
    }
    for (int off = 16; off > 0; off >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, off);
    __shared__ long long s[WARPS];
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s[w];
        b.blk[blockIdx.x] = t;
    }
}

// Write the kept cells of the box in lexicographic order, insert them in the
// table, and reduce their sum and maximum (their velocities, masks and rates
// come with the links). By rows: a block takes a tile of one row per thread,
// and its threads then share the tile's kept cells.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS, 4) k_init_write(const __grid_constant__ Model m, Bufs b,
                                                        const __grid_constant__ InitBox bx) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.error) return;
    __shared__ AxisTable s_tab;
    const Axes<N> ax = make_axes<N>(m, bx, s_tab);
    long long c0, c1;
    long long base = b.blk[blockIdx.x];
    long long d[NDIG] = {0, 0, 0, 0, 0, 0};
    T mx = -INFINITY;
    int err = 0;
    auto write = [&](long long c, const int* I, double g) {
        unsigned long long k;
        if (c >= m.cap) {
            set_error(sc, ST_ECAPACITY);
        } else if (!interior<N>(m, I) || !pack_key<N>(m, I, k)) {
            set_error(sc, ST_EKEYRANGE);
        } else {
            T v = (T)g;
            b.key[0][c] = k;
            static_cast<T*>(b.q[0])[c] = v;
            b.om[0][c] = 0;
            table_insert_new(m, b, k, c, b.slot[0]);
            acc_add(d, v, err);
            mx = vmax(mx, v);
        }
    };
    if (by_rows<N>(bx)) {
        __shared__ int s_first[THREADS], s_end[THREADS], s_w[WARPS];
        const int len = (int)bx.dims[N - 1];
        row_chunk(bx.total / len, c0, c1);
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
        for (long long t0 = c0; t0 < c1; t0 += blockDim.x) {
            const long long row = t0 + threadIdx.x;
            int n_in = 0, i_first = 0, i_last = -1;
            if (row < c1) {
                int I[N];
                row_index<N>(bx, row, I);
                const InitRow r = row_at<N>(m, bx, ax, I);
                for (int i = 0; i < len; ++i)
                    if (row_in<N>(m, bx, ax, r, I, i)) {
                        if (n_in == 0) i_first = i;
                        i_last = i;
                        ++n_in;
                    }
            }
            // inclusive scan of the rows' counts
            int x = n_in;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, off);
                if (lane >= off) x += y;
            }
            if (lane == 31) s_w[wid] = x;
            __syncthreads();
            int before = 0, total = 0;
            for (int w = 0; w < nw; ++w) {
                if (w < wid) before += s_w[w];
                total += s_w[w];
            }
            s_end[threadIdx.x] = before + x;
            // a row with a gap (rounding at the limit) is walked again: negative first index
            s_first[threadIdx.x] = i_last - i_first + 1 == n_in ? i_first : -1;
            __syncthreads();
            for (int q0 = threadIdx.x & ~31; q0 < total; q0 += blockDim.x) {
                const int q = q0 + lane;
                const bool on = q < total;
                int I[N];
                if (on) {
                    int lo = 0, hi = (int)blockDim.x - 1;  // the first row that ends beyond q
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (s_end[mid] > q) hi = mid;
                        else lo = mid + 1;
                    }
                    row_index<N>(bx, t0 + lo, I);
                    int left = q - (lo > 0 ? s_end[lo - 1] : 0), i = s_first[lo] + left;
                    if (s_first[lo] < 0) {
                        const InitRow r = row_at<N>(m, bx, ax, I);
                        for (i = 0; i < len; ++i)
                            if (row_in<N>(m, bx, ax, r, I, i) && left-- == 0) break;
                    }
                    I[N - 1] = bx.lo[N - 1] + i;
                }
                __syncwarp();  // (the FP64 part with the warp in one piece)
                const double g = on ? gauss_at<N>(m, bx, ax, I) : 0.0;
                if (on) write(base + q, I, g);
                __syncwarp();
            }
            base += total;
            __syncthreads();
        }
    } else {
        block_chunk(bx.total, c0, c1);
        for (long long t0 = c0; t0 < c1; t0 += blockDim.x) {
            long long lin = t0 + threadIdx.x;
            int I[N];
            double g = 0.0;
            int f = 0;
            if (lin < c1) {
                box_index<N>(bx, lin, I);
                g = gauss_at<N>(m, bx, ax, I);
                f = g > bx.pstar;
            }
            int total;
            int pos = block_exclusive_scan(f, total);
            if (f) write(base + pos, I, g);
            base += total;
        }
    }
    if (err) set_error(sc, ST_EDEGENERATE);
    block_reduce_acc_max(d, (double)mx, sc->acc, &sc->maxq_ord);
}

// ------------------------------------------------------------------ explicit cells

// Load N cells given as int32 indices (staged in device memory) and doubles
// (their velocities, masks and rates come with the links).
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_init_cells(const Model m, Bufs b, const int* __restrict__ idx,
                                                        const double* __restrict__ p, long long count) {
    DevScalars* sc = b.sc;
    double mx = -INFINITY;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < count;
         c += (long long)gridDim.x * blockDim.x) {
        int I[N];
#pragma unroll
        for (int k = 0; k < N; ++k) I[k] = idx[c * N + k];
        unsigned long long k;
        if (!interior<N>(m, I) || !pack_key<N>(m, I, k)) {
            set_error(sc, ST_EKEYRANGE);
            continue;
        }
        T v = (T)p[c];
        b.key[0][c] = k;
        static_cast<T*>(b.q[0])[c] = v;
        b.om[0][c] = 0;
        table_insert_new(m, b, k, c, b.slot[0]);
        mx = fmax(mx, (double)v);
    }
    mx = block_max(mx);
    if (threadIdx.x == 0 && mx > -INFINITY) atomicMax(&sc->maxq_ord, ord_key(mx));
}

// ------------------------------------------------------------------ grow

// Halo cells around the cells that grow made active (inserted ones: [N_prev, N)
// at entry; activated ones: the n_act entries listed in map). With STEP == 0
// (initial grid) it runs whatever the done flag says. The last block appends
// the new halo cells to the count.
template <int N, typename T, int STEP>
__global__ void __launch_bounds__(THREADS) k_halo(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.error || (STEP && h.done)) return;
    const StepView v = view_of(m, &h);
    halo_body<N, T>(m, b, v, v.N_prev, v.N, h.n_act);
    if (last_block(sc)) {
        if (threadIdx.x == 0) {
            sc->N = min(sc->N + sc->n_halo, m.cap);
            sc->n_halo = 0;
            sc->n_act = 0;
            sc->n_glist = 0;
            sc->ticket = 0;
        }
    }
}

// ------------------------------------------------------------------ step completion

// Time, step count, buffers, prune schedule and normalisation after the flux
// update of a step, from the combined partials of the update's blocks.
// fp64: of the storage type.
__device__ __forceinline__ void finish_step(const Model& m, DevScalars* sc, const Combined& cs, int pb, bool fp64) {
    sc->dt = sc->step_dt;
    sc->t = sc->step_t_new;
    sc->step += 1;
    sc->steps_call += 1;
    sc->updates_call += sc->NA;
    sc->done = sc->step_last;
    sc->pbuf = pb ^ 1;
    const long long K = m.prune_interval, into = K > 0 ? sc->step % K : 0;
    sc->prune_now = K > 0 && into == 0;
    // A large pool much of which is out of order (appended by growth since the last sort;
    // the halo of a new grid) is sorted at once, by the prune's kernels with every cell
    // kept, when that pays over the steps until the next prune or the end of the call
    // (resort_pays): no result depends on the order. (Pools below RESORT_MIN_ENTRIES
    // lose: a sort of 6.5e5 entries takes 0.5 ms and gains 0.02 ms per step.)
    if (!sc->prune_now && !sc->done && m.sort_order != 2 && sc->N > RESORT_MIN_ENTRIES &&
        (sc->N - sc->N_sorted) * 4 > sc->N) {
        double left = (sc->t_target - sc->t) / sc->dt;
        if (K > 0) left = fmin(left, (double)(K - into));
        if (resort_pays(sc->N, sc->N - sc->N_sorted, left, fp64)) sc->prune_now = RESORT;
    }
    sc->N_prev = sc->N;
    const double w = m.prod_h * acc_to_double(cs.acc);
    sc->w = w;
    if (!(w > 0.0) || !isfinite(w)) {
        set_error(sc, ST_EDEGENERATE);
        sc->scale = 0.0;
    } else {
        sc->scale = 1.0 / w;
    }
    sc->maxq = cs.maxq_ord ? ord_val(cs.maxq_ord) : 0.0;
    sc->ticket = 0;
}

// The grow of a large grid in two kernels: a sweep that lists the cells that grow,
// then every (listed cell, candidate) pair over the grid.
template <typename T>
__global__ void __launch_bounds__(THREADS) k_grow_mark(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.done | h.error) return;
    const StepView v = view_of(m, &h);
    const Above<T> above(m.thr_rel * v.maxq);
    for (WarpRuns wr(v.N_prev, v.nb, v.bi); wr.next();)
        if (wr.c < v.N_prev) grow_list_mark<T>(b, v, above, wr.c);
}

template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_grow_list(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.done | h.error) return;
    const StepView v = view_of(m, &h);
    join_rates(sc, grow_list_body<N, T>(m, b, v, h.n_glist), h.maxrate_bits);
}

// Update, pass 1 (after the links, with dt): jumps and transverse terms.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS, sizeof(T) == 8 ? 2 : 3) k_waves(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.done | h.error) return;
    waves_body<N, T>(m, b, view_of(m, &h));
}

// Update, pass 2 (FP64): the flux through every face that touches an active cell.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS, 3) k_faces(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.done | h.error) return;
    faces_body<N, T>(m, b, view_of(m, &h));
}

// The end of an update: exact per-block partial sums and maximum for the next
// normalisation; the last block ends the step.
template <typename T>
__device__ __forceinline__ void end_update(const Model& m, const Bufs& b, const StepView& v, long long (&d)[NDIG],
                                           double mx, int err) {
    if (err) set_error(b.sc, ST_EDEGENERATE);
    block_partial(b.part, d, mx, 0.0);
    if (last_block(b.sc)) {
        Combined cs = combine_partials(b.part, gridDim.x);
        if (threadIdx.x == 0) finish_step(m, b.sc, cs, v.pb, sizeof(T) == 8);
    }
}

// Update, pass 3 (FP64): the conservative update of every active cell from the
// fluxes of its 2n faces, divided by the last normaliser.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_apply(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.done | h.error) return;
    const StepView v = view_of(m, &h);
    long long d[NDIG] = {0, 0, 0, 0, 0, 0};
    double mx = -INFINITY;
    int err = 0;
    apply_body<N, T>(m, b, v, d, mx, err);
    end_update<T>(m, b, v, d, mx, err);
}

// Update, passes 2 and 3 in one (FP32).
template <int N, typename T>
__global__ void __launch_bounds__(THREADS, 2) k_update(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.done | h.error) return;
    const StepView v = view_of(m, &h);
    long long d[NDIG] = {0, 0, 0, 0, 0, 0};
    double mx = -INFINITY;
    int err = 0;
    update_body<N, T>(m, b, v, d, mx, err);
    end_update<T>(m, b, v, d, mx, err);
}

// ------------------------------------------------------------------ measurement update

struct Meas {
    int m;
    int H[MAXN];
    double y[MAXN];
    double Rinv[MAXN * MAXN];
    unsigned long long nonzero;  // bit a m + e: Rinv[a][e] != 0
};

// p <- exp(-1/2 (y - x_H)^T R^-1 (y - x_H)) p at the cell centres (Eq. 4); the
// maximum is reduced for the prune that follows.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_correct(const __grid_constant__ Model m, Bufs b,
                                                     const __grid_constant__ Meas ms) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (h.error) return;
    const long long ncell = min(h.N, m.cap);
    const int g = h.gen, pb = h.pbuf;
    T* Q = static_cast<T*>(b.q[pb]);
    const unsigned long long* key = b.key[g];
    T tmax = -INFINITY;
    for (WarpRuns wr(ncell); wr.next();) {
        const long long c = wr.c;
        if (c >= ncell) continue;
        const T q = Q[c];
        // a density of 0 (a halo cell's) stays 0: FP64 bounds this pass
        if (!nonzero(q)) {
            tmax = vmax(tmax, q);
            continue;
        }
        int I[N];
        unpack_key<N>(m, key[c], I);
        double r[MAXN];
        for (int a = 0; a < ms.m; ++a) r[a] = __dsub_rn(ms.y[a], centre64(m, ms.H[a], I[ms.H[a]]));
        double qf = 0.0;
        for (int a = 0; a < ms.m; ++a)
            for (int e = 0; e < ms.m; ++e)
                if ((ms.nonzero >> (a * ms.m + e)) & 1ull)  // (a zero adds a zero)
                    qf = __dadd_rn(qf, __dmul_rn(__dmul_rn(r[a], ms.Rinv[a * ms.m + e]), r[e]));
        const double L = exp(__dmul_rn(-0.5, qf));
        const T v = (T)__dmul_rn(L, (double)q);
        Q[c] = v;
        tmax = vmax(tmax, v);
    }
    const double mx = (double)tmax;
    long long zero[NDIG] = {0, 0, 0, 0, 0, 0};
    block_partial(b.part, zero, mx, 0.0);
    if (last_block(sc)) {
        Combined c = combine_partials(b.part, gridDim.x);
        if (threadIdx.x == 0) {
            sc->maxq = c.maxq_ord ? ord_val(c.maxq_ord) : 0.0;
            sc->ticket = 0;
            sc->prune_now = 1;
        }
    }
}

// ------------------------------------------------------------------ prune

__device__ __forceinline__ bool prune_due(const StepHead& h) { return h.prune_now && !h.error; }

// The prune kernels run to re-sort a grown pool, keeping every cell (finish_step).
__device__ __forceinline__ bool resort_due(const StepHead& h) { return h.prune_now == RESORT; }

// Prune (Algorithm 3), pass 1: mark the significant cells S.
template <typename T>
__global__ void __launch_bounds__(THREADS) k_prune_mark(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    if (!prune_due(h)) return;
    if (blockIdx.x == 0 && threadIdx.x < MAXN) {  // read and added to from the status pass on
        b.sc->sort_lo[threadIdx.x] = ~0u;
        b.sc->sort_hi[threadIdx.x] = 0u;
    }
    prune_mark_body<T>(m, b, view_of(m, &h), resort_due(h));
}

// Prune, pass 2: mark the downwind set D(S) of every significant cell (the
// directional rule of Sec. 3.3).
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_prune_scatter(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    if (!prune_due(h) || resort_due(h)) return;
    prune_scatter_body<N, T>(m, b, view_of(m, &h));
}

// Prune, pass 3: the status of every entry (active, halo or dropped) and the
// per-block counts of the survivors.
template <int N, bool SORTED>
__global__ void __launch_bounds__(THREADS) k_prune_count(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    if (!prune_due(h)) return;
    prune_count_body<N, SORTED>(m, b, view_of(m, &h));
}

// Prune, pass 4 without a sort: write the survivors into the other buffer set
// in storage order, active cells first, then the halo (stream compaction), with
// exact partial sums, maximum and CFL rates for the step scalars.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_prune_compact(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (!prune_due(h)) return;
    const StepView v = view_of(m, &h);
    const Survivors sv = block_offsets(b, v.nb, v.bi);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->N_new = sv.total_a + sv.total_g;
        sc->NA_new = sv.total_a;
    }
    long long d[NDIG] = {0, 0, 0, 0, 0, 0};
    double mx = -INFINITY, rmax = 0.0;
    int err = 0;
    prune_compact_body<N, T>(m, b, v, sv, d, mx, rmax, err, resort_due(h));
    if (err) set_error(sc, ST_EDEGENERATE);
    block_partial(b.part, d, mx, rmax);
}

// The end of a prune: swap the buffer sets, new count, normalisation scalars
// and CFL maximum of the survivors.
__device__ __forceinline__ void finish_prune(const Model& m, DevScalars* sc, const Combined& cp, long long n_new) {
    sc->N = n_new;
    sc->N_prev = n_new;
    sc->NA = sc->NA_new;
    sc->N_sorted = n_new;
    sc->gen ^= 1;
    sc->pbuf ^= 1;
    sc->maxrate_bits = cp.rate_bits;
    sc->prune_now = 0;
    const double w = m.prod_h * acc_to_double(cp.acc);
    sc->w = w;
    if (!(w > 0.0) || !isfinite(w)) {
        set_error(sc, ST_EDEGENERATE);
        sc->scale = 0.0;
    } else {
        sc->scale = 1.0 / w;
    }
    sc->maxq = cp.maxq_ord ? ord_val(cp.maxq_ord) : 0.0;
    sc->ticket = 0;
}

// Prune, pass 5: rehash the survivors and rebuild their links (Sec. 4.4.2);
// the last block swaps the buffer sets and sets the step scalars.
template <int N>
__global__ void __launch_bounds__(THREADS) k_prune_relink(const Model m, Bufs b, int nblk_compact) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (!prune_due(h)) return;
    prune_relink_body<N>(m, b, view_of(m, &h));
    if (last_block(sc)) {
        Combined cp = combine_partials(b.part, nblk_compact);
        if (threadIdx.x == 0) finish_prune(m, sc, cp, h.N_new);
    }
}

// Prune, passes 4 and 5 after a sort, in one: the survivors move into the other
// buffer set in the order of the sort, with their links and hashtable entries; the
// same partials, and the last block ends the prune.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_prune_move(const Model m, Bufs b) {
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    if (!prune_due(h)) return;
    const StepView v = view_of(m, &h);
    const Survivors sv = block_offsets(b, v.nb, v.bi);
    long long d[NDIG] = {0, 0, 0, 0, 0, 0};
    double mx = -INFINITY, rmax = 0.0;
    int err = 0;
    prune_move_body<N, T>(m, b, v, sv.total_a + sv.total_g, d, mx, rmax, err, resort_due(h));
    if (err) set_error(sc, ST_EDEGENERATE);
    block_partial(b.part, d, mx, rmax);
    if (last_block(sc)) {
        Combined cp = combine_partials(b.part, gridDim.x);
        if (threadIdx.x == 0) {
            sc->NA_new = sv.total_a;
            finish_prune(m, sc, cp, sv.total_a + sv.total_g);
        }
    }
}

// ------------------------------------------------------------------ read-out

// Read-out of the active cells in storage order: per-block counts
// (k_readout_count), an exclusive scan of them (k_scan_blocks), then every
// block writes its active cells at its offset.
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_readout(const Model m, Bufs b, int* __restrict__ idx,
                                                     double* __restrict__ p) {
    const StepHead& h = block_head(b.sc);
    const long long ncell = min(h.N, m.cap);
    const int g = h.gen, pb = h.pbuf;
    const T* Q = static_cast<const T*>(b.q[pb]);
    const unsigned short* om = b.om[g];
    const double w = h.w;
    long long c0, c1;
    block_chunk(ncell, c0, c1);
    long long base = b.blk[blockIdx.x];
    for (long long t0 = c0; t0 < c1; t0 += blockDim.x) {
        const long long c = t0 + threadIdx.x;
        const int f = c < c1 && !is_halo(om, c);
        int total;
        const int pos = block_exclusive_scan(f, total);
        if (f) {
            const long long r = base + pos;
            int I[N];
            unpack_key<N>(m, b.key[g][c], I);
#pragma unroll
            for (int k = 0; k < N; ++k) idx[r * N + k] = I[k];
            p[r] = __ddiv_rn((double)Q[c], w);
        }
        base += total;
    }
}

// Moments: PASS 0 sums x_a p (a < n) into mom_mean[a]; PASS 1 sums
// (x_a - mean_a)(x_b - mean_b) p (a <= b) into mom_out[pair], times prod h; exact
// sums, by the last block from the digits in mom, which it leaves at zero. Six
// sums per block row (blockIdx.y) in registers: the digits' atomics of all sums to
// shared memory bounded this pass (2.3e6 cells in six dimensions: 0.42 + 1.18 ms,
// now 0.35 ms for both; the cells of density 0 add nothing and are left out).
constexpr int MOM_SUMS = 6;
template <int N, int PASS>
constexpr int mom_slots() { return PASS == 0 ? N : N * (N + 1) / 2; }

template <int N, typename T, int PASS>
__global__ void __launch_bounds__(THREADS) k_moments(const Model m, Bufs b) {
    constexpr int SLOTS = mom_slots<N, PASS>(), ROWS = (SLOTS + MOM_SUMS - 1) / MOM_SUMS;
    constexpr int K = SLOTS < MOM_SUMS ? SLOTS : MOM_SUMS;
    DevScalars* sc = b.sc;
    const StepHead& h = block_head(sc);
    const long long ncell = min(h.N, m.cap);
    const int g = h.gen, pb = h.pbuf;
    const T* Q = static_cast<const T*>(b.q[pb]);
    const double w = h.w;
    const int row = ROWS > 1 ? blockIdx.y : 0;
    double mean[N];
#pragma unroll
    for (int k = 0; k < N; ++k) mean[k] = PASS ? *(volatile double*)&sc->mom_mean[k] : 0.0;
    long long d[K][NDIG];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int q = 0; q < NDIG; ++q) d[k][q] = 0;
    int err = 0;
    for (WarpRuns r(ncell); r.next();) {
        const T q = r.c < ncell ? Q[r.c] : (T)0;
        if (!nonzero(q)) continue;
        int I[N];
        unpack_key<N>(m, b.key[g][r.c], I);
        const double p = __ddiv_rn((double)q, w);
        double x[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            x[k] = centre64(m, k, I[k]);
            if (PASS) x[k] = __dsub_rn(x[k], mean[k]);
        }
        int slot = 0;
#pragma unroll
        for (int a = 0; a < N; ++a)
#pragma unroll
            for (int e = PASS ? a : 0; e < (PASS ? N : 1); ++e, ++slot) {
                if (ROWS > 1 && slot / MOM_SUMS != row) continue;
                const double v = PASS ? __dmul_rn(__dmul_rn(x[a], x[e]), p) : __dmul_rn(x[a], p);
                acc_add(d[slot % MOM_SUMS], v, err);
            }
    }
    if (err) set_error(sc, ST_EDEGENERATE);
    __shared__ long long s_acc[WARPS][K][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const long long t = warp_sum_digits(d[k]);
        if ((lane & 3) == 0) s_acc[wid][k][lane >> 2] = t;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < K * NDIG; i += blockDim.x) {
        const int k = i / NDIG, q = i - k * NDIG, slot = row * MOM_SUMS + k;
        long long t = 0;
        for (int x = 0; x < (int)(blockDim.x >> 5); ++x) t += s_acc[x][k][q];
        if (t && slot < SLOTS) atomicAdd((unsigned long long*)&sc->mom[slot][q], (unsigned long long)t);
    }
    if (!last_block(sc)) return;
    for (int s = threadIdx.x; s < SLOTS; s += blockDim.x) {
        long long D[NDIG];
        for (int q = 0; q < NDIG; ++q) {
            D[q] = __ldcg(&sc->mom[s][q]);
            sc->mom[s][q] = 0;
        }
        (PASS ? sc->mom_out : sc->mom_mean)[s] = __dmul_rn(m.prod_h, acc_to_double(D));
    }
    if (threadIdx.x == 0) sc->ticket = 0;
}

}  // namespace gbees
