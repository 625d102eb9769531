// Untemplated helper kernels of the host-side call sequences (begin, reset,
// finalisation, graph-loop control, scans, counts, moments). Included by one
// translation unit only.
#pragma once

#include "gbees_kernels.cuh"

namespace gbees {

// Start a propagate call: record the target and whether any step is due.
__global__ void k_begin(DevScalars* sc, double t_target) {
    sc->t_target = t_target;
    sc->done = !(sc->t < t_target) || sc->error != 0;
    sc->steps_call = 0;
    sc->updates_call = 0;
    sc->bar_seq = 0;
}

// Start a batched propagate call: k_begin for every grid of the batch.
__global__ void k_batch_begin(const BatchItem* items, int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        DevScalars* sc = items[i].b.sc;
        const double tt = items[i].t_end;
        sc->t_target = tt;
        sc->done = !(sc->t < tt) || sc->error != 0;
        sc->steps_call = 0;
        sc->updates_call = 0;
        sc->bar_seq = 0;
    }
}

// A further launch of the same batch: the teams' barriers count from zero.
__global__ void k_batch_again(const BatchItem* items, int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x)
        items[i].b.sc->bar_seq = 0;
}

// Copy the scalars of every grid of a batch into one array (one read-back).
__global__ void k_batch_collect(const BatchItem* items, int count, DevScalars* out) {
    constexpr int W = sizeof(DevScalars) / 8;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < (long long)count * W;
         k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k / W), q = (int)(k % W);
        reinterpret_cast<long long*>(out + i)[q] = __ldcg(reinterpret_cast<const long long*>(items[i].b.sc) + q);
    }
}

// Control of the device-side step loop of a graph launch (a WHILE node whose
// body is one step and an IF node around the prune): after the flux update of
// a step, decide whether the prune runs and whether another step follows.
// The loop ends when the target time is reached, on any error, or after
// max_iter iterations of this launch (the host then launches again).
__global__ void k_loop_reset(DevScalars* sc) {
    sc->loop_iter = 0;
    sc->graph_kernels += 1;
}

// step_kernels: kernels of one step up to and including this one; a prune adds
// prune_kernels.
__global__ void k_loop_ctl(DevScalars* sc, cudaGraphConditionalHandle h_while, cudaGraphConditionalHandle h_prune,
                           long long max_iter, int step_kernels, int prune_kernels) {
    const long long it = ++sc->loop_iter;
    const int err = sc->error;
    const bool prune = sc->prune_now && !err;
    sc->graph_kernels += step_kernels + (prune ? prune_kernels : 0);
    cudaGraphSetConditional(h_prune, prune ? 1u : 0u);
    cudaGraphSetConditional(h_while, (!sc->done && !err && it < max_iter) ? 1u : 0u);
}

// Exclusive scan of blk[0..nblk) by one block; the total goes to sc->N_new, and
// with count also becomes the pool of a new grid (its active cells; the halo
// kernel adds their halo).
__global__ void k_scan_blocks(Bufs b, int nblk, long long cap, int count) {
    __shared__ long long s_part[THREADS];
    const int per = (nblk + THREADS - 1) / THREADS;
    const int i0 = threadIdx.x * per;
    long long sum = 0;
    for (int i = i0; i < i0 + per && i < nblk; ++i) sum += b.blk[i];
    s_part[threadIdx.x] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long run = 0;
        for (int t = 0; t < THREADS; ++t) {
            long long v = s_part[t];
            s_part[t] = run;
            run += v;
        }
        b.sc->N_new = run;
        if (count) {
            b.sc->N = run;
            b.sc->NA = run;
            b.sc->N_prev = 0;
            b.sc->n_act = 0;
        }
        if (run > cap) set_error(b.sc, ST_ECAPACITY);
    }
    __syncthreads();
    long long run = s_part[threadIdx.x];
    for (int i = i0; i < i0 + per && i < nblk; ++i) {
        long long v = b.blk[i];
        b.blk[i] = run;
        run += v;
    }
}

// Reset the grid scalars.
__device__ __forceinline__ void reset_scalars(DevScalars* sc, double t0) {
    sc->N = 0;
    sc->N_prev = 0;
    sc->N_new = 0;
    sc->NA = 0;
    sc->NA_new = 0;
    sc->n_halo = 0;
    sc->n_act = 0;
    sc->n_glist = 0;
    sc->N_sorted = 0;
    sc->t = t0;
    sc->t_target = t0;
    sc->dt = 0.0;
    sc->maxrate_bits = 0;
    sc->maxq_ord = 0;
    sc->maxq = 0.0;
    sc->w = 1.0;
    sc->scale = 1.0;
    for (int q = 0; q < NDIG; ++q) sc->acc[q] = 0;
    sc->step = 0;
    sc->steps_call = 0;
    sc->updates_call = 0;
    sc->lookups_fallback = 0;
    sc->pbuf = 0;
    sc->gen = 0;
    sc->done = 1;
    sc->error = 0;
    sc->prune_now = 0;
    sc->ticket = 0;
    sc->tmp_ord = 0;
    sc->loop_iter = 0;
    sc->graph_kernels = 0;
    sc->bar_seq = 0;
    for (int e = 0; e < 2; ++e) {
        sc->loop_rate[e] = 0;
        sc->loop_maxq[e] = 0;
        for (int q = 0; q < NDIG; ++q) sc->loop_acc[e][q] = 0;
    }
    for (int q = 0; q < 8; ++q) sc->phase_cycles[q] = 0;
    for (int k = 0; k < 28; ++k)
        for (int q = 0; q < NDIG; ++q) sc->mom[k][q] = 0;
    sc->phase_steps = 0;
}

// A new context's scalars.
__global__ void k_reset(DevScalars* sc, double t0) { reset_scalars(sc, t0); }

// A new grid: scalars reset (count > 0: loaded from that many cells, after step0
// steps), every hashtable slot emptied.
__global__ void __launch_bounds__(THREADS) k_new_grid(const Model m, Bufs b, double t0, long long count,
                                                      long long step0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        reset_scalars(b.sc, t0);
        b.sc->N = count;
        b.sc->NA = count;
        b.sc->step = step0;
    }
    const unsigned long long T = m.tmask + 1;
    for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s < T;
         s += (unsigned long long)gridDim.x * blockDim.x) {
        reinterpret_cast<ulonglong2*>(b.table)[s] = make_ulonglong2(EMPTY_KEY, ~0ull);
    }
}

// ------------------------------------------------------------------ sorting
// The prune of a large grid gives the survivors a new storage order with a
// stable LSD radix sort of (order code, old index), 8 bits per pass: the
// lexicographic order of the cell indices (the packed key, dimension 0 most
// significant), so that the face neighbours of a warp's consecutive cells
// in any dimension are consecutive too and the neighbour gathers coalesce, or
// the Morton order of the indices. Scratch: the other generation's key/slot
// arrays (A) and its link/value arrays (B), free until the compaction writes
// them.
// A key's fields are mostly empty (10 bits of index per dimension in six
// dimensions, of which a grid uses 5 or 6): the code holds each field less its
// smallest value, in as many bits as the range needs, which sorts alike. 36 bits in
// place of 60 and five passes in place of eight on the 6-D grids; a pass beyond
// the code's digits returns at once.

constexpr int SORT_BLOCKS = 1024;  // blocks of the sort kernels at most (histogram rows)
constexpr int SORT_PASSES = 8;     // digits of a full code
constexpr int SORT_ITEMS = 4;      // elements per thread of a tile
constexpr int SORT_TILE = THREADS * SORT_ITEMS;

struct SortBufs {
    unsigned long long* key[2];
    unsigned int* val[2];
};

__device__ __forceinline__ SortBufs sort_bufs(const Bufs& b, int g, int pb) {
    SortBufs s;
    s.key[0] = b.key[g ^ 1];
    s.key[1] = reinterpret_cast<unsigned long long*>(b.link[g ^ 1]);
    s.val[0] = b.slot[g ^ 1];
    s.val[1] = static_cast<unsigned int*>(b.q[pb ^ 1]);
    return s;
}

// The compact code of a key: bits per field from the ranges in the scalars.
struct KeyCode {
    unsigned lo[MAXN];
    int bits[MAXN], total;
    __device__ __forceinline__ KeyCode(const Model& m, const DevScalars* sc) {
        total = 0;
        for (int j = 0; j < m.n; ++j) {
            lo[j] = sc->sort_lo[j];
            const unsigned hi = sc->sort_hi[j];
            bits[j] = hi > lo[j] ? 32 - __clz(hi - lo[j]) : 0;
            total += bits[j];
        }
    }
    __device__ __forceinline__ unsigned long long operator()(const Model& m, unsigned long long k) const {
        const unsigned long long mask = (1ull << m.key_bits) - 1;
        unsigned long long out = 0;
        for (int j = 0; j < m.n; ++j)
            out = (out << bits[j]) | (unsigned)(((k >> (m.key_bits * (m.n - 1 - j))) & mask) - lo[j]);
        return out;
    }
};

// keep[c] = status (0 drop, 1 active, 2 halo, from the status pass in map);
// A = (order code, c): active cells first, then the halo (each in the order of
// the configured code), or both interleaved in key order; dropped entries
// last (every result is independent of the storage order; only the speed
// depends on it). A survivor's full code is below 2^63: keys use at most 63 bits,
// and only an all-ones key has an all-ones Morton code, a key no cell that
// survives a prune has.
__global__ void __launch_bounds__(THREADS) k_sort_init(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    if (!prune_due(h)) return;
    const StepView v = view_of(m, &h);
    const SortBufs sb = sort_bufs(b, v.g, v.pb);
    const unsigned long long* key = b.key[v.g];
    long long c0, c1;
    block_chunk(v.N, c0, c1);
    const int order = m.sort_order;        // GBEES_ORDER_*
    const bool mixed = order == 3;          // halo cells among the active ones
    const KeyCode code(m, b.sc);
    const bool compact = (order == 0 || mixed) && code.total <= 62;
    const int region_bit = compact ? code.total : 63;
    if (blockIdx.x == 0 && threadIdx.x == 0) b.sc->sort_passes = compact ? (code.total + 2 + 7) / 8 : SORT_PASSES;
    for (long long c = c0 + threadIdx.x; c < c1; c += blockDim.x) {
        const int st = b.map[c];
        b.keep[c] = (unsigned char)st;
        const unsigned long long k = key[c];
        const unsigned long long x = compact      ? code(m, k)
                                     : order == 1 ? morton_code(k, m.n, m.key_bits)
                                     : order == 4 ? row_morton_code(k, m.n, m.key_bits)
                                                  : k;
        const unsigned long long region = (st == 2 && !mixed) ? (1ull << region_bit) : 0ull;
        const unsigned long long drop = compact ? 3ull << region_bit : ~0ull;
        sb.key[0][c] = st == 0 ? drop : (region | x);
        sb.val[0][c] = (unsigned int)c;
    }
}

// The entries of a sort: count of them, or (count < 0) the pool of a due prune.
// False: nothing to do in this pass.
__device__ __forceinline__ bool sort_pass(const Model& m, const Bufs& b, int pass, long long count, long long& n,
                                          SortBufs& sb) {
    const StepHead& h = block_head(b.sc);
    if (count < 0) {
        if (!prune_due(h) || pass >= h.sort_passes) return false;
        count = min(h.N, m.cap);
    }
    n = count;
    sb = sort_bufs(b, h.gen, h.pbuf);
    return true;
}

// Pass histogram: sorthist[d * nblk + block] = entries of this block's chunk
// whose digit is d. (One shared atomic per digit that occurs in a warp: the high
// digits of neighbouring entries are mostly alike.)
__global__ void __launch_bounds__(THREADS) k_sort_hist(const Model m, Bufs b, int pass, long long count) {
    long long n;
    SortBufs sb;
    if (!sort_pass(m, b, pass, count, n, sb)) return;
    __shared__ unsigned int cnt[256];
    const unsigned long long* in = sb.key[pass & 1];
    for (int d = threadIdx.x; d < 256; d += blockDim.x) cnt[d] = 0;
    __syncthreads();
    long long c0, c1;
    block_chunk(n, c0, c1);
    const int lane = threadIdx.x & 31, shift = 8 * pass;
    for (long long t0 = c0 + threadIdx.x; t0 - threadIdx.x < c1; t0 += SORT_TILE) {
        int d[SORT_ITEMS];
#pragma unroll
        for (int i = 0; i < SORT_ITEMS; ++i) {
            const long long c = t0 + i * THREADS;
            d[i] = c < c1 ? (int)((in[c] >> shift) & 255u) : 256;
        }
#pragma unroll
        for (int i = 0; i < SORT_ITEMS; ++i) {
            const unsigned same = __match_any_sync(0xffffffffu, d[i]);
            if (d[i] < 256 && (same & ((1u << lane) - 1u)) == 0) atomicAdd(&cnt[d[i]], (unsigned)__popc(same));
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += blockDim.x) b.sorthist[(long long)d * gridDim.x + blockIdx.x] = cnt[d];
}

// Exclusive prefixes of the histogram, block d along digit d's row of nblk (at
// most 4 THREADS) counters, in place; the row's total goes to the reductions'
// partials (free during a sort). The digits' offsets follow from the totals in the
// scatter. (256 blocks: 3 us; one block over all rows took 427 us, eight times
// the rest of the pass.)
__global__ void __launch_bounds__(THREADS) k_sort_scan(const Model m, Bufs b, int nblk, int pass,
                                                       long long count) {
    long long n;
    SortBufs sb;
    if (!sort_pass(m, b, pass, count, n, sb)) return;
    static_assert(SORT_BLOCKS <= 4 * THREADS, "a row has at most four counters per thread");
    __shared__ unsigned int s_w[WARPS];
    unsigned int* row = b.sorthist + (long long)blockIdx.x * nblk;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned v[4], sum = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = (int)threadIdx.x * 4 + k;
        v[k] = i < nblk ? row[i] : 0u;
        sum += v[k];
    }
    unsigned x = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
    }
    if (lane == 31) s_w[wid] = x;
    __syncthreads();
    unsigned before = x - sum, total = 0;
    for (int w = 0; w < WARPS; ++w) {
        if (w < wid) before += s_w[w];
        total += s_w[w];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = (int)threadIdx.x * 4 + k;
        if (i < nblk) row[i] = before;
        before += v[k];
    }
    if (threadIdx.x == 0) reinterpret_cast<unsigned int*>(b.part)[blockIdx.x] = total;
}

// Stable scatter of a pass: every block walks its chunk in tiles of SORT_ITEMS
// elements per thread (each warp a row of consecutive ones); an element's place is its
// digit's offset for the block, plus the elements of that digit in earlier tiles, in
// earlier warps of the tile, and before it in its warp's row. Bound by the chain of a
// tile (load, count, block barriers): one element per thread and tile, and sixteen tiles
// to a block, took 44 us at 6.5e5 entries, now 22 (k_sort_hist 22, now 13), and 0.14 ms
// at 4.9e6, now 0.10.
__global__ void __launch_bounds__(THREADS) k_sort_scatter(const Model m, Bufs b, int pass, long long count) {
    long long n;
    SortBufs sb;
    if (!sort_pass(m, b, pass, count, n, sb)) return;
    static_assert(THREADS == 256, "one thread per digit");
    __shared__ unsigned int wcnt[WARPS][256];
    __shared__ unsigned int s_w[WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, src = pass & 1, shift = 8 * pass;
    unsigned int base;  // place of the next element with digit threadIdx.x
    {
        // the digits' offsets: exclusive prefix of the rows' totals
        const unsigned tot = reinterpret_cast<const unsigned int*>(b.part)[threadIdx.x];
        unsigned x = tot;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        if (lane == 31) s_w[wid] = x;
        __syncthreads();
        unsigned before = x - tot;
        for (int w = 0; w < wid; ++w) before += s_w[w];
        base = before + b.sorthist[(long long)threadIdx.x * gridDim.x + blockIdx.x];
    }
    long long c0, c1;
    block_chunk(n, c0, c1);
    for (long long t0 = c0; t0 < c1; t0 += SORT_TILE) {
        unsigned long long k[SORT_ITEMS];
        unsigned int val[SORT_ITEMS], rank[SORT_ITEMS];
        int d[SORT_ITEMS];
#pragma unroll
        for (int i = 0; i < SORT_ITEMS; ++i) {
            const long long c = t0 + wid * (32 * SORT_ITEMS) + i * 32 + lane;
            k[i] = c < c1 ? sb.key[src][c] : 0;
            val[i] = c < c1 ? sb.val[src][c] : 0;
            d[i] = c < c1 ? (int)((k[i] >> shift) & 255u) : 256;  // 256: past the end
        }
        for (int i = lane; i < 256; i += 32) wcnt[wid][i] = 0;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < SORT_ITEMS; ++i) {
            const unsigned same = __match_any_sync(0xffffffffu, d[i]);
            const int in_row = __popc(same & ((1u << lane) - 1u));
            const unsigned before = d[i] < 256 ? wcnt[wid][d[i]] : 0u;
            rank[i] = before + in_row;
            __syncwarp();
            if (d[i] < 256 && in_row == 0) wcnt[wid][d[i]] = before + __popc(same);
            __syncwarp();
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {  // counts -> places, digit threadIdx.x
            const unsigned c = wcnt[w][threadIdx.x];
            wcnt[w][threadIdx.x] = base;
            base += c;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SORT_ITEMS; ++i) {
            if (d[i] == 256) continue;
            const unsigned int off = wcnt[wid][d[i]] + rank[i];
            sb.key[src ^ 1][off] = k[i];
            sb.val[src ^ 1][off] = val[i];
        }
        __syncwarp();  // (a warp clears its own row only)
    }
}

// New index of every survivor: its rank in the sorted order (survivors sort
// before the dropped entries), -1 for the dropped; and the survivors in that order.
__global__ void __launch_bounds__(THREADS) k_sort_map(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    if (!prune_due(h)) return;
    const StepView v = view_of(m, &h);
    const SortBufs sb = sort_bufs(b, v.g, v.pb);
    const unsigned int* val = sb.val[h.sort_passes & 1];
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < v.N; r += (long long)gridDim.x * blockDim.x) {
        const unsigned int c = val[r];
        const bool kept = b.keep[c] != 0;
        b.map[c] = kept ? (int)r : -1;
        if (kept) sorted_order(b)[r] = (int)c;
    }
}

// Per-block counts of the active cells (read-out, first pass).
__global__ void __launch_bounds__(THREADS) k_readout_count(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    const long long ncell = min(h.N, m.cap);
    const unsigned short* om = b.om[h.gen];
    long long c0, c1;
    block_chunk(ncell, c0, c1);
    int cnt = 0;
    for (long long c = c0 + threadIdx.x; c < c1; c += blockDim.x) cnt += !is_halo(om, c);
    const long long t = block_count(cnt);
    if (threadIdx.x == 0) b.blk[blockIdx.x] = t;
}

// ------------------------------------------------------------------ sorted read-out
// The active cells in lexicographic order of their indices, on the device: a sort
// on the host of the cells of one grid took longer than all the rest of a small
// grid's read-out (5 * 10^3 cells: 0.5 ms, 5.5 * 10^4: 1.5 ms).

// A pool of up to RANK_MAX entries: each active cell's place is the number of
// active cells with smaller keys, counted by RANK_LANES lanes per cell against all
// keys, staged through shared memory (no passes and no other launch; 27 us at
// 1.6 * 10^4 entries, where the sort's launches take about 60).
constexpr long long RANK_MAX = 1ll << 14;
constexpr int RANK_LANES = 8;
template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_readout_rank(const Model m, Bufs b, int* __restrict__ idx,
                                                          double* __restrict__ p) {
    constexpr int TILE = 1024;
    __shared__ unsigned long long s_key[TILE];
    const StepHead& h = block_head(b.sc);
    const int ncell = (int)min(h.N, m.cap);
    const int g = h.gen, pb = h.pbuf;
    const unsigned short* om = b.om[g];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = t / RANK_LANES, sub = t % RANK_LANES;
    const bool on = c < ncell && !is_halo(om, c);
    const unsigned long long k = on ? b.key[g][c] : 0ull;
    int rank = 0;
    for (int t0 = 0; t0 < ncell; t0 += TILE) {
        __syncthreads();
        for (int i = threadIdx.x; i < TILE; i += blockDim.x) {
            const int e = t0 + i;
            s_key[i] = e < ncell && !is_halo(om, e) ? b.key[g][e] : ~0ull;
        }
        __syncthreads();
#pragma unroll 8
        for (int i = sub; i < TILE; i += RANK_LANES) rank += s_key[i] < k;
    }
#pragma unroll
    for (int off = RANK_LANES / 2; off > 0; off >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, off);
    if (on && sub == 0) {
        int I[N];
        unpack_key<N>(m, k, I);
#pragma unroll
        for (int j = 0; j < N; ++j) idx[(long long)rank * N + j] = I[j];
        p[rank] = __ddiv_rn((double)static_cast<const T*>(b.q[pb])[c], h.w);
    }
}

// A larger pool: the ranges of the active cells' key fields (beside the counts),
// then (code, entry) of every active cell for the sort, and the read-out in the
// sorted order.
template <int N>
__global__ void __launch_bounds__(THREADS) k_readout_range(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    const long long ncell = min(h.N, m.cap);
    const int g = h.gen;
    FieldRange<N> range;
    for (WarpRuns r(ncell); r.next();)
        if (r.c < ncell && !is_halo(b.om[g], r.c)) range.see(m, b.key[g][r.c]);
    range.fold(b.sc);
}

__global__ void __launch_bounds__(THREADS) k_readout_keys(const Model m, Bufs b) {
    const StepHead& h = block_head(b.sc);
    const long long ncell = min(h.N, m.cap);
    const int g = h.gen;
    const SortBufs sb = sort_bufs(b, g, h.pbuf);
    const KeyCode code(m, b.sc);
    long long c0, c1;
    block_chunk(ncell, c0, c1);
    long long base = b.blk[blockIdx.x];
    for (long long t0 = c0; t0 < c1; t0 += blockDim.x) {
        const long long c = t0 + threadIdx.x;
        const int f = c < c1 && !is_halo(b.om[g], c);
        int total;
        const int pos = block_exclusive_scan(f, total);
        if (f) {
            sb.key[0][base + pos] = code(m, b.key[g][c]);
            sb.val[0][base + pos] = (unsigned)c;
        }
        base += total;
    }
}

template <int N, typename T>
__global__ void __launch_bounds__(THREADS) k_readout_order(const Model m, Bufs b, int passes, long long count,
                                                           int* __restrict__ idx, double* __restrict__ p) {
    const StepHead& h = block_head(b.sc);
    const int g = h.gen, pb = h.pbuf;
    const unsigned int* val = sort_bufs(b, g, pb).val[passes & 1];
    const double w = h.w;
    for (WarpRuns r(count); r.next();) {
        if (r.c >= count) continue;
        const unsigned c = val[r.c];
        int I[N];
        unpack_key<N>(m, b.key[g][c], I);
#pragma unroll
        for (int j = 0; j < N; ++j) idx[r.c * N + j] = I[j];
        p[r.c] = __ddiv_rn((double)static_cast<const T*>(b.q[pb])[c], w);
    }
}

}  // namespace gbees
