// Device-side building blocks of the GBEES library: layout of the workspace,
// packed cell keys, the open-addressing hashtable, the drift models, the exact
// fixed-point accumulator and block reductions.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "gbees_keys.cuh"

namespace gbees {

namespace cg = cooperative_groups;

constexpr int MAXN = 6;
constexpr int THREADS = 256;
constexpr int WARPS = THREADS / 32;
constexpr int PERSIST_THREADS = 512;                 // block of the persistent step loop
constexpr int MAX_WARPS = PERSIST_THREADS / 32;      // warps of the largest block that uses the block helpers
constexpr int GRID_MAX = 8192;                       // blocks of the fixed launch grid (upper bound)
constexpr unsigned long long EMPTY_KEY = ~0ull;      // free hashtable slot

// Exact accumulator: NDIG signed 64-bit cells, each collecting 32-bit digits of a
// fixed-point number whose lowest bit weighs 2^ACC_LSB. The window
// [2^-128, 2^64) holds every density sum and moment of the workloads; terms
// below 2^-128 are truncated (deterministically), terms of 2^64 or more raise
// an error. Up to 2^31 terms per reduction need no carry.
constexpr int NDIG = 6;
constexpr int ACC_LSB = -128;

enum { DYN_CONSTANT = 0, DYN_LINEAR = 1, DYN_LORENZ63 = 2, DYN_LORENZ63_SHIFTED = 3, DYN_LORENZ96 = 4 };
enum { LIM_MC = 0, LIM_NONE = 1, LIM_LW = 2 };
enum {
    ST_OK = 0,
    ST_EINVAL = -1,
    ST_ECAPACITY = -2,
    ST_EKEYRANGE = -3,
    ST_EDEGENERATE = -4,
    ST_ECUDA = -5,
    ST_ETIMEOUT = -6,
    ST_ETABLE = -7
};

struct alignas(16) Slot {
    unsigned long long key;
    long long val;  // cell index (low 32 bits used)
};

// The part of the state that the kernels of a step read when they start: two
// lines of memory, the counters that a step adds to by atomics and the words that
// stay as they are while a kernel runs. Copied by each block as a whole (block_head).
struct alignas(256) StepHead {
    long long N;          // pool entries, active cells and halo cells (grows during grow)
    long long N_prev;     // pool entries before the current grow
    long long N_new;      // pool entries surviving the current prune
    long long NA;         // active cells
    long long NA_new;     // active cells surviving the current prune
    long long n_halo;     // halo cells appended by the current halo phase
    long long n_act;      // halo cells made active by the current grow (listed in map)
    long long n_glist;    // cells listed for the current grow (listed form)
    long long N_sorted;   // entries that the last sort put in order
    unsigned long long maxrate_bits;  // max CFL rate over the cells (non-negative double bits)
    unsigned long long maxq_ord;      // order key of the running max of Q
    unsigned long long tmp_ord;       // scratch maximum (init)
    long long steps_call;    // steps of the current propagate call
    long long updates_call;  // cell updates of the current propagate call
    long long step;          // steps since init
    unsigned int ticket;  // last-block election
    int step_last;        // the step lands on t_target

    int pbuf;             // current Q buffer
    int gen;              // current key/link buffer
    int done;             // t reached t_target
    int error;            // first error status (0 = none)
    int prune_now;        // the step just taken is a prune step (1), or its pool is to be sorted (RESORT)
    int sort_passes;      // 8-bit digits of the current sort's codes
    double maxq;          // max of Q after the last finalisation
    double w;             // (prod h) * sum Q at the last finalisation
    double scale;         // 1 / w, applied by the next step
    // the current step (written by the last block of the link kernel)
    double step_dt;         // dt of the step being taken
    double step_t_new;      // time after it
    double coef_dth[MAXN];  // dt / h_j
    double t;               // time
    double t_target;        // end of the current propagate call
};
static_assert(sizeof(StepHead) == 256, "copied as 32 words of 8 bytes");

// Scalars that live on the device so that a whole step needs no host round trip.
struct DevScalars : StepHead {
    double dt;            // last step
    long long acc[NDIG];  // exact sum of Q
    long long lookups_fallback;  // hashtable lookups of the flux update (none: every stencil cell is linked)
    long long loop_iter;  // iterations of the device-side step loop in the current graph launch
    long long graph_kernels;  // kernels executed by graph launches (counted on the device)
    // grid barrier of the persistent kernel and of a team of a batched launch:
    // arrivals since the launch began (cleared before every such launch)
    unsigned long long bar_seq;
    // the step loop's running reductions, in global atomics: the largest CFL
    // rate of the current prune epoch (two epochs by parity), and the exact
    // sum and maximum of the apply phase (two steps by parity)
    unsigned long long loop_rate[2];
    long long loop_acc[2][NDIG];
    unsigned long long loop_maxq[2];
    // SM cycles spent by block 0 of the persistent kernel per phase (grow,
    // halo, link, faces, apply, prune, step scalars) and the steps they cover
    long long phase_cycles[8];
    long long phase_steps;
    unsigned sort_lo[MAXN], sort_hi[MAXN];  // range of the key fields to sort
    long long mom[28][NDIG];     // exact sums for moments
    double mom_mean[MAXN];       // mean, input of the covariance pass
    double mom_out[28];          // moments times prod h
};
static_assert(sizeof(DevScalars) == 2304, "part of every workspace");

// The head of the state as it was when the block began, for all its threads. One
// warp of each block reads it, two lines in one load. With every thread reading the
// dozen scalars that it needs, the 10^4 warps of a resident wave queued at the one L2
// slice that holds them, 25 to 40 us in each of a step's kernels (6.5e5 entries in
// six dimensions: the sweep of k_grow_mark took 43 us, now 7.5; k_halo 54, now 13).
__device__ __forceinline__ const StepHead& block_head(const DevScalars* sc) {
    __shared__ StepHead h;
    if (threadIdx.x < sizeof(StepHead) / 8)
        reinterpret_cast<unsigned long long*>(&h)[threadIdx.x] =
            reinterpret_cast<const volatile unsigned long long*>(static_cast<const StepHead*>(sc))[threadIdx.x];
    __syncthreads();
    return h;
}

// Everything a kernel needs to know about the model and the grid (by value).
struct Model {
    int n;
    int dyn;
    int limiter;
    int key_bits;
    int prune_interval;
    int probe_width;
    int sort_order;              // storage order after a sorting prune (GBEES_ORDER_*)
    int bar_extra;               // arrivals a grid barrier waits for beyond its blocks (0; > 0 only to test the bounded wait)
    long long spin_limit;        // polls of a grid barrier before it gives up with ST_ETIMEOUT
    long long cap;               // cell capacity
    unsigned long long tmask;    // hashtable slots - 1
    double a[64];                // model parameters
    double h[MAXN];
    double x0[MAXN];
    double thr_rel;
    double cfl;
    double prod_h;
    double inv_h[MAXN];    // 1 / h_j
    double inv_2h[MAXN];   // 1 / (2 h_j)
    int h_pow2;            // bit j: h_j is a power of two
    int h_plain;           // every h_j lies within [2^-128, 2^128] (div_round's range)
};

// One block's share of a grid-wide reduction, written without atomics and
// combined by whoever finishes the step (deterministic: integer digits, max).
struct alignas(64) Partial {
    long long acc[NDIG];           // exact-sum digits of the block's values
    unsigned long long maxq_ord;   // order key of the block's maximum value (0: none)
    unsigned long long rate_bits;  // the block's maximum CFL rate (non-negative double bits)
};

// Device buffers (by value). The pool holds the active cells and their halo:
// every face neighbour of an active cell that is not active itself is kept as
// a halo cell (p = 0, never updated, never counted), so that all cells of the
// update stencil (face neighbours, their face neighbours, the second
// neighbours) are reached through links. link[g] holds 2n direction-major
// int32 arrays of cap entries: link[g][(2j + s) * cap + c] is the index of the
// neighbour of entry c one step down (s = 0) or up (s = 1) in dimension j, or
// -1 when it is not in the pool (a warp's consecutive entries read one
// direction with one coalesced load).
//
// om[g][c]: bits 0..2n-1 are the outward directions of cell c (bit 2j+1: the
// flow leaves through the upper j-face, bit 2j: through the lower j-face),
// fixed at creation because the drift does not depend on time; bit 14 marks a
// halo cell; bit 15 marks an active cell whose downwind set is known to be
// active (cleared by every prune). Bits 12 and 13 mark a halo cell that a step
// of a persistent or batched step loop made active (by the step's parity in the
// launch; cleared by the next step or at the end of the launch).
//
// Face velocities (storage type, dimension-major: u[g][j * cap + c]): f_j at
// the centre of the lower j-face of entry c (Eq. 7), evaluated once in FP64 when
// the entry is created (the drift does not depend on time) and carried along
// by the prune's compaction.
//
// Update scratch (storage type, dimension-major: element d * cap + c, so that a
// warp's 32 consecutive entries read and write whole sectors). Step loop of a small
// grid: wl[d] the jump P_c - P_{c-e_d} across the lower d-face, wg[d] the
// d-direction wave entering the cell, tg the sum over d of wg[d] / (2 h_d) (one value
// per entry), fl[j] the flux through the lower j-face. Large grids: one pair per
// entry and dimension (Wave: the jump and the upwind base) from wl on, over wl and wg,
// which follow one another in one block of 2 n cap values; fl the flux in FP64; tg
// unused. The grow's list and a prune's new order are in fl meanwhile.
struct Bufs {
    unsigned long long* key[2];
    void* q[2];
    int* link[2];
    unsigned short* om[2];
    unsigned int* slot[2];  // hashtable slot of each cell
    unsigned char* keep;
    int* map;        // prune: status, then new index; grow: the halo cells it activated
    Slot* table;
    DevScalars* sc;
    long long* blk;  // per-block counts (active cells)
    long long* blk2; // per-block counts (halo cells)
    unsigned int* sorthist;  // digit histograms of the prune's radix sort
    void* u[2];  // face velocities (two generations, like the keys)
    double* rate[2];  // CFL rate sum_j |f_j(x_{c-e_j/2})| / h_j of every entry (Eq. 8, FP64, fixed at creation)
    void* wl;    // update scratch in the storage type (wl and wg: one block)
    void* wg;
    void* tg;
    void* fl;
    Partial* part;   // GRID_MAX per-block partials
};


constexpr int RESORT = 2;                            // DevScalars::prune_now
constexpr long long RESORT_MIN_ENTRIES = 1ll << 21;
constexpr long long SORT_MIN_ENTRIES = 1ll << 18;    // smaller pools (they fit in L2) are not sorted

constexpr unsigned short OM_COMPLETE = 0x8000;
constexpr unsigned short OM_GHOST = 0x4000;
constexpr unsigned short OM_NEW = 0x1000;  // two bits, by the parity of the loop's step

// The kernels of one time step for one dimension and precision: those before the
// link phase, those after it, and the persistent step-loop kernel.
struct Kernels {
    void* pre[3];
    int npre;
    void* post[3];
    int npost;
    void* persist;
    void* batch;
};

// One grid of a batched propagation (k_batch): its model, its buffers (in its
// own workspace) and the time to propagate it to.
struct BatchItem {
    Model m;
    Bufs b;
    double t_end;
};

// Block of a team launch (k_batch with slots): the grid it works on (-1: none), the
// team's size and this block's index in the team.
struct TeamSlot {
    int item, nb, bi;
};



// ------------------------------------------------------------------ cell iteration
// Cells are handed out in runs of 32 consecutive cells (one warp, coalesced),
// consecutive runs to consecutive blocks, so that a small grid still spreads
// over every SM. The blocks that share the work of one grid are nb blocks of
// index bi (the whole launch, or one block when a launch runs many grids).
// Usage:
//   for (WarpRuns r(ncell, nb, bi); r.next();) { const long long c = r.c; if (c >= ncell) continue; ... }
struct WarpRuns {
    long long k, step, n, c;
    __device__ __forceinline__ WarpRuns(long long ncell, int nb, int bi)
        : k(bi + (long long)nb * (threadIdx.x >> 5) - (long long)nb * (blockDim.x >> 5)),
          step((long long)nb * (blockDim.x >> 5)),
          n(ncell),
          c(0) {}
    __device__ __forceinline__ explicit WarpRuns(long long ncell) : WarpRuns(ncell, gridDim.x, blockIdx.x) {}
    __device__ __forceinline__ bool next() {
        k += step;
        c = k * 32 + (threadIdx.x & 31);
        return k * 32 < n;
    }
};

// The same for the step loop of a small grid, in 32-bit numbers (a pool has
// fewer than 2^31 entries): run k of n_runs, handed out from the block's first
// warp up (FIRST), or for the few runs that go beside a phase's many from its
// last warp down (LAST) or from its middle (MIDDLE).
enum { FIRST, MIDDLE, LAST };
struct Runs {
    int k, step, n;
    __device__ __forceinline__ Runs(int n_runs, int nb, int bi, int place = FIRST) {
        const int nw = (int)(blockDim.x >> 5);
        int w = (int)(threadIdx.x >> 5);
        if (place == LAST) w = nw - 1 - w;
        if (place == MIDDLE) w = w >= nw / 2 ? w - nw / 2 : w + nw - nw / 2;
        step = nb * nw;
        k = bi + nb * w - step;
        n = n_runs;
    }
    __device__ __forceinline__ bool next() {
        k += step;
        return k < n;
    }
    __device__ __forceinline__ int cell() const { return k * 32 + (int)(threadIdx.x & 31); }
};
__device__ __forceinline__ int runs_of(long long entries) { return (int)((entries + 31) >> 5); }

// ------------------------------------------------------------------ keys

template <int N>
__device__ __forceinline__ bool pack_key(const Model& m, const int* I, unsigned long long& k) {
    return pack_key_bits<N>(m.key_bits, I, k);
}

template <int N>
__device__ __forceinline__ void unpack_key(const Model& m, unsigned long long k, int* I) {
    unpack_key_bits<N>(m.key_bits, k, I);
}

// ------------------------------------------------------------------ hashtable
// Open addressing (Sec. 4.2) along table_home and table_next; keys are claimed with
// atomicCAS (the concurrent insertion of Algorithm 2 without staging).

__device__ __forceinline__ int table_find(const Model& m, const Slot* __restrict__ T, unsigned long long key) {
    unsigned long long h = table_home(key, m.tmask);
#pragma unroll 1
    for (unsigned long long probe = 0; probe <= m.tmask; ++probe) {
        ulonglong2 s = __ldcg(reinterpret_cast<const ulonglong2*>(T + h));
        if (s.x == key) return (int)(long long)s.y;
        if (s.x == EMPTY_KEY) return -1;
        h = table_next(h, probe, m.tmask);
    }
    return -1;
}

// Cooperative lookup: a tile of W lanes probes W slots of the sequence per round
// and the lowest lane that sees the key or an empty slot
// decides. All lanes of the tile must call it with the same key.
template <int W>
__device__ __forceinline__ int table_find_tile(const Model& m, const Slot* __restrict__ T, unsigned long long key,
                                               cg::thread_block_tile<W> tile) {
    const unsigned long long home = table_home(key, m.tmask);
    const int lane = tile.thread_rank();
#pragma unroll 1
    for (unsigned long long probe = 0; probe <= m.tmask; probe += W) {
        unsigned long long h = table_slot(home, (probe + lane) & m.tmask, m.tmask);
        ulonglong2 s = __ldcg(reinterpret_cast<const ulonglong2*>(T + h));
        unsigned hit = tile.ballot(s.x == key);
        unsigned emp = tile.ballot(s.x == EMPTY_KEY);
        if (hit | emp) {
            int first_hit = hit ? __ffs(hit) - 1 : W;
            int first_emp = emp ? __ffs(emp) - 1 : W;
            if (first_hit < first_emp) {
                long long v = tile.shfl((long long)s.y, first_hit);
                return (int)v;
            }
            return -1;
        }
    }
    return -1;
}

// A claim whose probes grow long looks at the error word now and then: a pool that has
// run out of capacity goes on claiming keys until its phase ends and fills the table,
// where every further claim would look at all slots (minutes on one block).
constexpr unsigned long long CLAIM_LOOK = 64;
__device__ __forceinline__ bool claim_hopeless(const DevScalars* sc, unsigned long long probe) {
    return (probe & (CLAIM_LOOK - 1)) == CLAIM_LOOK - 1 && *(volatile const int*)&sc->error;
}

// Insert key if absent. Returns 1 and the slot when this thread claimed a new
// slot, 0 when the key is present, -1 when the table is full (or an error is recorded).
__device__ __forceinline__ int table_claim(const Model& m, Slot* T, const DevScalars* sc, unsigned long long key,
                                           unsigned long long* slot) {
    unsigned long long h = table_home(key, m.tmask);
#pragma unroll 1
    for (unsigned long long probe = 0; probe <= m.tmask; ++probe) {
        unsigned long long k = *reinterpret_cast<volatile unsigned long long*>(&T[h].key);
        if (k == key) return 0;
        if (k == EMPTY_KEY) {
            unsigned long long old = atomicCAS(&T[h].key, EMPTY_KEY, key);
            if (old == EMPTY_KEY) {
                *slot = h;
                return 1;
            }
            if (old == key) return 0;
        }
        if (claim_hopeless(sc, probe)) return -1;
        h = table_next(h, probe, m.tmask);
    }
    return -1;
}

// ------------------------------------------------------------------ errors

__device__ __forceinline__ void set_error(DevScalars* sc, int code) { atomicCAS(&sc->error, 0, code); }

__device__ __forceinline__ long long warp_aggregated_add(long long* counter, int count = 1) {
    cg::coalesced_group g = cg::coalesced_threads();
    long long base = 0;
    int total = g.size() * count;
    if (g.thread_rank() == 0) base = (long long)atomicAdd((unsigned long long*)counter, (unsigned long long)total);
    base = g.shfl(base, 0);
    return base + (long long)g.thread_rank() * count;
}

// ------------------------------------------------------------------ drift models
// f_j(y) is evaluated with the order of operations written out and no fused
// multiply-add, so that the FP64 velocities that take the grow / prune / CFL
// decisions are the IEEE values of the textbook expressions.

struct Ar {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
};

// Centre coordinate x0_k + i_k h_k (one rounded product, one rounded sum).
__device__ __forceinline__ double centre64(const Model& m, int k, int i) {
    return __dadd_rn(m.x0[k], __dmul_rn((double)i, m.h[k]));
}

// x / h_j for x >= 0 as the IEEE division rounds it. For a width that is a power
// of two the reciprocal is exact, so the product rounds the same real number.
__device__ __forceinline__ double div_h(const Model& m, double x, int j) {
    if ((m.h_pow2 >> j) & 1) return __dmul_rn(x, m.inv_h[j]);
    const int e = (int)(__double_as_longlong(x) >> 52);
    if (m.h_plain && e > 256 && e < 1792) return div_round(x, m.h[j], m.inv_h[j]);
    return __ddiv_rn(x, m.h[j]);
}

// a * b + c rounded once, and the larger of two values, in the arithmetic
// type itself (explicit single-precision forms for float, so that nothing is
// widened to double).
__device__ __forceinline__ double fmadd(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fmadd(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }

// Sign tests, absolute value and negation. FP64 arithmetic is scarce on this
// chip, so for doubles they work on the two words of the bit pattern in the integer
// pipe. (The words, not the pattern as one 64-bit integer: the compiler knows that
// the pattern without its sign bit is the absolute value, and that the pattern
// shifted left by one is zero for a zero, and would put the FP64 instructions back;
// they were 8 of 13 per face of the flux pass and a third of the wave pass.)
__device__ __forceinline__ bool gt0(double x) {
    const int hi = __double2hiint(x);
    return hi > 0 || (hi == 0 && __double2loint(x) != 0);
}
__device__ __forceinline__ bool lt0(double x) {
    const int hi = __double2hiint(x);
    return hi < 0 && ((hi & 0x7fffffff) | __double2loint(x)) != 0;
}
__device__ __forceinline__ bool gt0(float x) { return x > 0.0f; }
__device__ __forceinline__ bool lt0(float x) { return x < 0.0f; }
__device__ __forceinline__ bool nonzero(double x) { return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) != 0; }
__device__ __forceinline__ bool nonzero(float x) { return x != 0.0f; }
// Whether a face's velocity carries a flux: it is not zero. (In FP32 a velocity that is
// no number carries none; in FP64 it does, and the step ends with ST_EDEGENERATE.)
__device__ __forceinline__ bool flows(double u) { return nonzero(u); }
__device__ __forceinline__ bool flows(float u) { return fabsf(u) > 0.0f; }
__device__ __forceinline__ double abs_bits(double x) {
    return __hiloint2double(__double2hiint(x) & 0x7fffffff, __double2loint(x));
}
// v >= 0 with the sign of s
__device__ __forceinline__ double with_sign(double v, double s) {
    return __hiloint2double(__double2hiint(v) | (__double2hiint(s) & (int)0x80000000), __double2loint(v));
}
__device__ __forceinline__ float with_sign(float v, float s) { return copysignf(v, s); }
__device__ __forceinline__ float abs_bits(float x) { return fabsf(x); }
// min of two non-negative finite values (integer order of the bits for doubles)
__device__ __forceinline__ double min_nonneg(double a, double b) {
    return __longlong_as_double(min(__double_as_longlong(a), __double_as_longlong(b)));
}
__device__ __forceinline__ float min_nonneg(float a, float b) { return fminf(a, b); }

// The significance test p > p* (p* >= 0) of a stored value, decided exactly
// as (double)p > p* but without FP64 arithmetic: for doubles on the bit
// patterns (signed integer order equals the order of doubles when one side is
// non-negative), for floats against the largest float not above p*.
template <typename T>
struct Above;
template <>
struct Above<double> {
    long long pb;
    __device__ __forceinline__ explicit Above(double pstar) { pb = __double_as_longlong(pstar); }
    __device__ __forceinline__ bool operator()(double q) const { return __double_as_longlong(q) > pb; }
};
template <>
struct Above<float> {
    float pf;
    __device__ __forceinline__ explicit Above(double pstar) {
        pf = (float)pstar;
        if ((double)pf > pstar) pf = nextafterf(pf, -INFINITY);  // round towards -inf
    }
    __device__ __forceinline__ bool operator()(float q) const { return q > pf; }
};

// 2x and x/2 of a non-negative double with the results of IEEE x + x and
// x * 0.5 (round to nearest even), in integer operations only (no FP64 pipe):
// the exponent field moves by one; a subnormal or overflowing case is formed
// on the bit pattern directly.
__device__ __forceinline__ double twice_nonneg(double x) {
    const long long b = __double_as_longlong(x);
    const long long e = b >> 52;
    long long r = e == 0 ? (b << 1)                                   // subnormal (or 0): the significand doubles
                : e <= 2045 ? b + (1ll << 52)                         // one more in the exponent
                : e == 2046 ? 0x7FF0000000000000ll                    // overflow to +inf
                : b;                                                  // inf, NaN
    return __longlong_as_double(r);
}
__device__ __forceinline__ double half_nonneg(double x) {
    const long long b = __double_as_longlong(x);
    const long long e = b >> 52;
    if (e >= 2) return __longlong_as_double(b - (1ll << 52));         // one less in the exponent (inf, NaN stay)
    // the result is subnormal: halve the significand, ties to even
    const long long sig = e == 0 ? b : (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
    long long q = sig >> 1;
    if ((sig & 1) && (q & 1)) q += 1;
    return __longlong_as_double(q);
}
__device__ __forceinline__ float twice_nonneg(float x) { return x + x; }
__device__ __forceinline__ float half_nonneg(float x) { return 0.5f * x; }

template <typename T>
__device__ __forceinline__ T limited_wave(int lim, T W, T Wup) {
    if (lim == LIM_LW) return W;
    // MC limiter phi(theta) = max(0, min((1+theta)/2, 2, 2 theta)) with theta = Wup / W,
    // multiplied by W and written without the division: zero unless W and Wup
    // have the same sign, else sign(W) min(|W + Wup| / 2, 2 |W|, 2 |Wup|).
    if ((gt0(W) && gt0(Wup)) || (lt0(W) && lt0(Wup))) {
        const T aW = abs_bits(W), aU = abs_bits(Wup);
        const T v = min_nonneg(min_nonneg(half_nonneg(aW + aU), twice_nonneg(aW)), twice_nonneg(aU));
        return with_sign(v, W);
    }
    return (T)0;
}

// ------------------------------------------------------------------ exact accumulator

// Add x (a finite double) to the digits. Sets err on a non-finite or too
// large term.
__device__ __forceinline__ void acc_add(long long (&d)[NDIG], double x, int& err) {
    unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    int ex = (int)((bits >> 52) & 0x7ff);
    unsigned long long mt = bits & 0xFFFFFFFFFFFFFull;
    if (ex == 0x7ff) { err = 1; return; }
    if (ex == 0) {
        if (mt == 0) return;
        ex = 1;
    } else {
        mt |= 1ull << 52;
    }
    int pos = ex - 1075 - ACC_LSB;  // x = mt * 2^(pos + ACC_LSB)
    if (pos < 0) {
        if (pos <= -64) return;
        mt >>= -pos;
        pos = 0;
        if (mt == 0) return;
    }
    if (pos > 32 * NDIG - 53 - 1) { err = 1; return; }
    const bool neg = (bits >> 63) != 0;
    const int k = pos >> 5, r = pos & 31;
    const unsigned long long lo = mt << r;
    const unsigned long long hi = r ? (mt >> (64 - r)) : 0ull;
    const long long d0 = (long long)(lo & 0xffffffffull), d1 = (long long)(lo >> 32), d2 = (long long)(hi & 0xffffffffull);
#pragma unroll
    for (int q = 0; q < NDIG; ++q) {
        long long v = (q == k) ? d0 : (q == k + 1) ? d1 : (q == k + 2) ? d2 : 0;
        d[q] += neg ? -v : v;
    }
}

// The same for a float (integer operations only; a float is exactly a double).
__device__ __forceinline__ void acc_add(long long (&d)[NDIG], float x, int& err) {
    const unsigned int bits = __float_as_uint(x);
    int ex = (int)((bits >> 23) & 0xff);
    unsigned long long mt = bits & 0x7FFFFFu;
    if (ex == 0xff) { err = 1; return; }
    if (ex == 0) {
        if (mt == 0) return;
        ex = 1;
    } else {
        mt |= 1u << 23;
    }
    int pos = ex - 150 - ACC_LSB;  // x = mt * 2^(pos + ACC_LSB)
    if (pos < 0) {
        if (pos <= -32) return;
        mt >>= -pos;
        pos = 0;
        if (mt == 0) return;
    }
    if (pos > 32 * NDIG - 24 - 1) { err = 1; return; }
    const bool neg = (bits >> 31) != 0;
    const int k = pos >> 5, r = pos & 31;
    const unsigned long long sh = mt << r;  // at most 55 bits
    const long long d0 = (long long)(sh & 0xffffffffull), d1 = (long long)(sh >> 32);
#pragma unroll
    for (int q = 0; q < NDIG; ++q) {
        long long v = (q == k) ? d0 : (q == k + 1) ? d1 : 0;
        d[q] += neg ? -v : v;
    }
}

// Round the exact value sum_q D[q] 2^(32 q + ACC_LSB) once to the nearest double
// (ties to even). Straight-line code on registers: one thread of each block
// runs it once per time step, on the critical path of a small grid's step.
static __host__ __device__ __noinline__ double acc_to_double(const long long* D) {
    // carries: base-2^32 digits below a signed top word
    unsigned int c[NDIG];
    long long carry = 0;
#pragma unroll
    for (int q = 0; q < NDIG; ++q) {
        const long long v = D[q] + carry;
        c[q] = (unsigned int)(unsigned long long)v;
        carry = v >> 32;  // floor division by 2^32
    }
    unsigned long long w0 = (unsigned long long)c[0] | ((unsigned long long)c[1] << 32);
    unsigned long long w1 = (unsigned long long)c[2] | ((unsigned long long)c[3] << 32);
    unsigned long long w2 = (unsigned long long)c[4] | ((unsigned long long)c[5] << 32);
    unsigned long long w3 = (unsigned long long)carry;
    const bool neg = carry < 0;
    if (neg) {  // the magnitude
        w0 = ~w0 + 1ull;
        w1 = ~w1 + (w0 == 0 ? 1ull : 0ull);
        w2 = ~w2 + (w0 == 0 && w1 == 0 ? 1ull : 0ull);
        w3 = ~w3 + (w0 == 0 && w1 == 0 && w2 == 0 ? 1ull : 0ull);
    }
    // the top non-zero word, the word below it, and whether anything lies below that
    unsigned long long hi = w0, lo = 0ull;
    bool rest = false;
    int base = 0;
    if (w3) {
        hi = w3; lo = w2; rest = (w1 | w0) != 0; base = 192;
    } else if (w2) {
        hi = w2; lo = w1; rest = w0 != 0; base = 128;
    } else if (w1) {
        hi = w1; lo = w0; base = 64;
    }
    if (hi == 0) return 0.0;
#if defined(__CUDA_ARCH__)
    const int z = __clzll((long long)hi);
#else
    const int z = __builtin_clzll(hi);
#endif
    // 64 significant bits and a sticky bit, then 53 bits
    const unsigned long long m = z ? (hi << z) | (lo >> (64 - z)) : hi;
    const bool sticky = rest || (z ? (lo << z) : lo) != 0;
    unsigned long long v = m >> 11;
    const unsigned int cut = (unsigned int)(m & 0x7FFull);
    if (cut > 0x400u || (cut == 0x400u && (sticky || (v & 1ull)))) v += 1;
    // v in [2^52, 2^53]: the exponent field takes a carry out of the mantissa;
    // the exponent is within [ACC_LSB, ACC_LSB + 255], far inside the normal range
    const int ex = base + 63 - z + ACC_LSB + 1023;
    unsigned long long bits = ((unsigned long long)ex << 52) + (v - (1ull << 52));
    if (neg) bits |= 1ull << 63;
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)bits);
#else
    double r;
    memcpy(&r, &bits, sizeof r);
    return r;
#endif
}

// Order-preserving map of doubles onto unsigned 64-bit keys (for atomicMax).
__device__ __forceinline__ unsigned long long ord_key(double x) {
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double ord_val(unsigned long long k) {
    unsigned long long b = (k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
    return __longlong_as_double((long long)b);
}

// Block-wide reduction of the digits and of a maximum, then one atomic per
// digit into global memory. All threads of the block must call it.
__device__ __forceinline__ void block_reduce_acc_max(long long (&d)[NDIG], double mx, long long* g_acc,
                                                     unsigned long long* g_ord) {
    __shared__ long long s_acc[MAX_WARPS][NDIG];
    __shared__ double s_mx[MAX_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NDIG; ++q) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) d[q] += __shfl_down_sync(0xffffffffu, d[q], off);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, off));
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < NDIG; ++q) s_acc[wid][q] = d[q];
        s_mx[wid] = mx;
    }
    __syncthreads();
    if (threadIdx.x < NDIG) {
        long long v = 0;
#pragma unroll 4
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += s_acc[w][threadIdx.x];
        if (v) atomicAdd((unsigned long long*)&g_acc[threadIdx.x], (unsigned long long)v);
    }
    if (threadIdx.x == 32 && g_ord) {
        double m = -INFINITY;
#pragma unroll 4
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, s_mx[w]);
        if (m > -INFINITY) atomicMax(g_ord, ord_key(m));
    }
    __syncthreads();
}

__device__ __forceinline__ double block_max(double mx) {
    __shared__ double s_m[MAX_WARPS];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_down_sync(0xffffffffu, mx, off));
    if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = mx;
    __syncthreads();
    double m = -INFINITY;
#pragma unroll 4
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, s_m[w]);
    __syncthreads();
    return m;
}

// True in every thread of exactly one block: the last one to arrive. One
// thread per block fences and takes a ticket (the block barrier before it
// orders the block's writes; fences are cumulative).
__device__ __forceinline__ bool last_block(DevScalars* sc) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned int t = atomicAdd(&sc->ticket, 1u);
        s_last = (t == gridDim.x * gridDim.y - 1);
        if (s_last) __threadfence();
    }
    __syncthreads();
    return s_last;
}

// Normalisation scalars of a new grid from the exact sum and the running
// maximum. mode bit 2: keep w = 1 (cells loaded as given).
__device__ __forceinline__ void finalise_norm(const Model& m, DevScalars* sc, int mode) {
    sc->N_prev = sc->N;
    sc->maxq = sc->maxq_ord ? ord_val(sc->maxq_ord) : 0.0;
    if (mode & 2) {
        sc->w = 1.0;
        sc->scale = 1.0;
    } else {
        long long D[NDIG];
        for (int q = 0; q < NDIG; ++q) D[q] = *(volatile long long*)&sc->acc[q];
        double s = acc_to_double(D);
        double w = m.prod_h * s;
        sc->w = w;
        if (!(w > 0.0) || !isfinite(w)) {
            set_error(sc, ST_EDEGENERATE);
            sc->scale = 0.0;
        } else {
            sc->scale = 1.0 / w;
        }
    }
    for (int q = 0; q < NDIG; ++q) sc->acc[q] = 0;
    sc->maxq_ord = 0;
    sc->ticket = 0;
    if (sc->N == 0 && !(mode & 2)) set_error(sc, ST_EDEGENERATE);
}

// Write this block's partial (exact digits, maximum value, maximum rate).
// All threads of the block must call it; d, mx, rate are per thread. The
// maxima are reduced as order-preserving integer keys (integer pipe).
__device__ __forceinline__ void block_partial(Partial* part, long long (&d)[NDIG], double mx, double rate,
                                              int bi) {
    __shared__ long long s_acc[MAX_WARPS][NDIG];
    __shared__ unsigned long long s_mx[MAX_WARPS], s_rt[MAX_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long mk = mx > -INFINITY ? ord_key(mx) : 0ull;
    unsigned long long rk = rate > 0.0 ? (unsigned long long)__double_as_longlong(rate) : 0ull;
#pragma unroll
    for (int q = 0; q < NDIG; ++q) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) d[q] += __shfl_down_sync(0xffffffffu, d[q], off);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        mk = max(mk, __shfl_down_sync(0xffffffffu, mk, off));
        rk = max(rk, __shfl_down_sync(0xffffffffu, rk, off));
    }
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < NDIG; ++q) s_acc[wid][q] = d[q];
        s_mx[wid] = mk;
        s_rt[wid] = rk;
    }
    __syncthreads();
    // one thread per digit and per maximum folds the warps' values
    const int q = threadIdx.x, nw = (int)(blockDim.x >> 5);
    if (q < NDIG) {
        long long a = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) a += s_acc[w][q];
        part[bi].acc[q] = a;
    } else if (q == NDIG) {
        unsigned long long mm = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) mm = max(mm, s_mx[w]);
        part[bi].maxq_ord = mm;
    } else if (q == NDIG + 1) {
        unsigned long long rr = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) rr = max(rr, s_rt[w]);
        part[bi].rate_bits = rr;
    }
    __syncthreads();
}
__device__ __forceinline__ void block_partial(Partial* part, long long (&d)[NDIG], double mx, double rate) {
    block_partial(part, d, mx, rate, blockIdx.x);
}

// Sum of the digits over a warp: the six digits (padded to eight) together, each
// exchange halves the values a lane carries, 9 shuffles of 64 bits instead of 30.
// Lane l returns the sum of digit l / 4 (0 of the padding).
__device__ __forceinline__ long long warp_sum_digits(const long long (&d)[NDIG]) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    long long a[4];
    const bool up = lane & 16;
    const long long hi[4] = {d[4], d[5], 0, 0};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long got = __shfl_xor_sync(full, up ? d[i] : hi[i], 16);
        a[i] = (up ? hi[i] : d[i]) + got;
    }
    const bool up2 = lane & 8;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const long long got = __shfl_xor_sync(full, up2 ? a[i] : a[i + 2], 8);
        a[i] = (up2 ? a[i + 2] : a[i]) + got;
    }
    const bool up4 = lane & 4;
    const long long got = __shfl_xor_sync(full, up4 ? a[0] : a[1], 4);
    a[0] = (up4 ? a[1] : a[0]) + got;
    a[0] += __shfl_xor_sync(full, a[0], 2);
    a[0] += __shfl_xor_sync(full, a[0], 1);
    return a[0];
}

// The block's digits and maximum value folded into global accumulators with
// atomics. Integer sums and maxima: the totals do not depend on the order of
// the blocks.
__device__ __forceinline__ void block_atomics(long long* acc, unsigned long long* maxq, const long long (&d)[NDIG],
                                              double mx) {
    __shared__ long long s_acc[MAX_WARPS][8];
    __shared__ unsigned long long s_mx[MAX_WARPS];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long mine = warp_sum_digits(d);
    const unsigned long long mk = mx > -INFINITY ? ord_key(mx) : 0ull;
    const unsigned top = __reduce_max_sync(full, (unsigned)(mk >> 32));
    const unsigned low = __reduce_max_sync(full, (unsigned)(mk >> 32) == top ? (unsigned)mk : 0u);
    if ((lane & 3) == 0) s_acc[wid][lane >> 2] = mine;
    if (lane == 0) s_mx[wid] = ((unsigned long long)top << 32) | low;
    __syncthreads();
    const int q = threadIdx.x, nw = (int)(blockDim.x >> 5);
    if (q < NDIG) {
        long long t = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) t += s_acc[w][q];
        if (t) atomicAdd((unsigned long long*)&acc[q], (unsigned long long)t);
    } else if (q == NDIG) {
        unsigned long long mm = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) mm = max(mm, s_mx[w]);
        if (mm) atomicMax(maxq, mm);
    }
}

// Combine the partials of blocks [0, nblk) in every thread of the calling
// block (the same result everywhere): digit sums, maximum value, maximum rate.
struct Combined {
    long long acc[NDIG];
    unsigned long long maxq_ord;
    unsigned long long rate_bits;
};
__device__ __forceinline__ Combined combine_partials(const Partial* part, int nblk) {
    __shared__ long long s_acc[MAX_WARPS][NDIG];
    __shared__ unsigned long long s_mo[MAX_WARPS], s_rt[MAX_WARPS];
    long long d[NDIG] = {0, 0, 0, 0, 0, 0};
    unsigned long long mo = 0, rt = 0;
#pragma unroll 1
    for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
        const Partial* p = part + i;
#pragma unroll
        for (int q = 0; q < NDIG; ++q) d[q] += __ldcg(&p->acc[q]);
        mo = max(mo, __ldcg(&p->maxq_ord));
        rt = max(rt, __ldcg(&p->rate_bits));
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NDIG; ++q)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) d[q] += __shfl_down_sync(0xffffffffu, d[q], off);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        mo = max(mo, __shfl_down_sync(0xffffffffu, mo, off));
        rt = max(rt, __shfl_down_sync(0xffffffffu, rt, off));
    }
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < NDIG; ++q) s_acc[wid][q] = d[q];
        s_mo[wid] = mo;
        s_rt[wid] = rt;
    }
    __syncthreads();
    // one thread per digit and per maximum folds the warps' values; every
    // thread then reads the results
    __shared__ unsigned long long s_fin[NDIG + 2];
    const int q = threadIdx.x, nw = (int)(blockDim.x >> 5);
    if (q < NDIG) {
        long long a = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) a += s_acc[w][q];
        s_fin[q] = (unsigned long long)a;
    } else if (q == NDIG) {
        unsigned long long mm = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) mm = max(mm, s_mo[w]);
        s_fin[q] = mm;
    } else if (q == NDIG + 1) {
        unsigned long long rr = 0;
#pragma unroll 4
        for (int w = 0; w < nw; ++w) rr = max(rr, s_rt[w]);
        s_fin[q] = rr;
    }
    __syncthreads();
    Combined c;
#pragma unroll
    for (int k = 0; k < NDIG; ++k) c.acc[k] = (long long)s_fin[k];
    c.maxq_ord = s_fin[NDIG];
    c.rate_bits = s_fin[NDIG + 1];
    __syncthreads();
    return c;
}

// Grid-wide barrier of a cooperative launch (all blocks resident). The wait is
// bounded: it gives up when another block has set an error or after
// spin_limit polls (BARRIER_SPIN_LIMIT by default: about 15 seconds, a poll being one
// load from L2 and, every 32nd time, the error word and a short sleep: 0.23 us), sets
// ST_ETIMEOUT, and returns false; callers then leave.
constexpr long long BARRIER_SPIN_LIMIT = 1ll << 26;

__device__ __forceinline__ unsigned long long atom_add_acq_rel_gpu(unsigned long long* p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.add.acq_rel.gpu.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}

__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Barrier k (1, 2, ...) of a launch whose nb blocks all take part in every
// barrier of the grid with scalars sc (the whole launch, or a team of a batched
// launch), on a counter that was zero when the launch began: the barrier is
// complete once k * nb arrivals are counted. One release-acquire add per block
// publishes the block's writes and counts the arrival; there is no reset, so the
// last arrival releases the waiters directly. All blocks must be resident
// (cooperative launch). Bounded: gives up with ST_ETIMEOUT.
// fetch runs in thread 0 after the barrier is complete, before the block goes
// on: it reads the scalars that the phase before produced, one reader per
// block, its loads in flight together with the error word's (read from every
// thread, the same few words queue up at one L2 slice).
__device__ __noinline__ static int barrier_wait(DevScalars* sc, unsigned long long target, long long spin_limit) {
    unsigned long long* cnt = &sc->bar_seq;
    if (atom_add_acq_rel_gpu(cnt, 1ull) + 1ull >= target) return 1;
    long long spins = 0;
    while (ld_acquire_gpu(cnt) < target) {
        ++spins;
        // the error word is read now and then: a second load per poll would
        // double the time until a waiter sees the barrier open
        if ((spins & 31) == 0) {
            if (*(volatile int*)&sc->error) return 0;
            __nanosleep(32);
        }
        if (spins > spin_limit) {
            set_error(sc, ST_ETIMEOUT);
            return 0;
        }
    }
    return 1;
}
template <typename F>
__device__ __forceinline__ bool grid_barrier_seq(DevScalars* sc, int nb, unsigned long long& k, long long spin_limit,
                                                 F&& fetch) {
    __shared__ int s_ok;
    __syncthreads();
    k += 1;
    if (threadIdx.x == 0) {
        const int ok = barrier_wait(sc, k * (unsigned long long)(unsigned int)nb, spin_limit);
        const int e = *(volatile int*)&sc->error;
        fetch();
        s_ok = ok && !e;
    }
    __syncthreads();
    return s_ok != 0;
}

// The same for a block that works alone: a block barrier, the error word read
// by one thread.
template <typename F>
__device__ __forceinline__ bool block_barrier(DevScalars* sc, F&& fetch) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int e = *(volatile int*)&sc->error;
        fetch();
        s_ok = !e;
    }
    __syncthreads();
    return s_ok != 0;
}

// Exclusive prefix of a 0/1 flag over the block (in thread order) and the total.
__device__ __forceinline__ int block_exclusive_scan(int flag, int& total) {
    __shared__ int s_w[MAX_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned bal = __ballot_sync(0xffffffffu, flag);
    int in_warp = __popc(bal & ((1u << lane) - 1u));
    if (lane == 0) s_w[wid] = __popc(bal);
    __syncthreads();
    int before = 0, tot = 0;
#pragma unroll 4
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        int v = s_w[w];
        if (w < wid) before += v;
        tot += v;
    }
    __syncthreads();
    total = tot;
    return before + in_warp;
}

}  // namespace gbees
