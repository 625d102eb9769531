// Packed cell keys, the hashtable's hash, the rule of the pool's order and the rounded
// division by a cell width: pure functions that the device code uses and that a host
// compiler can build too (the host tests pin them: round trip, key order, range limits,
// the probe sequence, and the probe lengths at load factor 1/2, Sec. 4.2).
//
// A cell index I (N signed ints) packs into one u64: each component biased by
// 2^(b-1) into b bits, dimension 0 in the most significant position, so that
// key order is the lexicographic order of the index vectors. A component
// outside [-2^(b-1), 2^(b-1)) has no key.
#pragma once

#include <math.h>

#if defined(__CUDACC__)
#define GBEES_HD __host__ __device__ __forceinline__
#else
#define GBEES_HD inline
#endif

namespace gbees {

template <int N>
GBEES_HD bool pack_key_bits(int b, const int* I, unsigned long long& k) {
    const long long bias = 1ll << (b - 1);
    const long long lim = 1ll << b;
    k = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        long long v = (long long)I[j] + bias;
        if (v < 0 || v >= lim) return false;
        k = (k << b) | (unsigned long long)v;
    }
    return true;
}

template <int N>
GBEES_HD void unpack_key_bits(int b, unsigned long long k, int* I) {
    const long long bias = 1ll << (b - 1);
    const unsigned long long mask = (b >= 64) ? ~0ull : ((1ull << b) - 1);
#pragma unroll
    for (int j = N - 1; j >= 0; --j) {
        I[j] = (int)((long long)(k & mask) - bias);
        k >>= b;
    }
}

// Component j of I one step up or down. False when there is no such 32-bit index: in
// one dimension an index takes all 32 bits, and a wrapped one would have a key (in more
// dimensions the index is there and has no key).
template <int N>
GBEES_HD bool step_index(int* I, int j, int up) {
    if (N == 1 && I[0] == (up ? 0x7fffffff : -0x7fffffff - 1)) return false;
    I[j] += up ? 1 : -1;
    return true;
}

// Morton (Z-order) code of a packed key of n fields of b bits: the bits of
// the n indices interleaved, from the most significant bit of every field
// down, dimension 0 first within each bit. A bijection of the n*b-bit keys
// that keeps cells near one another in all n dimensions near one another in
// code order (key order keeps them near only along the last dimension).
GBEES_HD unsigned long long morton_code(unsigned long long k, int n, int b) {
    unsigned long long out = 0;
    for (int bit = b - 1; bit >= 0; --bit)
        for (int j = 0; j < n; ++j) out = (out << 1) | ((k >> ((n - 1 - j) * b + bit)) & 1ull);
    return out;
}

// Row-Morton code of a packed key of n fields of b bits: the Morton code of
// the first n - 1 fields, then the last field. Cells that differ only in the
// last index keep their key order (a row of the grid along the last dimension
// stays contiguous, so the neighbours of a run of consecutive cells in any
// dimension are runs too), while the rows themselves follow the Z curve of
// the other n - 1 indices (rows near one another in those dimensions stay near
// one another in code order). A bijection of the n*b-bit keys.
GBEES_HD unsigned long long row_morton_code(unsigned long long k, int n, int b) {
    if (n <= 1) return k;
    const unsigned long long last = k & ((1ull << b) - 1);
    return (morton_code(k >> b, n - 1, b) << b) | last;
}

// Whether sorting a pool of n entries, `out` of them out of order, pays over the next
// `left` steps. A sort's time goes with n, a step's gain with out, and a sort pays when
// out left > c n, c falling as the pool outgrows what the L2 serves of its neighbours.
// Measured (Lorenz '96; time of a sort, gain per step; break-even in steps by the
// measurement and by this rule):
//   6-D FP64  2.2e6 entries, 65 % out  0.81 ms  0.038 ms  21 / 18
//             5.1e6, 60 %              1.9      0.123     16 / 15
//             8.2e6, 56 %              3.3      0.37       9 / 11
//             1.5e7, 53 %              6.3      0.96       7 / 7
//   5-D FP64  3.4e6, 40 %              1.0      0.033     31 / 27
//   6-D FP32  2.2e6, 65 %              0.76     0.098      8 / 8
//             5.1e6, 60 %              1.8      0.28       6 / 7
//             1.5e7, 53 %              5.6      1.19       5 / 5
//   5-D FP32  3.4e6, 40 %              0.89     0.081     11 / 12
GBEES_HD bool resort_pays(long long n, long long out, double left, bool fp64) {
    const double mi = (double)n / 1048576.0;
    const double c = fp64 ? fmax(14.0 - mi, 3.5) : fmax(5.5 - 0.25 * mi, 2.5);
    return (double)out * left > c * (double)n;
}

// murmur3 64-bit finaliser (a bijection of u64)
GBEES_HD unsigned long long mix64(unsigned long long x) {
    x ^= x >> 33;
    x *= 0xff51afd7ed558ccdull;
    x ^= x >> 33;
    x *= 0xc4ceb9fe1a85ec53ull;
    x ^= x >> 33;
    return x;
}

// Probe sequence of a key in a table of mask + 1 slots (a power of two, at
// least 64). Cells whose keys differ in the low 4 bits alone (16 neighbours along
// the last dimension) share a group of 16 consecutive slots: the group's place is
// hashed from the other bits, and the order within it is permuted by an XOR with
// bits of the same hash, so that a set that repeats with the period of a group
// (one cell in each, say) does not fill one slot of every group. A collision
// moves on to the same slot of the next group, so the sequences of 16 cells stay
// side by side; each of the 16 interleaved subtables is an ordinary table with
// linear probing at the same load. After all groups the sequence goes on with the
// next slot of each: it visits every slot once.
//
// Why groups: a random probe costs a translation miss and a DRAM sector, and
// translation misses bound the lookups of large pools. The cells of a warp follow
// one another along the last dimension, and so do their neighbours in any
// direction: a warp's 32 probes fall into 2 to 5 groups instead of 32 places.
constexpr int TABLE_GROUP_BITS = 4;
constexpr unsigned long long TABLE_GROUP = 1ull << TABLE_GROUP_BITS;

GBEES_HD unsigned long long table_home(unsigned long long key, unsigned long long mask) {
    const unsigned long long g = mix64(key >> TABLE_GROUP_BITS);
    return ((g << TABLE_GROUP_BITS) | ((key ^ (g >> 60)) & (TABLE_GROUP - 1))) & mask;
}

// The slot after `slot`, the probe-th of the sequence (0, 1, ...).
GBEES_HD unsigned long long table_next(unsigned long long slot, unsigned long long probe, unsigned long long mask) {
    slot = (slot + TABLE_GROUP) & mask;
    if (((probe + 1) & (mask >> TABLE_GROUP_BITS)) == 0)
        slot = (slot & ~(TABLE_GROUP - 1)) | ((slot + 1) & (TABLE_GROUP - 1));
    return slot;
}

// The probe-th slot of the sequence that starts at home.
GBEES_HD unsigned long long table_slot(unsigned long long home, unsigned long long probe, unsigned long long mask) {
    const unsigned long long groups = (mask >> TABLE_GROUP_BITS) + 1;
    return ((home + probe * TABLE_GROUP) & mask & ~(TABLE_GROUP - 1)) |
           ((home + probe / groups) & (TABLE_GROUP - 1));
}

// x / h for x >= 0 with y = RN(1 / h), x and h far from the ends of the exponent
// range, as the IEEE division rounds it: a quotient that is within an ulp becomes
// the correctly rounded one by its exact remainder times y (P. Markstein,
// Computation of elementary functions on the IBM RISC System/6000 processor,
// 1990). x y is within two ulp, the first correction brings it within one. Five
// FP64 instructions.
GBEES_HD double div_round(double x, double h, double y) {
    const double q0 = x * y;
    const double q1 = fma(fma(-q0, h, x), y, q0);
    return fma(fma(-q1, h, x), y, q1);
}

}  // namespace gbees
