// Near-field weights as matrix products (pm_quadmm.cu): what the table builders of the
// quadrilateral (pm_nearfield.cu) and triangle (pm_tri.cu) rules share with the engine.
#pragma once

#include <cuda_fp16.h>

#include <functional>

#include "pm_internal.cuh"

constexpr int kQmDigits = 6;       // base-512 digits a value is split into
constexpr int kQmPts = 64;         // quadrature points a tile
constexpr int kQmCols = 8;         // (target, patch) columns a block

// A table holds tiles of kQmPts quadrature points: the basis values' digits as float16
// [tile][digit][point][npad], npad = n rounded up to 16, most significant digit first, and
// per point (weight / (2 pi), twice the logarithm's correction).
struct QmTable {
    __half* dig = nullptr;
    double2* pt = nullptr;
    unsigned int* top = nullptr;   // largest |basis value|, as float bits: first pass only
    int* over = nullptr;           // set by a basis value of 2^eB or more
    int n = 0, npad = 0, eB = 0;   // |basis| < 2^eB
};

// v 2^(53 - e) for |v| < 2^e, e = top - 1022, rounded, as six base-512 digits in [-256, 256],
// each biased by 256 in nine bits of the result (ten for the first).  `guard` drops that many
// bits more.  Integer instructions only: the float64 pipe is what these kernels wait for.
__device__ __forceinline__ unsigned long long qm_fixed(double v, int top, int guard) {
    const int hi = __double2hiint(v);
    const int ex = (hi >> 20) & 0x7ff;
    const int sh = top - ex + guard;                 // >= guard
    unsigned long long m =
        ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned int)__double2loint(v);
    m = (ex == 0 || sh > 54) ? 0ull : sh > 0 ? (m + (1ull << (sh - 1))) >> sh : m;
    const long long s = hi < 0 ? -(long long)m : (long long)m;
    // bias: 256 (1 + 512 + ... + 512^5)
    return (unsigned long long)(s + 0x20100804020100ll);
}

// digit d (0 the most significant) of two biased values as a pair of float16
__device__ __forceinline__ unsigned int qm_digit2(unsigned long long a, unsigned long long b, int d) {
    const unsigned int mask = d == 0 ? 0x3ffu : 0x1ffu;
    const unsigned int da = (unsigned int)(a >> (9 * (kQmDigits - 1 - d))) & mask;
    const unsigned int db = (unsigned int)(b >> (9 * (kQmDigits - 1 - d))) & mask;
    const unsigned int w = da | (db << 16) | 0x64006400u;            // 1024 + digit + 256
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), __half2half2(__ushort_as_half(0x6500)));
    return *reinterpret_cast<const unsigned int*>(&h);               // 0x6500 = 1280
}

// c += a b: 16 x 16 digits by 16 x 8
__device__ __forceinline__ void qm_mma(float* c, const unsigned int* a, uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// Two neighbouring basis values k, k + 1 (k even) of a point into the table.
__device__ __forceinline__ void qm_put(const QmTable& T, size_t tile, int point, int k, double a,
                                       double b) {
    if (max(__double2hiint(a) & 0x7fffffff, __double2hiint(b) & 0x7fffffff) >= (1023 + T.eB) << 20)
        *T.over = 1;
    const unsigned long long fa = qm_fixed(a, T.eB + 1022, 0), fb = qm_fixed(b, T.eB + 1022, 0);
    unsigned int* row = reinterpret_cast<unsigned int*>(
        T.dig + (tile * kQmDigits * kQmPts + point) * T.npad + k);
    for (int d = 0; d < kQmDigits; ++d)
        row[(size_t)d * kQmPts * T.npad / 2] = qm_digit2(fa, fb, d);
}

// A surface type's rules for the engine.  With T.top set a table is not filled; its largest
// value is found instead.
struct QmRules {
    int n = 0;                                       // nodes (basis functions) a patch
    std::vector<int> tiles;                          // [n + 1] first tile of each node's self rule
    std::function<pm_status(int loc0, int nloc, const QmTable&)> self_table;
    int near_tiles = 4;                              // tiles of one cell's rule
    std::function<pm_status(const int* codes, int ncodes, const QmTable&)> near_table;
    // the leaf cells of npairs (target, patch) blocks: start and count of each in codes
    // (capacity cap, *used the total wanted)
    std::function<pm_status(const int* blocks, int npairs, int* start, int* count, int* codes,
                            int cap, int* used)> leaves;
};

// W_lb, W_g and W_k of every near block of s.
pm_status pm_quad_weights(pm_surface* s, const QmRules& R);
