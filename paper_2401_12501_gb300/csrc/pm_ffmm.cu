// Float-float smooth sums of many right-hand sides as matrix products on the tensor cores.
//
// The sums' matrix entries (log r^2, the remainder) are evaluated once per pair in the
// float-float arithmetic of pm_ff.cuh; their products with the columns' strengths, 12 float32
// instructions a pair and column in k_direct_multi_ff (pm_batch.cu), are integer arithmetic on
// the tensor cores, as in pm_quadmm.cu: entries and strengths in 54-bit fixed point (a power of
// two per target row, bounded over its pairs once per surface, and per column), six base-512
// digits in float16, float32 sums of 128 sources at a time, added up in 64 bits.  Those sums are
// integers, exact below 2^24: the two of largest weight always (128 256^2 and twice that), the
// others, of three products a source and more, unless nearly all digits of both operands sit at
// their extremes, which would cost 2^-24 of a sum that weighs 512^-2 or less.
// Surfaces whose nodes lie so unevenly that a row's largest entry dwarfs the rest of it, or with
// fewer nodes than a stage, keep k_direct_multi_ff (kFmSpread; pm_batch.cu kFfmmNodes).
// Of the digit products the remainder's matrices keep the 26 above 2^-58 of the scale, for a row's
// nearest neighbours set the scale and stand far above the rest of it; log r^2 varies little and
// keeps 21 (2^-54).
//
//   K    one matrix, log r^2, for the columns of every operator on a geometry
//   R1   one matrix, the remainder of one operator
//   RG   q^2 - H q and the three components of r/r^2 (q = n.r/r^2), for the columns of several
//        operators: the remainder of each is a/pi times the first and grad a/(2 pi) times the
//        others, factors of the target that multiply the finished sums
//
// Block: 512 threads, up to 64 columns; four row tiles of 16 (four tiles of targets, or RG's
// four matrices on one tile) by 128 sources a stage in shared memory, two buffers.  Every warp
// evaluates its share of the next stage's entries and multiplies its row tile by 16 columns
// of this stage, half the warps in one order and half in the other, so that float32 and tensor
// pipes run side by side.  The strengths' digits come from L2 a step ahead.
// GB300, 24,576 nodes: K with 64 columns 7.3 ms (k_direct_multi_ff 25.0), R1 with 8 columns 5.2
// (5.7) and with 16 6.5 (9.6), RG with 8 operators of 8 columns 24.4 (eight times 5.7).  An
// m16n8k16 takes two clocks an SM: RG keeps the tensor pipe 55 % busy; R1 and K are bound by the
// entries' latency.  Errors against float64 are at most 0.7 of
// k_direct_multi_ff's on even patches (kFmSpread).
#include "pm_ff.cuh"
#include "pm_quadmm.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace {

using namespace pmff;
enum { kK = 0, kR1 = 1, kRG = 2 };
constexpr int kFmThreads = 512;
constexpr int kFmK = 128;                  // sources a stage
constexpr int kKS = kFmK / 16;
constexpr int kFmCols = 64;
constexpr size_t kBufWords = (size_t)4 * kKS * kQmDigits * 4 * 32;
constexpr int kRecord = 20;                // floats of a target in shared memory
// The remainder's fixed point serves while no row's largest |q^2 - H q| or 1/r stands more than
// this factor above the row's root mean square.  Every entry of a row is rounded to some 2^-54 of
// its largest, which is S 2^-54 of their root mean square at a factor S, and float-float
// arithmetic rounds each to about 2^-44 of itself.  Surfaces of even patches have 2^5 to 2^10.3
// (1,500 to 400,000 nodes; 2^8.3 with the two kinks of a star); patches halved towards a point pass
// 2^11 at a size of 2^-8.  Errors against float64 over those of k_direct_multi_ff, 8 columns: 0.1
// to 0.2 at 2^7.4 (torus, 24,576 nodes), 0.04 to 0.1 at 2^8.3 (star, 24,576), 0.4 to 0.7 at 2^10.3
// (flat ellipsoid, 21,600), 0.7 to 1.3 at 2^15.4 and 49 to 53 at 2^21.4 (patches halved 12 and 18
// times).  log r^2 has no such rows and is taken whenever it is defined.
constexpr float kFmSpread = 2048.f;

// Columns of one launch: operators in order, first[q] <= column < first[q + 1]
struct Cols {
    int nops, first[PM_FFMM_OPS + 1];
    const double *sigma[PM_FFMM_OPS], *wa[PM_FFMM_OPS], *a[PM_FFMM_OPS], *g[PM_FFMM_OPS];
    long long ld;
};
__device__ __forceinline__ int op_of(const Cols& C, int col) {
    int q = 0;
    while (q + 1 < C.nops && col >= C.first[q + 1]) ++q;
    return q;
}

// What the fixed point of a row is laid out for, by target i: its pairs' largest |q^2 - H q| and
// 1/r, the sums of their squares over the sources, weighted as the strengths are by the quadrature,
// and the largest |log r^2|, of the sources of one split; part[(split 5 + k) N + i] in the order
// max, max, sum, sum, max, and the sum of the squared weights in sw[split N + i].  The sums are
// free of the surface's size L, L^2 its area: |q^2 - H q| L^2, L / r, weights N w / L^2.  The differences and n.r are those of the sums (float-float): n.r is of the
// order r^2, and of coordinates rounded to float32 its error grows past it where nodes are close.
__global__ void __launch_bounds__(128)
k_fm_rows(const float4* __restrict__ src, const double* __restrict__ nrm, const double* __restrict__ H,
          const double* __restrict__ w, int N, int chunk, double area, float* __restrict__ part,
          float* __restrict__ sw) {
    __shared__ float4 sa[128], sb[128];
    const int i = blockIdx.x * 128 + threadIdx.x, ii = min(i, N - 1);
    const float4 ta = src[2 * (size_t)ii], tb = src[2 * (size_t)ii + 1];
    ff n[3];
    for (int d = 0; d < 3; ++d) n[d] = ff_from_double(nrm[3 * (size_t)ii + d]);
    const float h = (float)H[ii];
    const float size2 = (float)area, size = sqrtf(size2);
    float top0 = 0.f, top1 = 0.f, toplog = 0.f, sum0 = 0.f, sum1 = 0.f, sumw = 0.f;
    const int s0 = blockIdx.y * chunk, s1 = min(s0 + chunk, N);
    for (int base = s0; base < s1; base += 128) {
        __syncthreads();
        const int j = min(base + (int)threadIdx.x, N - 1);
        sa[threadIdx.x] = src[2 * (size_t)j];
        sb[threadIdx.x] = src[2 * (size_t)j + 1];
        sb[threadIdx.x].w = (float)(w[j] * N / area);
        __syncthreads();
        const int len = min(128, s1 - base);
        for (int k = 0; k < len; ++k) {
            if (base + k == ii) continue;
            const float4 a = sa[k], b = sb[k];
            const ff dx = ff_sub(ff{ta.x, tb.x}, ff{a.x, b.x}), dy = ff_sub(ff{ta.y, tb.y}, ff{a.y, b.y}),
                     dz = ff_sub(ff{ta.z, tb.z}, ff{a.z, b.z});
            const float r2 = fmaf(dx.h, dx.h, fmaf(dy.h, dy.h, dz.h * dz.h)), inv = 1.f / r2;
            const ff nr = ff_norm(ff_add_lazy(ff_add_lazy(ff_mul_lazy(n[0], dx), ff_mul_lazy(n[1], dy)),
                                              ff_mul_lazy(n[2], dz)));
            const float q = nr.h * inv, e0 = fabsf(q * (q - h)), e1 = sqrtf(inv);
            const float f0 = b.w * size2 * e0, f1 = b.w * size * e1;
            sum0 = fmaf(f0, f0, sum0);           // an undefined pair leaves the sums undefined
            sum1 = fmaf(f1, f1, sum1);
            sumw = fmaf(b.w, b.w, sumw);
            top0 = fmaxf(top0, e0);
            top1 = fmaxf(top1, e1);
            toplog = fmaxf(toplog, fabsf(__logf(r2)));
        }
    }
    if (i >= N) return;
    float* p = part + (size_t)blockIdx.y * 5 * N + i;
    p[0] = top0;
    p[N] = top1;
    p[2 * (size_t)N] = sum0;
    p[3 * (size_t)N] = sum1;
    p[4 * (size_t)N] = toplog;
    sw[(size_t)blockIdx.y * N + i] = sumw;
}

// bound[i], bound[N + i], bound[2 N]: the largest |q^2 - H q| and 1/r of target i and the largest
// |log r^2| of all; bound[2 N + 1]: how far a row's largest entry stands above the row's root mean
// square, at worst (infinity where a pair is undefined)
__global__ void k_fm_bounds(int N, int nsplit, double area, const float* __restrict__ part,
                            const float* __restrict__ sw, unsigned int* __restrict__ bound) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float top0 = 0.f, top1 = 0.f, toplog = 0.f, sum0 = 0.f, sum1 = 0.f, sumw = 0.f;
    for (int s = 0; s < nsplit && i < N; ++s) {
        const float* p = part + (size_t)s * 5 * N + i;
        top0 = fmaxf(top0, p[0]);
        top1 = fmaxf(top1, p[N]);
        sum0 += p[2 * (size_t)N];
        sum1 += p[3 * (size_t)N];
        toplog = fmaxf(toplog, p[4 * (size_t)N]);
        sumw += sw[(size_t)s * N + i];
    }
    float over = 0.f;
    if (i < N) {
        bound[i] = __float_as_uint(top0);
        bound[N + i] = __float_as_uint(top1);
        const float size2 = (float)area, size = sqrtf(size2);
        const bool defined = sum0 < 3e38f && sum1 < 3e38f && sumw > 0.f && sumw < 3e38f;
        over = !defined && N > 1 ? __int_as_float(0x7f800000)
                                 : fmaxf(top0 > 0.f ? top0 * size2 * sqrtf(sumw / sum0) : 0.f,
                                         top1 > 0.f ? top1 * size * sqrtf(sumw / sum1) : 0.f);
    }
    for (int o = 16; o > 0; o >>= 1) {
        over = fmaxf(over, __shfl_xor_sync(0xffffffffu, over, o));
        toplog = fmaxf(toplog, __shfl_xor_sync(0xffffffffu, toplog, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(bound + 2 * (size_t)N, __float_as_uint(toplog));
        atomicMax(bound + 2 * (size_t)N + 1, __float_as_uint(over));
    }
}

// E with a bit to spare: bound < 2^(E - 1)
__device__ __forceinline__ int spare_exponent(float bound) {
    return (int)((__float_as_uint(bound + 1e-30f) >> 23) & 255) - 125;
}

// exponent field of each column's largest |strength|
__global__ void __launch_bounds__(256)
k_fm_strength_top(Cols C, int N, int* __restrict__ top, const int* __restrict__ skip) {
    if (skip && *skip) return;
    __shared__ int sh[8];
    const int col = blockIdx.x, q = op_of(C, col);
    const double* sg = C.sigma[q] + (size_t)(col - C.first[q]) * C.ld;
    const double* wa = C.wa[q];
    int t = 0;
    for (int j = threadIdx.x; j < N; j += 256) t = max(t, (__double2hiint(wa[j] * sg[j]) >> 20) & 0x7ff);
    t = __reduce_max_sync(0xffffffffu, t);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) t = max(t, sh[w]);
        top[col] = max(t, 64);
    }
}

// the strengths' digits in the mma's B order: [16 sources][8 columns][digit][lane][2]
__global__ void __launch_bounds__(256)
k_fm_strengths(Cols C, int N, int Npad, const int* __restrict__ top, unsigned int* __restrict__ S,
               const int* __restrict__ skip) {
    if (skip && *skip) return;
    const int jp = blockIdx.x * 256 + threadIdx.x, col = blockIdx.y;
    if (2 * jp >= Npad) return;
    unsigned long long v[2];
    if (col < C.first[C.nops]) {
        const int q = op_of(C, col);
        const double* sg = C.sigma[q] + (size_t)(col - C.first[q]) * C.ld;
        const double* wa = C.wa[q];
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * jp + h;
            v[h] = qm_fixed(j < N ? wa[j] * sg[j] : 0.0, top[col], 0);
        }
    } else {
        v[0] = v[1] = qm_fixed(0.0, 64, 0);
    }
    const int ks = jp >> 3, l = jp & 7;
    for (int d = 0; d < kQmDigits; ++d)
        S[((((size_t)ks * 8 + (col >> 3)) * kQmDigits + d) * 32 + (col & 7) * 4 + (l & 3)) * 2 + (l >> 2)] =
            qm_digit2(v[0], v[1], d);
}

// The base-512 digits of (h + l) 2^(8 - E) as floats: three from h, then three from what is left of
// it and l, so that they hold the value to 2^-51 of the scale.  All lie in [-256, 256] but the
// fourth, which takes in l and may reach 512 (float16 holds integers to 2,048).
struct FloatDigits {
    float r, l;
    __device__ __forceinline__ FloatDigits(ff v, int E) {
        const float sc = __int_as_float((127 + 8 - E) << 23);
        r = v.h * sc;
        l = v.l * sc;
    }
    __device__ __forceinline__ float next(int d) {
        if (d == 3) r = fmaf(l, 134217728.f, r);                 // 512^3
        const float q = (r + 12582912.f) - 12582912.f;           // to the nearest integer
        r = (r - q) * 512.f;
        return q;
    }
};

// entries of the pair (target record t, source at (A, B) hi and lo) into e[0 .. NM)
template <int KIND>
__device__ __forceinline__ void entries(const float* t, float4 A, float4 B, const float4* stab, ff* e) {
    if (KIND == kK) {
        const ff dx = ff_grid_sub(ff{t[0], t[3]}, A.x, B.x), dy = ff_grid_sub(ff{t[1], t[4]}, A.y, B.y),
                 dz = ff_grid_sub(ff{t[2], t[5]}, A.z, B.z);
        const ff r2 = ff_add_lazy(ff_add_lazy(ff_sqr_lazy(dx), ff_sqr_lazy(dy)), ff_sqr_lazy(dz));
        e[0] = ff_norm(ff_log_lazy(r2, stab));
        return;
    }
    const ff dx = ff_sub(ff{t[0], t[3]}, ff{A.x, B.x}), dy = ff_sub(ff{t[1], t[4]}, ff{A.y, B.y}),
             dz = ff_sub(ff{t[2], t[5]}, ff{A.z, B.z});
    const ff r2 = ff_add_lazy(ff_add_lazy(ff_sqr_lazy(dx), ff_sqr_lazy(dy)), ff_sqr_lazy(dz));
    const ff inv = ff_rcp_lazy(r2);
    const ff nr = ff_norm(ff_add_lazy(ff_add_lazy(ff_mul_lazy(ff{t[6], t[9]}, dx), ff_mul_lazy(ff{t[7], t[10]}, dy)),
                                      ff_mul_lazy(ff{t[8], t[11]}, dz)));
    if (KIND == kR1) {
        const ff mr = ff_add_lazy(ff_add_lazy(ff_mul_lazy(ff{t[12], t[15]}, dx), ff_mul_lazy(ff{t[13], t[16]}, dy)),
                                  ff_mul_lazy(ff{t[14], t[17]}, dz));
        const ff inner = ff_norm(ff_add_lazy(ff_mul_lazy(nr, ff_mul_lazy(nr, inv)), mr));
        e[0] = ff_mul(inv, inner);
    } else {
        const ff q = ff_mul(nr, inv);
        e[0] = ff_mul(q, ff_norm(ff_add_lazy(q, ff{-t[12], -t[13]})));      // q (q - H)
        e[1] = ff_mul(dx, inv);
        e[2] = ff_mul(dy, inv);
        e[3] = ff_mul(dz, inv);
    }
}

template <int KIND>
__global__ void __launch_bounds__(kFmThreads, 1)
k_ffmm(const float4* __restrict__ src, const float4* __restrict__ tg, const double* __restrict__ nrm,
       const double* __restrict__ H, const float4* __restrict__ log_tab,
       const uint2* __restrict__ S, const unsigned int* __restrict__ bound,
       const int* __restrict__ top, Cols C, int N, int chunk, float2* __restrict__ partial, const int* __restrict__ skip) {
    if (skip && *skip) return;
    constexpr int NM = KIND == kRG ? 4 : 1;
    constexpr int TB = 64 / NM;                 // targets of a block
    constexpr int kSums = KIND == kK ? 6 : 7;   // sums of digit products of equal weight
    extern __shared__ __align__(16) unsigned int sA[];           // [2][row tile][k-step][digit][reg][lane]
    __shared__ float srec[TB][kRecord];
    __shared__ float4 stab[KIND == kK ? 128 : 1];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const int i0 = blockIdx.x * TB;
    if (KIND == kK)
        for (int k = tid; k < 128; k += kFmThreads) stab[k] = log_tab[k];
    if (tid < TB) {
        const int i = min(i0 + tid, N - 1);
        float* t = srec[tid];
        if (KIND == kK) {
            const float4 a = src[2 * (size_t)i], b = src[2 * (size_t)i + 1];
            t[0] = a.x; t[1] = a.y; t[2] = a.z; t[3] = b.x; t[4] = b.y; t[5] = b.z;
            t[18] = __int_as_float(spare_exponent(__uint_as_float(bound[2 * (size_t)N])));
        } else {
            const float b0 = __uint_as_float(bound[i]), b1 = __uint_as_float(bound[N + i]);
            const float4* v = tg + 6 * (size_t)i;
            t[0] = v[0].x; t[1] = v[0].y; t[2] = v[0].z; t[3] = v[1].x; t[4] = v[1].y; t[5] = v[1].z;
            if (KIND == kR1) {
                t[6] = v[2].x; t[7] = v[2].y; t[8] = v[2].z; t[9] = v[3].x; t[10] = v[3].y; t[11] = v[3].z;
                t[12] = v[4].x; t[13] = v[4].y; t[14] = v[4].z; t[15] = v[5].x; t[16] = v[5].y; t[17] = v[5].z;
                // a/pi |q^2 - H q| + |grad a| / (2 pi r)
                const double* ga = C.g[0] + 3 * (size_t)i;
                const float gs = (float)(fabs(ga[0]) + fabs(ga[1]) + fabs(ga[2]));
                t[18] = __int_as_float(spare_exponent(0.32f * (float)fabs(C.a[0][i]) * b0 + 0.16f * gs * b1));
            } else {
                t[18] = __int_as_float(spare_exponent(b0));
                t[19] = __int_as_float(spare_exponent(b1));
                for (int d = 0; d < 3; ++d) {
                    const ff m = ff_from_double(nrm[3 * (size_t)i + d]);
                    t[6 + d] = m.h;
                    t[9 + d] = m.l;
                }
                const ff h = ff_from_double(H[i]);
                t[12] = h.h;
                t[13] = h.l;
            }
        }
    }
    const int s0 = blockIdx.y * chunk, s1 = min(s0 + chunk, N);

    // the stage of 128 sources from `base` into buffer b: a unit is one target and two
    // neighbouring sources
    auto fill = [&](int base, int b) {
        constexpr int kUnits = KIND == kRG ? 2 : 8;
#pragma unroll 1
        for (int u = 0; u < kUnits; ++u) {
            const int combo = w * kUnits + u;
            const int rh = combo & 1, kh = (combo >> 1) & 1, ks = (combo >> 2) & 7;
            const int tile = KIND == kRG ? 0 : combo >> 5;
            const int r = tile * 16 + g + 8 * rh, j = base + ks * 16 + 8 * kh + 2 * t4;
            ff e[2][NM];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int jj = min(j + h, N - 1);
                entries<KIND>(srec[r], src[2 * (size_t)jj], src[2 * (size_t)jj + 1], stab, e[h]);
                if (j + h >= s1 || j + h == i0 + r)
                    for (int m = 0; m < NM; ++m) e[h][m] = ff{0.f, 0.f};
            }
#pragma unroll
            for (int m = 0; m < NM; ++m) {
                const int E = __float_as_int(srec[r][m == 0 ? 18 : 19]);
                FloatDigits v0(e[0][m], E), v1(e[1][m], E);
                unsigned int* to = sA + b * kBufWords +
                                   ((((size_t)(KIND == kRG ? m : tile) * kKS + ks) * kQmDigits) * 4 + rh + 2 * kh) * 32 + lane;
#pragma unroll
                for (int d = 0; d < kQmDigits; ++d) {
                    const float q0 = v0.next(d), q1 = v1.next(d);
                    const __half2 q = __floats2half2_rn(q0, q1);
                    to[d * 128] = *reinterpret_cast<const unsigned int*>(&q);
                }
            }
        }
    };

    const int rt = w & 3, cg = w >> 2;          // this warp's row tile and 16 columns
    const int nts = min(2, (C.first[C.nops] - cg * 16 + 7) / 8);           // its n-tiles in use
    long long vh[2][4], vl[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h)
        for (int c = 0; c < 4; ++c) vh[h][c] = vl[h][c] = 0;
    auto multiply = [&](int base, int b) {
        if (nts <= 0) return;
        const unsigned int* ap = sA + b * kBufWords + ((size_t)rt * kKS * kQmDigits) * 128 + lane;
        const uint2* sp = S + (((size_t)(base / 16) * 8 + cg * 2) * kQmDigits) * 32 + lane;
        // strengths a step ahead: they come from L2
        uint2 bn[kQmDigits];
#pragma unroll
        for (int d = 0; d < kQmDigits; ++d) bn[d] = __ldg(sp + d * 32);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h >= nts) continue;
            float acc[kSums][4];
#pragma unroll
            for (int d = 0; d < kSums; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.f;
#pragma unroll 1
            for (int ks = 0; ks < kKS; ++ks) {
                unsigned int a[kQmDigits][4];
                uint2 bb[kQmDigits];
#pragma unroll
                for (int d = 0; d < kQmDigits; ++d) {
                    bb[d] = bn[d];
#pragma unroll
                    for (int q = 0; q < 4; ++q) a[d][q] = ap[(ks * kQmDigits + d) * 128 + q * 32];
                }
                const int next = ks + 1 < kKS ? (ks + 1) * 8 + h : 1;       // after h = 0: the second n-tile
#pragma unroll
                for (int d = 0; d < kQmDigits; ++d) bn[d] = __ldg(sp + ((size_t)next * kQmDigits + d) * 32);
#pragma unroll
                for (int da = 0; da < kQmDigits; ++da)
#pragma unroll
                    for (int db = 0; da + db < kSums && db < kQmDigits; ++db) qm_mma(acc[da + db], a[da], bb[db]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                vh[h][c] += ((long long)__float2int_rn(acc[0][c]) * 512 + __float2int_rn(acc[1][c])) * 512 +
                            __float2int_rn(acc[2][c]);
                vl[h][c] += ((long long)__float2int_rn(acc[3][c]) * 512 + __float2int_rn(acc[4][c])) * 512 +
                            __float2int_rn(acc[5][c]);
                if (kSums > 6) vl[h][c] += (__float2int_rn(acc[kSums - 1][c]) + 256) >> 9;
            }
        }
    };

    __syncthreads();                            // srec, stab
    if (s0 < s1) fill(s0, 0);
    __syncthreads();
    int b = 0;
    for (int base = s0; base < s1; base += kFmK, b ^= 1) {
        const int next = base + kFmK;
        if (w & 4) {
            if (next < s1) fill(next, b ^ 1);
            multiply(base, b);
        } else {
            multiply(base, b);
            if (next < s1) fill(next, b ^ 1);
        }
        __syncthreads();
    }

    // results in double
    const int ncols = C.first[C.nops];
    double* res = reinterpret_cast<double*>(sA);          // RG: [matrix][target][column]
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int col = cg * 16 + h * 8 + 2 * t4 + (c & 1), row = g + 8 * (c >> 1);
            const int ts = col < ncols ? top[col] : 64;
            const int E = __float_as_int(KIND == kRG ? srec[row][rt == 0 ? 18 : 19] : srec[rt * 16 + row][18]);
            const double unit = ldexp(1.0, E + (ts - 1022) - 61);
            double v = fma((double)vh[h][c], 134217728.0, (double)vl[h][c]) * unit;
            if (ts == 0x7ff) v = nan("");
            if (KIND == kRG) {
                res[((size_t)rt * 16 + row) * kFmCols + col] = v;
            } else {
                const int i = i0 + rt * 16 + row;
                if (KIND == kK) v *= 1.0 / (4.0 * M_PI);
                const float hi = (float)v;
                if (col < ncols && i < N)
                    partial[((size_t)col * gridDim.y + blockIdx.y) * N + i] = make_float2(hi, (float)(v - (double)hi));
            }
        }
    if (KIND == kRG) {
        __syncthreads();
        for (int e = tid; e < 16 * ncols; e += kFmThreads) {
            const int row = e & 15, col = e >> 4, i = i0 + row, q = op_of(C, col);
            if (i >= N) continue;
            const double* gq = C.g[q] + 3 * (size_t)i;
            const double* v = res + (size_t)row * kFmCols + col;
            constexpr int ms = 16 * kFmCols;
            const double s = C.a[q][i] * (1.0 / M_PI) * v[0] +
                             (0.5 / M_PI) * (gq[0] * v[ms] + gq[1] * v[2 * ms] + gq[2] * v[3 * ms]);
            const float hi = (float)s;
            partial[((size_t)col * gridDim.y + blockIdx.y) * N + i] = make_float2(hi, (float)(s - (double)hi));
        }
    }
}

template <int KIND>
pm_status launch(pm_surface* s, const PmFfmmWork& W, const Cols& C, int nsplit, float2* partial,
                 cudaStream_t st) {
    const size_t smem = 2 * kBufWords * sizeof(unsigned int);
    PM_CUDA_TRY(cudaFuncSetAttribute(k_ffmm<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int tb = KIND == kRG ? 16 : 64;
    const int chunk = pm_ceil_div(pm_ceil_div(s->N, nsplit), kFmK) * kFmK;
    k_ffmm<KIND><<<dim3(pm_ceil_div(s->N, tb), nsplit), kFmThreads, smem, st>>>(
        KIND == kK ? s->src_kg : s->src_ff, s->tgt_ff, s->n, s->H, s->log_tab,
        reinterpret_cast<const uint2*>(W.S), W.bound, W.top, C, s->N, chunk, partial, s->skip_flag);
    PM_CUDA_TRY(cudaGetLastError());
    s->launch_total++;
    return PM_OK;
}

}  // namespace

static size_t digit_words(int N) {
    return (size_t)pm_ceil_div(N, kFmK) * kFmK / 16 * 8 * kQmDigits * 64;
}
static size_t bound_words(int N) { return 2 * (size_t)N + 2; }

size_t pm_ffmm_bytes(int N) { return (digit_words(N) + bound_words(N) + kFmCols) * sizeof(int); }

void pm_ffmm_free(PmFfmmWork* W) {
    pm_dfree(W->S);
    pm_dfree(W->top);
    pm_dfree(W->bound);
}

// Buffers and the geometry's bounds (waits for them, once a workspace).  *room false: no room for
// the buffers, or a stream under capture, where nothing can be allocated; no error is left behind.
static pm_status ffmm_ready(pm_surface* s, PmFfmmWork* W, bool* room, cudaStream_t st) {
    *room = true;
    if (W->S) return PM_OK;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    PM_CUDA_TRY(cudaStreamIsCapturing(st, &capture));
    *room = capture == cudaStreamCaptureStatusNone;
    if (!*room) return PM_OK;
    const int N = s->N;
    pm_status r = pm_dmalloc(&W->S, digit_words(N));
    if (r == PM_OK) r = pm_dmalloc(&W->top, kFmCols);
    if (r == PM_OK) r = pm_dmalloc(&W->bound, bound_words(N));
    if (r == PM_OK) {
        const int blocks = pm_ceil_div(N, 128);
        const int ns = std::max(1, std::min({blocks, 16 * s->ctx->num_sms / blocks, 24}));
        const int chunk = pm_ceil_div(pm_ceil_div(N, ns), 128) * 128;
        // 6 ns N values in the digits' room of 192 N and more
        float *part = reinterpret_cast<float*>(W->S), *sw = part + (size_t)5 * ns * N;
        double area = 0.0;
        for (double v : s->h_w) area += std::fabs(v);
        cudaMemsetAsync(W->bound, 0, bound_words(N) * sizeof(int), st);
        k_fm_rows<<<dim3(blocks, ns), 128, 0, st>>>(s->src_ff, s->n, s->H, s->w, N, chunk, area, part, sw);
        k_fm_bounds<<<blocks, 128, 0, st>>>(N, ns, area, part, sw, W->bound);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&W->spread, W->bound + 2 * (size_t)N + 1, sizeof(float), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) {
            pm_set_error("bounds of the float-float sums: %s", cudaGetErrorString(e));
            r = PM_ERR_CUDA;
        }
    }
    if (r != PM_OK) pm_ffmm_free(W);
    if (r == PM_ERR_OOM) {
        cudaGetLastError();
        *room = false;
        return PM_OK;
    }
    return r;
}

pm_status pm_ffmm_sum(pm_surface* s, PmFfmmWork* W, int kind, int nops, pm_surface* const* ops,
                      const int* ncols, const double* const* sigma, long long ld, int nsplit,
                      float2* partial, bool* summed, cudaStream_t st) {
    PM_TRY(ffmm_ready(s, W, summed, st));
    *summed = *summed && W->spread <= (kind == kK ? 1e30f : kFmSpread);
    if (!*summed) return PM_OK;
    // launches of at most kFmCols columns of at most PM_FFMM_OPS operators
    int q = 0, done = 0;                 // operator, its columns already taken
    size_t out = 0;                      // first column of the launch
    while (q < nops) {
        Cols C{};
        C.ld = ld;
        while (q < nops && C.nops < PM_FFMM_OPS && C.first[C.nops] < kFmCols) {
            const int take = std::min(ncols[q] - done, kFmCols - C.first[C.nops]);
            C.sigma[C.nops] = sigma[q] + (size_t)done * ld;
            C.wa[C.nops] = ops[q]->wa;
            C.a[C.nops] = ops[q]->a;
            C.g[C.nops] = ops[q]->g;
            C.first[C.nops + 1] = C.first[C.nops] + take;
            ++C.nops;
            done += take;
            if (done == ncols[q]) {
                ++q;
                done = 0;
            }
        }
        const int n = C.first[C.nops], N = s->N, Npad = pm_ceil_div(N, kFmK) * kFmK;
        k_fm_strength_top<<<n, 256, 0, st>>>(C, N, W->top, s->skip_flag);
        k_fm_strengths<<<dim3(pm_ceil_div(Npad / 2, 256), kFmCols), 256, 0, st>>>(C, N, Npad, W->top, W->S,
                                                                                  s->skip_flag);
        PM_CUDA_TRY(cudaGetLastError());
        s->launch_total += 2;
        float2* to = partial + out * nsplit * (size_t)N;
        PM_TRY(kind == kK ? launch<kK>(s, *W, C, nsplit, to, st)
                          : kind == kR1 ? launch<kR1>(s, *W, C, nsplit, to, st)
                                        : launch<kRG>(s, *W, C, nsplit, to, st));
        out += n;
    }
    return PM_OK;
}
