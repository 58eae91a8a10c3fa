// Near-field weights (Sec. 6.1.1, 6.1.2) as matrix products on the tensor cores.
//
// The quadrature points of a rule depend on the reference cell alone: the polar points about a
// node position are the same for every patch, and so are the 256 Gauss points of a subdivision
// cell for every (target, patch) that has it as a leaf.  For the points q of one rule and the
// columns (target i, patch P) that use it, with B the basis values at the points,
//     Y = B [X_P - x_i, J_P]     offsets and surface element at the points       (contraction over nodes)
//     F = the five integrands of pm_nearfield.cu at Y, weighted                  (per point)
//     W = F^T B                  the weight sets                                 (contraction over points)
// GB300 runs two float64 multiply-adds a clock and SM, and both contractions together need
// about 9 n of them a point and column (n = 64: 590 of 870).  Here they run on the
// tensor cores in integer arithmetic (the error-free splitting of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012): every operand is a 54-bit fixed-point
// number under a power of two per column (per table for B), cut into six base-512 digits; the
// 26 digit products above 2^-58 of the result's scale are float16 mma with float32 accumulation
// (with the 21 above 2^-54 alone, what is dropped adds up over K to 2^-49, three times
// the float64 sums' error); sums of equal weight share one accumulator.  They are exact below
// 2^24: the two sums of largest weight always (K 256^2 and 2 K 256^2, K <= 128), the others
// unless nearly all digits of both operands sit at their extremes, which would cost 2^-24 of a
// sum that weighs 512^-2 or less.  The
// float64 pipe keeps the integrands (31 operations a point and column), the
// conversion of Y (8) and the accumulation of W (15 n / 64).
//
// Block: 256 threads, kQmCols columns, tiles of 64 points.  Warp w evaluates the integrands of
// column w (a lane two points), so a column's largest |F| of a tile is a warp reduction.
// Weights of an item (a range of tiles) go to a slot of `partial`; k_qm_reduce adds the slots of
// a block in a fixed order, so the results do not depend on which columns share a block.
// Two blocks an SM up to n = 64 (their shared memory is 113 KB), one above.
// GB300: a near field of 2,400 nodes (n = 100) 286 -> 59 ms with everything around it, 2,880
// nodes of triangles (n = 36) 705 -> 53 ms, against blocks that kept both contractions on the
// float64 pipe; that pipe is 73 % busy at n = 36 and n = 64, 45 % at n = 100, where one block
// an SM leaves it idle in the tensor phases.
#include "pm_quadmm.cuh"

#include "pm_fast64.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

namespace {

constexpr int kQmThreads = 256;
constexpr int kQmSums = 7;                // sums of digit products of equal weight that are kept
constexpr int kNT1 = kQmCols * 4 / 8;     // n-tiles of Y (4 fields a column)
constexpr int kNT2 = kQmCols * 5 / 8;     // n-tiles of W (5 kinds a column)
constexpr int kFStride = 72;              // words a k-step of an F n-tile (64 + 8: no bank conflicts)
constexpr int kYStride = kQmPts + 4;      // doubles a row of Y

template <int NK>
struct QmShape {
    static constexpr int np = 16 * NK;
    static constexpr int bstride = np + 8;                                  // halves
    static constexpr size_t b_bytes = (size_t)kQmDigits * kQmPts * bstride * 2;
    static constexpr size_t x_bytes = (size_t)kQmDigits * kNT1 * NK * 64 * 4;
    static constexpr size_t f_bytes = (size_t)kQmDigits * kNT2 * 4 * kFStride * 4;
    static constexpr size_t bytes = b_bytes + x_bytes + f_bytes + (kQmCols * 4 + kQmCols * 5) * 4;
    static constexpr int per_sm = NK <= 4 ? 2 : 1;
    static constexpr int tiles2 = NK * kNT2;                                // W tiles
    static constexpr int per_warp = (tiles2 + 7) / 8;
};

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(unsigned int* r, const __half* p) {
    const unsigned int a = (unsigned int)__cvta_generic_to_shared(p);
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}

// 2^e as a double, -1022 <= e <= 1023
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// v 2^e: the words' bits taken as 2^52 + 2^31 + hi and 2^52 + lo, the offsets removed by the two
// multiply-adds (the first is exact)
__device__ __forceinline__ double fixed_double(long long v, int e) {
    const double hi = __hiloint2double(0x43300000, (int)(v >> 32) ^ (int)0x80000000);
    const double lo = __hiloint2double(0x43300000, (int)v);
    // -(2^52 + 2^31 + 2^20) 2^(32 + e)
    const double off = __hiloint2double((int)0xc3300000 + ((32 + e) << 20), (int)0x80100000);
    return fma(lo, pow2d(e), fma(hi, pow2d(32 + e), off));
}

// columns: (target, patch, slot, 1 = own patch)
template <int NK>
__global__ void __launch_bounds__(kQmThreads, QmShape<NK>::per_sm)
k_qm(const int4* __restrict__ items, const int4* __restrict__ cols, const __half* __restrict__ dig,
     const double2* __restrict__ pt, int n, int eB, const double* __restrict__ x,
     const double* __restrict__ J, const double* __restrict__ nself, const double* __restrict__ nrm,
     const double* __restrict__ H, double* __restrict__ partial) {
    using S = QmShape<NK>;
    extern __shared__ __align__(16) unsigned char smem[];
    __half* sB = reinterpret_cast<__half*>(smem);                                  // [digit][point][bstride]
    unsigned int* sX = reinterpret_cast<unsigned int*>(smem + S::b_bytes);         // [digit][ntile][k-step][lane][2]
    unsigned int* sF = reinterpret_cast<unsigned int*>(smem + S::b_bytes + S::x_bytes);  // [digit][ntile][k-step][kFStride]
    double* sY = reinterpret_cast<double*>(sF);                                    // [column 4 + field][kYStride]
    int* sEx = reinterpret_cast<int*>(smem + S::b_bytes + S::x_bytes + S::f_bytes);
    int* sEf = sEx + kQmCols * 4;
    static_assert(sizeof(double) * kQmCols * 4 * kYStride <= S::f_bytes, "Y shares F's storage");
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, g = lane >> 2, t4 = lane & 3;
    const int4 it = items[blockIdx.x];                // first tile, tiles, first column, columns
    const int4 col = cols[it.z + min(w, it.w - 1)];   // a missing column repeats the last one
    const int i = col.x;

    // this warp's column: the fields' digits
    {
        const double xi[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
        const size_t P0 = (size_t)col.y * n;
        for (int f = 0; f < 4; ++f) {
            const int cidx = w * 4 + f, nt = cidx >> 3, cg = cidx & 7;
            int top = 0;
            for (int k = lane; k < n; k += 32) {
                const double v = f < 3 ? x[3 * (P0 + k) + f] - xi[f] : J[P0 + k];
                top = max(top, (__double2hiint(v) >> 20) & 0x7ff);
            }
            top = __reduce_max_sync(0xffffffffu, top);
            top = max(top, 64);
            if (lane == 0) sEx[cidx] = top - 1022;
            for (int kp = lane; kp < S::np / 2; kp += 32) {
                unsigned long long v[2];
                for (int h = 0; h < 2; ++h) {
                    const int k = 2 * kp + h;
                    double d = 0.0;
                    if (k < n) d = f < 3 ? x[3 * (P0 + k) + f] - xi[f] : J[P0 + k];
                    v[h] = qm_fixed(d, top, 1);      // a bit for |Y| > 2^ex
                }
                const int ks = kp >> 3, l = kp & 7;
                for (int d = 0; d < kQmDigits; ++d)
                    sX[(((d * kNT1 + nt) * NK + ks) * 32 + cg * 4 + (l & 3)) * 2 + (l >> 2)] =
                        qm_digit2(v[0], v[1], d);
            }
        }
    }
    const double* np_ = col.w ? nself : nrm;
    const double n0 = np_[3 * i], n1 = np_[3 * i + 1], n2 = np_[3 * i + 2], Hi = H[i];

    double out[S::per_warp][4];
#pragma unroll
    for (int k = 0; k < S::per_warp; ++k)
        for (int c = 0; c < 4; ++c) out[k][c] = 0.0;

    for (int tile = it.x; tile < it.x + it.y; ++tile) {
        __syncthreads();                              // sB, sF of the previous tile are read
        {
            const uint4* src = reinterpret_cast<const uint4*>(dig + (size_t)tile * kQmDigits * kQmPts * S::np);
            constexpr int per_row = S::np / 8;
            for (int e = tid; e < kQmDigits * kQmPts * per_row; e += kQmThreads) {
                const int row = e / per_row, c = e - row * per_row;
                const unsigned int dst = (unsigned int)__cvta_generic_to_shared(sB + row * S::bstride + c * 8);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + e));
            }
            asm volatile("cp.async.commit_group;");
            asm volatile("cp.async.wait_group 0;");
        }
        const double2 pw0 = pt[(size_t)tile * kQmPts + 2 * lane], pw1 = pt[(size_t)tile * kQmPts + 2 * lane + 1];
        __syncthreads();

        // Y: warp w takes points 16 (w & 3).. of n-tiles 2 (w >> 2), 2 (w >> 2) + 1
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const int nt = 2 * (w >> 2) + h, m0 = 16 * (w & 3);
            float acc[kQmSums][4];
#pragma unroll
            for (int d = 0; d < kQmSums; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.f;
#pragma unroll 1
            for (int ks = 0; ks < NK; ++ks) {
                unsigned int a[kQmDigits][4];
                uint2 b[kQmDigits];
#pragma unroll
                for (int d = 0; d < kQmDigits; ++d) {
                    ldmatrix4<false>(a[d], sB + (d * kQmPts + m0 + (lane & 15)) * S::bstride + ks * 16 + (lane >> 4) * 8);
                    b[d] = *reinterpret_cast<const uint2*>(sX + (((d * kNT1 + nt) * NK + ks) * 32 + lane) * 2);
                }
#pragma unroll
                for (int da = 0; da < kQmDigits; ++da)
#pragma unroll
                    for (int db = 0; da + db < kQmSums && db < kQmDigits; ++db)
                        qm_mma(acc[da + db], a[da], b[db]);
            }
            // sum over the digits' weights in units 512^-5, then to double: two exact steps
            const int c0 = nt * 8 + 2 * t4;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                long long v = (long long)__float2int_rn(acc[0][c]);
#pragma unroll
                for (int d = 1; d < kQmDigits; ++d) v = v * 512 + (long long)__float2int_rn(acc[d][c]);
                v += (__float2int_rn(acc[kQmDigits][c]) + 256) >> 9;
                const int cc = c0 + (c & 1), row = m0 + g + 8 * (c >> 1);
                const int sc = eB + sEx[cc] - 60;
                sY[cc * kYStride + row] = fixed_double(v, sc);
            }
        }
        __syncthreads();

        // F: column w, points 2 lane and 2 lane + 1
        double f[5][2];
        {
            const double2 d0 = *reinterpret_cast<const double2*>(sY + (w * 4 + 0) * kYStride + 2 * lane);
            const double2 d1 = *reinterpret_cast<const double2*>(sY + (w * 4 + 1) * kYStride + 2 * lane);
            const double2 d2 = *reinterpret_cast<const double2*>(sY + (w * 4 + 2) * kYStride + 2 * lane);
            const double2 jj = *reinterpret_cast<const double2*>(sY + (w * 4 + 3) * kYStride + 2 * lane);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const double a = h ? d0.y : d0.x, b = h ? d1.y : d1.x, c = h ? d2.y : d2.x;
                const double wj = (h ? pw1.x : pw0.x) * (h ? jj.y : jj.x);
                const double r2 = fma(a, a, fma(b, b, c * c));
                const double inv = pm_rcp64(r2);
                const double q = fma(n0, a, fma(n1, b, n2 * c)) * inv;       // -n.r / r^2
                f[0][h] = wj * (q * (q + Hi));
                const double gf = wj * inv;
                f[1][h] = gf * a;                                            // minus the integrand
                f[2][h] = gf * b;
                f[3][h] = gf * c;
                f[4][h] = wj * (pm_log64(r2) + (h ? pw1.y : pw0.y));
            }
        }
        __syncthreads();                              // every warp has read its Y
        {
            const int ks = lane >> 3, word = lane & 3, half = (lane >> 2) & 1;
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const int cidx = w * 5 + k, nt = cidx >> 3, cg = cidx & 7;
                int top = max((__double2hiint(f[k][0]) >> 20) & 0x7ff, (__double2hiint(f[k][1]) >> 20) & 0x7ff);
                top = max(__reduce_max_sync(0xffffffffu, top), 64);
                if (lane == 0) sEf[cidx] = top - 1022;
                const unsigned long long a = qm_fixed(f[k][0], top, 0), b = qm_fixed(f[k][1], top, 0);
#pragma unroll
                for (int d = 0; d < kQmDigits; ++d)
                    sF[((d * kNT2 + nt) * 4 + ks) * kFStride + (cg * 4 + word) * 2 + half] = qm_digit2(a, b, d);
            }
        }
        __syncthreads();

        // W += B^T F: tiles (16 nodes, 8 sums) dealt to the warps
#pragma unroll
        for (int k = 0; k < S::per_warp; ++k) {
            const int id = w + 8 * k;
            if (id < S::tiles2) {
                const int mt = id / kNT2, nt = id - mt * kNT2;
                float acc[kQmSums][4];
#pragma unroll
                for (int d = 0; d < kQmSums; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.f;
#pragma unroll 1
                for (int ks = 0; ks < kQmPts / 16; ++ks) {
                    unsigned int a[kQmDigits][4];
                    uint2 b[kQmDigits];
#pragma unroll
                    for (int d = 0; d < kQmDigits; ++d) {
                        // A = B^T: matrices (nodes 0-7 | 8-15) x (points 0-7 | 8-15), stored by point
                        ldmatrix4<true>(a[d], sB + (d * kQmPts + ks * 16 + (lane & 7) + 8 * (lane >> 4)) * S::bstride +
                                                  mt * 16 + 8 * ((lane >> 3) & 1));
                        b[d] = *reinterpret_cast<const uint2*>(sF + ((d * kNT2 + nt) * 4 + ks) * kFStride + lane * 2);
                    }
#pragma unroll
                    for (int da = 0; da < kQmDigits; ++da)
#pragma unroll
                        for (int db = 0; da + db < kQmSums && db < kQmDigits; ++db)
                            qm_mma(acc[da + db], a[da], b[db]);
                }
                // a tile's sum to 2^-52 of its largest term (58 bits), two exact steps
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    long long v = (long long)__float2int_rn(acc[0][c]);
#pragma unroll
                    for (int d = 1; d < kQmDigits - 1; ++d) v = v * 512 + (long long)__float2int_rn(acc[d][c]);
                    v += (__float2int_rn(acc[kQmDigits - 1][c]) + (__float2int_rn(acc[kQmDigits][c]) >> 9) + 256) >> 9;
                    const int ef = sEf[nt * 8 + 2 * t4 + (c & 1)];
                    double s = fixed_double(v, eB + ef - 52);
                    if (ef == 0x7ff - 1022) s = nan("");         // an infinite or undefined integrand
                    out[k][c] += s;
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < S::per_warp; ++k) {
        const int id = w + 8 * k;
        if (id < S::tiles2) {
            const int mt = id / kNT2, nt = id - mt * kNT2;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int node = mt * 16 + g + 8 * (c >> 1), cidx = nt * 8 + 2 * t4 + (c & 1);
                const int cc = cidx / 5, kind = cidx - cc * 5;
                if (node < n && cc < it.w) {
                    // the points' weights carry 1/(2 pi): lb needs 1/pi, the gradient's sign is
                    // turned, the logarithm is of r^2
                    const double v = kind == 0 ? 2.0 * out[k][c] : kind == 4 ? 0.5 * out[k][c] : -out[k][c];
                    partial[((size_t)cols[it.z + cc].z * 5 + kind) * n + node] = v;
                }
            }
        }
    }
}

// a near block's weights from its slots: red (block, first slot, slots)
__global__ void k_qm_reduce(int nout, int n, int nblk, const int* __restrict__ blk,
                            const int* __restrict__ slot0, const int* __restrict__ nslot,
                            const double* __restrict__ partial, double* __restrict__ W_lb,
                            double* __restrict__ W_g, double* __restrict__ W_k) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t per = (size_t)5 * n;
    if (e >= nout * per) return;
    const int o = (int)(e / per), r = (int)(e - o * per), kind = r / n, node = r - kind * n;
    const double* p = partial + (size_t)slot0[o] * per + r;
    double s = 0.0;
    for (int k = 0; k < nslot[o]; ++k) s += p[(size_t)k * per];
    const size_t b = (size_t)blk[o];
    if (kind == 0) W_lb[b * n + node] = s;
    else if (kind == 4) W_k[b * n + node] = s;
    else W_g[((size_t)(kind - 1) * nblk + b) * n + node] = s;
}

// The leaves of a batch by cell: a hash of the codes gives each its index and count, then every
// leaf finds a place among its cell's columns.  The order within a cell does not matter.
constexpr int kQmHash = 1 << 16;
__global__ void k_qm_cells(int nleaf, const int* __restrict__ codes, int* __restrict__ key,
                           int* __restrict__ cnt, int* __restrict__ where) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nleaf) return;
    const int c = codes[l] + 1;                              // 0 marks a free entry
    unsigned int h = (unsigned int)c * 2654435761u >> 16;
    for (int tries = 0; tries < kQmHash; ++tries, h = (h + 1) & (kQmHash - 1)) {
        const int old = atomicCAS(key + h, 0, c);
        if (old == 0 || old == c) {
            atomicAdd(cnt + h, 1);
            where[l] = (int)h;
            return;
        }
    }
    where[l] = -1;
}
__global__ void k_qm_place(int npairs, const int* __restrict__ blocks, const int* __restrict__ start,
                           const int* __restrict__ count, const int* __restrict__ where,
                           int* __restrict__ pos, const int* __restrict__ blk_row,
                           const int* __restrict__ blk_patch, int4* __restrict__ cols) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npairs) return;
    const int b = blocks[p], s0 = start[p];
    for (int k = 0; k < count[p]; ++k) {
        const int h = where[s0 + k];
        if (h < 0) continue;
        cols[atomicAdd(pos + h, 1)] = make_int4(blk_row[b], blk_patch[b], s0 + k, 0);
    }
}

template <int NK>
pm_status launch(const pm_surface* s, int nitems, const int4* items, const int4* cols,
                 const QmTable& T, double* partial) {
    PM_CUDA_TRY(cudaFuncSetAttribute(k_qm<NK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)QmShape<NK>::bytes));
    k_qm<NK><<<nitems, kQmThreads, QmShape<NK>::bytes>>>(items, cols, T.dig, T.pt, T.n, T.eB, s->x,
                                                         s->J, s->npatch_n, s->n, s->H, partial);
    PM_CUDA_TRY(cudaGetLastError());
    return PM_OK;
}

pm_status run(const pm_surface* s, int nitems, const int4* items, const int4* cols,
              const QmTable& T, double* partial) {
    switch (T.npad / 16) {
        case 1: return launch<1>(s, nitems, items, cols, T, partial);
        case 2: return launch<2>(s, nitems, items, cols, T, partial);
        case 3: return launch<3>(s, nitems, items, cols, T, partial);
        case 4: return launch<4>(s, nitems, items, cols, T, partial);
        case 5: return launch<5>(s, nitems, items, cols, T, partial);
        case 6: return launch<6>(s, nitems, items, cols, T, partial);
        case 7: return launch<7>(s, nitems, items, cols, T, partial);
        case 8: return launch<8>(s, nitems, items, cols, T, partial);
    }
    pm_set_error("near-field weights: %d nodes a patch are not supported", T.n);
    return PM_ERR_INTERNAL;
}

// device buffers of one build, given back together
struct Buffers {
    std::vector<void*> p;
    ~Buffers() {
        for (void* q : p) cudaFree(q);
    }
    template <typename T>
    pm_status get(T** d, size_t count) {
        PM_TRY(pm_dmalloc(d, count));
        p.push_back(*d);
        return PM_OK;
    }
};

// Room for a batch's table and slots.  Larger batches leave fewer half-empty last waves; these
// keep what a build takes beside its results below 0.4 GB.  On a device without that much left
// the batches are halved, up to five times, which cuts the self rules into other pieces: the weights
// change by rounding alone (2e-15 of the largest).
constexpr size_t kTableBytes = 192u << 20, kSlotBytes = 128u << 20;

}  // namespace

namespace {

pm_status weights(pm_surface* s, const QmRules& R, int eB, int halved, bool* over);

}  // namespace

pm_status pm_quad_weights(pm_surface* s, const QmRules& R) {
    // the tables' power of two: three times the largest basis value at the whole cell's Gauss
    // points (the rules reach a little closer to its corners); more if a value passes that all
    // the same, as it may for triangle nodes of the caller's own choice
    unsigned int top = 0;
    {
        Buffers B;
        QmTable T;
        T.n = R.n;
        T.npad = (R.n + 15) / 16 * 16;
        int* whole = nullptr;
        PM_TRY(B.get(&T.top, 1));
        PM_TRY(B.get(&whole, 1));
        PM_CUDA_TRY(cudaMemset(T.top, 0, sizeof(int)));
        PM_CUDA_TRY(cudaMemset(whole, 0, sizeof(int)));      // code 0: the whole cell
        PM_TRY(R.near_table(whole, 1, T));
        PM_CUDA_TRY(cudaMemcpy(&top, T.top, sizeof(top), cudaMemcpyDeviceToHost));
    }
    float ftop = 0.f;
    std::memcpy(&ftop, &top, sizeof(ftop));
    int eB = (int)std::ceil(std::log2(std::min(1e30, std::max(1.0, 3.0 * (double)ftop))));
    int halved = 0;
    for (;;) {
        bool over = false;
        const pm_status st = weights(s, R, eB, halved, &over);
        if (st == PM_ERR_OOM && halved < 5) {
            cudaGetLastError();
            ++halved;
            continue;
        }
        PM_TRY(st);
        if (!over) return PM_OK;
        eB += 3;
        if (eB > 200) {
            pm_set_error("near-field weights: basis values above 2^%d", eB);
            return PM_ERR_INTERNAL;
        }
    }
}

namespace {

pm_status weights(pm_surface* s, const QmRules& R, int eB, int halved, bool* over) {
    const int n = R.n, npatch = s->npatch;
    QmTable T;
    T.n = n;
    T.npad = (n + 15) / 16 * 16;
    T.eB = eB;
    const size_t tile_bytes = (size_t)kQmDigits * kQmPts * T.npad * 2 + kQmPts * sizeof(double2);
    int max_loc = 0;
    for (int l = 0; l < n; ++l) max_loc = std::max(max_loc, R.tiles[l + 1] - R.tiles[l]);
    const int cap_tiles = std::max<int>(std::max(max_loc, R.near_tiles), (int)((kTableBytes >> halved) / tile_bytes));
    const int cap_slots = (int)std::max<size_t>(4096, (kSlotBytes >> halved) / (5 * (size_t)n * sizeof(double)));
    Buffers B;
    double* partial = nullptr;
    PM_TRY(B.get(&T.dig, (size_t)cap_tiles * kQmDigits * kQmPts * T.npad));
    PM_TRY(B.get(&T.pt, (size_t)cap_tiles * kQmPts));
    PM_TRY(B.get(&T.over, 1));
    PM_CUDA_TRY(cudaMemset(T.over, 0, sizeof(int)));
    PM_TRY(B.get(&partial, (size_t)cap_slots * 5 * n));
    int4 *items = nullptr, *cols = nullptr;
    int *out_blk = nullptr, *out_slot = nullptr, *out_n = nullptr;
    PM_TRY(B.get(&items, cap_slots));
    PM_TRY(B.get(&cols, cap_slots));
    PM_TRY(B.get(&out_blk, cap_slots));
    PM_TRY(B.get(&out_slot, cap_slots));
    PM_TRY(B.get(&out_n, cap_slots));

    std::vector<int> rp(s->N + 1);
    PM_CUDA_TRY(cudaMemcpy(rp.data(), s->row_ptr, sizeof(int) * rp.size(), cudaMemcpyDeviceToHost));
    std::vector<int4> hi, hc;
    std::vector<int> ob, os, on;
    auto reduce = [&]() -> pm_status {
        const int nout = (int)ob.size();
        PM_CUDA_TRY(cudaMemcpyAsync(out_blk, ob.data(), sizeof(int) * nout, cudaMemcpyHostToDevice));
        PM_CUDA_TRY(cudaMemcpyAsync(out_slot, os.data(), sizeof(int) * nout, cudaMemcpyHostToDevice));
        PM_CUDA_TRY(cudaMemcpyAsync(out_n, on.data(), sizeof(int) * nout, cudaMemcpyHostToDevice));
        k_qm_reduce<<<pm_ceil_div((long long)nout * 5 * n, 256), 256>>>(
            nout, n, s->nblk, out_blk, out_slot, out_n, partial, s->W_lb, s->W_g, s->W_k);
        PM_CUDA_TRY(cudaGetLastError());
        return PM_OK;
    };

    // ---- self rules: the node positions of a batch share the table; each takes every patch in
    // groups of kQmCols, its tiles cut into pieces until the device has about four blocks a slot
    const int ngroup = pm_ceil_div(npatch, kQmCols);
    const int want = 4 * s->ctx->num_sms * (T.npad <= 64 ? 2 : 1);
    for (int l0 = 0; l0 < n;) {
        int l1 = l0 + 1;
        while (l1 < n && R.tiles[l1 + 1] - R.tiles[l0] <= cap_tiles) ++l1;
        PM_TRY(R.self_table(l0, l1 - l0, T));
        const int pieces = std::max(1, std::min({max_loc / 4, pm_ceil_div(want, (long long)ngroup * (l1 - l0)),
                                                 cap_slots / ((l1 - l0) * kQmCols)}));
        // patches at a time that the slots hold (all but on very large surfaces)
        const int gstep = std::max(1, (int)std::min<long long>(ngroup, cap_slots / ((long long)(l1 - l0) * pieces * kQmCols)));
        for (int g0 = 0; g0 < ngroup; g0 += gstep) {
            const int p0 = g0 * kQmCols, p1 = std::min(npatch, (g0 + gstep) * kQmCols);
            hi.clear(); hc.clear(); ob.clear(); os.clear(); on.clear();
            int slot = 0;
            for (int l = l0; l < l1; ++l) {
                const int nt = R.tiles[l + 1] - R.tiles[l], np = std::min(pieces, nt);
                for (int q0 = p0; q0 < p1; q0 += kQmCols) {
                    const int m = std::min(kQmCols, p1 - q0);
                    for (int c = 0; c < m; ++c) {
                        ob.push_back(rp[(q0 + c) * n + l]);
                        os.push_back(slot + c * np);
                        on.push_back(np);
                    }
                    for (int k = 0; k < np; ++k) {
                        const int a = (int)((long long)nt * k / np), b = (int)((long long)nt * (k + 1) / np);
                        hi.push_back(make_int4(R.tiles[l] - R.tiles[l0] + a, b - a, (int)hc.size(), m));
                        for (int c = 0; c < m; ++c)
                            hc.push_back(make_int4((q0 + c) * n + l, q0 + c, slot + c * np + k, 1));
                    }
                    slot += m * np;
                }
            }
            if (slot > cap_slots) {
                pm_set_error("near-field weights: %d slots wanted, %d held", slot, cap_slots);
                return PM_ERR_INTERNAL;
            }
            PM_CUDA_TRY(cudaMemcpyAsync(items, hi.data(), sizeof(int4) * hi.size(), cudaMemcpyHostToDevice));
            PM_CUDA_TRY(cudaMemcpyAsync(cols, hc.data(), sizeof(int4) * hc.size(), cudaMemcpyHostToDevice));
            PM_TRY(run(s, (int)hi.size(), items, cols, T, partial));
            PM_TRY(reduce());
            PM_CUDA_TRY(cudaDeviceSynchronize());          // the host lists are rebuilt
        }
        l0 = l1;
    }

    // ---- near rules: (target, patch) blocks in batches whose leaves fit the slots; the leaves
    // are grouped by cell, a cell's columns in groups of kQmCols
    std::vector<int> near;
    for (int i = 0; i < s->N; ++i)
        for (int b = rp[i] + 1; b < rp[i + 1]; ++b) near.push_back(b);
    auto passed = [&]() -> pm_status {
        int o = 0;
        PM_CUDA_TRY(cudaMemcpy(&o, T.over, sizeof(int), cudaMemcpyDeviceToHost));
        *over = o != 0;
        return PM_OK;
    };
    if (near.empty()) return passed();
    int *blocks = nullptr, *start = nullptr, *count = nullptr, *codes = nullptr, *where = nullptr,
        *key = nullptr, *cnt = nullptr, *used = nullptr, *cells = nullptr;
    const int max_pairs = cap_slots / 4;
    PM_TRY(B.get(&blocks, max_pairs));
    PM_TRY(B.get(&start, max_pairs));
    PM_TRY(B.get(&count, max_pairs));
    PM_TRY(B.get(&codes, cap_slots));
    PM_TRY(B.get(&where, cap_slots));
    PM_TRY(B.get(&key, kQmHash));
    PM_TRY(B.get(&cnt, kQmHash));
    PM_TRY(B.get(&cells, kQmHash));
    PM_TRY(B.get(&used, 1));
    std::vector<int> hstart(max_pairs), hcount(max_pairs), hkey(kQmHash), hcnt(kQmHash), hpos(kQmHash), hcells;
    size_t at = 0;
    int take = std::max(1, std::min(max_pairs, cap_slots / 40));
    while (at < near.size()) {
        const int np = (int)std::min<size_t>(take, near.size() - at);
        PM_CUDA_TRY(cudaMemcpy(blocks, near.data() + at, sizeof(int) * np, cudaMemcpyHostToDevice));
        PM_CUDA_TRY(cudaMemset(used, 0, sizeof(int)));
        PM_TRY(R.leaves(blocks, np, start, count, codes, cap_slots, used));
        int nleaf = 0;
        PM_CUDA_TRY(cudaMemcpy(&nleaf, used, sizeof(int), cudaMemcpyDeviceToHost));
        if (nleaf > cap_slots) {                           // more leaves than slots: fewer blocks
            if (np == 1) {
                pm_set_error("near-field weights: %d leaves of one block", nleaf);
                return PM_ERR_INTERNAL;
            }
            take = std::max(1, std::min(np / 2, (int)((long long)np * cap_slots / nleaf * 9 / 10)));
            continue;
        }
        PM_CUDA_TRY(cudaMemset(key, 0, sizeof(int) * kQmHash));
        PM_CUDA_TRY(cudaMemset(cnt, 0, sizeof(int) * kQmHash));
        k_qm_cells<<<pm_ceil_div(nleaf, 256), 256>>>(nleaf, codes, key, cnt, where);
        PM_CUDA_TRY(cudaGetLastError());
        PM_CUDA_TRY(cudaMemcpy(hkey.data(), key, sizeof(int) * kQmHash, cudaMemcpyDeviceToHost));
        PM_CUDA_TRY(cudaMemcpy(hcnt.data(), cnt, sizeof(int) * kQmHash, cudaMemcpyDeviceToHost));
        PM_CUDA_TRY(cudaMemcpy(hstart.data(), start, sizeof(int) * np, cudaMemcpyDeviceToHost));
        PM_CUDA_TRY(cudaMemcpy(hcount.data(), count, sizeof(int) * np, cudaMemcpyDeviceToHost));
        hcells.clear();
        int c0 = 0;
        std::vector<std::pair<int, int>> cell_cols;        // first column and count by cell
        for (int h = 0; h < kQmHash; ++h) {
            hpos[h] = c0;
            if (!hcnt[h]) continue;
            hcells.push_back(hkey[h] - 1);
            cell_cols.emplace_back(c0, hcnt[h]);
            c0 += hcnt[h];
        }
        if (c0 != nleaf) {                                 // more different cells than kQmHash
            if (np == 1) {
                pm_set_error("near-field weights: more than %d different cells in a block", kQmHash);
                return PM_ERR_INTERNAL;
            }
            take = np / 2;
            continue;
        }
        PM_CUDA_TRY(cudaMemcpy(cnt, hpos.data(), sizeof(int) * kQmHash, cudaMemcpyHostToDevice));
        k_qm_place<<<pm_ceil_div(np, 128), 128>>>(np, blocks, start, count, where, cnt, s->blk_row,
                                                  s->blk_patch, cols);
        PM_CUDA_TRY(cudaGetLastError());
        const int per = cap_tiles / R.near_tiles;
        for (size_t q0 = 0; q0 < hcells.size(); q0 += per) {
            const int nc = (int)std::min<size_t>(per, hcells.size() - q0);
            PM_CUDA_TRY(cudaMemcpyAsync(cells, hcells.data() + q0, sizeof(int) * nc, cudaMemcpyHostToDevice));
            PM_TRY(R.near_table(cells, nc, T));
            hi.clear();
            for (int c = 0; c < nc; ++c) {
                const auto& cc = cell_cols[q0 + c];
                for (int k = 0; k < cc.second; k += kQmCols)
                    hi.push_back(make_int4(c * R.near_tiles, R.near_tiles, cc.first + k,
                                           std::min(kQmCols, cc.second - k)));
            }
            PM_CUDA_TRY(cudaMemcpyAsync(items, hi.data(), sizeof(int4) * hi.size(), cudaMemcpyHostToDevice));
            PM_TRY(run(s, (int)hi.size(), items, cols, T, partial));
            PM_CUDA_TRY(cudaDeviceSynchronize());
        }
        ob.assign(near.begin() + at, near.begin() + at + np);
        os.assign(hstart.begin(), hstart.begin() + np);
        on.assign(hcount.begin(), hcount.begin() + np);
        PM_TRY(reduce());
        PM_CUDA_TRY(cudaDeviceSynchronize());
        at += np;
        take = std::max(1, std::min(max_pairs, (int)((double)np * cap_slots / std::max(1, nleaf) * 0.9)));
    }
    return passed();
}

}  // namespace
