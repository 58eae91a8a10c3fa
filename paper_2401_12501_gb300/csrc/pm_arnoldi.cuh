// Arnoldi steps of the float64 solvers with a host-side Hessenberg system (pm_helm.cu complex,
// pm_bvp.cu real): classical Gram-Schmidt applied twice and the normalisation, all on the
// device, so that a step's coefficients travel to the host while the next step already runs.
//   dots, subtract, dots, subtract (with |w|^2), next basis vector
// Each kernel sums its predecessor's per-block partials itself, in a fixed order: no separate
// reductions, and results that do not depend on timing.  Bound by launch latency at the sizes
// solved here (a few thousand unknowns): five launches of 3-5 us a step.
#pragma once

#include "pm_internal.cuh"

#include <algorithm>

namespace pm_arnoldi {

constexpr int kThreads = 256;
constexpr int kPerBlock = 1024;      // elements a block of the dots

__device__ __forceinline__ double cdot(double a, double b) { return a * b; }
__device__ __forceinline__ double2 cdot(double2 a, double2 b) {      // conj(a) b
    return make_double2(fma(a.x, b.x, a.y * b.y), fma(a.x, b.y, -a.y * b.x));
}
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double2 add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double submul(double acc, double v, double h) { return fma(-v, h, acc); }
__device__ __forceinline__ double2 submul(double2 acc, double2 v, double2 h) {
    return make_double2(fma(-v.x, h.x, fma(v.y, h.y, acc.x)), fma(-v.x, h.y, fma(-v.y, h.x, acc.y)));
}
__device__ __forceinline__ double norm2(double a) { return a * a; }
__device__ __forceinline__ double norm2(double2 a) { return fma(a.x, a.x, a.y * a.y); }
__device__ __forceinline__ double scaled(double a, double s) { return a * s; }
__device__ __forceinline__ double2 scaled(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double down(double v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double2 down(double2 v, int o) {
    return make_double2(__shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o));
}

// sum over the block, valid in thread 0
template <typename T>
__device__ __forceinline__ T block_add(T v, T* sh) {
    for (int o = 16; o > 0; o >>= 1) v = add(v, down(v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 1; k < kThreads / 32; ++k) v = add(v, sh[k]);
    return v;
}

// part[j][b] = conj(V_j) . w over block b's elements
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_dots(const T* __restrict__ V, long long ldv, const T* __restrict__ w, int n, T* __restrict__ part) {
    __shared__ T sh[kThreads / 32];
    const T* v = V + blockIdx.y * ldv;
    T acc{};
    const int e1 = min(n, (int)(blockIdx.x + 1) * kPerBlock);
    for (int i = blockIdx.x * kPerBlock + threadIdx.x; i < e1; i += kThreads) acc = add(acc, cdot(v[i], w[i]));
    acc = block_add(acc, sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = acc;
}

// h_j = sum_b part[j][b] (block 0 keeps them), w -= sum_j V_j h_j; nrm[block] = |w|^2 of its share
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_subtract(const T* __restrict__ V, long long ldv, int ncols, const T* __restrict__ part, int nparts,
           T* __restrict__ hout, T* __restrict__ w, int n, double* __restrict__ nrm) {
    extern __shared__ __align__(16) unsigned char smem[];
    T* h = reinterpret_cast<T*>(smem);
    __shared__ double sh[kThreads / 32];
    for (int j = threadIdx.x; j < ncols; j += kThreads) {
        T s = part[(size_t)j * nparts];
        for (int b = 1; b < nparts; ++b) s = add(s, part[(size_t)j * nparts + b]);
        h[j] = s;
        if (blockIdx.x == 0) hout[j] = s;
    }
    __syncthreads();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    double q = 0.0;
    if (i < n) {
        T acc = w[i];
#pragma unroll 4
        for (int j = 0; j < ncols; ++j) acc = submul(acc, V[j * ldv + i], h[j]);
        w[i] = acc;
        q = norm2(acc);
    }
    if (nrm) {
        q = block_add(q, sh);
        if (threadIdx.x == 0) nrm[blockIdx.x] = q;
    }
}

// *hn = sqrt(sum of the blocks' squares), next = w / *hn
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_next(const T* __restrict__ w, int n, const double* __restrict__ nrm, int nblk,
       T* __restrict__ next, double* __restrict__ hn) {
    __shared__ double sh[kThreads / 32];
    __shared__ double inv;
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += kThreads) s += nrm[b];
    s = block_add(s, sh);
    if (threadIdx.x == 0) {
        const double r = sqrt(s);
        inv = r > 0.0 ? 1.0 / r : 0.0;
        if (blockIdx.x == 0) *hn = r;
    }
    __syncthreads();
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i < n) next[i] = scaled(w[i], inv);
}

// x += sum_j V_j y_j
template <typename T>
__global__ void __launch_bounds__(kThreads)
k_combine(const T* __restrict__ V, long long ldv, int ncols, const T* __restrict__ y, T* __restrict__ x,
          int n) {
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    T acc = x[i];
#pragma unroll 4
    for (int j = 0; j < ncols; ++j) acc = submul(acc, V[j * ldv + i], scaled(y[j], -1.0));
    x[i] = acc;
}

// Scratch and pinned host copies of the steps' coefficients; two steps may be in flight.
// Slot k & 1 holds step k's 2 (k + 1) coefficients (first pass, second pass) and |w|.
template <typename T>
struct Steps {
    int n = 0, m = 0, nparts = 0, nblk = 0;
    T *part = nullptr, *dev = nullptr, *host = nullptr;      // dev, host: [2][2 (m + 1) + 1]
    double* nrm = nullptr;
    cudaEvent_t ev[2] = {nullptr, nullptr};

    size_t slot() const { return 2 * (size_t)(m + 1) + 1; }
    pm_status create(int n_, int m_) {
        n = n_;
        m = m_;
        nparts = pm_ceil_div(n, kPerBlock);
        nblk = pm_ceil_div(n, kThreads);
        PM_TRY(pm_dmalloc(&part, (size_t)nparts * (m + 1)));
        PM_TRY(pm_dmalloc(&dev, 2 * slot()));
        PM_TRY(pm_dmalloc(&nrm, nblk));
        PM_CUDA_TRY(cudaMallocHost((void**)&host, sizeof(T) * 2 * slot()));
        for (cudaEvent_t& e : ev) PM_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
        return PM_OK;
    }
    void release() {
        pm_dfree(part);
        pm_dfree(dev);
        pm_dfree(nrm);
        if (host) cudaFreeHost(host);
        host = nullptr;
        for (cudaEvent_t& e : ev) {
            if (e) cudaEventDestroy(e);
            e = nullptr;
        }
    }
    // V_0 = r / |r|, and |r| (waits for it), NaN or infinite where r is or its squares overflow: a
    // solve that met one has not converged
    pm_status begin(T* r, T* V0, cudaStream_t st, double* beta) {
        k_subtract<T><<<nblk, kThreads, 0, st>>>(nullptr, 0, 0, nullptr, 0, nullptr, r, n, nrm);
        k_next<T><<<nblk, kThreads, 0, st>>>(r, n, nrm, nblk, V0, reinterpret_cast<double*>(dev));
        PM_CUDA_TRY(cudaGetLastError());
        PM_CUDA_TRY(cudaMemcpyAsync(host, dev, sizeof(double), cudaMemcpyDeviceToHost, st));
        PM_CUDA_TRY(cudaStreamSynchronize(st));
        *beta = *reinterpret_cast<const double*>(host);
        return PM_OK;
    }
    // x += sum_{j < k} V_j y_j with y on the host (the stream's earlier steps have been waited for,
    // or keep to the other slot)
    pm_status combine(const T* V, long long ldv, int k, const T* y, T* x, cudaStream_t st) {
        const size_t o = (size_t)((k - 1) & 1) * slot();      // the slot of the last step taken
        std::copy(y, y + k, host + o);
        PM_CUDA_TRY(cudaMemcpyAsync(dev + o, host + o, sizeof(T) * k, cudaMemcpyHostToDevice, st));
        k_combine<T><<<nblk, kThreads, 0, st>>>(V, ldv, k, dev + o, x, n);
        PM_CUDA_TRY(cudaGetLastError());
        return PM_OK;
    }
    // orthogonalise w = A V_k against V_0..V_k into V_{k+1}, the coefficients on their way to the host
    pm_status step(T* V, long long ldv, int k, T* w, cudaStream_t st) {
        T* d = dev + (k & 1) * slot();
        const dim3 grid(nparts, k + 1);
        const size_t smem = sizeof(T) * (k + 1);
        k_dots<T><<<grid, kThreads, 0, st>>>(V, ldv, w, n, part);
        k_subtract<T><<<nblk, kThreads, smem, st>>>(V, ldv, k + 1, part, nparts, d, w, n, nullptr);
        k_dots<T><<<grid, kThreads, 0, st>>>(V, ldv, w, n, part);
        k_subtract<T><<<nblk, kThreads, smem, st>>>(V, ldv, k + 1, part, nparts, d + (k + 1), w, n, nrm);
        k_next<T><<<nblk, kThreads, 0, st>>>(w, n, nrm, nblk, V + (size_t)(k + 1) * ldv,
                                             reinterpret_cast<double*>(d + 2 * (k + 1)));
        PM_CUDA_TRY(cudaGetLastError());
        PM_CUDA_TRY(cudaMemcpyAsync(host + (k & 1) * slot(), d, sizeof(T) * (2 * (size_t)(k + 1) + 1),
                                    cudaMemcpyDeviceToHost, st));
        PM_CUDA_TRY(cudaEventRecord(ev[k & 1], st));
        return PM_OK;
    }
    // wait for step k; its coefficients h_j = c[j] + c[k + 1 + j] and |w|, 0 where it is undefined,
    // which ends the cycle
    pm_status wait(int k, const T** c, double* hn) {
        PM_CUDA_TRY(cudaEventSynchronize(ev[k & 1]));
        *c = host + (k & 1) * slot();
        const double norm = *reinterpret_cast<const double*>(*c + 2 * (k + 1));
        *hn = norm > 0.0 ? norm : 0.0;
        return PM_OK;
    }
};

}  // namespace pm_arnoldi
