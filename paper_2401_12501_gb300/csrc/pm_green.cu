// Host entry point of the c != 0 Green's function evaluators (pm_green.cuh):
// lets the host-side tests compare the library's own g, g', g'' with an
// independent evaluation before any device kernel uses them.

#include "pm_internal.cuh"
#include "pm_green.cuh"

#include <cmath>

extern "C" pm_status pm_selftest_green(const double* r, int n, double q, double* out) {
    if (!r || !out || n < 0 || !std::isfinite(q) || q == 0.0) {
        pm_set_error("pm_selftest_green: NULL array, negative n, or q not finite and non-zero");
        return PM_ERR_INVALID_ARG;
    }
    for (int i = 0; i < n; ++i)
        if (!(r[i] > 0.0) || !std::isfinite(r[i])) {
            pm_set_error("pm_selftest_green: r must be finite and positive");
            return PM_ERR_INVALID_ARG;
        }
    for (int i = 0; i < n; ++i) pm_green::green_scaled(r[i], q, out + 6 * i);
    return PM_OK;
}

extern "C" pm_status pm_selftest_green_c(const double* r, int n, double q_re, double q_im,
                                         double* out) {
    if (!r || !out || n < 0 || !std::isfinite(q_re) || !std::isfinite(q_im) ||
        (q_re == 0.0 && q_im == 0.0)) {
        pm_set_error("pm_selftest_green_c: NULL array, negative n, or q not finite and non-zero");
        return PM_ERR_INVALID_ARG;
    }
    for (int i = 0; i < n; ++i)
        if (!(r[i] > 0.0) || !std::isfinite(r[i])) {
            pm_set_error("pm_selftest_green_c: r must be finite and positive");
            return PM_ERR_INVALID_ARG;
        }
    QuadTables T;
    pm_build_tables(2, &T);
    for (int i = 0; i < n; ++i) {
        if (q_im == 0.0)
            pm_green::green_scaled(r[i], q_re, out + 6 * i);
        else
            pm_green::green_scaled_cz(r[i], pm_green::cplx_d{q_re, q_im}, T.g16t, T.g16w, out + 6 * i);
    }
    return PM_OK;
}

extern "C" pm_status pm_selftest_green_f32(const float* r, int n, float q, float* out) {
    if (!r || !out || n < 0 || !std::isfinite(q) || q == 0.0f) {
        pm_set_error("pm_selftest_green_f32: NULL array, negative n, or q not finite and non-zero");
        return PM_ERR_INVALID_ARG;
    }
    for (int i = 0; i < n; ++i)
        if (!(r[i] > 0.0f) || !std::isfinite(r[i])) {
            pm_set_error("pm_selftest_green_f32: r must be finite and positive");
            return PM_ERR_INVALID_ARG;
        }
    for (int i = 0; i < n; ++i) pm_green::green_scaled_f32(r[i], q, out + 6 * i);
    return PM_OK;
}

extern "C" pm_status pm_selftest_smooth_c_f32(int N, const float* x, const float* n,
                                              const float* H, const float* a, const float* gb,
                                              const float* c, const float* s, double* out) {
    if (N < 0 || !x || !n || !H || !a || !gb || !c || !s || !out) {
        pm_set_error("pm_selftest_smooth_c_f32: NULL array or negative N");
        return PM_ERR_INVALID_ARG;
    }
    for (int i = 0; i < N; ++i)
        if (!(a[i] > 0.0f) || !std::isfinite(c[i]) || c[i] == 0.0f) {
            pm_set_error("pm_selftest_smooth_c_f32: a must be positive and c finite and non-zero");
            return PM_ERR_INVALID_ARG;
        }
    for (int i = 0; i < N; ++i) {
        double sum[4] = {0.0, 0.0, 0.0, 0.0};
        for (int j = 0; j < N; ++j) {
            if (j == i) continue;
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            pm_green::pair_rk_c_f32(x[3 * i] - x[3 * j], x[3 * i + 1] - x[3 * j + 1],
                                    x[3 * i + 2] - x[3 * j + 2], n[3 * i], n[3 * i + 1],
                                    n[3 * i + 2], H[i], a[i], gb[3 * i], gb[3 * i + 1],
                                    gb[3 * i + 2], c[i], c[j] / a[j], s[2 * j], s[2 * j + 1],
                                    acc);
            for (int m = 0; m < 4; ++m) sum[m] += acc[m];
        }
        for (int m = 0; m < 4; ++m) out[4 * i + m] = sum[m];
    }
    return PM_OK;
}

// ------------------------------------------------------------------ device smooth sums, c != 0
// One thread per target; sources (x, y, z, q = c/a) and s = w sigma / a staged
// through shared memory in stages of kCStage; every kCTile sources the partial
// is folded into a (hi, lo) pair with TwoSum, as in the c = 0 float32 sums.  The
// self pair j = i is skipped by index (the Hankel kernels have no removable
// value at r = 0).  Threads past N compute on a dummy target and write nothing.
namespace {

constexpr int kCThreads = 128;
constexpr int kCStage = 512;
constexpr int kCTile = 128;

__device__ __forceinline__ void two_sum_c(float& hi, float& lo, float v) {
    const float t = hi + v;
    const float bp = t - hi;
    lo += (hi - (t - bp)) + (v - bp);
    hi = t;
}

__global__ void __launch_bounds__(kCThreads)
k_smooth_c32(int N, const float* __restrict__ x, const float* __restrict__ n,
             const float* __restrict__ H, const float* __restrict__ a,
             const float* __restrict__ gb, const float* __restrict__ c,
             const float* __restrict__ s, double* __restrict__ out) {
    __shared__ float4 sp[kCStage];
    __shared__ float2 ss[kCStage];
    const int i = blockIdx.x * kCThreads + threadIdx.x;
    const bool live = i < N;
    float tx = 0.f, ty = 0.f, tz = 0.f, nx = 0.f, ny = 0.f, nz = 0.f, Hi = 0.f, ai = 1.f,
          gx = 0.f, gy = 0.f, gz = 0.f, ci = 0.f;
    if (live) {
        tx = x[3 * i]; ty = x[3 * i + 1]; tz = x[3 * i + 2];
        nx = n[3 * i]; ny = n[3 * i + 1]; nz = n[3 * i + 2];
        Hi = H[i]; ai = a[i]; ci = c[i];
        gx = gb[3 * i]; gy = gb[3 * i + 1]; gz = gb[3 * i + 2];
    }
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
    for (int base = 0; base < N; base += kCStage) {
        const int len = min(kCStage, N - base);
        __syncthreads();
        for (int j = threadIdx.x; j < len; j += kCThreads) {
            const int g = base + j;
            sp[j] = make_float4(x[3 * g], x[3 * g + 1], x[3 * g + 2], c[g] / a[g]);
            ss[j] = make_float2(s[2 * g], s[2 * g + 1]);
        }
        __syncthreads();
        for (int j0 = 0; j0 < len; j0 += kCTile) {
            const int j1 = min(j0 + kCTile, len);
            float part[4] = {0.f, 0.f, 0.f, 0.f};
            for (int j = j0; j < j1; ++j) {
                if (base + j == i) continue;
                const float4 p = sp[j];
                const float2 w = ss[j];
                pm_green::pair_rk_c_f32(tx - p.x, ty - p.y, tz - p.z, nx, ny, nz, Hi, ai, gx,
                                        gy, gz, ci, p.w, w.x, w.y, part);
            }
#pragma unroll
            for (int m = 0; m < 4; ++m) two_sum_c(hi[m], lo[m], part[m]);
        }
    }
    if (live) {
#pragma unroll
        for (int m = 0; m < 4; ++m) out[4 * (size_t)i + m] = (double)hi[m] + (double)lo[m];
    }
}

constexpr int kSmoothCMaxN = 1 << 26;

}  // namespace

extern "C" pm_status pm_smooth_c_f32(int N, const float* x, const float* n, const float* H,
                                     const float* a, const float* gb, const float* c,
                                     const float* s, double* out, void* stream) {
    if (N < 1 || N > kSmoothCMaxN) {
        pm_set_error("pm_smooth_c_f32: N = %d outside 1..%d", N, kSmoothCMaxN);
        return PM_ERR_INVALID_ARG;
    }
    if (!x || !n || !H || !a || !gb || !c || !s || !out) {
        pm_set_error("pm_smooth_c_f32: NULL argument");
        return PM_ERR_INVALID_ARG;
    }
    const int grid = (N + kCThreads - 1) / kCThreads;
    k_smooth_c32<<<grid, kCThreads, 0, (cudaStream_t)stream>>>(N, x, n, H, a, gb, c, s, out);
    PM_CUDA_TRY(cudaGetLastError());
    return PM_OK;
}

namespace {

using pm_green::cplx_d;
__constant__ double cG16[2 * PM_GL16];     // 16-point Gauss-Legendre nodes, weights

// Taylor coefficients a_2.. about c from a_0, a_1 by c (n+2)(n+1) a_{n+2} =
// s (c a_n + a_{n-1}) - (n+1)^2 a_{n+1}, s = 1 (K) or -1 (H)
__device__ void taylor(cplx_d c, double s, int terms, cplx_d* a) {
    const cplx_d ic = pm_green::cz_rcp(c);
    for (int n = 0; n + 2 < terms; ++n) {
        cplx_d v = pm_green::cz_mul(c, a[n]);
        if (n > 0) v = pm_green::cz_add(v, a[n - 1]);
        v = pm_green::cz_sub(pm_green::cz_scale(v, s), pm_green::cz_scale(a[n + 1], (n + 1.0) * (n + 1.0)));
        a[n + 2] = pm_green::cz_scale(pm_green::cz_mul(v, ic), 1.0 / ((n + 2.0) * (n + 1.0)));
    }
}

__global__ void k_green_rows(double2* __restrict__ k1, double2* __restrict__ h1) {
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= pm_green::kTabRows) return;
    const int oct = row >> 3;
    const double z = oct < pm_green::kTabOctaves
                         ? ldexp(1.0 + ((row & 7) + 0.5) / 8.0, oct + pm_green::kTabLow)
                         : row - pm_green::kTabOctaves * 8 + 16.5;
    cplx_d a[15];
    double K0, K1;
    pm_green::bessel_k01(z, &K0, &K1);
    a[0] = {K0, 0.0};
    a[1] = {-K1, 0.0};
    taylor({z, 0.0}, 1.0, 15, a);
    k1[row * 8] = make_double2(z, a[0].re);
    for (int n = 1; n < 8; ++n) k1[row * 8 + n] = make_double2(a[2 * n - 1].re, a[2 * n].re);
    if (z < 8.0) {
        a[0] = {j0(z), y0(z)};
        a[1] = {-j1(z), -y1(z)};
    } else if (z >= 32.0) {
        // H_nu = sqrt(2 / (pi z)) e^{i (z - nu pi/2 - pi/4)} sum_k i^k a_k / z^k,
        // a_k = a_{k-1} (4 nu^2 - (2k - 1)^2) / (8k) (A&S 9.2.7); its smallest term is below e^{-2z}
        double sn, cs;
        sincos(z, &sn, &cs);
        const double m = sqrt(1.0 / (M_PI * z));              // times e^{i z} (1 - i) = e^{i (z - pi/4)} sqrt 2
        const cplx_d e = {m * (cs + sn), m * (sn - cs)};
        for (int nu = 0; nu < 2; ++nu) {
            cplx_d sum = {1.0, 0.0};
            double t = 1.0;
            for (int k = 1; k < 40; ++k) {
                t *= (4.0 * nu * nu - (2.0 * k - 1.0) * (2.0 * k - 1.0)) / (8.0 * k * z);
                if (fabs(t) < 1e-18) break;
                const double v = (k & 2) ? -t : t;            // i^k t
                if (k & 1) sum.im += v;
                else sum.re += v;
            }
            const cplx_d h = pm_green::cz_mul(e, sum);
            // e^{-i pi/2} turns H1; a_1 = H0' = -H1
            a[nu] = nu ? cplx_d{-h.im, h.re} : h;
        }
    } else {                            // H0 = (2 / (pi i)) K0(-i z), H1 = -(2 / pi) K1(-i z)
        cplx_d C0, C1;
        pm_green::bessel_k01_c({0.0, -z}, cG16, cG16 + PM_GL16, &C0, &C1);
        a[0] = {2.0 / M_PI * C0.im, -2.0 / M_PI * C0.re};
        a[1] = pm_green::cz_scale(C1, 2.0 / M_PI);
    }
    taylor({z, 0.0}, -1.0, 15, a);
    h1[row * 16] = make_double2(z, 0.0);
    for (int n = 0; n < 15; ++n) h1[row * 16 + 1 + n] = make_double2(a[n].re, a[n].im);
}

__global__ void k_green_cells(double2* __restrict__ c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pm_green::kTabCells) return;
    cplx_d c;
    double s;
    if (i < pm_green::kTabOctaves * 1024) {
        s = ldexp(1.0, (i >> 10) + pm_green::kTabLow - 3);
        c = {(((i >> 5) & 31) - 15.5) * s, ((i & 31) - 15.5) * s};
    } else {
        const int q = i - pm_green::kTabOctaves * 1024;
        s = 1.0;
        c = {(q >> 6) - 31.5, (q & 63) - 31.5};
    }
    cplx_d a[16];
    for (int n = 0; n < 16; ++n) a[n] = {0.0, 0.0};
    // arguments of w lie in (-3 pi/4, pi/4]; cells of the smaller octaves inside are not read
    const double th = atan2(c.im, c.re);
    if (th > -0.75 * M_PI - 0.4 && th < 0.25 * M_PI + 0.4 && fmax(fabs(c.re), fabs(c.im)) > 7.0 * s) {
        cplx_d K0, K1;
        pm_green::bessel_k01_c(c, cG16, cG16 + PM_GL16, &K0, &K1);
        a[0] = K0;
        a[1] = pm_green::cz_scale(K1, -1.0);
        taylor(c, 1.0, 16, a);
    }
    for (int n = 0; n < 16; ++n) c2[(size_t)i * 16 + n] = make_double2(a[n].re, a[n].im);
}

}  // namespace

pm_status pm_green_tables(pm_ctx* ctx, bool complex_q, pm_green::GreenTab* T) {
    std::lock_guard<std::mutex> lock(ctx->green_mu);
    if (!ctx->green_h1 || (complex_q && !ctx->green_c2)) {
        QuadTables Q;
        pm_build_tables(2, &Q);
        double g16[2 * PM_GL16];
        for (int k = 0; k < PM_GL16; ++k) {
            g16[k] = Q.g16t[k];
            g16[PM_GL16 + k] = Q.g16w[k];
        }
        PM_CUDA_TRY(cudaMemcpyToSymbol(cG16, g16, sizeof(g16)));
        PM_CUDA_TRY(pm_green::upload_cheb_k01());
    }
    if (!ctx->green_h1) {
        double2 *k1 = nullptr, *h1 = nullptr;
        PM_TRY(pm_dmalloc(&k1, (size_t)pm_green::kTabRows * 8));
        const pm_status st = pm_dmalloc(&h1, (size_t)pm_green::kTabRows * 16);
        if (st != PM_OK) {
            pm_dfree(k1);
            return st;
        }
        k_green_rows<<<pm_ceil_div(pm_green::kTabRows, 32), 32>>>(k1, h1);
        const cudaError_t e = cudaGetLastError() == cudaSuccess ? cudaDeviceSynchronize() : cudaErrorUnknown;
        if (e != cudaSuccess) {
            pm_dfree(k1);
            pm_dfree(h1);
            pm_set_error("Green's function tables: %s", cudaGetErrorString(e));
            return PM_ERR_CUDA;
        }
        ctx->green_k1 = k1;
        ctx->green_h1 = h1;
    }
    if (complex_q && !ctx->green_c2) {
        double2* c2 = nullptr;
        PM_TRY(pm_dmalloc(&c2, (size_t)pm_green::kTabCells * 16));
        k_green_cells<<<pm_ceil_div(pm_green::kTabCells, 128), 128>>>(c2);
        const cudaError_t e = cudaGetLastError() == cudaSuccess ? cudaDeviceSynchronize() : cudaErrorUnknown;
        if (e != cudaSuccess) {
            pm_dfree(c2);
            pm_set_error("Green's function tables: %s", cudaGetErrorString(e));
            return PM_ERR_CUDA;
        }
        ctx->green_c2 = c2;
    }
    T->k1 = ctx->green_k1;
    T->h1 = ctx->green_h1;
    T->c2 = ctx->green_c2;
    return PM_OK;
}
