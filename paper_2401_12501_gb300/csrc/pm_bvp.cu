// Boundary-value systems on an open surface: Neumann (Sec. 5.2, eq. NeuBVPsystem) and,
// for a constant coefficient, Dirichlet (Sec. 5.3, eq. DirBVPsystem).
//
// Gamma is a surface built from an open surface's patches (pm_surface_create +
// pm_surface_set_coeff); its boundary gamma is a union of closed curves given at
// edge nodes t_k = 2 pi (k + 1/2) / M of a periodic parameter and at F M oversampled
// points t_j = 2 pi j / (F M).  Unknowns sigma [N] and mu [Me]:
//
//   sigma + R~_Gamma sigma + R_gamma mu                          = f        (surface rows)
//   -mu / (2a) + K'_Gamma sigma + K'_gamma mu + (sum_k w_k mu_k)  = f_gamma  (edge rows)
//   u = K~_Gamma sigma + K_gamma mu                               (eq. BC_rep)
//
// with K = log r / (2 pi a(x')), R of eq. explicit_remainder (c = 0), K' = nu . grad_x K
// at edge nodes (nu the binormal).  The rank-one term removes the one-dimensional null
// space (constants solve the homogeneous Neumann problem); any multiple of it gives the
// same u up to a constant for consistent data.
//
// Dirichlet, a constant (the paper proves T_gamma compact for constant a only):
//
//   sigma + R~_Gamma sigma + T_gamma mu                 = f        (surface rows)
//   +mu / (2a) + K~_Gamma sigma + N_gamma mu            = f_gamma  (edge rows: the trace)
//   u = K~_Gamma sigma + N_gamma mu
//
// N_gamma the double layer nu(x') . grad_x' K, T_gamma = nu(x') . grad_x' R; the trace of
// the double layer from inside is +mu/(2a) plus its value on gamma (the paper prints
// -mu/(2a); Gauss's lemma fixes the sign), and the edge row carries K_Gamma[sigma], as
// the trace theorem states (the printed system writes N_Gamma there).  K~_Gamma at the
// edge nodes: smooth rule plus corrections (polar rule with dyadic radial panels on the
// edge patch, quadtree near rule on the others); N_gamma on gamma: trapezoid rule, its
// diagonal the limit -nu . gamma'' / (4 pi a |gamma'|^2); T_gamma and N_gamma off gamma:
// the oversampled trapezoid rule.
//
// Discretisation (Sec. 6.1.4 with the surface rules of Sec. 6.1):
// * R~_Gamma, K~_Gamma: the surface's float64 applies (smooth sums + near corrections).
// * R_gamma, K_gamma: trapezoid rule on the oversampled points, mu carried there by the
//   trigonometric interpolant (degree < M/2 and the symmetric Nyquist term), the paper's
//   Fourier oversampling; a(x') at the oversampled points.
// * K'_gamma: trapezoid rule on the edge nodes, the diagonal entry the limit of the smooth
//   kernel along the curve, nu . (x - y) / |x - y|^2 -> -nu . gamma'' / (2 |gamma'|^2).
// * K'_Gamma: the smooth rule over all surface nodes plus corrections on the patches near
//   each edge node (pm_nearfield.cu k_bvp_kp_quad: polar rule about the edge point on its
//   own patch, the quadtree near rule on the others).
// Everything runs in float64; a solve applies the system through its dense matrix where
// that fits the device (else pair by pair); the solver is restarted GMRES
// (pm_arnoldi.cuh), the Hessenberg system on the host.
#include "pm_arnoldi.cuh"
#include "pm_fast64.cuh"
#include "pm_internal.cuh"

#include <algorithm>
#include <chrono>
#include <cmath>
#include <vector>

pm_status pm_bvp_kp_weights(pm_surface* s, int nb, const int* blk_edge, const int* blk_patch,
                            const int* blk_own, const double* xe, const double* nue,
                            const double* uv, int log_kernel, double* W);

struct pm_bvp {
    pm_surface* s = nullptr;
    int kind = 0;                        // 0 Neumann, 1 Dirichlet
    long long coeff_epoch = 0;           // the surface's coefficient epoch at creation
    int N = 0, Me = 0, Fo = 0, ncurves = 0;
    std::vector<int> M, F, off, offo;
    std::vector<double> h_we;
    double *xe = nullptr, *nue = nullptr, *we = nullptr, *ae = nullptr, *uv = nullptr;
    double *xo = nullptr, *wo = nullptr, *ao = nullptr, *nuo = nullptr;
    double *interp = nullptr;            // per curve [F M][M], curve blocks concatenated
    int *interp_off = nullptr;           // five rows of [ncurves + 1]: offset into interp, first
                                         // oversampled point, first edge node, M, offset into fourier
    double *fourier = nullptr;           // per curve [F M / 4 + 1][M] and [M][M] (k_bvp_fill_edge_fourier)
    bool foldable = false;               // every curve has them
    int *curve_of = nullptr;             // [Fo] curve of an oversampled point
    double *Kpg = nullptr;               // [Me][Me] K'_gamma (Neumann) or N_gamma (Dirichlet), weighted
    int *kp_ptr = nullptr, *kp_patch = nullptr, *kp_edge = nullptr;
    double *kp_C = nullptr;              // [nblk][pp] K'_Gamma (K_Gamma) corrections
    int kp_nblk = 0;
    double *mu_o = nullptr;              // [Fo]
    cudaStream_t st = nullptr;
};

namespace {

constexpr int kT = 256;

// mu_o[j] = sum_k I_c[j][k] mu[off_c + k] for the curve c of oversampled point j
__global__ void k_bvp_interp(const double* __restrict__ I, const int* __restrict__ ioff,
                             const int* __restrict__ curve_of, const int* __restrict__ offo,
                             const int* __restrict__ off, const int* __restrict__ Mc,
                             const double* __restrict__ mu, double* __restrict__ mu_o, int Fo) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= Fo) return;
    const int c = curve_of[j];
    const int m = Mc[c], jl = j - offo[c];
    const double* row = I + ioff[c] + (size_t)jl * m;
    const double* mc = mu + off[c];
    double s = 0.0;
    for (int k = 0; k < m; ++k) s += row[k] * mc[k];
    mu_o[j] = s;
}

// out[i] += sum_j wo_j mu_o_j G(x_i, xo_j) with r = x_i - xo_j: KIND 0 the remainder
// R / a(x') (target n, H, a, grad a), 1 the parametrix log r / (2 pi a(x')), 2 T =
// nu' . grad' R for constant a (the a's cancel), 3 the double layer
// -nu' . r / (2 pi a r^2)
enum { kEdgeR = 0, kEdgeK = 1, kEdgeT = 2, kEdgeN = 3 };

// a target's data (n, H, a and g for the remainder kinds only)
struct EdgeTarget {
    double x[3], n[3], g[3], H, a;
};

template <int KIND>
__device__ __forceinline__ EdgeTarget edge_target(int i, const double* x, const double* n,
                                                  const double* H, const double* a, const double* g) {
    EdgeTarget t{};
    for (int d = 0; d < 3; ++d) t.x[d] = x[3 * i + d];
    if (KIND == kEdgeR || KIND == kEdgeT) {
        for (int d = 0; d < 3; ++d) {
            t.n[d] = n[3 * i + d];
            t.g[d] = g[3 * i + d];
        }
        t.H = H[i];
        t.a = a[i];
    }
    return t;
}

// the kernel of one (target, oversampled point y with binormal u) pair, all its constants in
// (R and K without 1 / a(x'), which the strength carries)
template <int KIND>
__device__ __forceinline__ double edge_pair(const EdgeTarget& t, double y0, double y1, double y2,
                                            double u0, double u1, double u2) {
    const double r0 = t.x[0] - y0, r1 = t.x[1] - y1, r2 = t.x[2] - y2;
    const double rr = r0 * r0 + r1 * r1 + r2 * r2;
    if (KIND == kEdgeK) return pm_log64(rr) * (0.25 / M_PI);
    const double inv = pm_rcp64(rr);
    if (KIND == kEdgeN) return -(u0 * r0 + u1 * r1 + u2 * r2) * inv * (0.5 / M_PI);
    const double nr = t.n[0] * r0 + t.n[1] * r1 + t.n[2] * r2;
    if (KIND == kEdgeR) {
        const double qn = nr * inv;
        return t.a * (qn * qn - t.H * qn) * (1.0 / M_PI) +
               (t.g[0] * r0 + t.g[1] * r1 + t.g[2] * r2) * inv * (0.5 / M_PI);
    }
    // -(1/pi) [2 (n.r)(n.nu')/r^4 - 4 (n.r)^2 (r.nu')/r^6 - H (n.nu')/r^2
    //          + 2 H (n.r)(r.nu')/r^4], with q = (n.r)/r^2 a product of two factors
    const double nnu = t.n[0] * u0 + t.n[1] * u1 + t.n[2] * u2;
    const double rnu = r0 * u0 + r1 * u1 + r2 * u2;
    const double q = nr * inv;
    return (-(1.0 / M_PI) * inv) * ((2.0 * q - t.H) * (nnu - 2.0 * q * rnu));
}

// A warp a target, its lanes over the oversampled points: float64-pipe work, for which a
// thread a target left most SMs without any (9.6 ms for 2,048 targets x 4,096 points).
template <int KIND>
__global__ void __launch_bounds__(kT)
k_bvp_edge_to_surface(int N, const double* __restrict__ x, const double* __restrict__ n,
                      const double* __restrict__ H, const double* __restrict__ a,
                      const double* __restrict__ g, int Fo, const double* __restrict__ xo,
                      const double* __restrict__ wo, const double* __restrict__ ao,
                      const double* __restrict__ nuo, const double* __restrict__ mu_o,
                      double* __restrict__ out) {
    const int i = (blockIdx.x * kT + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= N) return;
    const EdgeTarget t = edge_target<KIND>(i, x, n, H, a, g);
    double acc = 0.0;
    for (int j = lane; j < Fo; j += 32) {
        const double s = KIND == kEdgeT ? wo[j] * mu_o[j] : wo[j] * mu_o[j] / ao[j];
        acc += s * edge_pair<KIND>(t, xo[3 * j], xo[3 * j + 1], xo[3 * j + 2], nuo[3 * j],
                                   nuo[3 * j + 1], nuo[3 * j + 2]);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) out[i] += acc;
}

// ------------------------------------------------------------------ the dense system
// A solve forms the system's matrix once, A [n][n] over z = [sigma; mu] (n = N + Me), and
// its Krylov steps stream it: 8 n^2 bytes a step instead of the float64 pair sums of
// apply_sys.  Dirichlet, 2,048 nodes and 128 edge nodes (a matrix of 38 MB, so it stays in
// L2): a solve of 15 steps 176 -> 3.2 ms.

// surface rows, sigma columns: delta_ij + w_j R(x_i, x_j) / a_j (kDI targets x kDJ sources a block)
constexpr int kDI = 32, kDJ = 128;
__global__ void __launch_bounds__(kDJ)
k_bvp_fill_surface(int N, const double* __restrict__ x, const double* __restrict__ nrm,
                   const double* __restrict__ H, const double* __restrict__ a,
                   const double* __restrict__ g, const double* __restrict__ wa, int ld,
                   double* __restrict__ A) {
    __shared__ double st[kDI][9];        // x, sqrt(a/pi) n, -(a H/pi) n + grad a/(2 pi)
    const int i0 = blockIdx.y * kDI, rows = min(kDI, N - i0);
    for (int e = threadIdx.x; e < rows * 3; e += kDJ) {
        const int r = e / 3, d = e - r * 3, i = i0 + r;
        st[r][d] = x[3 * i + d];
        st[r][3 + d] = sqrt(a[i] / M_PI) * nrm[3 * i + d];
        st[r][6 + d] = -a[i] * H[i] / M_PI * nrm[3 * i + d] + 0.5 / M_PI * g[3 * i + d];
    }
    __syncthreads();
    const int j = blockIdx.x * kDJ + threadIdx.x;
    if (j >= N) return;
    const double y0 = x[3 * j], y1 = x[3 * j + 1], y2 = x[3 * j + 2], w = wa[j];
    for (int r = 0; r < rows; ++r) {
        const double* t = st[r];
        const double r0 = t[0] - y0, r1 = t[1] - y1, r2 = t[2] - y2;
        const double inv = pm_rcp64(r0 * r0 + r1 * r1 + r2 * r2);
        const double nr = t[3] * r0 + t[4] * r1 + t[5] * r2;
        const double mr = t[6] * r0 + t[7] * r1 + t[8] * r2;
        A[(size_t)(i0 + r) * ld + j] = i0 + r == j ? 1.0 : w * inv * (nr * nr * inv + mr);
    }
}

// corrections of surface rows (row_of = blk_row) or edge rows (the edge node of each block)
__global__ void k_bvp_fill_near(int nblk, int pp, const int* __restrict__ row_of, int row0,
                                const int* __restrict__ blk_patch, const double* __restrict__ C,
                                int ld, double* __restrict__ A) {
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)nblk * pp) return;
    const int b = (int)(e / pp), k = (int)(e - (size_t)b * pp);
    A[(size_t)(row0 + row_of[b]) * ld + (size_t)blk_patch[b] * pp + k] += C[e];
}

// surface rows, mu columns: sum over curve c's oversampled points of the pair kernel times the
// interpolation row.  Block: kEI targets x 128 edge nodes of one curve; the points pass in
// tiles of 128, a thread evaluating its point for every target, then its edge node's sums.
// For the curves that k_bvp_fill_edge_fourier does not take.
constexpr int kEI = 4;
template <int KIND>
__global__ void __launch_bounds__(128)
k_bvp_fill_edge_columns(int N, const double* __restrict__ x, const double* __restrict__ n,
                        const double* __restrict__ H, const double* __restrict__ a,
                        const double* __restrict__ g, int ncurves, const double* __restrict__ xo,
                        const double* __restrict__ wo, const double* __restrict__ ao,
                        const double* __restrict__ nuo, const double* __restrict__ I,
                        const int* __restrict__ ioff, int ld, double* __restrict__ A) {
    __shared__ double sk[kEI][128];
    const int c = blockIdx.y, nc1 = ncurves + 1;
    const int o0 = ioff[nc1 + c], o1 = ioff[nc1 + c + 1], off = ioff[2 * nc1 + c], M = ioff[3 * nc1 + c];
    const int e = blockIdx.z * 128 + threadIdx.x;
    if (blockIdx.z * 128 >= M) return;
    const int i0 = blockIdx.x * kEI;
    EdgeTarget t[kEI];
    for (int r = 0; r < kEI; ++r) t[r] = edge_target<KIND>(min(i0 + r, N - 1), x, n, H, a, g);
    double acc[kEI] = {};
    for (int base = o0; base < o1; base += 128) {
        const int j = base + threadIdx.x;
        if (j < o1) {
            const double w = KIND == kEdgeT ? wo[j] : wo[j] / ao[j];
            for (int r = 0; r < kEI; ++r)
                sk[r][threadIdx.x] = w * edge_pair<KIND>(t[r], xo[3 * j], xo[3 * j + 1], xo[3 * j + 2],
                                                         nuo[3 * j], nuo[3 * j + 1], nuo[3 * j + 2]);
        }
        __syncthreads();
        if (e < M) {
            const double* row = I + ioff[c] + (size_t)(base - o0) * M + e;
            const int cnt = min(128, o1 - base);
            for (int q = 0; q < cnt; ++q) {
                const double v = row[(size_t)q * M];
                for (int r = 0; r < kEI; ++r) acc[r] = fma(v, sk[r][q], acc[r]);
            }
        }
        __syncthreads();
    }
    if (e < M)
        for (int r = 0; r < kEI && i0 + r < N; ++r) A[(size_t)(i0 + r) * ld + N + off + e] = acc[r];
}

// The same columns by the trigonometric interpolant's own basis, for curves of n = F M points,
// n a multiple of 4 and M <= kEM.  Interpolating at t_j = 2 pi j / n from the M nodes is the
// sum over M functions cos(q t), sin(q t), so the weights of the nodes are those functions'
// sums over the points, C_q = sum_j f_j cos(q t_j) and S_q, times an M x M matrix; and the four
// points t, -t, pi - t, pi + t of a quarter share every function up to its sign, so a quarter
// of the products remains once their values are added with the four patterns of signs (even
// and odd q of the cosines, then of the sines).  Bound by the float64 pipe (two multiply-adds a
// clock an SM): at 2,048 targets, two curves of 64 nodes and 2,048 points, 0.5 ms of pair
// kernels stay and the products are 0.25 ms instead of 0.95 (by operation counts; the whole
// Dirichlet solve of 2,048 + 128 unknowns 3.70 -> 3.16 ms).
// fourier[off]: [n / 4 + 1][M] functions at t_j, then [M][M] functions at the nodes, scaled;
// order: even q cosines, odd q cosines, even q sines, odd q sines.
constexpr int kEM = 512;              // [M][kEI] beside sk in 48 KB of shared memory
__host__ __device__ __forceinline__ int cosines(int M, int odd) {    // q = 0 .. ceil(M / 2) - 1
    return ((M + 1) / 2 + 1 - odd) / 2;
}
__host__ __device__ __forceinline__ int sines(int M, int odd) {      // q = 1 .. floor(M / 2)
    return (M / 2 + odd) / 2;
}
template <int KIND>
__global__ void __launch_bounds__(128)
k_bvp_fill_edge_fourier(int N, const double* __restrict__ x, const double* __restrict__ n,
                        const double* __restrict__ H, const double* __restrict__ a,
                        const double* __restrict__ g, int ncurves, const double* __restrict__ xo,
                        const double* __restrict__ wo, const double* __restrict__ ao,
                        const double* __restrict__ nuo, const double* __restrict__ fourier,
                        const int* __restrict__ ioff, int ld, double* __restrict__ A) {
    __shared__ EdgeTarget t[kEI];
    __shared__ double sk[4][128][kEI];
    extern __shared__ double coef[];     // [M][kEI]
    const int c = blockIdx.y, nc1 = ncurves + 1, tid = threadIdx.x;
    const int o0 = ioff[nc1 + c], np = ioff[nc1 + c + 1] - o0, off = ioff[2 * nc1 + c], M = ioff[3 * nc1 + c];
    const double* F = fourier + ioff[4 * nc1 + c];
    const int i0 = blockIdx.x * kEI, quarter = np / 4;
    const int k1 = cosines(M, 0), k2 = k1 + cosines(M, 1), k3 = k2 + sines(M, 0);
    if (tid < kEI) t[tid] = edge_target<KIND>(min(i0 + tid, N - 1), x, n, H, a, g);
    for (int e = tid; e < M * kEI; e += 128) coef[e] = 0.0;
    __syncthreads();
    for (int base = 0; base <= quarter; base += 128) {
        const int j = base + tid;
        if (j <= quarter) {
            // t_j, -t_j, pi - t_j, pi + t_j; at j = 0 and n / 4 two of them are one point
            const int pt[4] = {j, np - j, np / 2 - j, np / 2 + j};
            const bool end = j == 0 || j == quarter;
            double v[4][kEI];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int y = o0 + pt[s];
                if (end && !(s == 0 || s == (j == 0 ? 2 : 1))) {
#pragma unroll
                    for (int r = 0; r < kEI; ++r) v[s][r] = 0.0;
                    continue;
                }
                const double w = KIND == kEdgeT ? wo[y] : wo[y] / ao[y];
#pragma unroll
                for (int r = 0; r < kEI; ++r)
                    v[s][r] = w * edge_pair<KIND>(t[r], xo[3 * y], xo[3 * y + 1], xo[3 * y + 2],
                                                  nuo[3 * y], nuo[3 * y + 1], nuo[3 * y + 2]);
            }
#pragma unroll
            for (int r = 0; r < kEI; ++r) {
                const double sum0 = v[0][r] + v[1][r], dif0 = v[0][r] - v[1][r];
                const double sum1 = v[2][r] + v[3][r], dif1 = v[2][r] - v[3][r];
                sk[0][tid][r] = sum0 + sum1;
                sk[1][tid][r] = sum0 - sum1;
                sk[2][tid][r] = dif0 - dif1;
                sk[3][tid][r] = dif0 + dif1;
            }
        }
        __syncthreads();
        const int cnt = min(128, quarter + 1 - base);
        for (int e = tid; e < M; e += 128) {
            const double(*f)[kEI] = sk[(e >= k1) + (e >= k2) + (e >= k3)];
            const double* col = F + (size_t)base * M + e;
            double acc[kEI];
#pragma unroll
            for (int r = 0; r < kEI; ++r) acc[r] = coef[e * kEI + r];
#pragma unroll 4
            for (int q = 0; q < cnt; ++q) {
                const double b = col[(size_t)q * M];
#pragma unroll
                for (int r = 0; r < kEI; ++r) acc[r] = fma(b, f[q][r], acc[r]);
            }
#pragma unroll
            for (int r = 0; r < kEI; ++r) coef[e * kEI + r] = acc[r];
        }
        __syncthreads();
    }
    const double* D = F + (size_t)(quarter + 1) * M;
    for (int e = tid; e < M; e += 128) {
        double acc[kEI] = {};
#pragma unroll 4
        for (int q = 0; q < M; ++q) {
            const double b = D[(size_t)q * M + e];
#pragma unroll
            for (int r = 0; r < kEI; ++r) acc[r] = fma(b, coef[q * kEI + r], acc[r]);
        }
#pragma unroll
        for (int r = 0; r < kEI; ++r)
            if (i0 + r < N) A[(size_t)(i0 + r) * ld + N + off + e] = acc[r];
    }
}

// fourier of one curve of m nodes and f m points
void fourier_tables(int m, int f, std::vector<double>* out) {
    const int n = f * m;
    auto function = [m](int e, int* q, bool* sine) {
        const int k1 = cosines(m, 0), k2 = k1 + cosines(m, 1), k3 = k2 + sines(m, 0);
        *sine = e >= k2;
        *q = e < k1 ? 2 * e : e < k2 ? 2 * (e - k1) + 1 : e < k3 ? 2 * (e - k2) + 2 : 2 * (e - k3) + 1;
    };
    // function e at the angle 2 pi num / den
    auto value = [&](int e, long long num, int den) {
        int q;
        bool sine;
        function(e, &q, &sine);
        const double t = 2.0 * M_PI * (double)(num * q % den) / den;
        return sine ? std::sin(t) : std::cos(t);
    };
    for (int j = 0; j <= n / 4; ++j)
        for (int e = 0; e < m; ++e) out->push_back(value(e, j, n));
    for (int e = 0; e < m; ++e) {
        int q;
        bool sine;
        function(e, &q, &sine);
        const double scale = (q == 0 || 2 * q == m ? 1.0 : 2.0) / m;
        for (int k = 0; k < m; ++k) out->push_back(scale * value(e, 2 * k + 1, 2 * m));
    }
}

// edge rows (as k_bvp_edge_row, without the corrections)
__global__ void k_bvp_fill_edge_rows(int dirichlet, int N, int Me, const double* __restrict__ x,
                                     const double* __restrict__ wa, const double* __restrict__ xe,
                                     const double* __restrict__ nue, const double* __restrict__ ae,
                                     const double* __restrict__ we, const double* __restrict__ Kpg,
                                     int ld, double* __restrict__ A) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x, e = blockIdx.y;
    if (j >= N + Me) return;
    double v;
    if (j < N) {
        const double r0 = xe[3 * e] - x[3 * j], r1 = xe[3 * e + 1] - x[3 * j + 1],
                     r2 = xe[3 * e + 2] - x[3 * j + 2];
        const double rr = r0 * r0 + r1 * r1 + r2 * r2;
        v = wa[j] * (0.5 / M_PI) *
            (dirichlet ? 0.5 * pm_log64(rr)
                       : (nue[3 * e] * r0 + nue[3 * e + 1] * r1 + nue[3 * e + 2] * r2) * pm_rcp64(rr));
    } else {
        const int k = j - N;
        v = Kpg[(size_t)e * Me + k] + (dirichlet ? 0.0 : we[k]);
        if (k == e) v += (dirichlet ? 0.5 : -0.5) / ae[e];
    }
    A[(size_t)(N + e) * ld + j] = v;
}

// out = A z, four rows a block
__global__ void __launch_bounds__(128)
k_bvp_gemv(int n, const double* __restrict__ A, const double* __restrict__ z, double* __restrict__ out) {
    __shared__ double sh[4][4];
    const int i0 = blockIdx.x * 4;
    const double* row[4];
    double acc[4] = {};
    for (int r = 0; r < 4; ++r) row[r] = A + (size_t)min(i0 + r, n - 1) * n;
#pragma unroll 4
    for (int j = threadIdx.x; j < n; j += 128) {
        const double v = z[j];
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = fma(row[r][j], v, acc[r]);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int r = 0; r < 4; ++r) {
        for (int o = 16; o > 0; o >>= 1) acc[r] += __shfl_down_sync(0xffffffffu, acc[r], o);
        if (lane == 0) sh[r][wid] = acc[r];
    }
    __syncthreads();
    const int r = threadIdx.x;
    if (r < 4 && i0 + r < n) out[i0 + r] = (sh[r][0] + sh[r][1]) + (sh[r][2] + sh[r][3]);
}

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    return t;
}

// edge rows: one block per edge node e; Neumann (dirichlet = 0): K'_Gamma sigma +
// K'_gamma mu - mu/(2a) + sum w mu; Dirichlet: K_Gamma sigma + N_gamma mu + mu/(2a)
__global__ void __launch_bounds__(kT)
k_bvp_edge_row(int dirichlet, int N, int Me, int pp, const double* __restrict__ x,
               const double* __restrict__ wa,
               const double* __restrict__ xe, const double* __restrict__ nue,
               const double* __restrict__ ae, const double* __restrict__ we,
               const int* __restrict__ kp_ptr, const int* __restrict__ kp_patch,
               const double* __restrict__ kp_C, const double* __restrict__ Kpg,
               const double* __restrict__ sigma, const double* __restrict__ mu,
               double* __restrict__ out) {
    __shared__ double red[kT / 32];
    const int e = blockIdx.x;
    const double x0 = xe[3 * e], x1 = xe[3 * e + 1], x2 = xe[3 * e + 2];
    const double n0 = nue[3 * e], n1 = nue[3 * e + 1], n2 = nue[3 * e + 2];
    double acc = 0.0;
    for (int j = threadIdx.x; j < N; j += kT) {
        const double r0 = x0 - x[3 * j], r1 = x1 - x[3 * j + 1], r2 = x2 - x[3 * j + 2];
        const double rr = r0 * r0 + r1 * r1 + r2 * r2;
        acc += wa[j] * sigma[j] * (dirichlet ? 0.5 * log(rr) : (n0 * r0 + n1 * r1 + n2 * r2) / rr);
    }
    acc *= 0.5 / M_PI;
    for (int b = kp_ptr[e]; b < kp_ptr[e + 1]; ++b) {
        const double* C = kp_C + (size_t)b * pp;
        const double* sg = sigma + (size_t)kp_patch[b] * pp;
        for (int k = threadIdx.x; k < pp; k += kT) acc += C[k] * sg[k];
    }
    for (int k = threadIdx.x; k < Me; k += kT)
        acc += (Kpg[(size_t)e * Me + k] + (dirichlet ? 0.0 : we[k])) * mu[k];
    const double t = block_sum(acc, red);
    if (threadIdx.x == 0) out[e] = t + (dirichlet ? 0.5 : -0.5) * mu[e] / ae[e];
}

// C[b][k] = W[b][k] / a_k - w_k G(x_e, x_k) / a_k with G = nu_e . (x_e - x_k) / (2 pi |.|^2)
// (Neumann) or log|x_e - x_k| / (2 pi) (Dirichlet)
__global__ void k_bvp_combine(int dirichlet, int nblk, int pp, const int* __restrict__ blk_edge,
                              const int* __restrict__ blk_patch, const double* __restrict__ x,
                              const double* __restrict__ a, const double* __restrict__ w,
                              const double* __restrict__ xe, const double* __restrict__ nue,
                              double* __restrict__ C) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (size_t)nblk * pp) return;
    const int b = (int)(q / pp), k = (int)(q - (size_t)b * pp);
    const int e = blk_edge[b];
    const size_t j = (size_t)blk_patch[b] * pp + k;
    const double r0 = xe[3 * e] - x[3 * j], r1 = xe[3 * e + 1] - x[3 * j + 1],
                 r2 = xe[3 * e + 2] - x[3 * j + 2];
    const double rr = r0 * r0 + r1 * r1 + r2 * r2;
    const double G = dirichlet ? 0.5 * log(rr)
                               : (nue[3 * e] * r0 + nue[3 * e + 1] * r1 + nue[3 * e + 2] * r2) / rr;
    const double smooth = w[j] * G * (0.5 / M_PI) / a[j];
    C[q] = C[q] / a[j] - smooth;
}

__global__ void k_bvp_axpy(int n, double alpha, const double* __restrict__ xv, double* __restrict__ y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] += alpha * xv[i];
}

// r = b - r
__global__ void k_bvp_rsub(int n, const double* __restrict__ b, double* __restrict__ r) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = b[i] - r[i];
}

// the system's operator on z = [sigma; mu] (device), out = [surface rows; edge rows]
pm_status apply_sys(pm_bvp* b, const double* z, double* out) {
    pm_surface* s = b->s;
    const int N = b->N;
    cudaStream_t st = b->st;
    PM_TRY(pm_apply_dev(s, 0, 1, 1, z, out, PM_PREC_FP64, st));
    k_bvp_axpy<<<pm_ceil_div(N, kT), kT, 0, st>>>(N, 1.0, z, out);
    if (b->Me > 0) {
        k_bvp_interp<<<pm_ceil_div(b->Fo, kT), kT, 0, st>>>(
            b->interp, b->interp_off, b->curve_of, b->interp_off + b->ncurves + 1,
            b->interp_off + 2 * (b->ncurves + 1), b->interp_off + 3 * (b->ncurves + 1), z + N,
            b->mu_o, b->Fo);
        if (b->kind)
            k_bvp_edge_to_surface<kEdgeT><<<pm_ceil_div((long long)N * 32, kT), kT, 0, st>>>(
                N, s->x, s->n, s->H, s->a, s->g, b->Fo, b->xo, b->wo, b->ao, b->nuo, b->mu_o, out);
        else
            k_bvp_edge_to_surface<kEdgeR><<<pm_ceil_div((long long)N * 32, kT), kT, 0, st>>>(
                N, s->x, s->n, s->H, s->a, s->g, b->Fo, b->xo, b->wo, b->ao, b->nuo, b->mu_o, out);
        k_bvp_edge_row<<<b->Me, kT, 0, st>>>(b->kind, N, b->Me, s->pp, s->x, s->wa, b->xe, b->nue, b->ae,
                                             b->we, b->kp_ptr, b->kp_patch, b->kp_C, b->Kpg, z,
                                             z + N, out + N);
    }
    PM_CUDA_TRY(cudaGetLastError());
    return PM_OK;
}

// The system's matrix into A [n][n] (device).
pm_status fill_sys(pm_bvp* b, double* A) {
    pm_surface* s = b->s;
    const int N = b->N, Me = b->Me, ld = N + Me;
    cudaStream_t st = b->st;
    k_bvp_fill_surface<<<dim3(pm_ceil_div(N, kDJ), pm_ceil_div(N, kDI)), kDJ, 0, st>>>(
        N, s->x, s->n, s->H, s->a, s->g, s->wa, ld, A);
    k_bvp_fill_near<<<pm_ceil_div((long long)s->nblk * s->pp, kT), kT, 0, st>>>(
        s->nblk, s->pp, s->blk_row, 0, s->blk_patch, s->cR64, ld, A);
    if (Me > 0) {
        const int mmax = *std::max_element(b->M.begin(), b->M.end());
        dim3 grid(pm_ceil_div(N, kEI), b->ncurves, b->foldable ? 1 : pm_ceil_div(mmax, 128));
        if (b->foldable)
            (b->kind ? k_bvp_fill_edge_fourier<kEdgeT> : k_bvp_fill_edge_fourier<kEdgeR>)
                <<<grid, 128, (size_t)mmax * kEI * sizeof(double), st>>>(
                    N, s->x, s->n, s->H, s->a, s->g, b->ncurves, b->xo, b->wo, b->ao, b->nuo,
                    b->fourier, b->interp_off, ld, A);
        else
            (b->kind ? k_bvp_fill_edge_columns<kEdgeT> : k_bvp_fill_edge_columns<kEdgeR>)
                <<<grid, 128, 0, st>>>(N, s->x, s->n, s->H, s->a, s->g, b->ncurves, b->xo, b->wo,
                                       b->ao, b->nuo, b->interp, b->interp_off, ld, A);
        k_bvp_fill_edge_rows<<<dim3(pm_ceil_div(ld, kT), Me), kT, 0, st>>>(
            b->kind, N, Me, s->x, s->wa, b->xe, b->nue, b->ae, b->we, b->Kpg, ld, A);
        k_bvp_fill_near<<<pm_ceil_div((long long)b->kp_nblk * s->pp, kT), kT, 0, st>>>(
            b->kp_nblk, s->pp, b->kp_edge, N, b->kp_patch, b->kp_C, ld, A);
    }
    PM_CUDA_TRY(cudaGetLastError());
    return PM_OK;
}

// the operator through its matrix where the solve holds one
pm_status apply_any(pm_bvp* b, const double* A, const double* z, double* out) {
    if (!A) return apply_sys(b, z, out);
    const int n = b->N + b->Me;
    k_bvp_gemv<<<pm_ceil_div(n, 4), 128, 0, b->st>>>(n, A, z, out);
    PM_CUDA_TRY(cudaGetLastError());
    return PM_OK;
}

pm_status represent(pm_bvp* b, const double* z, double* u) {
    pm_surface* s = b->s;
    const int N = b->N;
    cudaStream_t st = b->st;
    PM_TRY(pm_apply_dev(s, 1, 1, 1, z, u, PM_PREC_FP64, st));
    if (b->Me > 0) {
        k_bvp_interp<<<pm_ceil_div(b->Fo, kT), kT, 0, st>>>(
            b->interp, b->interp_off, b->curve_of, b->interp_off + b->ncurves + 1,
            b->interp_off + 2 * (b->ncurves + 1), b->interp_off + 3 * (b->ncurves + 1), z + N,
            b->mu_o, b->Fo);
        if (b->kind)
            k_bvp_edge_to_surface<kEdgeN><<<pm_ceil_div((long long)N * 32, kT), kT, 0, st>>>(
                N, s->x, s->n, s->H, s->a, s->g, b->Fo, b->xo, b->wo, b->ao, b->nuo, b->mu_o, u);
        else
            k_bvp_edge_to_surface<kEdgeK><<<pm_ceil_div((long long)N * 32, kT), kT, 0, st>>>(
                N, s->x, s->n, s->H, s->a, s->g, b->Fo, b->xo, b->wo, b->ao, b->nuo, b->mu_o, u);
    }
    PM_CUDA_TRY(cudaGetLastError());
    return PM_OK;
}

void free_bvp(pm_bvp* b) {
    if (!b) return;
    if (b->s) cudaSetDevice(b->s->ctx->device);
    pm_dfree(b->xe); pm_dfree(b->nue); pm_dfree(b->we); pm_dfree(b->ae); pm_dfree(b->uv);
    pm_dfree(b->xo); pm_dfree(b->wo); pm_dfree(b->ao); pm_dfree(b->nuo); pm_dfree(b->interp);
    pm_dfree(b->interp_off); pm_dfree(b->fourier);
    pm_dfree(b->curve_of); pm_dfree(b->Kpg); pm_dfree(b->kp_ptr); pm_dfree(b->kp_patch);
    pm_dfree(b->kp_C); pm_dfree(b->kp_edge); pm_dfree(b->mu_o);
    delete b;
}

template <typename T>
pm_status upload(T** d, const T* h, size_t n) {
    PM_TRY(pm_dmalloc(d, n));
    if (n) PM_CUDA_TRY(cudaMemcpy(*d, h, sizeof(T) * n, cudaMemcpyHostToDevice));
    return PM_OK;
}

pm_status create_impl(pm_bvp* b, const double* edge_x, const double* edge_d1,
                      const double* edge_d2, const double* edge_nu, const double* edge_a,
                      const int* edge_patch, const double* edge_uv, const double* over_x,
                      const double* over_nu, const double* over_speed, const double* over_a) {
    pm_surface* s = b->s;
    const int Me = b->Me, Fo = b->Fo, pp = s->pp;
    // trapezoid weights, K'_gamma (host, dense), interpolation matrices
    b->h_we.resize(Me);
    std::vector<double> wo(Fo), Kpg((size_t)Me * Me), I, fourier;
    std::vector<int> ioff(5 * (b->ncurves + 1), 0), curve_of(Fo);
    for (int c = 0; c < b->ncurves; ++c) {
        const int m = b->M[c], f = b->F[c];
        for (int k = 0; k < m; ++k) {
            const int e = b->off[c] + k;
            const double* d1 = edge_d1 + 3 * e;
            b->h_we[e] = (2.0 * M_PI / m) * std::sqrt(d1[0] * d1[0] + d1[1] * d1[1] + d1[2] * d1[2]);
        }
        for (int j = 0; j < f * m; ++j) {
            wo[b->offo[c] + j] = (2.0 * M_PI / (f * m)) * over_speed[b->offo[c] + j];
            curve_of[b->offo[c] + j] = c;
        }
        ioff[c] = (int)I.size();
        const int nyq = (m % 2 == 0) ? m / 2 : 0;
        for (int j = 0; j < f * m; ++j) {
            const double tj = 2.0 * M_PI * j / (f * m);
            for (int k = 0; k < m; ++k) {
                const double d = tj - 2.0 * M_PI * (k + 0.5) / m;
                double v = 1.0;
                for (int q = 1; q <= (m - 1) / 2; ++q) v += 2.0 * std::cos(q * d);
                if (nyq) v += std::cos(nyq * d);
                I.push_back(v / m);
            }
        }
    }
    const int nc1 = b->ncurves + 1;
    ioff[b->ncurves] = (int)I.size();
    b->foldable = b->ncurves > 0;
    for (int c = 0; c < b->ncurves; ++c)
        b->foldable = b->foldable && b->M[c] <= kEM && b->M[c] * b->F[c] % 4 == 0;
    for (int c = 0; c < b->ncurves && b->foldable; ++c) {
        ioff[4 * nc1 + c] = (int)fourier.size();
        fourier_tables(b->M[c], b->F[c], &fourier);
    }
    for (int c = 0; c < nc1; ++c) {
        ioff[nc1 + c] = c < b->ncurves ? b->offo[c] : Fo;
        ioff[2 * nc1 + c] = c < b->ncurves ? b->off[c] : Me;
        ioff[3 * nc1 + c] = c < b->ncurves ? b->M[c] : 0;
    }
    for (int e = 0; e < Me; ++e) {
        const double* xe_ = edge_x + 3 * e;
        const double* ne = edge_nu + 3 * e;
        for (int k = 0; k < Me; ++k) {
            double v;
            if (k == e) {
                const double* d1 = edge_d1 + 3 * e;
                const double* d2 = edge_d2 + 3 * e;
                const double sp2 = d1[0] * d1[0] + d1[1] * d1[1] + d1[2] * d1[2];
                v = -(ne[0] * d2[0] + ne[1] * d2[1] + ne[2] * d2[2]) / (2.0 * sp2);
            } else {
                const double r0 = xe_[0] - edge_x[3 * k], r1 = xe_[1] - edge_x[3 * k + 1],
                             r2 = xe_[2] - edge_x[3 * k + 2];
                // Neumann: nu(x_e) . r;  Dirichlet (double layer): -nu(x_k) . r
                const double* nn = b->kind ? edge_nu + 3 * k : ne;
                const double sg = b->kind ? -1.0 : 1.0;
                v = sg * (nn[0] * r0 + nn[1] * r1 + nn[2] * r2) / (r0 * r0 + r1 * r1 + r2 * r2);
            }
            Kpg[(size_t)e * Me + k] = b->h_we[k] * v / (2.0 * M_PI * edge_a[k]);
        }
    }
    // near patches of each edge node: its own patch first, then every patch within
    // near_factor radii of the node
    std::vector<double> cen(3 * (size_t)s->npatch), rad(s->npatch);
    PM_CUDA_TRY(cudaMemcpy(cen.data(), s->centroid, sizeof(double) * cen.size(), cudaMemcpyDeviceToHost));
    PM_CUDA_TRY(cudaMemcpy(rad.data(), s->radius, sizeof(double) * rad.size(), cudaMemcpyDeviceToHost));
    std::vector<int> kp_ptr(Me + 1, 0), kp_patch, blk_edge, blk_own;
    for (int e = 0; e < Me; ++e) {
        const int own = edge_patch[e];
        kp_patch.push_back(own);
        blk_edge.push_back(e);
        blk_own.push_back(1);
        for (int P = 0; P < s->npatch; ++P) {
            if (P == own) continue;
            const double d0 = edge_x[3 * e] - cen[3 * P], d1 = edge_x[3 * e + 1] - cen[3 * P + 1],
                         d2 = edge_x[3 * e + 2] - cen[3 * P + 2];
            if (std::sqrt(d0 * d0 + d1 * d1 + d2 * d2) < s->opts.near_factor * rad[P]) {
                kp_patch.push_back(P);
                blk_edge.push_back(e);
                blk_own.push_back(0);
            }
        }
        kp_ptr[e + 1] = (int)kp_patch.size();
    }
    b->kp_nblk = (int)kp_patch.size();
    int* d_own = nullptr;
    PM_TRY(upload(&b->xe, edge_x, 3 * (size_t)Me));
    PM_TRY(upload(&b->nue, edge_nu, 3 * (size_t)Me));
    PM_TRY(upload(&b->we, b->h_we.data(), (size_t)Me));
    PM_TRY(upload(&b->ae, edge_a, (size_t)Me));
    PM_TRY(upload(&b->uv, edge_uv, 2 * (size_t)Me));
    PM_TRY(upload(&b->xo, over_x, 3 * (size_t)Fo));
    PM_TRY(upload(&b->wo, wo.data(), (size_t)Fo));
    PM_TRY(upload(&b->ao, over_a, (size_t)Fo));
    PM_TRY(upload(&b->nuo, over_nu, 3 * (size_t)Fo));
    PM_TRY(upload(&b->interp, I.data(), I.size()));
    PM_TRY(upload(&b->fourier, fourier.data(), fourier.size()));
    PM_TRY(upload(&b->interp_off, ioff.data(), ioff.size()));
    PM_TRY(upload(&b->curve_of, curve_of.data(), curve_of.size()));
    PM_TRY(upload(&b->Kpg, Kpg.data(), Kpg.size()));
    PM_TRY(upload(&b->kp_ptr, kp_ptr.data(), kp_ptr.size()));
    PM_TRY(upload(&b->kp_patch, kp_patch.data(), kp_patch.size()));
    PM_TRY(pm_dmalloc(&b->kp_C, (size_t)b->kp_nblk * pp));
    PM_TRY(pm_dmalloc(&b->mu_o, (size_t)std::max(Fo, 1)));
    pm_status stt = upload(&b->kp_edge, blk_edge.data(), blk_edge.size());
    if (stt == PM_OK) stt = upload(&d_own, blk_own.data(), blk_own.size());
    if (stt == PM_OK)
        stt = pm_bvp_kp_weights(s, b->kp_nblk, b->kp_edge, b->kp_patch, d_own, b->xe, b->nue, b->uv,
                                b->kind, b->kp_C);
    if (stt == PM_OK && b->kp_nblk > 0) {
        k_bvp_combine<<<pm_ceil_div((long long)b->kp_nblk * pp, kT), kT>>>(
            b->kind, b->kp_nblk, pp, b->kp_edge, b->kp_patch, s->x, s->a, s->w, b->xe, b->nue, b->kp_C);
        if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
            pm_set_error("pm_bvp_create: correction kernel failed");
            stt = PM_ERR_CUDA;
        }
    }
    pm_dfree(d_own);
    return stt;
}

}  // namespace

extern "C" pm_status pm_bvp_create(pm_surface* s, int kind, int ncurves, const int* M,
                                   const int* F, const double* edge_x, const double* edge_d1,
                                   const double* edge_d2, const double* edge_nu,
                                   const double* edge_a, const int* edge_patch,
                                   const double* edge_uv, const double* over_x,
                                   const double* over_nu, const double* over_speed,
                                   const double* over_a, pm_bvp** out) {
    if (!out) { pm_set_error("pm_bvp_create: out is NULL"); return PM_ERR_INVALID_ARG; }
    *out = nullptr;
    if (!s || ncurves < 0 || (ncurves > 0 && (!M || !F || !edge_x || !edge_d1 || !edge_d2 ||
                                              !edge_nu || !edge_a || !edge_patch || !edge_uv ||
                                              !over_x || !over_nu || !over_speed || !over_a))) {
        pm_set_error("pm_bvp_create: NULL argument");
        return PM_ERR_INVALID_ARG;
    }
    if (kind != PM_BVP_NEUMANN && kind != PM_BVP_DIRICHLET) {
        pm_set_error("pm_bvp_create: kind %d is neither PM_BVP_NEUMANN nor PM_BVP_DIRICHLET", kind);
        return PM_ERR_INVALID_ARG;
    }
    if (!s->has_coeff) { pm_set_error("pm_bvp_create: call pm_surface_set_coeff first"); return PM_ERR_NO_COEFF; }
    if (s->has_c || s->tri) {
        pm_set_error("pm_bvp_create: built for quadrilateral patches with c = 0");
        return PM_ERR_INVALID_ARG;
    }
    PM_CUDA_TRY(cudaSetDevice(s->ctx->device));
    pm_bvp* b = new pm_bvp();
    b->s = s;
    b->kind = kind == PM_BVP_DIRICHLET ? 1 : 0;
    b->coeff_epoch = s->coeff_epoch;
    b->N = s->N;
    b->ncurves = ncurves;
    for (int c = 0; c < ncurves; ++c) {
        if (M[c] < 2 || F[c] < 1 || (long long)M[c] * F[c] > (1 << 24)) {
            pm_set_error("pm_bvp_create: curve %d has M = %d, F = %d (need M >= 2, F >= 1)", c, M[c], F[c]);
            delete b;
            return PM_ERR_INVALID_ARG;
        }
        b->M.push_back(M[c]);
        b->F.push_back(F[c]);
        b->off.push_back(b->Me);
        b->offo.push_back(b->Fo);
        b->Me += M[c];
        b->Fo += M[c] * F[c];
    }
    long long interp_entries = 0;        // the interpolation matrices: F M x M per curve
    for (int c = 0; c < ncurves; ++c) interp_entries += (long long)F[c] * M[c] * M[c];
    if (b->Me > 4096 || interp_entries > (1LL << 26)) {
        pm_set_error("pm_bvp_create: %d edge nodes (at most 4096), %lld interpolation entries "
                     "sum F M^2 (at most 2^26)", b->Me, interp_entries);
        delete b;
        return PM_ERR_INVALID_ARG;
    }
    for (int e = 0; e < b->Me; ++e) {
        const double u0 = edge_uv[2 * e], v0 = edge_uv[2 * e + 1];
        const bool on_edge = std::fabs(std::fabs(u0) - 1.0) < 1e-12 || std::fabs(std::fabs(v0) - 1.0) < 1e-12;
        if (edge_patch[e] < 0 || edge_patch[e] >= s->npatch || !on_edge || std::fabs(u0) > 1.0 ||
            std::fabs(v0) > 1.0 || !(edge_a[e] > 0.0)) {
            pm_set_error("pm_bvp_create: edge node %d: patch %d, (u, v) = (%g, %g), a = %g (the node "
                         "must lie on an edge of its patch, a > 0)", e, edge_patch[e], u0, v0, edge_a[e]);
            delete b;
            return PM_ERR_INVALID_ARG;
        }
    }
    if (b->kind) {
        // Dirichlet: a constant over the surface, the edge nodes and the oversampled points
        std::vector<double> ah(s->N), gh(3 * (size_t)s->N);
        cudaError_t ce = cudaMemcpy(ah.data(), s->a, sizeof(double) * s->N, cudaMemcpyDeviceToHost);
        if (ce == cudaSuccess)
            ce = cudaMemcpy(gh.data(), s->g, sizeof(double) * gh.size(), cudaMemcpyDeviceToHost);
        if (ce != cudaSuccess) {
            pm_set_error("pm_bvp_create: %s", cudaGetErrorString(ce));
            delete b;
            return PM_ERR_CUDA;
        }
        const double a0 = ah[0];
        bool ok = true;
        for (double v : ah) ok = ok && std::fabs(v - a0) <= 1e-14 * a0;
        for (double v : gh) ok = ok && v == 0.0;
        for (int e = 0; e < b->Me; ++e) ok = ok && std::fabs(edge_a[e] - a0) <= 1e-14 * a0;
        for (int j = 0; j < b->Fo; ++j) ok = ok && std::fabs(over_a[j] - a0) <= 1e-14 * a0;
        if (!ok) {
            pm_set_error("pm_bvp_create: the Dirichlet system needs a constant coefficient "
                         "(on the surface, the edge nodes and the oversampled points)");
            delete b;
            return PM_ERR_INVALID_ARG;
        }
    }
    const pm_status st = create_impl(b, edge_x, edge_d1, edge_d2, edge_nu, edge_a, edge_patch,
                                     edge_uv, over_x, over_nu, over_speed, over_a);
    if (st != PM_OK) {
        free_bvp(b);
        return st;
    }
    *out = b;
    return PM_OK;
}

extern "C" void pm_bvp_destroy(pm_bvp* b) { free_bvp(b); }

extern "C" pm_status pm_bvp_apply(pm_bvp* b, const double* sigma, const double* mu, double* out_s,
                                  double* out_e) {
    if (!b || !sigma || !out_s || (b->Me > 0 && (!mu || !out_e))) {
        pm_set_error("pm_bvp_apply: NULL argument");
        return PM_ERR_INVALID_ARG;
    }
    if (b->coeff_epoch != b->s->coeff_epoch) {
        pm_set_error("pm_bvp_apply: the surface's coefficient changed after pm_bvp_create");
        return PM_ERR_INVALID_ARG;
    }
    PM_CUDA_TRY(cudaSetDevice(b->s->ctx->device));
    const size_t n = (size_t)b->N + b->Me;
    double *z = nullptr, *y = nullptr;
    PM_TRY(pm_dmalloc(&z, n));
    pm_status st = pm_dmalloc(&y, n);
    if (st == PM_OK) {
        cudaError_t e = cudaMemcpy(z, sigma, sizeof(double) * b->N, cudaMemcpyHostToDevice);
        if (e == cudaSuccess && b->Me)
            e = cudaMemcpy(z + b->N, mu, sizeof(double) * b->Me, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) {
            pm_set_error("pm_bvp_apply: %s", cudaGetErrorString(e));
            st = PM_ERR_CUDA;
        }
    }
    if (st == PM_OK) st = apply_sys(b, z, y);
    if (st == PM_OK) {
        cudaError_t e = cudaMemcpy(out_s, y, sizeof(double) * b->N, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && b->Me) e = cudaMemcpy(out_e, y + b->N, sizeof(double) * b->Me, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) { pm_set_error("pm_bvp_apply: %s", cudaGetErrorString(e)); st = PM_ERR_CUDA; }
    }
    pm_dfree(z);
    pm_dfree(y);
    return st;
}

extern "C" pm_status pm_bvp_solve(pm_bvp* b, const double* f, const double* f_gamma, double tol,
                                  int maxit, double* u, double* sigma_out, double* mu_out,
                                  pm_solve_info* info) {
    if (!b || !f || !u || (b->Me > 0 && !f_gamma) || !(tol > 0.0) || maxit < 1) {
        pm_set_error("pm_bvp_solve: NULL argument, tol <= 0 or maxit < 1");
        return PM_ERR_INVALID_ARG;
    }
    if (b->coeff_epoch != b->s->coeff_epoch) {
        pm_set_error("pm_bvp_solve: the surface's coefficient changed after pm_bvp_create");
        return PM_ERR_INVALID_ARG;
    }
    PM_CUDA_TRY(cudaSetDevice(b->s->ctx->device));
    const int n = b->N + b->Me;
    const int m = std::max(2, std::min(b->s->opts.gmres_restart, 120));
    double *V = nullptr, *w = nullptr, *rhs = nullptr, *x = nullptr, *ud = nullptr;
    pm_arnoldi::Steps<double> steps;
    double* A = nullptr;                 // the system's matrix, where the device has room for it
    pm_status st = pm_dmalloc(&V, (size_t)(m + 1) * n);
    if (st == PM_OK) st = pm_dmalloc(&w, (size_t)n);
    if (st == PM_OK) st = pm_dmalloc(&rhs, (size_t)n);
    if (st == PM_OK) st = pm_dmalloc(&x, (size_t)n);
    if (st == PM_OK) st = steps.create(n, m);
    if (st == PM_OK) st = pm_dmalloc(&ud, (size_t)b->N);
    auto cleanup = [&]() {
        pm_dfree(V); pm_dfree(w); pm_dfree(rhs); pm_dfree(x); pm_dfree(ud);
        steps.release();
        if (A) cudaFreeAsync(A, b->st);
    };
    if (st != PM_OK) { cleanup(); return st; }
    const auto t0 = std::chrono::steady_clock::now();
    {
        cudaError_t e = cudaMemcpy(rhs, f, sizeof(double) * b->N, cudaMemcpyHostToDevice);
        if (e == cudaSuccess && b->Me)
            e = cudaMemcpy(rhs + b->N, f_gamma, sizeof(double) * b->Me, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemset(x, 0, sizeof(double) * n);
        if (e != cudaSuccess) {
            pm_set_error("pm_bvp_solve: %s", cudaGetErrorString(e));
            cleanup();
            return PM_ERR_CUDA;
        }
    }
    const int grid = pm_ceil_div(n, kT);
    double bnorm = 0.0;
    if ((st = steps.begin(rhs, V, b->st, &bnorm)) != PM_OK) { cleanup(); return st; }   // x = 0: r = rhs
    int iters = 0;
    double relres = bnorm == 0.0 ? 0.0 : std::isfinite(bnorm) ? 1.0 : NAN;
    std::vector<double> H((size_t)(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
    if (relres > tol) {
        const size_t need = sizeof(double) * (size_t)n * n;
        if (pm_matrix_fits(need) && cudaMallocAsync((void**)&A, need, b->st) != cudaSuccess)
            A = nullptr;
        cudaGetLastError();
        if (A && (st = fill_sys(b, A)) != PM_OK) { cleanup(); return st; }
    }
    double beta = bnorm;
    // A V_k and its orthogonalisation; through the matrix the next step is started before this
    // one's coefficients are looked at (the last one in vain)
    auto step = [&](int k) -> pm_status {
        PM_TRY(apply_any(b, A, V + (size_t)k * n, w));
        return steps.step(V, n, k, w, b->st);
    };
    while (st == PM_OK && relres > tol && iters < maxit) {       // an undefined residual ends it
        std::fill(g.begin(), g.end(), 0.0);
        g[0] = beta;
        int k = 0, started = 0;
        for (; k < m && iters < maxit; ++k, ++iters) {
            if (started == k && (st = step(started++)) != PM_OK) break;
            if (A && started < m && iters + 1 < maxit && (st = step(started++)) != PM_OK) break;
            const double* c = nullptr;
            double hn = 0.0;
            if ((st = steps.wait(k, &c, &hn)) != PM_OK) break;
            for (int j = 0; j <= k; ++j) H[(size_t)j * m + k] = c[j] + c[k + 1 + j];
            H[(size_t)(k + 1) * m + k] = hn;
            // Givens rotations
            for (int j = 0; j < k; ++j) {
                const double a0 = H[(size_t)j * m + k], a1 = H[(size_t)(j + 1) * m + k];
                H[(size_t)j * m + k] = cs[j] * a0 + sn[j] * a1;
                H[(size_t)(j + 1) * m + k] = -sn[j] * a0 + cs[j] * a1;
            }
            const double a0 = H[(size_t)k * m + k], a1 = H[(size_t)(k + 1) * m + k];
            const double rr = std::hypot(a0, a1);
            cs[k] = rr > 0 ? a0 / rr : 1.0;
            sn[k] = rr > 0 ? a1 / rr : 0.0;
            H[(size_t)k * m + k] = rr;
            H[(size_t)(k + 1) * m + k] = 0.0;
            g[k + 1] = -sn[k] * g[k];
            g[k] = cs[k] * g[k];
            relres = std::fabs(g[k + 1]) / bnorm;
            if (relres <= tol || hn == 0.0) { ++k; ++iters; break; }
        }
        if (st != PM_OK) break;
        // x += V y, H y = g (upper triangular k x k)
        for (int i = k - 1; i >= 0; --i) {
            double t = g[i];
            for (int j = i + 1; j < k; ++j) t -= H[(size_t)i * m + j] * y[j];
            y[i] = t / H[(size_t)i * m + i];
        }
        if (k > 0 && (st = steps.combine(V, n, k, y.data(), x, b->st)) != PM_OK) break;
        // the true residual r = b - A x
        if ((st = apply_any(b, A, x, w)) != PM_OK) break;
        k_bvp_rsub<<<grid, kT, 0, b->st>>>(n, rhs, w);
        if ((st = steps.begin(w, V, b->st, &beta)) != PM_OK) break;
        relres = beta / bnorm;
    }
    if (st == PM_OK) st = represent(b, x, ud);
    if (st == PM_OK) {
        cudaError_t e = cudaMemcpy(u, ud, sizeof(double) * b->N, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && sigma_out) e = cudaMemcpy(sigma_out, x, sizeof(double) * b->N, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess && mu_out && b->Me)
            e = cudaMemcpy(mu_out, x + b->N, sizeof(double) * b->Me, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) { pm_set_error("pm_bvp_solve: %s", cudaGetErrorString(e)); st = PM_ERR_CUDA; }
    }
    if (st == PM_OK && !(relres <= tol)) {
        pm_set_error("pm_bvp_solve: relative residual %.3e above %.3e after %d iterations", relres, tol, iters);
        st = PM_ERR_NOT_CONVERGED;
    }
    if (info) {
        info->iterations = iters;
        info->refinements = 0;
        info->residual = relres;
        info->removed_mean = 0.0;
        info->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        info->residual_updates = 0;
    }
    cleanup();
    return st;
}
