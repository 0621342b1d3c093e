// Ensemble diagnostics (arXiv 2308.03972, Section 4.1 energy spectrum):
// E(s) = mean over members of sum_{s - 1/2 <= |k'| < s + 1/2} |u-hat(k')|^2 / 2,
// u-hat(k') = N^{-1} sum_xi u(xi) exp(-i k'.xi), both velocity components.
//
// One complex transform serves both components: with z = u + i v,
// |u-hat(k')|^2 + |v-hat(k')|^2 = (|z-hat(k')|^2 + |z-hat(-k')|^2) / 2, and k' and
// -k' lie in the same shell, so a shell's sum is that of |z-hat|^2 / 2.
// Three passes, all FP64:
//  (1) rows: per lattice row and member group, the velocity is formed from
//      the nine f's and transformed along x;
//  (2) columns: per kx and member group, the x-transforms are transformed
//      along y and |z-hat|^2 / 2 is summed over the group's members and, per
//      shell in ky order, into a partial row;
//  (3) reduce: per shell, the partials in a fixed order (the result does not
//      depend on scheduling).
// The transforms are Stockham FFTs in shared memory (Cochran et al., "What is
// the fast Fourier transform?", 1967; Van Loan, "Computational Frameworks for
// the FFT", 1992) of any length: radix 4 and 2, and direct sums over pairs of
// inputs and outputs for the odd prime factors (one by one, 1613 x 4 x 1 took
// 2.75 ms, 257 x 251 x 8 2.16 and 500 x 428 x 9 2.93; in pairs 0.82, 0.66 and
// 1.51). Bound by GB300's FP64 pipe (two operations per SM cycle):
// 7 operations per point and radix-4 stage, so about 56 per point at 256^2.
// Direct transforms, O(nx + ny) per point, took 13.7 + 4.2 ms at
// 256^2 x 64 and their one-thread-per-shell sum 1.0 ms; rows, columns and
// reduction now take 0.61, 0.49 and 0.005 ms.
#include <cmath>

#include "lbm_internal.cuh"
#include "vec.cuh"

namespace lbmgpu {
namespace {

constexpr int kFftThreads = 256;
constexpr int kFftStages = 32;  // prime factors of a 32-bit length

// Stages of a length-n transform: radices in order (4s, then 2, then odd
// primes in increasing order).
struct FftPlan {
    int n, stages;
    int radix[kFftStages];
};

FftPlan fft_plan(int n) {
    FftPlan p{};
    p.n = n;
    int m = n;
    while (m % 4 == 0) {
        p.radix[p.stages++] = 4;
        m /= 4;
    }
    for (int r = 2; (long long)r * r <= m; ++r)
        while (m % r == 0) {
            p.radix[p.stages++] = r;
            m /= r;
        }
    if (m > 1) p.radix[p.stages++] = m;
    return p;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// tw[j] = exp(-2 pi i j / n), the angle reduced to j / n in [0, 1).
__device__ __forceinline__ void fft_twiddles(double2* tw, int n) {
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double sn, cs;
        sincospi(2.0 * (double)j / (double)n, &sn, &cs);
        tw[j] = make_double2(cs, -sn);
    }
}

// Forward transforms of G interleaved sequences x[j * G + m], ping-pong
// between a and b; returns the buffer that holds the result. Stage with
// radix r after a product L of earlier radices: for j < n / r, kk = j mod L,
//   y[(j / L) L r + kk + p L] = sum_q x[j + q n / r] w^{q kk n / (L r)} w^{p q n / r},
// w = exp(-2 pi i / n). Consecutive threads take consecutive members, then
// consecutive j, so shared accesses are contiguous. Block-wide; begins and
// ends with a barrier.
__device__ double2* fft_block(double2* a, double2* b, const double2* tw, const FftPlan& p, int G) {
    const int n = p.n;
    int L = 1;
    for (int st = 0; st < p.stages; ++st) {
        const int r = p.radix[st], nr = n / r, step = nr / L;  // step = n / (L r)
        __syncthreads();
        if (r == 4) {
            for (int t = threadIdx.x; t < nr * G; t += kFftThreads) {
                const int j = t / G, m = t - j * G, hi = j / L, kk = j - hi * L;
                double2 x0 = a[t], x1 = a[t + nr * G], x2 = a[t + 2 * nr * G], x3 = a[t + 3 * nr * G];
                if (L > 1) {
                    x1 = cmul(x1, tw[kk * step]);
                    x2 = cmul(x2, tw[2 * kk * step]);
                    x3 = cmul(x3, tw[3 * kk * step]);
                }
                const double2 s02 = cadd(x0, x2), d02 = csub(x0, x2), s13 = cadd(x1, x3), d13 = csub(x1, x3);
                double2* y = b + (size_t)(hi * L * 4 + kk) * G + m;
                y[0] = cadd(s02, s13);
                y[L * G] = make_double2(d02.x + d13.y, d02.y - d13.x);
                y[2 * L * G] = csub(s02, s13);
                y[3 * L * G] = make_double2(d02.x - d13.y, d02.y + d13.x);
            }
        } else if (r == 2) {
            for (int t = threadIdx.x; t < nr * G; t += kFftThreads) {
                const int j = t / G, m = t - j * G, hi = j / L, kk = j - hi * L;
                const double2 x0 = a[t];
                double2 x1 = a[t + nr * G];
                if (L > 1) x1 = cmul(x1, tw[kk * step]);
                double2* y = b + (size_t)(hi * L * 2 + kk) * G + m;
                y[0] = cadd(x0, x1);
                y[L * G] = csub(x0, x1);
            }
        } else {
            // Odd r: with s_q = x_q + x_{r-q} and d_q = x_q - x_{r-q} (formed in
            // place, the stage's twiddles first), outputs p and r - p are
            // x_0 + sum_q s_q Re w^{pq n/r} +- i sum_q d_q Im w^{pq n/r}, q < r/2:
            // r^2 multiply-adds per transform instead of 4 r^2.
            const int h = (r - 1) / 2;
            for (int t = threadIdx.x; t < h * nr * G; t += kFftThreads) {
                const int q = t / (nr * G) + 1, jm = t - (q - 1) * nr * G, kk = (jm / G) % L;
                double2 &u = a[q * nr * G + jm], &v = a[(r - q) * nr * G + jm];
                const double2 x = cmul(u, tw[q * kk * step]), z = cmul(v, tw[(r - q) * kk * step]);
                u = cadd(x, z);
                v = csub(x, z);
            }
            __syncthreads();
            for (int t = threadIdx.x; t < (h + 1) * nr * G; t += kFftThreads) {
                const int pp = t / (nr * G), jm = t - pp * nr * G, j = jm / G, m = jm - j * G;
                const int hi = j / L, kk = j - hi * L;
                const int ex = pp * nr;
                double2 e = a[jm], o = make_double2(0.0, 0.0);
                int idx = 0;
                for (int q = 1; q <= h; ++q) {
                    idx += ex;
                    if (idx >= n) idx -= n;
                    const double2 w = tw[idx], sq = a[q * nr * G + jm], dq = a[(r - q) * nr * G + jm];
                    e.x = fma(sq.x, w.x, e.x);
                    e.y = fma(sq.y, w.x, e.y);
                    o.x = fma(-dq.y, w.y, o.x);
                    o.y = fma(dq.x, w.y, o.y);
                }
                double2* y = b + (size_t)(hi * L * r + kk) * G + m;
                y[(size_t)pp * L * G] = cadd(e, o);
                if (pp > 0) y[(size_t)(r - pp) * L * G] = csub(e, o);
            }
        }
        L *= r;
        double2* c = a;
        a = b;
        b = c;
    }
    __syncthreads();
    return a;
}

// Pass 1. Grid (ny, groups of G members). Shared: two buffers [nx][G]
// complex, twiddles [nx]. Output F1 [ny][nx][k] complex.
template <typename T, bool SHIFT>
__global__ void __launch_bounds__(kFftThreads) spectrum_rows_kernel(const T* __restrict__ f, int nx, int ny, int k,
                                                                    int G, const __grid_constant__ FftPlan plan,
                                                                    double2* __restrict__ F1,
                                                                    int* __restrict__ flags) {
    extern __shared__ __align__(16) double2 shz[];
    double2 *za = shz, *zb = za + (size_t)nx * G, *tw = zb + (size_t)nx * G;
    const int y = blockIdx.x;
    const int m0 = blockIdx.y * G;
    const size_t plane = (size_t)nx * ny * k;
    fft_twiddles(tw, nx);
    bool bad = false;
    for (int t = threadIdx.x; t < nx * G; t += kFftThreads) {
        const int x = t / G, m = m0 + t - x * G;
        double2 z = make_double2(0.0, 0.0);
        if (m < k) {
            const size_t i = ((size_t)y * nx + x) * k + m;
            double g[9], r;
#pragma unroll
            for (int a = 0; a < 9; ++a) g[a] = widen(f[a * plane + i]);
            moments_of<SHIFT>(g, r, z.x, z.y);
            bad |= !(r > 0.0) || !(z.x * z.x + z.y * z.y <= kUMax2);
        }
        za[t] = z;
    }
    if (bad) atomicOr(flags, FLAG_DIVERGED);
    const double2* z = fft_block(za, zb, tw, plan, G);
    for (int t = threadIdx.x; t < nx * G; t += kFftThreads) {
        const int x = t / G, m = m0 + t - x * G;
        if (m < k) F1[((size_t)y * nx + x) * k + m] = z[t];
    }
}

// Pass 2. Grid (nx, groups of G members). Shared: two buffers [ny][G]
// complex, twiddles [ny]; the energies and the shell of each ky [ny] take the
// buffer that the transform leaves free. Output P [groups][nx][nsh].
__global__ void __launch_bounds__(kFftThreads) spectrum_cols_kernel(const double2* __restrict__ F1, int nx, int ny,
                                                                    int k, int G,
                                                                    const __grid_constant__ FftPlan plan, int nsh,
                                                                    double* __restrict__ P) {
    extern __shared__ __align__(16) double2 shz[];
    double2 *za = shz, *zb = za + (size_t)ny * G, *tw = zb + (size_t)ny * G;
    const int x = blockIdx.x;
    const int m0 = blockIdx.y * G;
    fft_twiddles(tw, ny);
    for (int t = threadIdx.x; t < ny * G; t += kFftThreads) {
        const int y = t / G, m = m0 + t - y * G;
        za[t] = m < k ? F1[((size_t)y * nx + x) * k + m] : make_double2(0.0, 0.0);
    }
    const double2* z = fft_block(za, zb, tw, plan, G);
    double* e = reinterpret_cast<double*>(z == za ? zb : za);
    int* shell = reinterpret_cast<int*>(e + ny);
    const int kx = 2 * x > nx ? x - nx : x;
    const double inv_n = 1.0 / ((double)nx * (double)ny);
    for (int y = threadIdx.x; y < ny; y += kFftThreads) {
        double s = 0.0;
        for (int m = 0; m < G; ++m) {
            const double2 v = z[(size_t)y * G + m];
            s += v.x * v.x + v.y * v.y;
        }
        e[y] = 0.5 * inv_n * inv_n * s;
        const int ky = 2 * y > ny ? y - ny : y;
        shell[y] = (int)floor(sqrt((double)kx * kx + (double)ky * ky) + 0.5);
    }
    __syncthreads();
    double* out = P + ((size_t)blockIdx.y * nx + x) * nsh;
    for (int s = threadIdx.x; s < nsh; s += kFftThreads) {
        double acc = 0.0;
        for (int y = 0; y < ny; ++y)
            if (shell[y] == s) acc += e[y];
        out[s] = acc;
    }
}

// Pass 3. One block per shell: rows of P in a fixed order.
__global__ void __launch_bounds__(kFftThreads) spectrum_reduce_kernel(const double* __restrict__ P, long long rows,
                                                                      int k, int nsh, double* __restrict__ E) {
    __shared__ double red[kFftThreads];
    const int s = blockIdx.x;
    double acc = 0.0;
    for (long long r = threadIdx.x; r < rows; r += kFftThreads) acc += P[(size_t)r * nsh + s];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int h = kFftThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) E[s] = red[0] / k;
}

// RMSE of two velocity fields (Section 4.3 scores the ensemble mean
// against the truth): sum over cells of (u1 - u2)^2 + (v1 - v2)^2 in FP64,
// block partials in a fixed order, then one block sums the partials in
// order and writes sqrt(sum / n).
constexpr int kRmseBlocks = 256, kRmseThreads = 256;

__global__ void __launch_bounds__(kRmseThreads) rmse_partial_kernel(const double* __restrict__ u1,
                                                                   const double* __restrict__ v1,
                                                                   const double* __restrict__ u2,
                                                                   const double* __restrict__ v2, size_t n,
                                                                   double* __restrict__ partial) {
    __shared__ double red[kRmseThreads];
    double s = 0.0;
    for (size_t i = (size_t)blockIdx.x * kRmseThreads + threadIdx.x; i < n; i += (size_t)kRmseBlocks * kRmseThreads) {
        const double du = u1[i] - u2[i], dv = v1[i] - v2[i];
        s += du * du + dv * dv;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = kRmseThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(kRmseThreads) rmse_final_kernel(const double* __restrict__ partial, size_t n,
                                                                 double* __restrict__ out) {
    __shared__ double red[kRmseThreads];
    red[threadIdx.x] = threadIdx.x < kRmseBlocks ? partial[threadIdx.x] : 0.0;
    __syncthreads();
    for (int h = kRmseThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sqrt(red[0] / (double)n);
}

}  // namespace

constexpr size_t kMaxShared = 227 * 1024;

static size_t fft_shared(int n, int G) { return (2 * (size_t)G + 1) * n * sizeof(double2); }

// Members per block: eight (32- or 64-byte runs of f, 128-byte runs of F1)
// while two blocks fit an SM, fewer on long rows and columns.
static int spectrum_group(int n) {
    int G = 8;
    while (G > 1 && fft_shared(n, G) > kMaxShared / 2) G /= 2;
    return G;
}

size_t spectrum_work_bytes(int nx, int ny, int k, int nshells) {
    const int G = spectrum_group(ny);
    return (size_t)k * ny * nx * sizeof(double2) + (size_t)((k + G - 1) / G) * nx * nshells * sizeof(double);
}

cudaError_t launch_energy_spectrum(const void* f, int fp32, int nx, int ny, int k, double* E,
                                   int nshells, void* work, int* flags, cudaStream_t s) {
    // The lattice sizes the diagnostic takes: rows of up to 1,614 cells, and
    // columns and shells within 227 KB at 56 bytes a cell and 8 a shell. One
    // member per block needs 48 bytes a cell, so all of them fit.
    const size_t lim1 = (size_t)nx * 144, lim2 = 56 * (size_t)ny + 8 * (size_t)nshells;
    if (lim1 > kMaxShared || lim2 > kMaxShared) return cudaErrorInvalidValue;
    const int G1 = spectrum_group(nx), G2 = spectrum_group(ny);
    const size_t sh1 = fft_shared(nx, G1), sh2 = fft_shared(ny, G2);
    const int n1 = (k + G1 - 1) / G1, n2 = (k + G2 - 1) / G2;
    double2* F1 = reinterpret_cast<double2*>(work);
    double* P = reinterpret_cast<double*>(F1 + (size_t)k * ny * nx);
    const FftPlan px = fft_plan(nx), py = fft_plan(ny);
    auto rows = [&](auto kern, auto* ff) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh1);
        if (e != cudaSuccess) return e;
        kern<<<dim3((unsigned)ny, (unsigned)n1), kFftThreads, sh1, s>>>(ff, nx, ny, k, G1, px, F1, flags);
        return cudaGetLastError();
    };
    cudaError_t e = fp32 ? rows(spectrum_rows_kernel<float, true>, (const float*)f)
                         : rows(spectrum_rows_kernel<double, false>, (const double*)f);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(spectrum_cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh2);
    if (e != cudaSuccess) return e;
    spectrum_cols_kernel<<<dim3((unsigned)nx, (unsigned)n2), kFftThreads, sh2, s>>>(F1, nx, ny, k, G2, py, nshells, P);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    spectrum_reduce_kernel<<<(unsigned)nshells, kFftThreads, 0, s>>>(P, (long long)n2 * nx, k, nshells, E);
    return cudaGetLastError();
}

size_t rmse_work_doubles() { return kRmseBlocks; }

cudaError_t launch_velocity_rmse(const double* u1, const double* v1, const double* u2, const double* v2, size_t n,
                                 double* work, double* out, cudaStream_t s) {
    if (n == 0) return cudaErrorInvalidValue;
    rmse_partial_kernel<<<kRmseBlocks, kRmseThreads, 0, s>>>(u1, v1, u2, v2, n, work);
    rmse_final_kernel<<<1, kRmseThreads, 0, s>>>(work, n, out);
    return cudaGetLastError();
}

}  // namespace lbmgpu
