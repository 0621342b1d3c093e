// Ensemble-space Gram C = a I + Yh^T Yh and b = Yh^T d-hat of the
// mixed-precision analysis in double-binary32 (arXiv 2308.03972, Section
// 3.2; sm_103a).
//
// All nvar scalars of an observation point share its localisation weight G,
// so C = a I + sum_j G_j O_j with O_j = sum_q y_q y_q^T / sigma_q^2 over the
// scalars q of point j, the same for every grid point. The upper triangles
// of the O_j are formed once per analysis in FP64 and kept as binary32 pairs
// (outer_kernel); the pass over the grid points is then one product of the
// weights with them: per grid point k (k + 1) / 2 entries times the local
// points, against k^2 entries times nvar as many scalars when the rows
// themselves are multiplied (up to 32 members; gram_by_outer says why).
//
// gram_outer_kernel is bound by the binary32 pipe (twelve operations per
// multiply-add: the exact product, the two cross terms, TwoSum and the error
// sum, two grid points per packed instruction). A block takes kPts
// consecutive grid points, whose local sets are nearly the same: an entry of
// O_j is read once (from L2) for all of them. 256^2 lattice, rows multiplied
// against this: 16 members with 32^2 points 7.4 -> 1.8 ms, 32 members with
// 16^2 points 3.9 -> 1.3 ms (both figures include the weights' part: 5.3 and
// 2.0 ms before their table).
#include <cmath>
#include <cstdint>

#include "lbm_internal.cuh"
#include "letkf_device.cuh"

namespace lbmgpu {
namespace {

constexpr int kPts = 8;    // grid points per block
constexpr int kThr = 288;  // most threads per block, and observation points per stage

// Row and column (i <= m) of entry e of an upper triangle stored by rows.
__device__ __forceinline__ void entry_at(int e, int k, int& i, int& m) {
    const float t = (float)(2 * k + 1);
    int r = (int)((t - sqrtf(fmaxf(t * t - 8.0f * (float)e, 0.0f))) * 0.5f);
    r = r < 0 ? 0 : (r > k - 1 ? k - 1 : r);
    while (r > 0 && r * k - r * (r - 1) / 2 > e) --r;
    while ((r + 1) * k - (r + 1) * r / 2 <= e) ++r;
    i = r;
    m = r + e - (r * k - r * (r - 1) / 2);
}

// O_j as (high, low) pairs [npts][k (k + 1) / 2] and R_j = sum_q y_q d_q / sigma_q^2
// [npts][k], one block per observation point.
__global__ void outer_kernel(ObsParams o, int k, float2* __restrict__ O, double* __restrict__ R) {
    __shared__ double ys[3][kOuterMaxK], yw[3][kOuterMaxK];
    const int j = blockIdx.x, nv = o.nvar, ne = k * (k + 1) / 2;
    for (int e = threadIdx.x; e < nv * k; e += blockDim.x) {
        const int q = e / k, m = e % k;
        const double s = q == 0 ? o.sigma_u : (q == 1 ? o.sigma_v : o.sigma_r);
        const double y = o.dY[(size_t)(nv * j + q) * k + m];
        ys[q][m] = y;
        yw[q][m] = y / (s * s);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < ne; e += blockDim.x) {
        int i, m;
        entry_at(e, k, i, m);
        double v = 0.0;
        for (int q = 0; q < nv; ++q) v = fma(ys[q][i], yw[q][m], v);
        const float h = (float)v;
        O[(size_t)j * ne + e] = make_float2(h, (float)(v - (double)h));
    }
    for (int m = threadIdx.x; m < k; m += blockDim.x) {
        double v = 0.0;
        for (int q = 0; q < nv; ++q) v = fma(yw[q][m], o.d[nv * j + q], v);
        R[(size_t)j * k + m] = v;
    }
}

// ENT: entries of C per thread and pass; blockDim.x <= kThr threads.
template <int ENT>
__global__ void __launch_bounds__(kThr, 2) gram_outer_kernel(GramArgs g, double aa) {
    __shared__ __align__(16) float Wh[kThr][kPts], Wl[kThr][kPts];  // G = Wh + Wl of (point j, grid point)
    __shared__ double Wd[kThr][kPts];
    __shared__ int U[kThr], wcount[kThr / 32], pcnt[kPts];
    const ObsParams& o = g.o;
    const int tid = threadIdx.x, nt = blockDim.x, w = tid >> 5, lane = tid & 31;
    const int li0 = blockIdx.x * kPts;
    const int k = g.k, ne = k * (k + 1) / 2;
    const int npt = min(kPts, g.ncell - li0);
    const long long lim2 = support_lim2(g.d_cut);
    const float aah = (float)aa, aal = (float)(aa - (double)aah);
    constexpr int NB = (kPts * kOuterMaxK + 95) / 96;  // entries of b per thread, at least 96 threads
    double bacc[NB];
#pragma unroll
    for (int t = 0; t < NB; ++t) bacc[t] = 0.0;
    if (tid < kPts) pcnt[tid] = 0;
    __syncthreads();

    // Adds the first `rows` staged points to C (from zero when first; with
    // the diagonal a and renormalised when last) and to b.
    auto add = [&](int rows, bool first, bool last) {
        for (int e0 = 0; e0 < ne; e0 += nt * ENT) {
            int e[ENT], ei[ENT], em[ENT];
            f2x S[ENT][kPts / 2], C[ENT][kPts / 2];
#pragma unroll
            for (int u = 0; u < ENT; ++u) {
                const int t = e0 + u * nt + tid;
                e[u] = t < ne ? t : ne - 1;
                entry_at(e[u], k, ei[u], em[u]);
#pragma unroll
                for (int p = 0; p < kPts / 2; ++p) {
                    S[u][p] = C[u][p] = 0ull;
                    if (!first) {
                        float s[2] = {0.0f, 0.0f}, c[2] = {0.0f, 0.0f};
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (2 * p + h < npt) {
                                const size_t at = ((size_t)(li0 + 2 * p + h) * k + ei[u]) * k + em[u];
                                s[h] = g.C32[at];
                                c[h] = g.Clo[at];
                            }
                        S[u][p] = f2pack(s[0], s[1]);
                        C[u][p] = f2pack(c[0], c[1]);
                    }
                }
            }
#pragma unroll 4
            for (int r = 0; r < rows; ++r) {
                const float2* row = g.O + (size_t)U[r] * ne;
                float2 ov[ENT];
#pragma unroll
                for (int u = 0; u < ENT; ++u) ov[u] = __ldg(row + e[u]);
                const ulonglong2 h0 = *reinterpret_cast<const ulonglong2*>(&Wh[r][0]);
                const ulonglong2 h1 = *reinterpret_cast<const ulonglong2*>(&Wh[r][4]);
                const ulonglong2 l0 = *reinterpret_cast<const ulonglong2*>(&Wl[r][0]);
                const ulonglong2 l1 = *reinterpret_cast<const ulonglong2*>(&Wl[r][4]);
                const f2x wh[4] = {h0.x, h0.y, h1.x, h1.y}, wl[4] = {l0.x, l0.y, l1.x, l1.y};
#pragma unroll
                for (int u = 0; u < ENT; ++u) {
                    const f2x H = f2pack(ov[u].x, ov[u].x), NH = f2pack(-ov[u].x, -ov[u].x);
                    const f2x L = f2pack(ov[u].y, ov[u].y);
#pragma unroll
                    for (int p = 0; p < kPts / 2; ++p) {
                        df2_acc(S[u][p], C[u][p], wh[p], wl[p], H, NH);
                        C[u][p] = f2fma(wh[p], L, C[u][p]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < ENT; ++u) {
                if (e0 + u * nt + tid >= ne) continue;
#pragma unroll
                for (int p = 0; p < kPts / 2; ++p) {
                    float s[2], c[2];
                    f2unpack(S[u][p], s[0], s[1]);
                    f2unpack(C[u][p], c[0], c[1]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (2 * p + h >= npt) continue;
                        float hi = s[h], lo = c[h];
                        if (last) df_pair_out(s[h], c[h], ei[u] == em[u], aah, aal, hi, lo);
                        const size_t base = (size_t)(li0 + 2 * p + h) * k * k;
                        g.C32[base + (size_t)ei[u] * k + em[u]] = hi;
                        g.Clo[base + (size_t)ei[u] * k + em[u]] = lo;
                        if (last && ei[u] != em[u]) {
                            g.C32[base + (size_t)em[u] * k + ei[u]] = hi;
                            g.Clo[base + (size_t)em[u] * k + ei[u]] = lo;
                        }
                    }
                }
            }
        }
        // b in FP64: thread t takes entries t, t + nt, ... of [kPts][k].
#pragma unroll
        for (int t = 0; t < NB; ++t) {
            const int e = tid + t * nt;
            if (e >= kPts * k) break;
            const int q = e / k, m = e % k;
            double s = bacc[t];
#pragma unroll 4
            for (int r = 0; r < rows; ++r) s = fma(Wd[r][q], __ldg(g.R + (size_t)U[r] * k + m), s);
            bacc[t] = s;
            if (last && q < npt) g.b64[(size_t)(li0 + q) * k + m] = s;
        }
    };

    int total = 0;
    bool first = true;
    for (int j0 = 0; j0 < o.npts; j0 += nt) {
        const int j = j0 + tid;
        double gw[kPts];
        bool in = false;
#pragma unroll
        for (int q = 0; q < kPts; ++q) {
            gw[q] = 0.0;
            if (j < o.npts && q < npt) {
                const int cell = g.cell0 + li0 + q;
                gw[q] = point_weight(o, j, cell % g.nx, cell / g.nx, g.nx, g.ny, g.d_cut, lim2, 0);
            }
            const unsigned bq = __ballot_sync(kFull, gw[q] > 0.0);
            if (lane == 0 && bq) atomicAdd(&pcnt[q], __popc(bq));
            in |= gw[q] > 0.0;
        }
        const unsigned bal = __ballot_sync(kFull, in);
        if (lane == 0) wcount[w] = __popc(bal);
        __syncthreads();
        int off = 0, n = 0;
        for (int q = 0; q < nt / 32; ++q) {
            if (q < w) off += wcount[q];
            n += wcount[q];
        }
        if (total + n > kThr) {  // the stage is full (n <= nt)
            add(total, first, false);
            first = false;
            total = 0;
            __syncthreads();
        }
        if (in) {
            const int r = total + off + __popc(bal & ((1u << lane) - 1u));
            U[r] = j;
#pragma unroll
            for (int q = 0; q < kPts; ++q) {
                const float h = (float)gw[q];
                Wh[r][q] = h;
                Wl[r][q] = (float)(gw[q] - (double)h);
                Wd[r][q] = gw[q];
            }
        }
        total += n;
        __syncthreads();
    }
    bool any_ens = false;
    for (int q = 0; q < npt; ++q) any_ens |= pcnt[q] * o.nvar >= k;
    if (!any_ens) return;
    add(total, first, true);
}

}  // namespace

size_t gram_outer_bytes(int npts, int k) {
    return (size_t)npts * ((size_t)k * (k + 1) / 2 * sizeof(float2) + (size_t)k * sizeof(double));
}

void gram_outer_at(void* base, int npts, int k, GramArgs* g) {
    g->R = reinterpret_cast<double*>(base);
    g->O = reinterpret_cast<float2*>(g->R + (size_t)npts * k);
}

cudaError_t launch_outer(const GramArgs& g, cudaStream_t s) {
    if (g.k > kOuterMaxK || g.o.npts < 1) return cudaErrorInvalidValue;
    outer_kernel<<<(unsigned)g.o.npts, 256, 0, s>>>(g.o, g.k, g.O, g.R);
    return cudaGetLastError();
}

cudaError_t launch_gram_outer(const GramArgs& g, double aa, cudaStream_t s) {
    if (g.k > kOuterMaxK) return cudaErrorInvalidValue;
    // Threads and entries per thread that leave the fewest lanes idle in the
    // passes over the triangle (k = 16: 160 threads of one entry, 85% busy
    // against 27% of 256 threads of two; k = 32: 288 of two, 92% against 52%).
    const int ne = g.k * (g.k + 1) / 2;
    int best = 1 << 30, nt = 96, ent = 1;
    for (int t = kThr; t >= 96; t -= 32)
        for (int u = 2; u >= 1; --u) {
            const int slots = (ne + t * u - 1) / (t * u) * t * u;
            if (slots < best) {
                best = slots;
                nt = t;
                ent = u;
            }
        }
    const unsigned grid = (unsigned)((g.ncell + kPts - 1) / kPts);
    if (ent == 2)
        gram_outer_kernel<2><<<grid, nt, 0, s>>>(g, aa);
    else
        gram_outer_kernel<1><<<grid, nt, 0, s>>>(g, aa);
    return cudaGetLastError();
}

}  // namespace lbmgpu
