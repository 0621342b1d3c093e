// Kernel (B) of the mixed-precision analysis for local problems of 33..128,
// and of some of 27..32 (launch_analyze draws the line; sm_103a): the refinement and transform of analyze_mixed_kernel
// (letkf_kernels.cu; arXiv 2308.03972, Section 3.2) by a block per grid
// point, with every n^3 product from register tiles.
//
// A thread owns an 8 x 4 tile of a product (two groups of four rows). Each
// entry's sum runs over the inner index in order with the roundings of the
// one-column-per-lane form, and S' is corrected in FP64 as there, so the
// results agree with it to the bit (but for entries of E and S whose sum of
// two halves is a binary32 tie after rounding to binary64, which that form
// rounds twice: about one in 2^29); per multiply-add it needs 3 / 32 shared
// 16-byte loads where that form needed two to four 4-byte ones and was bound
// by them. Three matrices are held in
// shared memory (A and then A Y as binary32 halves, and the basis), reused as
// the analysis proceeds; above 64 the older form kept A and A Y in global
// scratch.
//
// Double-binary32 products bound the kernel: A Y (eleven operations per
// multiply-add), and E = Y^T Y - I and S = Y^T (A Y), of which only the tiles
// that reach the upper triangle are formed. Per analysis, one column per lane
// against tiles: n = 64 at 256^2 points 59 -> 19.6 ms, n = 88..104 at 128^2
// 54 -> 26.1 ms.
#include <cmath>
#include <cstdint>

#include "lbm_internal.cuh"
#include "letkf_device.cuh"
#include "vec.cuh"

namespace lbmgpu {
namespace {

template <int KP>
struct WideB {
    static_assert(KP % 16 == 0, "tiles of 8 x 4");
    static constexpr int NCG = KP / 4;  // column groups
    static constexpr int NRG = KP / 8;  // row groups of the first half
    static constexpr int T = NCG * NRG;
    static constexpr int LD = (KP + 31) / 32 * 32;
    static constexpr int MAT = KP * LD;
    // 32: 16 KB, one warp, twelve per SM; 64: 55 KB, four blocks; 80: 101 KB, two;
    // above, one. kdx: members whose perturbations are staged (k, or 0).
    static constexpr size_t bytes(int kdx) {
        return sizeof(float) * (3 * (size_t)MAT + 10 * (size_t)KP + 9 * (size_t)kdx + 32) +
               KP * (3 * sizeof(double) + sizeof(int));
    }
};

constexpr size_t kMaxShared = 227 * 1024;

// Element group g (four columns) of row i: groups are permuted within
// 128-byte lines by the row's group, so that walking a column block along
// rows (a transposed tile) meets all banks.
template <int LD>
__device__ __forceinline__ int at4(int i, int g) {
    return i * LD + ((g ^ ((i >> 2) & 7)) << 2);
}
template <int LD>
__device__ __forceinline__ int at(int i, int j) {
    return at4<LD>(i, j >> 2) + (j & 3);
}

// Row of tile row q (0..7) for row group ti: two groups of four, half a
// matrix apart.
template <int KP>
__device__ __forceinline__ int tile_row(int ti, int q) {
    return (q < 4 ? 0 : KP / 2) + 4 * ti + (q & 3);
}

// acc[p][j] += sum_{k < n4} A[k][rows 2p, 2p+1] B[k][col j] of this thread's tile, k in order.
template <int KP>
__device__ __forceinline__ void tile_mul(const float* __restrict__ A, const float* __restrict__ B, int n4, int ti,
                                         int tj, f2x (&acc)[4][4]) {
    using RS = WideB<KP>;
    for (int k0 = 0; k0 < n4; k0 += 4) {
        const int sw = (k0 >> 2) & 7;
        const float* a0 = A + k0 * RS::LD + ((ti ^ sw) << 2);
        const float* a1 = A + k0 * RS::LD + (((RS::NRG + ti) ^ sw) << 2);
        const float* b0 = B + k0 * RS::LD + ((tj ^ sw) << 2);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(a0 + kk * RS::LD);
            const ulonglong2 p1 = *reinterpret_cast<const ulonglong2*>(a1 + kk * RS::LD);
            const float4 b = *reinterpret_cast<const float4*>(b0 + kk * RS::LD);
            const f2x ap[4] = {p0.x, p0.y, p1.x, p1.y};
            const float bj[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const f2x bb = f2pack(bj[j], bj[j]);
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[p][j] = f2fma(ap[p], bb, acc[p][j]);
            }
        }
    }
}

// The same in double-binary32, left factor A = Ah + Al, right factor B:
// (s, c)[p][j] over rows 2p, 2p + 1.
template <int KP>
__device__ __forceinline__ void tile_mul_df(const float* __restrict__ Ah, const float* __restrict__ Al,
                                            const float* __restrict__ B, int n, int ti, int tj, f2x (&s)[4][4],
                                            f2x (&c)[4][4]) {
    using RS = WideB<KP>;
    // One iteration is ~160 packed instructions; unrolled by four the three
    // products overflow the instruction cache up to 64 (B at 256^2: 5.9 -> 3.6 ms
    // at n = 32, 21.9 -> 18.9 at 64); above, one block per SM gains by it.
#pragma unroll (KP <= 64 ? 1 : 4)
    for (int k = 0; k < n; ++k) {
        const int sw = (k >> 2) & 7;
        const int o0 = k * RS::LD + ((ti ^ sw) << 2), o1 = k * RS::LD + (((RS::NRG + ti) ^ sw) << 2);
        const ulonglong2 h0 = *reinterpret_cast<const ulonglong2*>(Ah + o0);
        const ulonglong2 h1 = *reinterpret_cast<const ulonglong2*>(Ah + o1);
        const ulonglong2 l0 = *reinterpret_cast<const ulonglong2*>(Al + o0);
        const ulonglong2 l1 = *reinterpret_cast<const ulonglong2*>(Al + o1);
        const float4 b = *reinterpret_cast<const float4*>(B + k * RS::LD + ((tj ^ sw) << 2));
        const f2x ah[4] = {h0.x, h0.y, h1.x, h1.y}, al[4] = {l0.x, l0.y, l1.x, l1.y};
        const float bj[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const f2x bb = f2pack(bj[j], bj[j]), nb = f2pack(-bj[j], -bj[j]);
#pragma unroll
            for (int p = 0; p < 4; ++p) df2_acc(s[p][j], c[p][j], ah[p], al[p], bb, nb);
        }
    }
}

// Tile of eight consecutive rows 8 ri .. and four columns of A^T B in
// double-binary32, right factor B = Bh + Bl (LO) or Bh.
template <int KP, bool LO>
__device__ __forceinline__ void sym_mul_df(const float* __restrict__ A, const float* __restrict__ Bh,
                                           const float* __restrict__ Bl, int n, int ri, int tj, f2x (&s)[4][4],
                                           f2x (&c)[4][4]) {
    using RS = WideB<KP>;
#pragma unroll (KP <= 64 ? 1 : 4)
    for (int k = 0; k < n; ++k) {
        const int sw = (k >> 2) & 7;
        const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(A + k * RS::LD + (((2 * ri) ^ sw) << 2));
        const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(A + k * RS::LD + (((2 * ri + 1) ^ sw) << 2));
        const int ob = k * RS::LD + ((tj ^ sw) << 2);
        const float4 b = *reinterpret_cast<const float4*>(Bh + ob);
        float4 l = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (LO) l = *reinterpret_cast<const float4*>(Bl + ob);
        const f2x ap[4] = {a0.x, a0.y, a1.x, a1.y};
        const float bj[4] = {b.x, b.y, b.z, b.w}, lj[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const f2x bb = f2pack(bj[j], bj[j]), nb = f2pack(-bj[j], -bj[j]), ll = f2pack(lj[j], lj[j]);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                // df_acc with the halves on B's side: the product, its error
                // and the cross term are those of (bh + bl) a.
                const f2x NP = f2mul(ap[p], nb);
                f2x E = f2fma(ap[p], bb, NP);
                if (LO) E = f2fma(ap[p], ll, E);
                const f2x S1 = f2sub(s[p][j], NP);
                const f2x Z = f2sub(S1, s[p][j]);
                const f2x T = f2sub(f2sub(s[p][j], f2sub(S1, Z)), f2add(Z, NP));
                c[p][j] = f2add(c[p][j], f2add(T, E));
                s[p][j] = S1;
            }
        }
    }
}

__device__ __forceinline__ void tile_zero(f2x (&acc)[4][4]) {
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[p][j] = 0ull;
}

// v[q][j] of a tile held as packed row pairs.
__device__ __forceinline__ void tile_unpack(const f2x (&acc)[4][4], float (&v)[8][4]) {
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int j = 0; j < 4; ++j) f2unpack(acc[p][j], v[2 * p][j], v[2 * p + 1][j]);
}

template <int KP>
__device__ __forceinline__ void tile_load(const float* M, int ti, int tj, float (&v)[8][4]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 t = *reinterpret_cast<const float4*>(M + at4<WideB<KP>::LD>(tile_row<KP>(ti, q), tj));
        v[q][0] = t.x;
        v[q][1] = t.y;
        v[q][2] = t.z;
        v[q][3] = t.w;
    }
}
template <int KP>
__device__ __forceinline__ void tile_store(float* M, int ti, int tj, const float (&v)[8][4]) {
#pragma unroll
    for (int q = 0; q < 8; ++q)
        *reinterpret_cast<float4*>(M + at4<WideB<KP>::LD>(tile_row<KP>(ti, q), tj)) =
            make_float4(v[q][0], v[q][1], v[q][2], v[q][3]);
}
// Transposed store: M[column j][row q] = v[q][j].
template <int KP>
__device__ __forceinline__ void tile_store_t(float* M, int ti, int tj, const float (&v)[8][4]) {
    using RS = WideB<KP>;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        *reinterpret_cast<float4*>(M + at4<RS::LD>(4 * tj + j, ti)) = make_float4(v[0][j], v[1][j], v[2][j], v[3][j]);
        *reinterpret_cast<float4*>(M + at4<RS::LD>(4 * tj + j, RS::NRG + ti)) =
            make_float4(v[4][j], v[5][j], v[6][j], v[7][j]);
    }
}

// STAGED: the perturbations dX [9][k] are held in shared memory. Otherwise
// (ensembles that do not fit beside the matrices: from 751 members at KP = 128,
// from 1,464 at 112; always in observation space) they are formed from the
// state at each use; a thread's own values are the last it reads before it
// writes them.
template <int KP, bool STAGED>
__global__ void __launch_bounds__(WideB<KP>::T, KP <= 32 ? 12 : (KP <= 64 ? 4 : (KP <= 80 ? 2 : 1))) analyze_wide_kernel(WideArgs g) {
    using RS = WideB<KP>;
    constexpr int LD = RS::LD, T = RS::T, NW = T / 32;  // full warps
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* M1 = reinterpret_cast<float*>(smem_raw);  // A^T high half, A Y high half, S' off the diagonal, F, ...
    float* M2 = M1 + RS::MAT;                        // A^T low half, A Y low half, E, Y^T
    float* Y = M2 + RS::MAT;                         // the basis (binary32, exact); then the row arrays
    float* vf = Y + RS::MAT;                         // [KP] each:
    float* vu = vf + KP;
    float* vinv = vu + KP;
    float* t1 = vinv + KP;
    float* t2 = t1 + KP;
    float* vb = t2 + KP;  // and four more, for the nine rows of R0 below
    float* dX = vf + 10 * KP;  // [9][k]
    const int kdx = STAGED ? g.k : 0;
    float* xbar = dX + 9 * kdx;
    float* zv = xbar + 10;
    double* dS = reinterpret_cast<double*>(dX + 9 * kdx + 32 - (kdx & 1));
    double* lsq = dS + KP;
    double* ldh = lsq + KP;
    int* lidx = reinterpret_cast<int*>(ldh + KP);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ti = tid / RS::NCG, tj = tid % RS::NCG;
    const int k = g.k, nobs = g.o.nvar * g.o.npts;
    const int li = blockIdx.x;
    const int cell = g.cell0 + li;
    const int cap = g.o.plmax > 0 ? g.o.plmax : nobs;
    const size_t plane = (size_t)g.nx * g.ny * k;
    float* fc = g.f + (size_t)cell * k;

    // Ensemble mean and perturbations in binary32.
    for (int a = wid; a < 9 && wid < NW; a += NW) {
        float s = 0.0f;
        for (int m = lane; m < k; m += 32) {
            const float xv = fc[a * plane + m];
            if (STAGED) dX[a * k + m] = xv;
            s += xv;
        }
        const float mean = warp_sum(s) / (float)k;
        if (STAGED)
            for (int m = lane; m < k; m += 32) dX[a * k + m] -= mean;
        if (lane == 0) xbar[a] = mean;
    }
    auto dx = [&](int a, int m) { return STAGED ? dX[a * k + m] : __fsub_rn(fc[a * plane + m], xbar[a]); };
    const int p = g.pcount[li];
    if (p > cap) {
        if (tid == 0) atomicOr(g.flags, FLAG_TOOLARGE);
        return;
    }
    const bool obs_space = p < k;
    const int n = obs_space ? p : k;
    if (p > 0 && n > g.nm) {
        if (tid == 0) atomicOr(g.flags, FLAG_TOOLARGE);
        return;
    }
    if (obs_space)
        for (int i = tid; i < p; i += T) {
            const int oi = g.lidx[(size_t)li * cap + i];
            const double si = g.lsq[(size_t)li * cap + i];
            lidx[i] = oi;
            lsq[i] = si;
            ldh[i] = si * g.o.d[oi];
        }
    __syncthreads();
    if (p == 0) {
        const float sb = (float)sqrt(g.beta);
        for (int a = 0; a < 9; ++a)
            for (int m = tid; m < k; m += T) fc[a * plane + m] = xbar[a] + sb * dx(a, m);
        return;
    }
    const double aa = (k - 1) / g.beta;

    // A^T as two binary32 halves, and the basis; zero outside n x n.
    const float* Xp = g.X + (size_t)li * g.xr * g.xr;
    for (int e = tid; e < KP * KP; e += T) {
        const int i = e / KP, c = e % KP;
        float h = 0.0f, l = 0.0f, y = 0.0f;
        if (i < n && c < n) {
            const size_t at0 = (size_t)li * k * k + (size_t)i * k + c;
            if (obs_space || g.C64) {
                const double v = obs_space ? lsq[i] * g.o.G[(size_t)lidx[i] * nobs + lidx[c]] * lsq[c] : g.C64[at0];
                h = __double2float_rn(v);
                l = __double2float_rn(v - (double)h);
            } else {
                h = g.C32[at0];
                l = g.Clo ? g.Clo[at0] : 0.0f;
            }
            y = Xp[(size_t)i * g.xr + c];
        }
        M1[at<LD>(c, i)] = h;
        M2[at<LD>(c, i)] = l;
        Y[at<LD>(i, c)] = y;
    }
    if (!obs_space)
        for (int c = tid; c < n; c += T) vb[c] = g.b64 ? (float)g.b64[(size_t)li * k + c] : g.b32[(size_t)li * k + c];
    else
        for (int c = tid; c < n; c += T) vb[c] = (float)ldh[c];
    __syncthreads();

    // A Y in double-binary32, over A's halves.
    {
        f2x s[4][4], c[4][4];
        tile_zero(s);
        tile_zero(c);
        tile_mul_df<KP>(M1, M2, Y, n, ti, tj, s, c);
        float vs[8][4], vc[8][4];
        tile_unpack(s, vs);
        tile_unpack(c, vc);
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float hi, lo;
                two_sum(vs[q][j], vc[q][j], hi, lo);
                vs[q][j] = hi;
                vc[q][j] = lo;
            }
        __syncthreads();
        tile_store<KP>(M1, ti, tj, vs);
        tile_store<KP>(M2, ti, tj, vc);
        __syncthreads();
    }
    // E = Y^T Y - I and S = Y^T (A Y): tiles (ri, cj) of eight rows and four
    // columns that hold entries on or above the diagonal.
    {
        int ri = 0, cj = tid;
        while (ri < RS::NRG && cj >= RS::NCG - 2 * ri) {
            cj -= RS::NCG - 2 * ri;
            ++ri;
        }
        cj += 2 * ri;
        const bool mine = ri < RS::NRG;
        float ev[8][4], sv[8][4];
        if (mine) {
            f2x s[4][4], c[4][4];
            float vc[8][4];
            tile_zero(s);
            tile_zero(c);
            sym_mul_df<KP, false>(Y, Y, nullptr, n, ri, cj, s, c);
            tile_unpack(s, ev);
            tile_unpack(c, vc);
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    ev[q][j] = __fadd_rn(8 * ri + q == 4 * cj + j ? __fsub_rn(ev[q][j], 1.0f) : ev[q][j], vc[q][j]);
            tile_zero(s);
            tile_zero(c);
            sym_mul_df<KP, true>(Y, M1, M2, n, ri, cj, s, c);
            tile_unpack(s, sv);
            tile_unpack(c, vc);
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int i = 8 * ri + q;
                    if (i == 4 * cj + j) dS[i] = df_value(sv[q][j], vc[q][j]);
                    sv[q][j] = __fadd_rn(sv[q][j], vc[q][j]);
                }
        }
        __syncthreads();
        // S' = S - E o (d_i + d_j)/2 off the diagonal, to both triangles, in
        // FP64 with one rounding to binary32 (two operations per entry, the
        // conversions on the integer units: 0.2 ms per 256^2 points at n = 32,
        // 0.7 at 64).
        if (mine) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int i = 8 * ri + q, c = 4 * cj + j;
                    if (i > c) continue;
                    const float e = ev[q][j];
                    const float s = narrow(fma(-widen(0.5f * e), dS[i] + dS[c], widen(sv[q][j])));
                    M1[at<LD>(i, c)] = s;
                    M1[at<LD>(c, i)] = s;
                    M2[at<LD>(i, c)] = e;
                    M2[at<LD>(c, i)] = e;
                }
        }
        __syncthreads();
    }
    for (int c = tid; c < n; c += T) dS[c] -= (double)M2[at<LD>(c, c)] * dS[c];
    __syncthreads();
    const float sk = (float)sqrt((double)(k - 1));
    const float af = (float)aa, rf = sqrtf(af);
    for (int c = tid; c < n; c += T) {
        if (obs_space) {
            const float ap = af + (float)dS[c];  // a + s_ii
            const float u = sqrtf(ap);
            vu[c] = u;
            vinv[c] = 1.0f / (u * (u + rf));  // alpha_i
            vf[c] = 1.0f / ap;                // h_i
        } else {
            const float lam = (float)dS[c];
            vu[c] = sqrtf(lam);
            vinv[c] = 1.0f / lam;
            vf[c] = vinv[c];
        }
        float t = 0.0f;
        for (int l = 0; l < n; ++l) t += Y[at<LD>(l, c)] * vb[l];
        t1[c] = t;  // Y^T d-hat or Y^T b
    }
    __syncthreads();
    // t2 = h(S') t1, h the inverse (of a + S' in observation space), with the
    // basis factor.
    for (int c = tid; c < n; c += T) {
        const float hi = vf[c];
        float t = 0.0f, te = 0.0f;
        for (int j = 0; j < n; ++j) {
            const float hj = vf[j];
            if (j != c) t += M1[at<LD>(j, c)] * (hj * t1[j]);
            te += M2[at<LD>(j, c)] * (0.5f * (hi + hj)) * t1[j];
        }
        t2[c] = hi * (t1[c] - t) - te;
    }
    __syncthreads();
    // F = g(S') or S'^{-1/2} over S', then Y^T over E.
    float v[8][4];
    {
        float s[8][4], e[8][4];
        tile_load<KP>(M1, ti, tj, s);
        tile_load<KP>(M2, ti, tj, e);
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = tile_row<KP>(ti, q), c = 4 * tj + j;
                float r = 0.0f;
                if (i < n && c < n) {
                    if (obs_space) {
                        const float ai = vinv[c], ui = vu[c], aj = vinv[i], uj = vu[i];
                        const float gc = -ai / rf;
                        const float o = i == c ? gc : s[q][j] * (ui + uj + rf) * ai * aj / (rf * (ui + uj));
                        r = o - e[q][j] * (0.5f * (gc - aj / rf));
                    } else {
                        const float si = vu[c], sj = vu[i];
                        const float o = i == c ? 1.0f / si : -s[q][j] / (si * sj * (si + sj));
                        r = o - e[q][j] * (0.5f * (1.0f / si + 1.0f / sj));
                    }
                }
                s[q][j] = r;
            }
        tile_store<KP>(M1, ti, tj, s);
        tile_load<KP>(Y, ti, tj, v);
        __syncthreads();  // E read
        tile_store_t<KP>(M2, ti, tj, v);
        __syncthreads();
    }
    const float* Yt = M2;
    // w-bar (ensemble space) or v = (a I + A)^{-1} d-hat.
    for (int c = tid; c < n; c += T) {
        float t = 0.0f;
        for (int l = 0; l < n; ++l) t += Yt[at<LD>(l, c)] * t2[l];
        vf[c] = t;
    }
    if (STAGED && !obs_space) {  // n = k <= KP: staged
        const int n4 = (n + 3) & ~3;
        f2x acc[4][4];
        tile_zero(acc);
        tile_mul<KP>(Yt, M1, n4, ti, tj, acc);  // Y F
        __syncthreads();
        tile_unpack(acc, v);
        tile_store_t<KP>(M1, ti, tj, v);
        __syncthreads();
        tile_zero(acc);
        tile_mul<KP>(M1, Yt, n4, ti, tj, acc);  // Y F Y^T
        __syncthreads();
        tile_unpack(acc, v);
        // T = sqrt(k-1) Y F Y^T + w-bar 1^T.
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int j = 0; j < 4; ++j) v[q][j] = sk * v[q][j] + vf[tile_row<KP>(ti, q)];
        tile_store<KP>(M1, ti, tj, v);
        __syncthreads();
        for (int e = tid; e < 9 * k; e += T) {
            const int a = e / k, m = e % k;
            float s = 0.0f;
            for (int j = 0; j < k; ++j) s += dX[a * k + j] * M1[at<LD>(j, m)];
            fc[a * plane + m] = xbar[a] + s;
        }
        return;
    }
    // Observation space: Z = dX Yh^T, then Z Y, Z Y g(S') and B =
    // sqrt(k-1) Z Y g(S') Y^T diag(sqrt(rho)), [9][KP] each. A thread takes
    // three components of one column.
    constexpr int IT = (3 * KP + T - 1) / T;
    float* R0 = vu;  // nine vectors that are no longer needed
    float* R1 = Y;
    __syncthreads();
    for (int e = tid; e < 3 * n; e += T) {
        const int c = e % n, a0 = e / n * 3;
        const float* row = g.o.dY32 + (size_t)lidx[c] * k;
        float acc[3] = {0.0f, 0.0f, 0.0f};
        for (int m = 0; m < k; ++m) {
            const float dy = row[m];
#pragma unroll
            for (int a = 0; a < 3; ++a) acc[a] += dx(a0 + a, m) * dy;
        }
        const float sl = (float)lsq[c];
#pragma unroll
        for (int a = 0; a < 3; ++a) R0[(a0 + a) * KP + c] = sl * acc[a];
    }
    __syncthreads();
    if (tid < 9) {
        float s = 0.0f;
        for (int i = 0; i < n; ++i) s += R0[tid * KP + i] * vf[i];
        zv[tid] = s;
    }
    // dst = src M, after every thread has read.
    auto rows_by = [&](const float* src, const float* M, float* dst, bool scale) {
        float acc[IT][3];
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const int e = tid + it * T;
            acc[it][0] = acc[it][1] = acc[it][2] = 0.0f;
            if (e >= 3 * n) continue;
            const int c = e % n, a0 = e / n * 3;
            for (int i = 0; i < n; ++i) {
                const float y = M[at<LD>(i, c)];
#pragma unroll
                for (int a = 0; a < 3; ++a) acc[it][a] += src[(a0 + a) * KP + i] * y;
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            const int e = tid + it * T;
            if (e >= 3 * n) continue;
            const int c = e % n, a0 = e / n * 3;
            const float sl = scale ? sk * (float)lsq[c] : 1.0f;
#pragma unroll
            for (int a = 0; a < 3; ++a) dst[(a0 + a) * KP + c] = sl * acc[it][a];
        }
        __syncthreads();
    };
    rows_by(R0, Y, R1, false);
    rows_by(R1, M1, R0, false);
    rows_by(R0, Yt, R1, true);
    const float sb = (float)sqrt(g.beta);
    for (int e = tid; e < 3 * k; e += T) {
        const int m = e % k, a0 = e / k * 3;
        float acc[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) acc[a] = xbar[a0 + a] + zv[a0 + a] + sb * dx(a0 + a, m);
        for (int i = 0; i < n; ++i) {
            const float dy = g.o.dY32[(size_t)lidx[i] * k + m];
#pragma unroll
            for (int a = 0; a < 3; ++a) acc[a] += R1[(a0 + a) * KP + i] * dy;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) fc[(a0 + a) * plane + m] = acc[a];
    }
}

template <int KP>
cudaError_t launch_kp(const WideArgs& g, int ncell, cudaStream_t s) {
    size_t sh = WideB<KP>::bytes(g.k);
    auto kern = analyze_wide_kernel<KP, true>;
    if constexpr (WideB<KP>::bytes(kObsMaxMembers) > kMaxShared)
        if (sh > kMaxShared) {
            sh = WideB<KP>::bytes(0);
            kern = analyze_wide_kernel<KP, false>;
        }
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)ncell, WideB<KP>::T, sh, s>>>(g);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_analyze_wide(const WideArgs& g, int ncell, cudaStream_t s) {
    if (g.nm <= 32) return launch_kp<32>(g, ncell, s);
    if (g.nm <= 48) return launch_kp<48>(g, ncell, s);
    if (g.nm <= 64) return launch_kp<64>(g, ncell, s);
    if (g.nm <= 80) return launch_kp<80>(g, ncell, s);
    if (g.nm <= 96) return launch_kp<96>(g, ncell, s);
    if (g.nm <= 112) return launch_kp<112>(g, ncell, s);
    return launch_kp<128>(g, ncell, s);
}

}  // namespace lbmgpu
