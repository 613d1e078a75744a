// Solve and left update of one middle level (Alg. 1, middle factors): per
// slice, Cholesky of K + lambda I from the record of the Gram kernels (Rec),
// the new slice, and h_{m+1} = h_m^T Z for the slice's entries.
//
// One CTA per slice.  The record lies in shared memory in its
// panel layout and is factored in place, right-looking, 8 columns at a time:
//  (1) warp 0 factors the 8 x 8 diagonal block in registers (lane = row and
//      two columns, values passed by shuffles) and, in the precision form,
//      inverts it on the way;
//  (2) a thread per row solves the panel rows below it, conj(y) among them;
//  (3) threads own 4 x 4 tiles of the trailing matrix: 8 rows of the panel are
//      read as 16-byte pieces for 64 complex multiply-adds, done as packed
//      pairs of neighbouring k (f32x2 in the precision form; 2 x 2 tiles in FP64).
// The row of conj(y) ends as conj(z), z the forward solution, so only the
// backward substitution is left; the refinement's solves run in warp 0, block
// by block, with the inverted diagonal blocks.
//
// Bound by latency: shared memory and registers hold 8 slices of rank 8 per SM
// and the diagonal blocks and triangular solves are one warp's chains (ncu,
// n = 16384, r = 8: 36 % issue slots, 29 % of the stalls at barriers, L1
// throughput 61 %).  Measured, all middle levels of a sweep, against the
// kernel before (one warp per slice on a packed triangle, a lane per row):
// n = 65536, r = 8 6.48 -> 5.74 ms; n = 4096, r = 12 8.8 -> 3.1 ms; n = 4096,
// r = 6, FP64 3.75 -> 1.67 ms; n = 3072, r = 5 0.47 -> 0.38 ms.  One warp per
// slice: 7.3 ms at n = 65536, three: 6.8 (r = 12: 7.2 and 4.0, eight: 3.3).
// Also slower or no faster: lanes sharing the rows of the left update (the
// lines of a load or store fewer, the shuffles more), two lanes per row of the
// residual, two residual accumulators with the next panel prefetched, 112
// registers for a ninth CTA per SM (spills).
#pragma once

#include "bfc_kernels.cuh"

namespace bfc {

// Arithmetic on pairs of neighbouring k of two rows: packed FP32 pairs, whose
// two partial sums are added at the end, or FP64 scalars.
template <typename T> struct KPair;
template <> struct KPair<float> {
    typedef uint64_t P;
    typedef uint64_t A;
    static __device__ __forceinline__ A zero() { return 0ull; }
    static __device__ __forceinline__ A fma(A a, P x, P l) { return c2fma(x, l, a); }
    static __device__ __forceinline__ P make(float x, float y) { return c2pack(x, y); }
    static __device__ __forceinline__ P neg(P x)
    {
        float a, b;
        c2unpack(x, a, b);
        return c2pack(-a, -b);
    }
    static __device__ __forceinline__ float sum(A a)
    {
        float x, y;
        c2unpack(a, x, y);
        return x + y;
    }
    // four consecutive values: two pairs
    static __device__ __forceinline__ void load4(const float* p, P (&d)[2])
    {
        const float4 v = *reinterpret_cast<const float4*>(p);
        d[0] = c2pack(v.x, v.y);
        d[1] = c2pack(v.z, v.w);
    }
};
template <> struct KPair<double> {
    typedef double2 P;
    typedef double A;
    static __device__ __forceinline__ A zero() { return 0.0; }
    static __device__ __forceinline__ A fma(A a, P x, P l) { return ::fma(x.y, l.y, ::fma(x.x, l.x, a)); }
    static __device__ __forceinline__ P make(double x, double y) { return make_double2(x, y); }
    static __device__ __forceinline__ P neg(P x) { return make_double2(-x.x, -x.y); }
    static __device__ __forceinline__ double sum(A a) { return a; }
};
__device__ __forceinline__ void load8(const float* p, uint64_t (&d)[4])
{
    uint64_t a[2], b[2];
    KPair<float>::load4(p, a);
    KPair<float>::load4(p + 4, b);
    d[0] = a[0]; d[1] = a[1]; d[2] = b[0]; d[3] = b[1];
}
// four consecutive values of shared memory
__device__ __forceinline__ void ld4(const float* p, float (&v)[4])
{
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4])
{
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4])
{
    const double2 x = *reinterpret_cast<const double2*>(p), y = *reinterpret_cast<const double2*>(p + 2);
    v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}
__device__ __forceinline__ void st4(double* p, const double (&v)[4])
{
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}

template <typename T> __device__ __forceinline__ void ld8(const T* p, T (&v)[8])
{
    T a[4], b[4];
    ld4(p, a);
    ld4(p + 4, b);
#pragma unroll
    for (int q = 0; q < 4; ++q) { v[q] = a[q]; v[4 + q] = b[q]; }
}

template <typename T, int R> struct SolveCfg {
    static constexpr int D = R * R;
    static constexpr int NS = (D + 31) / 32;
    static constexpr bool MIXED = sizeof(T) == 4;
    typedef Rec<T, R> RC;
    // Warps of a slice's CTA: shared memory holds 9 records of rank 8 per SM, 2
    // of rank 12, and the diagonal blocks and triangular solves are chains of
    // one warp.  FP64 at r = 6: the entries' left update is most of the work, 2
    // warps leave its loads exposed and 8 lose the CTAs per SM that overlap
    // (S = 512: 208 / 209 / 281 us per launch with 2 / 4 / 8, S = 128: 316 / 204
    // / 199 us; 256 and 360 us with 2 warps and 4 x 4 tiles)
    static constexpr int NW = R <= 8 ? (MIXED || R <= 2 ? 2 : 4) : R <= 10 ? 4 : 8;
    // Small ranks also in a form of one warp, for levels with more slices than
    // CTAs of two warps are resident (8 per SM): the second warp finds little to
    // do between the barriers.  us per launch, two warps / one: r = 3, S = 4096, 20
    // entries per row 49 / 32, S = 512, 300 entries per row 32 / 40; r = 5, S =
    // 16384 358 / 196, S = 512, 300 entries 53 / 60; FP64, r = 1, S = 4096 (four
    // warps / one) 31 / 20
    static constexpr bool ONE_WARP = R <= (MIXED ? 5 : 2);
    static constexpr int ONE_WARP_FROM = 8;   // slices per SM
    static constexpr int NTH = 32 * NW;
    static constexpr int FBT = 128;      // threads of a k_mid_fallback CTA
    // record (+ slack: short blocks and tiles read, but do not write, rows past its
    // end), solution (double-float or FP64), residual / new slice, exchange
    // buffer of warp 0, flags, mbarrier
    static constexpr size_t LBYTES = (size_t)(RC::SIZE + 128) * sizeof(T);
    static constexpr size_t XBYTES = (size_t)D * 16;
    static constexpr size_t ZBYTES = ((size_t)D * 2 * sizeof(T) + 15) / 16 * 16;
    static constexpr size_t EBYTES = 32 * sizeof(T);
    static constexpr size_t SMEM = LBYTES + XBYTES + ZBYTES + EBYTES + 32;
    static_assert(SMEM <= 227 * 1024, "shared memory of a CTA");
};

// (1) Diagonal block of panel J (warp 0, nb <= 8 columns): L, with 1 / L_cc in
// the imaginary slot of the diagonal, into the block; in the precision form
// this lane's two elements of the inverse (rows >= nb: identity) into X.
// Returns false (warp-uniform) when a pivot is <= tol.
template <typename T, int R>
__device__ __forceinline__ bool solve_diag(T* Lm, int J, int nb, T tol, int lane, T (&xr)[2], T (&xi)[2])
{
    typedef Rec<T, R> RC;
    constexpr bool INV = sizeof(T) == 4;
    constexpr unsigned FULL = 0xffffffffu;
    const int i = lane >> 2, cp = lane & 3, c0 = 2 * cp;
    T* rp = Lm + RC::row(J, i) + c0;
    T ar[2] = {rp[0], rp[1]}, ai[2] = {rp[8], rp[9]};
    xr[0] = i == c0 ? T(1) : T(0);
    xr[1] = i == c0 + 1 ? T(1) : T(0);
    xi[0] = xi[1] = T(0);
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        if (c < nb) {
            const T d = __shfl_sync(FULL, ar[c & 1], c * 4 + (c >> 1));
            ok = ok && d > tol;
            const T inv = rsqrt(d);
            if (cp == (c >> 1) && i > c) {
                ar[c & 1] *= inv;
                ai[c & 1] *= inv;
            }
            // L[i][c], L[c0][c], L[c0 + 1][c]
            const int s0 = (lane & ~3) | (c >> 1), s1 = c0 * 4 + (c >> 1), s2 = s1 + 4;
            const T lr = __shfl_sync(FULL, ar[c & 1], s0), li = __shfl_sync(FULL, ai[c & 1], s0);
            const T ur = __shfl_sync(FULL, ar[c & 1], s1), ui = __shfl_sync(FULL, ai[c & 1], s1);
            const T vr = __shfl_sync(FULL, ar[c & 1], s2), vi = __shfl_sync(FULL, ai[c & 1], s2);
            const bool below = i > c && i < nb;
            if (below && c0 > c) {
                ar[0] -= lr * ur + li * ui;
                ai[0] -= li * ur - lr * ui;
            }
            if (below && c0 + 1 > c) {
                ar[1] -= lr * vr + li * vi;
                ai[1] -= li * vr - lr * vi;
            }
            if constexpr (INV) {
                if (i == c) {
                    xr[0] *= inv; xr[1] *= inv;
                    xi[0] *= inv; xi[1] *= inv;
                }
                const int sx = c * 4 + cp;
                const T x0r = __shfl_sync(FULL, xr[0], sx), x0i = __shfl_sync(FULL, xi[0], sx);
                const T x1r = __shfl_sync(FULL, xr[1], sx), x1i = __shfl_sync(FULL, xi[1], sx);
                if (below) {
                    xr[0] -= lr * x0r - li * x0i;
                    xi[0] -= lr * x0i + li * x0r;
                    xr[1] -= lr * x1r - li * x1i;
                    xi[1] -= lr * x1i + li * x1r;
                }
            }
            if (i == c && cp == (c >> 1)) {
                ar[c & 1] = d * inv;
                ai[c & 1] = inv;
            }
        }
    }
    if (i < nb) {
        // only the lower triangle: the row of conj(y) follows in a short block
        if (c0 <= i) { rp[0] = ar[0]; rp[8] = ai[0]; }
        if (c0 + 1 <= i) { rp[1] = ar[1]; rp[9] = ai[1]; }
    }
    return ok;
}

// (2) One row of panel J below its diagonal block: x L_dd^H = row (columns < nb).
template <typename T, int R> __device__ __forceinline__ void solve_panel_row(T* Lm, int J, int nb, int rho)
{
    typedef Rec<T, R> RC;
    typedef KPair<T> K;
    typedef typename K::P P;
    T* rp = Lm + RC::row(J, rho);
    T ar[8], ai[8];
    {
        T v[4];
        ld4(rp, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) ar[q] = v[q];
        ld4(rp + 4, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) ar[4 + q] = v[q];
        ld4(rp + 8, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) ai[q] = v[q];
        ld4(rp + 12, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) ai[4 + q] = v[q];
    }
    P x2r[4], x2i[4], n2r[4];   // solved columns in pairs, and -re
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        if (c < nb) {
            const T* lp = Lm + RC::row(J, c);
            typename K::A sr = K::zero(), si = K::zero();
#pragma unroll
            for (int h = 0; 2 * h + 1 < c; ++h) {
                if constexpr (sizeof(T) == 4) {
                    const float2 vr = *reinterpret_cast<const float2*>(lp + 2 * h);
                    const float2 vi = *reinterpret_cast<const float2*>(lp + 8 + 2 * h);
                    const P lr = K::make(vr.x, vr.y), li = K::make(vi.x, vi.y);
                    sr = K::fma(K::fma(sr, x2r[h], lr), x2i[h], li);
                    si = K::fma(K::fma(si, x2i[h], lr), n2r[h], li);
                } else {
                    const P lr = *reinterpret_cast<const P*>(lp + 2 * h), li = *reinterpret_cast<const P*>(lp + 8 + 2 * h);
                    sr = K::fma(K::fma(sr, x2r[h], lr), x2i[h], li);
                    si = K::fma(K::fma(si, x2i[h], lr), n2r[h], li);
                }
            }
            T tr = ar[c] - K::sum(sr), ti = ai[c] - K::sum(si);
            if (c & 1) {
                const T lr = lp[c - 1], li = lp[8 + c - 1];
                tr -= ar[c - 1] * lr + ai[c - 1] * li;
                ti -= ai[c - 1] * lr - ar[c - 1] * li;
            }
            const T inv = lp[8 + c];
            ar[c] = tr * inv;
            ai[c] = ti * inv;
            if (c & 1) {
                x2r[c >> 1] = K::make(ar[c - 1], ar[c]);
                x2i[c >> 1] = K::make(ai[c - 1], ai[c]);
                n2r[c >> 1] = K::neg(x2r[c >> 1]);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const T vr[4] = {ar[4 * q], ar[4 * q + 1], ar[4 * q + 2], ar[4 * q + 3]};
        const T vi[4] = {ai[4 * q], ai[4 * q + 1], ai[4 * q + 2], ai[4 * q + 3]};
        st4(rp + 4 * q, vr);
        st4(rp + 8 + 4 * q, vi);
    }
}

// (3) Precision form: tile (I, Jt) of the trailing matrix of panel J: rows 8J + 8 + 4 I .. + 3,
// columns 8J + 8 + 4 Jt .. + 3, minus the product of the panel's rows.
template <int R> __device__ __forceinline__ void solve_tile(float* Lm, int J, int I, int Jt)
{
    typedef Rec<float, R> RC;
    typedef KPair<float> K;
    typedef K::P P;
    const float* xp = Lm + RC::row(J, 8 + 4 * I);   // four consecutive rows, 16 values apart
    const float* lp = Lm + RC::row(J, 8 + 4 * Jt);
    K::A sr[4][4], si[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) { sr[u][v] = K::zero(); si[u][v] = K::zero(); }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        P lr[4][2], li[4][2];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            K::load4(lp + 16 * v + 4 * h, lr[v]);
            K::load4(lp + 16 * v + 8 + 4 * h, li[v]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            P xr[2], xi[2], nr[2];
            K::load4(xp + 16 * u + 4 * h, xr);
            K::load4(xp + 16 * u + 8 + 4 * h, xi);
            nr[0] = K::neg(xr[0]);
            nr[1] = K::neg(xr[1]);
#pragma unroll
            for (int v = 0; v < 4; ++v)
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    sr[u][v] = K::fma(K::fma(sr[u][v], xr[t], lr[v][t]), xi[t], li[v][t]);
                    si[u][v] = K::fma(K::fma(si[u][v], xi[t], lr[v][t]), nr[t], li[v][t]);
                }
        }
    }
    const int c = 8 * J + 8 + 4 * Jt, Jd = c >> 3, r0 = 8 * J + 8 + 4 * I;
    float* dp = Lm + RC::row(Jd, r0 - 8 * Jd) + (c & 7);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (r0 + u <= RC::D) {
            float a[4], b[4];
            ld4(dp + 16 * u, a);
            ld4(dp + 16 * u + 8, b);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                a[v] -= K::sum(sr[u][v]);
                b[v] -= K::sum(si[u][v]);
            }
            st4(dp + 16 * u, a);
            st4(dp + 16 * u + 8, b);
        }
    }
}

// The row of conj(y) (row D) of the trailing matrix, columns 8J + 8 + 4 Jt ..
// + 3, where D is a multiple of 4 (otherwise it lies in the last full tiles).
template <int R> __device__ __forceinline__ void solve_y_tile(float* Lm, int J, int Jt)
{
    typedef Rec<float, R> RC;
    typedef KPair<float> K;
    typedef K::P P;
    const float* xp = Lm + RC::row(J, RC::D - 8 * J);
    const float* lp = Lm + RC::row(J, 8 + 4 * Jt);
    P xr[4], xi[4], nr[4];
    load8(xp, xr);
    load8(xp + 8, xi);
#pragma unroll
    for (int t = 0; t < 4; ++t) nr[t] = K::neg(xr[t]);
    float a[4], b[4];
    const int c = 8 * J + 8 + 4 * Jt, Jd = c >> 3;
    float* dp = Lm + RC::row(Jd, RC::D - 8 * Jd) + (c & 7);
    ld4(dp, a);
    ld4(dp + 8, b);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        P lr[4], li[4];
        load8(lp + 16 * v, lr);
        load8(lp + 16 * v + 8, li);
        K::A sr = K::zero(), si = K::zero();
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            sr = K::fma(K::fma(sr, xr[t], lr[t]), xi[t], li[t]);
            si = K::fma(K::fma(si, xi[t], lr[t]), nr[t], li[t]);
        }
        a[v] -= K::sum(sr);
        b[v] -= K::sum(si);
    }
    st4(dp, a);
    st4(dp + 8, b);
}

// FP64: a 2 x 2 tile (I, Jt) of the trailing matrix of panel J.  A warp
// instruction takes the FP64 pipe as long with one active lane as with 32, and
// 4 x 4 tiles leave most lanes of the later panels idle.
template <int R> __device__ __forceinline__ void solve_tile2(double* Lm, int J, int I, int Jt)
{
    typedef Rec<double, R> RC;
    const double* xp = Lm + RC::row(J, 8 + 2 * I);
    const double* lp = Lm + RC::row(J, 8 + 2 * Jt);
    double sr[2][2] = {}, si[2][2] = {};
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        double2 lr[2], li[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            lr[v] = *reinterpret_cast<const double2*>(lp + 16 * v + 2 * h);
            li[v] = *reinterpret_cast<const double2*>(lp + 16 * v + 8 + 2 * h);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const double2 xr = *reinterpret_cast<const double2*>(xp + 16 * u + 2 * h);
            const double2 xi = *reinterpret_cast<const double2*>(xp + 16 * u + 8 + 2 * h);
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                sr[u][v] += xr.x * lr[v].x;
                si[u][v] += xi.x * lr[v].x;
                sr[u][v] += xi.x * li[v].x;
                si[u][v] -= xr.x * li[v].x;
                sr[u][v] += xr.y * lr[v].y;
                si[u][v] += xi.y * lr[v].y;
                sr[u][v] += xi.y * li[v].y;
                si[u][v] -= xr.y * li[v].y;
            }
        }
    }
    const int c = 8 * J + 8 + 2 * Jt, Jd = c >> 3, r0 = 8 * J + 8 + 2 * I;
    double* dp = Lm + RC::row(Jd, r0 - 8 * Jd) + (c & 7);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (r0 + u <= RC::D) {
            double2* a = reinterpret_cast<double2*>(dp + 16 * u);
            double2* b = reinterpret_cast<double2*>(dp + 16 * u + 8);
            const double2 av = *a, bv = *b;
            *a = make_double2(av.x - sr[u][0], av.y - sr[u][1]);
            *b = make_double2(bv.x - si[u][0], bv.y - si[u][1]);
        }
    }
}

// Factorization of the record in Lm by all threads of the CTA.  In the
// precision form the diagonal blocks end inverted, in FP64 as L (1 / L_cc in
// the imaginary slot of the diagonal).  False (CTA-uniform) when a pivot is
// <= tol.  *fail is a shared word, zero on entry.
template <typename T, int R>
__device__ __forceinline__ bool solve_chol(T* Lm, T tol, volatile int* fail, int tid, int nthr)
{
    typedef Rec<T, R> RC;
    constexpr int D = RC::D;
    const int lane = tid & 31;
    for (int J = 0; J < RC::NPAN; ++J) {
        const int nb = min(8, D - 8 * J);
        T xr[2], xi[2];
        if (tid < 32) {
            const bool ok = solve_diag<T, R>(Lm, J, nb, tol, lane, xr, xi);
            if (!ok && lane == 0) *fail = 1;
        }
        __syncthreads();
        if (*fail) return false;
        for (int rho = nb + tid; rho < RC::DR - 8 * J; rho += nthr) solve_panel_row<T, R>(Lm, J, nb, rho);
        __syncthreads();
        if (sizeof(T) == 4 && tid < 32) {
            // the panel is done with L_dd: keep its inverse (zeros above the diagonal)
            const int i = lane >> 2, c0 = 2 * (lane & 3);
            if (i < nb) {
                T* rp = Lm + RC::row(J, i) + c0;
                rp[0] = xr[0]; rp[1] = xr[1];
                rp[8] = xi[0]; rp[9] = xi[1];
            }
        }
        // tile columns hold columns < D; the row of conj(y) is in the last tile
        // row, or (D a multiple of 4) has tiles of one row, by the last threads
        // (as full tiles they would take a round of their own)
        auto tri = [](int x) {   // the row of element x of a packed lower triangle
            int I = (int)((sqrtf(8.f * (float)x + 1.f) - 1.f) * 0.5f);
            if (I * (I + 1) / 2 > x) --I;
            if ((I + 1) * (I + 2) / 2 <= x) ++I;
            return I;
        };
        if constexpr (sizeof(T) == 8) {
            // columns 8J + 8 .. D - 1 in pairs, rows to D: with an even number of
            // columns the row of conj(y) is a row of tiles of its own
            const int M = max(0, D - 8 * J - 8), mc = (M + 1) / 2;
            const int nt = mc * (mc + 1) / 2 + (M % 2 == 0 ? mc : 0);
            for (int x = tid; x < nt; x += nthr) {
                const int I = tri(x);
                solve_tile2<R>(Lm, J, I, x - I * (I + 1) / 2);
            }
        } else {
            const int mc = max(0, (D - 8 * J - 5) / 4), nt = mc * (mc + 1) / 2;
            if constexpr (D % 4 == 0)
                for (int x = nthr - 1 - tid; x < mc; x += nthr) solve_y_tile<R>(Lm, J, x);
            for (int x = tid; x < nt; x += nthr) {
                const int I = tri(x);
                solve_tile<R>(Lm, J, I, x - I * (I + 1) / 2);
            }
        }
        __syncthreads();
    }
    return true;
}

// Triangular solves of warp 0, row p of the vector in slot p / 32 of lane
// p % 32 (zero past D).  xb: 32 values of shared memory (the block's part of
// the right-hand side, then of the solution).  Precision form only: the
// diagonal blocks are inverted.
template <int R> __device__ __forceinline__ void solve_fwd(const float* Lm, float2 (&bv)[SolveCfg<float, R>::NS],
                                                           float* xb, int lane)
{
    typedef Rec<float, R> RC;
    typedef KPair<float> K;
    constexpr int D = RC::D, NS = SolveCfg<float, R>::NS;
    for (int J = 0; J < RC::NPAN; ++J) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int p = lane + 32 * s;
            if ((p >> 3) == J) { xb[p & 7] = bv[s].x; xb[8 + (p & 7)] = bv[s].y; }
        }
        __syncwarp();
        uint64_t rr[4], ri[4], lr[4], li[4];
        load8(xb, rr);
        load8(xb + 8, ri);
        const int i = lane & 7;
        load8(Lm + RC::row(J, i), lr);
        load8(Lm + RC::row(J, i) + 8, li);
        uint64_t a = 0ull, b = 0ull, c = 0ull;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            a = c2fma(lr[h], rr[h], a);
            b = c2fma(li[h], ri[h], b);
            c = c2fma(lr[h], ri[h], c);
            c = c2fma(li[h], rr[h], c);
        }
        if (lane < 8) {
            const bool in = 8 * J + i < D;
            xb[16 + i] = in ? K::sum(a) - K::sum(b) : 0.f;
            xb[24 + i] = in ? K::sum(c) : 0.f;
        }
        __syncwarp();
        load8(xb + 16, rr);
        load8(xb + 24, ri);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int p = lane + 32 * s;
            if ((p >> 3) == J) { bv[s].x = xb[16 + (p & 7)]; bv[s].y = xb[24 + (p & 7)]; }
            if (p >= 8 * J + 8 && p < D) {
                const float* rp = Lm + RC::row(J, p - 8 * J);
                load8(rp, lr);
                load8(rp + 8, li);
                a = b = c = 0ull;
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    a = c2fma(lr[h], rr[h], a);
                    b = c2fma(li[h], ri[h], b);
                    c = c2fma(lr[h], ri[h], c);
                    c = c2fma(li[h], rr[h], c);
                }
                bv[s].x -= K::sum(a) - K::sum(b);
                bv[s].y -= K::sum(c);
            }
        }
    }
}

// L^H x = z, both forms.
template <typename T, int R>
__device__ __forceinline__ void solve_bwd(const T* Lm, typename cvec<T>::type (&bv)[SolveCfg<T, R>::NS], T* xb,
                                          int lane)
{
    typedef Rec<T, R> RC;
    typedef typename cvec<T>::type V;
    constexpr int D = RC::D, NS = SolveCfg<T, R>::NS;
    for (int J = RC::NPAN - 1; J >= 0; --J) {
        const int nb = min(8, D - 8 * J);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int p = lane + 32 * s;
            if ((p >> 3) == J) { xb[p & 7] = bv[s].x; xb[8 + (p & 7)] = bv[s].y; }
        }
        __syncwarp();
        const int i = lane & 7;
        V x;
        if constexpr (sizeof(T) == 4) {
            // column i of the inverse, conjugated
            x = czero<V>();
            const T* cp = Lm + RC::row(J, 0) + i;
            T rr[8], ri[8];
            ld8(xb, rr);
            ld8(xb + 8, ri);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (D % 8 == 0 || k < nb) {
                    const T* e = cp + k * 16 + (k >> 2) * RC::PADT;
                    V l, r;
                    l.x = e[0]; l.y = e[8];
                    r.x = rr[k]; r.y = ri[k];
                    cmacc(x, l, r);
                }
        } else {
            x.x = xb[i];
            x.y = xb[8 + i];
            for (int c = nb - 1; c >= 0; --c) {
                const T* e = Lm + RC::row(J, c);
                const T inv = e[8 + c];
                V xc;
                xc.x = __shfl_sync(0xffffffffu, x.x, c) * inv;
                xc.y = __shfl_sync(0xffffffffu, x.y, c) * inv;
                if (i == c) x = xc;
                if (i < c) {
                    V l;
                    l.x = -e[i]; l.y = -e[8 + i];
                    cmacc(x, l, xc);
                }
            }
        }
        if (lane < 8) {
            const bool in = i < nb;
            xb[16 + i] = in ? x.x : T(0);
            xb[24 + i] = in ? x.y : T(0);
        }
        __syncwarp();
        T xr[8], xi[8];
        ld8(xb + 16, xr);
        ld8(xb + 24, xi);
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int q = lane + 32 * s;
            if ((q >> 3) == J) { bv[s].x = xb[16 + (q & 7)]; bv[s].y = xb[24 + (q & 7)]; }
            if (q < 8 * J) {
                const T* cp = Lm + RC::row(q >> 3, 8 * J - (q & ~7)) + (q & 7);
                V acc = czero<V>();
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (D % 8 == 0 || k < nb) {
                        const T* e = cp + k * 16 + (k >> 2) * RC::PADT;
                        V l, xk;
                        l.x = e[0]; l.y = e[8];
                        xk.x = xr[k]; xk.y = xi[k];
                        cmacc(acc, l, xk);
                    }
                bv[s].x -= acc.x;
                bv[s].y -= acc.y;
            }
        }
    }
}

// Double-float residual y - (K + lambda I) s, row p, of the record in global
// memory (K above the diagonal by conjugation); s_df[q] = {re_hi, im_hi,
// re_lo, im_lo}.
template <int R>
__device__ __forceinline__ float2 solve_residual(const float* __restrict__ K, const float4* s_df, float lamf, int p)
{
    typedef Rec<float, R> RC;
    constexpr int D = RC::D;
    const float* yp = K + RC::re(D, p);
    uint64_t hi = c2pack(yp[0], -yp[8]), lo = 0ull;
    const float4 sp = s_df[p];
    df2_sub_cmul(hi, lo, make_float2(lamf, 0.f), df2_prep(make_float2(sp.x, sp.y), make_float2(sp.z, sp.w)));
    // element (q, p) below the diagonal, seen as K_pq^*: a fixed offset per row
    // p plus 16 q + 4 (q / 4)
    const int Jp = p >> 3;
    const float* col = K + (RC::base(Jp) - Jp * (128 + 2 * RC::PADT) + (p & 7));
    for (int J = 0; J < RC::NPAN; ++J) {
        const int nb = min(8, D - 8 * J);
        float kr[8], ki[8];
        if (p >= 8 * J) {
            // columns of the row itself
            ld8(K + RC::row(J, p - 8 * J), kr);
            ld8(K + RC::row(J, p - 8 * J) + 8, ki);
        }
        if (p < 8 * J + 7) {
            const float* cq = col + J * (128 + 2 * RC::PADT);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if ((D % 8 == 0 || i < nb) && 8 * J + i > p) {
                    kr[i] = cq[i * 16 + (i >> 2) * RC::PADT];
                    ki[i] = -cq[i * 16 + (i >> 2) * RC::PADT + 8];
                }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (D % 8 == 0 || i < nb) {
                const float4 sq = s_df[8 * J + i];
                df2_sub_cmul(hi, lo, make_float2(kr[i], ki[i]),
                             df2_prep(make_float2(sq.x, sq.y), make_float2(sq.z, sq.w)));
            }
    }
    float2 r;
    c2unpack(c2add(hi, lo), r.x, r.y);
    return r;
}

// Left environment update of slice k: h_{m+1}(e) = h_m(e)^T Z^{m+1}(k) for the
// slice's entries (threads tid of nthr over entries), scattered into order m+1.
template <typename T, int R>
__device__ __forceinline__ void slice_h_update(const typename cvec<T>::type* __restrict__ H,
                                               const typename cvec<T>::type* zt_s, const int32_t* __restrict__ nxt,
                                               typename cvec<T>::type* __restrict__ Hn, int s0, int s1, int tid,
                                               int nthr)
{
    typedef typename cvec<T>::type V;
    constexpr bool VEC = sizeof(V) == 8 && R % 2 == 0;   // rows as 16-byte vectors
    auto load_row = [&](int p, V* h) {
        if constexpr (VEC) {
            const float4* src = reinterpret_cast<const float4*>(H + (size_t)p * R);
#pragma unroll
            for (int a = 0; a < R / 2; ++a) {
                const float4 v = __ldg(src + a);
                h[2 * a].x = v.x; h[2 * a].y = v.y;
                h[2 * a + 1].x = v.z; h[2 * a + 1].y = v.w;
            }
        } else {
#pragma unroll
            for (int a = 0; a < R; ++a) h[a] = H[(size_t)p * R + a];
        }
    };
    auto store_row = [&](size_t o, const V* x) {
        if constexpr (VEC) {
            float4* dst = reinterpret_cast<float4*>(Hn + o);
#pragma unroll
            for (int a = 0; a < R / 2; ++a) dst[a] = make_float4(x[2 * a].x, x[2 * a].y, x[2 * a + 1].x, x[2 * a + 1].y);
        } else {
#pragma unroll
            for (int a = 0; a < R; ++a) Hn[o + a] = x[a];
        }
    };
    // NE entries per thread and step: their loads are in flight together
    constexpr int NE = R <= 8 ? 2 : 1;
    for (int p = s0 + tid; p < s1; p += NE * nthr) {
        asm volatile("" ::: "memory");   // the slice stays in shared memory, not hoisted into registers
        V h[NE][R], r[NE][R];
        size_t o[NE];
#pragma unroll
        for (int n = 0; n < NE; ++n) {
            const int q = min(p + n * nthr, s1 - 1);   // past the end: the last entry, not stored
            load_row(q, h[n]);
            o[n] = (size_t)nxt[q] * R;
        }
        if constexpr (sizeof(V) == 8) {
            // packed: h z = h.re (z.re, z.im) + h.im (-z.im, z.re), the second
            // product taken as h.im (z.re, z.im) and turned at the end
            uint64_t a1[NE][R], a2[NE][R];
#pragma unroll
            for (int n = 0; n < NE; ++n)
#pragma unroll
                for (int c = 0; c < R; ++c) a1[n][c] = a2[n][c] = 0ull;
#pragma unroll
            for (int a = 0; a < R; ++a) {
                uint64_t z[R];
                if constexpr (VEC) {
#pragma unroll
                    for (int c = 0; c < R / 2; ++c) {
                        const float4 v = *reinterpret_cast<const float4*>(zt_s + a * R + 2 * c);
                        z[2 * c] = c2pack(v.x, v.y);
                        z[2 * c + 1] = c2pack(v.z, v.w);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < R; ++c) z[c] = c2pack(zt_s[a * R + c].x, zt_s[a * R + c].y);
                }
#pragma unroll
                for (int n = 0; n < NE; ++n) {
                    const uint64_t hr = c2pack(h[n][a].x, h[n][a].x), hi = c2pack(h[n][a].y, h[n][a].y);
#pragma unroll
                    for (int c = 0; c < R; ++c) {
                        a1[n][c] = c2fma(hr, z[c], a1[n][c]);
                        a2[n][c] = c2fma(hi, z[c], a2[n][c]);
                    }
                }
            }
#pragma unroll
            for (int n = 0; n < NE; ++n)
#pragma unroll
                for (int c = 0; c < R; ++c) {
                    float xr, xi, yr, yi;
                    c2unpack(a1[n][c], xr, xi);
                    c2unpack(a2[n][c], yr, yi);
                    r[n][c].x = xr - yi;
                    r[n][c].y = xi + yr;
                }
        } else {
#pragma unroll
            for (int n = 0; n < NE; ++n)
#pragma unroll
                for (int c = 0; c < R; ++c) {
                    V acc = czero<V>();
#pragma unroll
                    for (int a = 0; a < R; ++a) cmac(acc, h[n][a], zt_s[a * R + c]);
                    r[n][c] = acc;
                }
        }
#pragma unroll
        for (int n = 0; n < NE; ++n)
            if (p + n * nthr < s1) store_row(o[n], r[n]);
    }
}

// Middle level m, stage 2 (solve + left update): one CTA per slice, see the
// head of this file.  Precision form (float): the record arrives in shared
// memory by one bulk copy; complex64 Cholesky of K + lambda I and solve, then
// up to three steps of iterative refinement: the residual y - (K + lambda I) s
// in double-float arithmetic (TwoSum-compensated float pairs, rows over the
// threads, K from the record in L2) against a solution kept as a double-float
// pair, and the correction through the complex64 factor.  If the factorization
// breaks down or the refinement does not contract, the slice goes on a list
// for the FP64 Cholesky of k_mid_fallback.  FP64 path (double): FP64 Cholesky
// directly.  The slice is written row-major in FP64 and the compute type; then
// h_{m+1}(e) = h_m(e)^T Z^{m+1}(k) for the slice's entries is scattered into
// order m+1.  A singular system keeps its old slice.
template <typename T, int R, int NW>
__global__ void __launch_bounds__(32 * NW, sizeof(T) == 4 ? 16 / NW : 1)   // 128 registers in the precision form
k_mid_solve(const T* __restrict__ rec, const typename cvec<T>::type* __restrict__ H,
            const int32_t* __restrict__ seg, const int32_t* __restrict__ nxt,
            typename cvec<T>::type* __restrict__ Hn, double2* __restrict__ Zd,
            typename cvec<T>::type* __restrict__ Zt, double lambda_in, double ridge,
            unsigned long long* __restrict__ nsing, unsigned long long* __restrict__ nfb,
            unsigned long long* __restrict__ nsteps, int32_t* __restrict__ fblist,
            unsigned long long* __restrict__ terr, int skip_copy)
{
    // nfb: slices handed to the FP64 fallback (length of fblist); nsteps: refinement steps;
    // terr: raised when the bulk copy of a record does not complete within the wait limit;
    // skip_copy (failure injection of the tests, bfc_inject_fault): the bulk copy is not
    // issued and the wait gives up after a few tries
    typedef typename cvec<T>::type V;
    typedef SolveCfg<T, R> C;
    typedef Rec<T, R> RC;
    constexpr int D = C::D, NS = C::NS;
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int nthr = 32 * NW;
    const int tid = threadIdx.x, lane = tid & 31, k = blockIdx.x;
    T* Lm = (T*)smem;
    float4* s_df = (float4*)(smem + C::LBYTES);      // double-float solution
    double2* s_x = (double2*)(smem + C::LBYTES);     // FP64 solution
    V* zt_s = (V*)(smem + C::LBYTES + C::XBYTES);    // residual, then the new slice
    T* xb = (T*)(smem + C::LBYTES + C::XBYTES + C::ZBYTES);
    volatile int* flag = (volatile int*)((unsigned char*)xb + C::EBYTES);   // [0] breakdown, [1] refinement goes on
    const T* K = rec + (size_t)k * RC::SIZE;
    bool pending = false;     // a copy that was issued and then given up on
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared((unsigned char*)flag + 16);
    if (tid == 0) { flag[0] = 0; flag[1] = 0; }
    bool have = false;
    if constexpr (C::MIXED) {
        constexpr uint32_t BYTES = (uint32_t)(RC::SIZE * sizeof(T));   // a multiple of 16
        if (tid == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
                         ::"r"(bar), "r"(BYTES) : "memory");
            if (!skip_copy)
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"((uint32_t)__cvta_generic_to_shared(Lm)), "l"(K), "r"(BYTES), "r"(bar)
                             : "memory");
        }
        __syncthreads();
        bool done = false;
        const uint32_t wait_limit = skip_copy ? 64u : (1u << 22);
        for (uint32_t it = 0; it < wait_limit && !done; ++it) {
            uint32_t ok;
            asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                         "selp.u32 %0, 1, 0, p;\n}\n"
                         : "=r"(ok) : "r"(bar), "r"(0u) : "memory");
            done = ok != 0;
        }
        // the phase completes once for every thread: any thread that saw it
        // completed makes the copy valid for the CTA
        have = __syncthreads_or(done) != 0;
        if (!have) {
            // the copy did not complete: report it and load by plain loads
            // (the call's results are undefined)
            if (tid == 0) atomicExch(terr, 1ull);
            pending = !skip_copy;
        }
    }
    if (!have) {
        const float4* src = reinterpret_cast<const float4*>(K);
        float4* dst = reinterpret_cast<float4*>(Lm);
        constexpr int NV = (int)(RC::SIZE * sizeof(T) / 16);
#pragma unroll 4
        for (int q = tid; q < NV; q += nthr) dst[q] = src[q];
        __syncthreads();
    }
    // every warp forms the trace (the same value in all)
    double tr = 0.0;
    for (int p = lane; p < D; p += 32) tr += (double)Lm[RC::re(p, p)];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    // lambda, raised to the ridge floor (relative to the mean diagonal) when set
    const double lambda = fmax(lambda_in, ridge * tr / D);
    const double tol = lambda > 0.0 ? 0.0 : 1e-14 * (tr + D * lambda);
    __syncthreads();
    for (int p = tid; p < D; p += nthr) Lm[RC::re(p, p)] += (T)lambda;
    __syncthreads();
    bool ok = solve_chol<T, R>(Lm, (T)tol, flag, tid, nthr);
    if constexpr (C::MIXED) {
        if (ok) {
            float2 bv[NS], sh[NS], sl[NS];
            if (tid < 32) {
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int p = lane + 32 * s;
                    bv[s] = make_float2(0.f, 0.f);
                    if (p < D) {
                        const T* zp = Lm + RC::re(D, p);   // conj(z)
                        bv[s] = make_float2(zp[0], -zp[8]);
                    }
                }
                solve_bwd<T, R>(Lm, bv, xb, lane);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int p = lane + 32 * s;
                    sh[s] = bv[s];
                    sl[s] = make_float2(0.f, 0.f);
                    if (p < D) s_df[p] = make_float4(sh[s].x, sh[s].y, 0.f, 0.f);
                }
            }
            const float lamf = (float)lambda;
            bool conv = false;
            for (int it = 0; it < 3; ++it) {
                __syncthreads();
                static_assert(D <= nthr, "a row of the residual per thread");
                if (tid < D) zt_s[tid] = solve_residual<R>(K, s_df, lamf, tid);
                __syncthreads();
                if (tid < 32) {
                    float rmax = 0.f;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const int p = lane + 32 * s;
                        bv[s] = p < D ? zt_s[p] : make_float2(0.f, 0.f);
                        rmax = fmaxf(rmax, fmaxf(fabsf(bv[s].x), fabsf(bv[s].y)));
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
                    // (a residual below the normal range: its reciprocal would be infinite)
                    const float sc = fmaxf(rmax, 1.17549435e-38f);
                    const float isc = 1.f / sc;
#pragma unroll
                    for (int s = 0; s < NS; ++s) { bv[s].x *= isc; bv[s].y *= isc; }
                    solve_fwd<R>(Lm, bv, xb, lane);
                    solve_bwd<T, R>(Lm, bv, xb, lane);
                    float dmax = 0.f, smax = 0.f;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const float dx = bv[s].x * sc, dy = bv[s].y * sc;
                        float t, e;
                        two_sum(sh[s].x, dx, t, e); sh[s].x = t; sl[s].x += e;
                        two_sum(sh[s].y, dy, t, e); sh[s].y = t; sl[s].y += e;
                        dmax = fmaxf(dmax, fmaxf(fabsf(dx), fabsf(dy)));
                        smax = fmaxf(smax, fmaxf(fabsf(sh[s].x), fabsf(sh[s].y)));
                        const int p = lane + 32 * s;
                        if (p < D) s_df[p] = make_float4(sh[s].x, sh[s].y, sl[s].x, sl[s].y);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
                        smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
                    }
                    // after a step with relative correction rho the remaining error is
                    // about rho^2: stop once that is below 1e-10
                    if (lane == 0) {
                        atomicAdd(nsteps, 1ull);
                        flag[1] = (dmax <= 1e-5f * smax ? 1 : 0) | (dmax <= 1e-4f * smax ? 2 : 0);
                    }
                }
                __syncthreads();
                const int f = flag[1];
                conv = (f & 2) != 0;
                if (f & 1) break;
            }
            ok = conv;
        }
        if (!ok) {
            // solved afterwards in FP64 by k_mid_fallback (slice and its entries untouched here)
            if (tid == 0) fblist[atomicAdd(nfb, 1ull)] = k;
        } else {
            for (int p = tid; p < D; p += nthr) {
                const float4 s = s_df[p];
                const double2 v = make_double2((double)s.x + (double)s.z, (double)s.y + (double)s.w);
                Zd[(size_t)k * D + p] = v;
                const V st = from_d2<V>(v);
                Zt[(size_t)k * D + p] = st;
                zt_s[p] = st;
            }
        }
    } else {
        if (ok) {
            if (tid < 32) {
                V bv[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int p = lane + 32 * s;
                    bv[s] = czero<V>();
                    if (p < D) {
                        const T* zp = Lm + RC::re(D, p);   // conj(z)
                        bv[s].x = zp[0];
                        bv[s].y = -zp[8];
                    }
                }
                solve_bwd<T, R>(Lm, bv, xb, lane);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int p = lane + 32 * s;
                    if (p < D) s_x[p] = to_d2(bv[s]);
                }
            }
            __syncthreads();
        } else if (tid == 0) {
            atomicAdd(nsing, 1ull);
        }
        for (int p = tid; p < D; p += nthr) {
            if (ok) {
                const V st = from_d2<V>(s_x[p]);
                Zd[(size_t)k * D + p] = s_x[p];
                Zt[(size_t)k * D + p] = st;
                zt_s[p] = st;
            } else {
                zt_s[p] = Zt[(size_t)k * D + p];
            }
        }
    }
    __syncthreads();
    if (ok || !C::MIXED) slice_h_update<T, R>(H, zt_s, nxt, Hn, seg[k], seg[k + 1], tid, nthr);
    if (pending) {
        // a copy that was given up on may still land: wait for it (bounded)
        // before the CTA's shared memory is released
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            uint32_t done;
            asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                         "selp.u32 %0, 1, 0, p;\n}\n"
                         : "=r"(done) : "r"(bar), "r"(0u) : "memory");
            if (done) break;
        }
    }
}

// FP64 fallback of the precision form: a CTA per slice listed by k_mid_solve
// (complex64 factorization broke down or refinement did not contract): FP64
// Cholesky of K + lambda I in shared memory, solve, slice write (or keep the
// old slice and count it singular), left update.
template <typename T, int R>
__global__ void __launch_bounds__(SolveCfg<double, R>::FBT)
k_mid_fallback(const T* __restrict__ rec, const typename cvec<T>::type* __restrict__ H,
               const int32_t* __restrict__ seg, const int32_t* __restrict__ nxt,
               typename cvec<T>::type* __restrict__ Hn, double2* __restrict__ Zd,
               typename cvec<T>::type* __restrict__ Zt, double lambda_in, double ridge,
               unsigned long long* __restrict__ nsing, const unsigned long long* __restrict__ nfb,
               const int32_t* __restrict__ fblist, unsigned long long* __restrict__ nfb_sweep)
{
    typedef typename cvec<T>::type V;
    typedef SolveCfg<double, R> C;
    typedef Rec<double, R> RD;
    typedef Rec<T, R> RC;
    constexpr int D = C::D, NS = C::NS;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x;
    double* Lm = (double*)smem;
    double2* s_x = (double2*)(smem + C::LBYTES);
    V* zt_s = (V*)(smem + C::LBYTES + C::XBYTES);
    double* xb = (double*)(smem + C::LBYTES + C::XBYTES + C::ZBYTES);
    volatile int* flag = (volatile int*)((unsigned char*)xb + C::EBYTES);
    const long long count = (long long)*nfb;
    // the level's fallbacks join the sweep's count (one thread; nothing else
    // writes it while this kernel runs)
    if (blockIdx.x == 0 && tid == 0) *nfb_sweep += (unsigned long long)count;
    for (long long idx = blockIdx.x; idx < count; idx += gridDim.x) {
        const int k = fblist[idx];
        const T* K = rec + (size_t)k * RC::SIZE;
        __syncthreads();   // the previous slice's readers are done
        if (tid == 0) flag[0] = 0;
        for (int J = 0; J < RC::NPAN; ++J)
            for (int x = tid; x < (RC::DR - 8 * J) * 16; x += nthr)
                Lm[RD::row(J, x >> 4) + (x & 15)] = (double)K[RC::row(J, x >> 4) + (x & 15)];
        double tr = 0.0;
        for (int p = lane; p < D; p += 32) tr += (double)K[RC::re(p, p)];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        const double lambda = fmax(lambda_in, ridge * tr / D);
        const double tol = lambda > 0.0 ? 0.0 : 1e-14 * (tr + D * lambda);
        __syncthreads();
        for (int p = tid; p < D; p += nthr) Lm[RD::re(p, p)] += lambda;
        __syncthreads();
        const bool ok = solve_chol<double, R>(Lm, tol, flag, tid, nthr);
        if (ok && tid < 32) {
            double2 bv[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int p = lane + 32 * s;
                bv[s] = make_double2(0.0, 0.0);
                if (p < D) {
                    const double* zp = Lm + RD::re(D, p);   // conj(z)
                    bv[s] = make_double2(zp[0], -zp[8]);
                }
            }
            solve_bwd<double, R>(Lm, bv, xb, lane);
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int p = lane + 32 * s;
                if (p < D) s_x[p] = bv[s];
            }
        } else if (!ok && tid == 0) {
            atomicAdd(nsing, 1ull);
        }
        __syncthreads();
        for (int p = tid; p < D; p += nthr) {
            if (ok) {
                const V st = from_d2<V>(s_x[p]);
                Zd[(size_t)k * D + p] = s_x[p];
                Zt[(size_t)k * D + p] = st;
                zt_s[p] = st;
            } else {
                zt_s[p] = Zt[(size_t)k * D + p];
            }
        }
        __syncthreads();
        slice_h_update<T, R>(H, zt_s, nxt, Hn, seg[k], seg[k + 1], tid, nthr);
    }
}

}  // namespace bfc
