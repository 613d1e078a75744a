// Device kernels of the butterfly-completion hot path (Alg. 1 / Eqs.
// grad_butterfly_*), templated on the compute type T (float for the
// precision form, double for the FP64 path) and the rank R.
//
// Orders and buffers (see bfc_internal.h): every training entry has a
// position in each level order l = 0..L+1.  Level-l work reads contiguous
// per-position data (environment vectors, values) of its own order and
// scatters what the next level needs through the precomputed maps nxt / prv.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bfc {

template <typename T> struct cvec;
template <> struct cvec<float> { typedef float2 type; };
template <> struct cvec<double> { typedef double2 type; };

template <typename V> __device__ __forceinline__ V czero() { V v; v.x = 0; v.y = 0; return v; }

// a * b
template <typename V> __device__ __forceinline__ V cmul(V a, V b)
{
    V r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
// acc += a * b
template <typename V> __device__ __forceinline__ void cmac(V& acc, V a, V b)
{
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}
// acc += conj(a) * b
template <typename V> __device__ __forceinline__ void cmacc(V& acc, V a, V b)
{
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(-a.y, b.x, acc.y);
}

template <typename V> __device__ __forceinline__ double2 to_d2(V a)
{
    return make_double2((double)a.x, (double)a.y);
}
template <typename V> __device__ __forceinline__ V from_d2(double2 a)
{
    V v;
    v.x = (decltype(v.x))a.x;
    v.y = (decltype(v.y))a.y;
    return v;
}

// Kahan step: s + x with running compensation c (true sum ~ s - c).  The
// steps are explicitly rounded so that no product of the caller's x can be
// contracted into them.
__device__ __forceinline__ void kahan(float& s, float& c, float x)
{
    const float y = __fsub_rn(x, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

// Four consecutive complex values from 16-byte-aligned shared memory.
__device__ __forceinline__ void load4(float2 (&d)[4], const float2* p)
{
    const float4 a = *reinterpret_cast<const float4*>(p);
    const float4 b = *reinterpret_cast<const float4*>(p + 2);
    d[0] = make_float2(a.x, a.y);
    d[1] = make_float2(a.z, a.w);
    d[2] = make_float2(b.x, b.y);
    d[3] = make_float2(b.z, b.w);
}
__device__ __forceinline__ void load4(double2 (&d)[4], const double2* p)
{
#pragma unroll
    for (int u = 0; u < 4; ++u) d[u] = p[u];
}

// Slice id of the middle factor S^{m+1}: psi^{-1}(i_0..i_{L-m}, j_0..j_{m-1}).
__device__ __forceinline__ int slice_of(int pi, int pj, int m, int L)
{
    return ((pi >> (m - 1)) << m) | (pj >> (L - m));
}

// Packed lower-triangular index (p >= q).
__host__ __device__ __forceinline__ constexpr int tri(int p, int q) { return (p * (p + 1) >> 1) + q; }

// ------------------------------------------------------------------------
// Right environments, one level: w_{m-1} = Z^{m+1}(k) w_m for every entry of
// slice k (Alg. 1: the right vector v, built from the right end).  One CTA
// per slice; the slice is staged in shared memory and read by broadcast.
// (8 CTAs of 128 threads per SM: the slice stays in shared memory instead of
// being hoisted into registers, so enough loads are in flight to cover DRAM
// latency; rows of an even number of complex64 values move as 16-byte
// vectors.)
template <typename T, int R>
__global__ void __launch_bounds__(128, 8)
k_env_right(const typename cvec<T>::type* __restrict__ Win,
            typename cvec<T>::type* __restrict__ Wout,
            const typename cvec<T>::type* __restrict__ Zm,
            const int32_t* __restrict__ seg, const int32_t* __restrict__ prv, int S)
{
    typedef typename cvec<T>::type V;
    constexpr bool VEC = sizeof(V) == 8 && R % 2 == 0;
    __shared__ V z[R * R];
    for (int k = blockIdx.x; k < S; k += gridDim.x) {
        const int s0 = seg[k], s1 = seg[k + 1];
        if (s0 == s1) continue;
        __syncthreads();
        for (int q = threadIdx.x; q < R * R; q += blockDim.x) z[q] = Zm[(size_t)k * R * R + q];
        __syncthreads();
        if constexpr (VEC) {
            for (int p = s0 + threadIdx.x; p < s1; p += blockDim.x) {
                V w[R];
                const float4* src = reinterpret_cast<const float4*>(Win + (size_t)p * R);
#pragma unroll
                for (int c = 0; c < R / 2; ++c) {
                    const float4 v = __ldg(src + c);
                    w[2 * c].x = v.x; w[2 * c].y = v.y;
                    w[2 * c + 1].x = v.z; w[2 * c + 1].y = v.w;
                }
                const size_t o = (size_t)prv[p] * R;
                V res[R];
#pragma unroll
                for (int a = 0; a < R; ++a) {
                    V acc = czero<V>();
#pragma unroll
                    for (int c = 0; c < R; ++c) cmac(acc, z[a * R + c], w[c]);
                    res[a] = acc;
                }
                float4* dst = reinterpret_cast<float4*>(Wout + o);
#pragma unroll
                for (int a = 0; a < R / 2; ++a)
                    dst[a] = make_float4(res[2 * a].x, res[2 * a].y, res[2 * a + 1].x, res[2 * a + 1].y);
            }
        } else {
            for (int p = s0 + threadIdx.x; p < s1; p += blockDim.x) {
                V w[R];
#pragma unroll
                for (int c = 0; c < R; ++c) w[c] = Win[(size_t)p * R + c];
                const size_t o = (size_t)prv[p] * R;
                // one output value at a time, stored at once (not unrolled,
                // so the slice is read from shared memory, not held in
                // registers across entries)
#pragma unroll 1
                for (int a = 0; a < R; ++a) {
                    V acc = czero<V>();
#pragma unroll
                    for (int c = 0; c < R; ++c) cmac(acc, z[a * R + c], w[c]);
                    Wout[o + a] = acc;
                }
            }
        }
    }
}

// w_L = zL(j, :) for the entries in order L.
template <typename T, int R>
__global__ void k_env_init(typename cvec<T>::type* __restrict__ WL,
                           const typename cvec<T>::type* __restrict__ zL,
                           const int32_t* __restrict__ jL, int64_t N)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N * R) return;
    int64_t p = q / R;
    int c = (int)(q - p * R);
    WL[q] = zL[(int64_t)jL[p] * R + c];
}

// ------------------------------------------------------------------------
// Normal equations of Alg. 1 (complex form): for a block (one fiber of S^1 or
// S^{L+2}, or one slice of a middle factor) with design vectors a_e,
//   K = sum conj(a_e) a_e^T + lambda I,   y = sum conj(a_e) t_e,   K s = y.
// Every kernel that accumulates K and y writes them, packed lower-triangular
// (element (p, q), p >= q, at tri(p, q)) followed by y, to a per-block
// record; a solve kernel then factors and solves.
//
// FP64 on this GPU runs at 1/64 of the FP32 rate and a warp-wide FP64
// instruction holds an SM sub-partition's FP64 pipe for tens of cycles
// whatever the number of active lanes, so every FP64 stage below keeps all 32
// lanes busy: small systems are solved one per thread, large ones with rows
// spread over the lanes.

// Packed pairs of FP32 values (the f32x2 arithmetic of sm_100 and later): one
// instruction does two lanes' worth of adds or fused multiply-adds.
__device__ __forceinline__ uint64_t c2pack(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void c2unpack(uint64_t r, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t c2fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ uint64_t c2add(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t c2sub(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t c2mul(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

template <typename E> __device__ __forceinline__ void csub_mul_conj(E& acc, E a, E b)
{
    // acc -= a * conj(b)
    acc.x -= a.x * b.x + a.y * b.y;
    acc.y -= a.y * b.x - a.x * b.y;
}

// Error-free transformations (Knuth TwoSum, FMA-based TwoProd) for
// double-float ("hi + lo" float pair, about 48 significant bits) arithmetic
// on the FP32 pipes.  Every operation whose rounding the transformation
// relies on is an explicitly rounded intrinsic (__fadd_rn, __fsub_rn,
// __fmul_rn): nvcc contracts a plain product feeding an addition into one
// FMA by default (--fmad=true), which would make s = a + b exact in the
// product and leave e counting the product's rounding error twice.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// Double-float complex update acc -= k (sh + sl) for a complex64 k and a
// double-float complex s, on packed (re, im) pairs: hi = (re_hi, im_hi), lo =
// (re_lo, im_lo), so each step is one f32x2 instruction for both components.  Every operation is an explicitly rounded packed
// instruction (inline PTX is never contracted), so TwoSum and the FMA-based
// TwoProd stay exact.  DfS2 holds the packed forms of s = sh + sl that the
// products need (prepared once per column and shared by a lane's rows).
struct DfS2 {
    uint64_t sh, shn, shr, shrn, sl, slr;
};
__device__ __forceinline__ DfS2 df2_prep(float2 sh, float2 sl)
{
    DfS2 r;
    r.sh = c2pack(sh.x, sh.y);
    r.shn = c2pack(-sh.x, -sh.y);
    r.shr = c2pack(-sh.y, sh.x);
    r.shrn = c2pack(sh.y, -sh.x);
    r.sl = c2pack(sl.x, sl.y);
    r.slr = c2pack(-sl.y, sl.x);
    return r;
}
__device__ __forceinline__ void two_sum2(uint64_t a, uint64_t b, uint64_t& s, uint64_t& e)
{
    s = c2add(a, b);
    const uint64_t bb = c2sub(s, a);
    e = c2add(c2sub(a, c2sub(s, bb)), c2sub(b, bb));
}
// hi + lo -= k (sh + sl).  With A = k.re (sh.re, sh.im) and B = k.im (-sh.im,
// sh.re), k sh = A + B; fl(-A), fl(-B) enter hi by TwoSum and their exact
// product errors, with k sl, enter lo.
__device__ __forceinline__ void df2_sub_cmul(uint64_t& hi, uint64_t& lo, float2 k, const DfS2& s)
{
    const uint64_t kx = c2pack(k.x, k.x), ky = c2pack(k.y, k.y);
    const uint64_t pa = c2mul(kx, s.shn);     // -fl(A)
    const uint64_t ea = c2fma(kx, s.sh, pa);  // A - fl(A)
    const uint64_t pb = c2mul(ky, s.shrn);    // -fl(B)
    const uint64_t eb = c2fma(ky, s.shr, pb); // B - fl(B)
    uint64_t t, e;
    two_sum2(hi, pa, t, e);
    hi = t;
    lo = c2add(lo, e);
    two_sum2(hi, pb, t, e);
    hi = t;
    lo = c2add(lo, e);
    uint64_t w = c2fma(kx, s.sl, ea);
    w = c2fma(ky, s.slr, w);
    lo = c2sub(lo, c2add(w, eb));
}

// Hermitian Cholesky + two triangular solves for one small system held by one
// thread (R compile-time: the loops unroll and K, y stay in registers).
// K: packed lower (R(R+1)/2), y: right-hand side, overwritten by the solution.
template <int R>
__device__ __forceinline__ bool thread_chol_solve(double2 (&K)[R * (R + 1) / 2], double2 (&y)[R], double tol)
{
#pragma unroll
    for (int c = 0; c < R; ++c) {
        double d = K[tri(c, c)].x;
#pragma unroll
        for (int q = 0; q < c; ++q) d -= K[tri(c, q)].x * K[tri(c, q)].x + K[tri(c, q)].y * K[tri(c, q)].y;
        if (!(d > tol)) return false;
        const double piv = sqrt(d), inv = 1.0 / piv;
        K[tri(c, c)] = make_double2(piv, inv);  // .y keeps 1/piv for the solves
#pragma unroll
        for (int row = c + 1; row < R; ++row) {
            double2 acc = K[tri(row, c)];
#pragma unroll
            for (int q = 0; q < c; ++q) csub_mul_conj(acc, K[tri(row, q)], K[tri(c, q)]);
            K[tri(row, c)] = make_double2(acc.x * inv, acc.y * inv);
        }
    }
#pragma unroll
    for (int row = 0; row < R; ++row) {
        double2 acc = y[row];
#pragma unroll
        for (int q = 0; q < row; ++q) {
            const double2 l = K[tri(row, q)], z = y[q];
            acc.x -= l.x * z.x - l.y * z.y;
            acc.y -= l.x * z.y + l.y * z.x;
        }
        const double inv = K[tri(row, row)].y;
        y[row] = make_double2(acc.x * inv, acc.y * inv);
    }
#pragma unroll
    for (int row = R - 1; row >= 0; --row) {
        double2 acc = y[row];
#pragma unroll
        for (int q = row + 1; q < R; ++q) {
            const double2 l = K[tri(q, row)], z = y[q];
            acc.x -= l.x * z.x + l.y * z.y;
            acc.y -= l.x * z.y - l.y * z.x;
        }
        const double inv = K[tri(row, row)].y;
        y[row] = make_double2(acc.x * inv, acc.y * inv);
    }
    return true;
}

// ------------------------------------------------------------------------
// Sums of one warp over the rows s0 .. s1 of A (R values each) and the values
// tv: K[p][q] = sum conj(a_p) a_q for p >= q and y[p] = sum conj(a_p) t.  Lanes
// own the R(R+1)/2 + R items; chunks of 32 rows pass through the warp's own
// shared memory (a_s: 32 R values, t_s: 32); in float the per-chunk partials
// are folded into Kahan-compensated sums.  emit(item, p, q, sum, comp) hands
// out every item once (q = -2: y), its value being sum - comp.
template <typename T, int R, typename F>
__device__ __forceinline__ void warp_sums(const typename cvec<T>::type* __restrict__ A,
                                          const typename cvec<T>::type* __restrict__ tv, int s0, int s1,
                                          typename cvec<T>::type* a_s, typename cvec<T>::type* t_s, int lane, F emit)
{
    typedef typename cvec<T>::type V;
    constexpr bool COMP = sizeof(T) == 4;
    constexpr int NP = R * (R + 1) / 2;
    constexpr int NI = NP + R;
    constexpr int IPL = (NI + 31) / 32;

    int ip[IPL], iq[IPL];
#pragma unroll
    for (int u = 0; u < IPL; ++u) {
        const int it = lane + 32 * u;
        ip[u] = -1;
        iq[u] = -1;
        if (it < NP) {
            int p = 0;
            while ((p + 1) * (p + 2) / 2 <= it) ++p;
            ip[u] = p;
            iq[u] = it - p * (p + 1) / 2;
        } else if (it < NI) {
            ip[u] = it - NP;
            iq[u] = -2;  // right-hand side item
        }
    }
    V acc[IPL], sum[IPL], cmp[IPL];
#pragma unroll
    for (int u = 0; u < IPL; ++u) { acc[u] = czero<V>(); sum[u] = czero<V>(); cmp[u] = czero<V>(); }

    for (int base = s0; base < s1; base += 32) {
        const int cnt = min(32, s1 - base);
        __syncwarp();
        // the chunk's rows are contiguous: copy them as one coalesced block
        // (16-byte moves in complex64 at even rank, where every row starts on
        // a 16-byte boundary)
        {
            const V* src = A + (size_t)base * R;
            const int nv = cnt * R;
            if constexpr (sizeof(V) == 8 && R % 2 == 0) {
                for (int x = lane; x < nv / 2; x += 32)
                    reinterpret_cast<float4*>(a_s)[x] = reinterpret_cast<const float4*>(src)[x];
            } else {
                for (int x = lane; x < nv; x += 32) a_s[x] = src[x];
            }
            if (lane < cnt) t_s[lane] = tv[base + lane];
        }
        __syncwarp();
        for (int e = 0; e < cnt; ++e) {
            const V* ae = &a_s[e * R];
#pragma unroll
            for (int u = 0; u < IPL; ++u) {
                if (ip[u] >= 0) {   // Gram item (iq >= 0) or right-hand side (iq == -2): one code path
                    const V* bp = iq[u] >= 0 ? ae + iq[u] : &t_s[e];
                    cmacc(acc[u], ae[ip[u]], *bp);
                }
            }
        }
        if (COMP) {
#pragma unroll
            for (int u = 0; u < IPL; ++u) {
                float sx = (float)sum[u].x, sy = (float)sum[u].y, cx = (float)cmp[u].x, cy = (float)cmp[u].y;
                kahan(sx, cx, (float)acc[u].x);
                kahan(sy, cy, (float)acc[u].y);
                sum[u].x = sx; sum[u].y = sy; cmp[u].x = cx; cmp[u].y = cy;
                acc[u] = czero<V>();
            }
        }
    }
#pragma unroll
    for (int u = 0; u < IPL; ++u) {
        const int it = lane + 32 * u;
        if (it < NI) emit(it, ip[u], iq[u], COMP ? sum[u] : acc[u], cmp[u]);
    }
}

// Outer fibers, stage 1: one warp per fiber accumulates K and y (r x r) over
// the fiber's entries (warp_sums).  A: design vectors in the level order (w_0
// for the S^1 rows, h_{L+1} for the S^{L+2} columns).
// Output record per fiber: [K packed (R(R+1)/2) | y (R)] in FP64.
template <typename T, int R>
__global__ void __launch_bounds__(128)
k_outer_gram(const typename cvec<T>::type* __restrict__ A, const typename cvec<T>::type* __restrict__ tv,
             const int32_t* __restrict__ seg, int nfib, double2* __restrict__ rec)
{
    typedef typename cvec<T>::type V;
    constexpr int NI = R * (R + 1) / 2 + R;
    constexpr int WPB = 4;
    __shared__ __align__(16) V a_s[WPB][32 * R];
    __shared__ V t_s[WPB][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int f = blockIdx.x * WPB + wib;
    if (f >= nfib) return;  // whole warp leaves; only warp-level barriers below
    warp_sums<T, R>(A, tv, seg[f], seg[f + 1], a_s[wib], t_s[wib], lane, [&](int it, int, int, V s, V c) {
        rec[(size_t)f * NI + it] = make_double2((double)s.x - (double)c.x, (double)s.y - (double)c.y);
    });
}

// Outer fibers, stage 2: one thread per fiber solves K + lambda I in FP64
// (32 independent fibers per warp keep every lane of the FP64 pipe busy).
// A system whose pivot falls to <= tol keeps its old fiber and is counted.
template <typename T, int R>
__global__ void __launch_bounds__(64)
k_outer_solve(const double2* __restrict__ rec, int nfib, double lambda, double ridge, double2* __restrict__ zd,
              typename cvec<T>::type* __restrict__ zt, unsigned long long* __restrict__ nsing)
{
    typedef typename cvec<T>::type V;
    constexpr int NP = R * (R + 1) / 2;
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nfib) return;
    double2 K[NP], y[R];
    const double2* src = rec + (size_t)f * (NP + R);
#pragma unroll
    for (int q = 0; q < NP; ++q) K[q] = src[q];
#pragma unroll
    for (int q = 0; q < R; ++q) y[q] = src[NP + q];
    double tr0 = 0.0;
#pragma unroll
    for (int p = 0; p < R; ++p) tr0 += K[tri(p, p)].x;
    const double lam = fmax(lambda, ridge * tr0 / R);
#pragma unroll
    for (int p = 0; p < R; ++p) K[tri(p, p)].x += lam;
    const double tol = lam > 0.0 ? 0.0 : 1e-14 * (tr0 + R * lam);
    if (thread_chol_solve<R>(K, y, tol)) {
#pragma unroll
        for (int c = 0; c < R; ++c) {
            zd[(size_t)f * R + c] = y[c];
            zt[(size_t)f * R + c] = from_d2<V>(y[c]);
        }
    } else {
        atomicAdd(nsing, 1ull);
    }
}

// Outer fibers, stage 3 (one warp per fiber).  Rows (S^1): h_1 = z1(i, :) for
// every entry, written into order 1.  Columns (S^{L+2}): x = h_{L+1}^T zL(j),
// per-fiber sums of |t - x|^2 and |t|^2 for the training error.
template <typename T, int R, bool COLS>
__global__ void __launch_bounds__(128)
k_outer_post(const typename cvec<T>::type* __restrict__ A, const typename cvec<T>::type* __restrict__ tv,
             const int32_t* __restrict__ seg, int nfib, const typename cvec<T>::type* __restrict__ zt,
             const int32_t* __restrict__ nxt, typename cvec<T>::type* __restrict__ Hn,
             double* __restrict__ err_part)
{
    typedef typename cvec<T>::type V;
    const int lane = threadIdx.x & 31;
    const int f = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (f >= nfib) return;
    const int s0 = seg[f], s1 = seg[f + 1];
    // complex64 rows of an even rank are written as 16-byte vectors
    constexpr bool VEC = sizeof(V) == 8 && R % 2 == 0;
    V zf[R];
#pragma unroll
    for (int c = 0; c < R; ++c) zf[c] = zt[(size_t)f * R + c];
    if (!COLS) {
        for (int p = s0 + lane; p < s1; p += 32) {
            const size_t o = (size_t)nxt[p] * R;
            if constexpr (VEC) {
                float4* d4 = reinterpret_cast<float4*>(Hn + o);
#pragma unroll
                for (int c = 0; c < R / 2; ++c)
                    d4[c] = make_float4(zf[2 * c].x, zf[2 * c].y, zf[2 * c + 1].x, zf[2 * c + 1].y);
            } else {
#pragma unroll
                for (int c = 0; c < R; ++c) Hn[o + c] = zf[c];
            }
        }
    } else {
        // lane sums in the compute type (about two entries per lane), the
        // warp reduction in FP64
        T numl = T(0), denl = T(0);
        for (int p = s0 + lane; p < s1; p += 32) {
            V x = czero<V>();
#pragma unroll
            for (int c = 0; c < R; ++c) cmac(x, A[(size_t)p * R + c], zf[c]);
            const V t = tv[p];
            const T dx = t.x - x.x, dy = t.y - x.y;
            numl += dx * dx + dy * dy;
            denl += t.x * t.x + t.y * t.y;
        }
        double num = (double)numl, den = (double)denl;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            num += __shfl_xor_sync(0xffffffffu, num, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        if (lane == 0) {
            err_part[2 * (size_t)f] = num;
            err_part[2 * (size_t)f + 1] = den;
        }
    }
}

// ------------------------------------------------------------------------
// Middle level m, stage 1 (Gram): one CTA per slice k of S^{m+1}
// (persistent over slices).
//   a_e = h_m(e) (x) w_m(e), a[p r + c] = h_p w_c, K = sum conj(a) a^T,
//   y = sum conj(a) t over the slice's entries (Alg. 1 middle branch).
// Threads own 4x4 complex tiles of the lower triangle of K (split over G
// entry groups for small ranks); the diagonal-tile threads also accumulate y.
// Software pipeline over chunks of CE entries with one barrier per chunk:
// while chunk c is multiplied out of one design-vector buffer, chunk c+1 is
// formed into the other from its staged h, w, t, and chunk c+2 is fetched
// into the other staging buffer with cp.async.  In float every FOLD chunks
// the register partials are folded into Kahan-compensated running sums
// (sums in registers, compensation in shared memory).
// Output record per slice: [K packed lower | y] in the compute type.
template <typename T, int R> struct GramCfg {
    static constexpr int D = R * R;
    static constexpr int DP = (D + 3) / 4 * 4;
    static constexpr int NB = DP / 4;
    static constexpr int NT = NB * (NB + 1) / 2;
    static constexpr int CE = 32;
    static constexpr int GT = (160 / NT) < 1 ? 1 : (160 / NT);
    static constexpr int G = GT > CE ? CE : GT;
    static constexpr int NTH = ((NT * G + 31) / 32) * 32;
    static constexpr int FOLD = 2;
    static constexpr bool COMP = sizeof(T) == 4;
    static constexpr int NPK = D * (D + 1) / 2;
    static constexpr int CSTRIDE = 40;  // compensation floats per thread (32 K + 8 y)
    static constexpr size_t VS = sizeof(typename cvec<T>::type);
    static constexpr size_t RING = 2 * (size_t)CE * DP * VS + 2 * (size_t)CE * VS;  // a and t rings
    static constexpr size_t STAGE1 = ((2 * (size_t)CE * R + CE) * VS + 15) / 16 * 16;
    static constexpr size_t CBYTES = COMP ? (size_t)NTH * CSTRIDE * sizeof(float) : 0;
    static constexpr size_t KBYTES = G > 1 ? (size_t)(NPK + D) * sizeof(double2) : 0;
    static constexpr size_t UBYTES = ((CBYTES > KBYTES ? CBYTES : KBYTES) + 15) / 16 * 16;
    static constexpr size_t SMEM = RING + 2 * STAGE1 + UBYTES + 16;
    static constexpr int MINB0 = 65536 / (NTH * 128);
    static constexpr int MINB = MINB0 < 1 ? 1 : (MINB0 > 3 ? 3 : MINB0);
};

// Asynchronous global -> shared copy of one complex value (8 or 16 bytes).
__device__ __forceinline__ void cp_async_v(float2* smem_dst, const float2* gmem_src)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_v(double2* smem_dst, const double2* gmem_src)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <typename T, int R>
__global__ void __launch_bounds__(GramCfg<T, R>::NTH, GramCfg<T, R>::MINB)
k_mid_gram(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Wm,
           const typename cvec<T>::type* __restrict__ tv, const int32_t* __restrict__ seg,
           typename cvec<T>::type* __restrict__ rec, int S)
{
    typedef typename cvec<T>::type V;
    typedef GramCfg<T, R> C;
    constexpr int D = C::D, DP = C::DP, NPK = C::NPK, CE = C::CE, NTH = C::NTH;
    extern __shared__ __align__(16) unsigned char smem[];
    V* ring = (V*)smem;                                      // [2][CE][DP]
    V* tring = ring + 2 * CE * DP;                           // [2][CE]
    unsigned char* stage_base = smem + C::RING;              // 2 x { h [CE][R], w [CE][R], t [CE] }
    unsigned char* U = stage_base + 2 * C::STAGE1;
    float* c_s = (float*)U;                                  // compensation [CSTRIDE][NTH]
    double2* Kacc = (double2*)U;                             // group reduction (G > 1)

    const int tid = threadIdx.x;
    const bool worker = tid < C::NT * C::G;
    const int grp = tid / C::NT, tile = tid - (tid / C::NT) * C::NT;
    int I = 0;
    while ((I + 1) * (I + 2) / 2 <= tile) ++I;
    const int J = tile - I * (I + 1) / 2;
    const bool diag = (I == J);

    // fetch chunk (base, cnt) of the current slice into staging buffer sb
    auto fetch = [&](int sb, int base, int cnt) {
        V* hs = (V*)(stage_base + sb * C::STAGE1);
        V* ws = hs + CE * R;
        V* ts = ws + CE * R;
        for (int q = tid; q < cnt * R; q += NTH) {
            cp_async_v(hs + q, H + (size_t)base * R + q);
            cp_async_v(ws + q, Wm + (size_t)base * R + q);
        }
        for (int e = tid; e < cnt; e += NTH) cp_async_v(ts + e, tv + base + e);
        cp_async_commit();
    };
    // form the design vectors (and copy t) of staging buffer sb into ring buffer rb
    auto form = [&](int sb, int rb, int cnt) {
        const V* hs = (const V*)(stage_base + sb * C::STAGE1);
        const V* ws = hs + CE * R;
        const V* ts = ws + CE * R;
        V* buf = ring + (size_t)rb * CE * DP;
        for (int idx = tid; idx < CE * DP; idx += NTH) {
            const int e = idx / DP, q = idx - e * DP;
            V a = czero<V>();
            if (q < D && e < cnt) a = cmul(hs[e * R + q / R], ws[e * R + q % R]);
            buf[idx] = a;
        }
        for (int e = tid; e < CE; e += NTH) tring[rb * CE + e] = e < cnt ? ts[e] : czero<V>();
    };

    for (int k = blockIdx.x; k < S; k += gridDim.x) {
        const int s0 = seg[k], s1 = seg[k + 1];
        const int nch = (s1 - s0 + CE - 1) / CE;
        V acc[4][4], sum[4][4], yacc[4], ysum[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            yacc[u] = czero<V>();
            ysum[u] = czero<V>();
#pragma unroll
            for (int v = 0; v < 4; ++v) { acc[u][v] = czero<V>(); sum[u][v] = czero<V>(); }
        }
        __syncthreads();  // previous slice done with every shared buffer
        if (C::COMP && worker)
            for (int x = 0; x < C::CSTRIDE; ++x) c_s[x * NTH + tid] = 0.0f;
        // prologue: chunk 0 staged and formed, chunk 1 in flight
        if (nch > 0) {
            fetch(0, s0, min(CE, s1 - s0));
            cp_async_wait_all();
            __syncthreads();
            form(0, 0, min(CE, s1 - s0));
            if (nch > 1) fetch(1, s0 + CE, min(CE, s1 - s0 - CE));
        }
        int pend = 0;
        for (int c = 0; c < nch; ++c) {
            const int base = s0 + c * CE;
            const int cnt = min(CE, s1 - base);
            // chunk c formed (ring c&1) and chunk c+1 staged (stage (c+1)&1) by everybody
            cp_async_wait_all();
            __syncthreads();
            if (c + 1 < nch) {
                form((c + 1) & 1, (c + 1) & 1, min(CE, s1 - base - CE));
                if (c + 2 < nch) fetch(c & 1, base + 2 * CE, min(CE, s1 - base - 2 * CE));
            }
            if (worker) {
                const V* buf = ring + (size_t)(c & 1) * CE * DP;
                const V* ts = tring + (c & 1) * CE;
                for (int e = grp; e < cnt; e += C::G) {
                    const V* ae = buf + e * DP;
                    V ap[4], aq[4];
                    load4(ap, ae + I * 4);
                    load4(aq, ae + J * 4);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int v = 0; v < 4; ++v) cmacc(acc[u][v], ap[u], aq[v]);
                    if (diag) {
                        const V te = ts[e];
#pragma unroll
                        for (int u = 0; u < 4; ++u) cmacc(yacc[u], ap[u], te);
                    }
                }
                if (C::COMP && (++pend == C::FOLD || c + 1 == nch)) {
                    pend = 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            float sx = (float)sum[u][v].x, sy = (float)sum[u][v].y;
                            float& cx = c_s[(2 * (u * 4 + v)) * NTH + tid];
                            float& cy = c_s[(2 * (u * 4 + v) + 1) * NTH + tid];
                            kahan(sx, cx, (float)acc[u][v].x);
                            kahan(sy, cy, (float)acc[u][v].y);
                            sum[u][v].x = sx; sum[u][v].y = sy;
                            acc[u][v] = czero<V>();
                        }
                        if (diag) {
                            float sx = (float)ysum[u].x, sy = (float)ysum[u].y;
                            float& cx = c_s[(32 + 2 * u) * NTH + tid];
                            float& cy = c_s[(32 + 2 * u + 1) * NTH + tid];
                            kahan(sx, cx, (float)yacc[u].x);
                            kahan(sy, cy, (float)yacc[u].y);
                            ysum[u].x = sx; ysum[u].y = sy;
                            yacc[u] = czero<V>();
                        }
                    }
                }
            }
        }
        if (C::COMP && worker) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    acc[u][v].x = sum[u][v].x - c_s[(2 * (u * 4 + v)) * NTH + tid];
                    acc[u][v].y = sum[u][v].y - c_s[(2 * (u * 4 + v) + 1) * NTH + tid];
                }
                if (diag) {
                    yacc[u].x = ysum[u].x - c_s[(32 + 2 * u) * NTH + tid];
                    yacc[u].y = ysum[u].y - c_s[(32 + 2 * u + 1) * NTH + tid];
                }
            }
        }
        V* out = rec + (size_t)k * (NPK + D);
        if (C::G == 1) {
            if (worker) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int p = I * 4 + u;
                    if (p < D) {
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int q = J * 4 + v;
                            if (q <= p) out[tri(p, q)] = acc[u][v];
                        }
                        if (diag) out[NPK + p] = yacc[u];
                    }
                }
            }
        } else {
            __syncthreads();  // compensation reads done before Kacc overwrites them
            for (int q = tid; q < NPK + D; q += NTH) Kacc[q] = make_double2(0.0, 0.0);
            __syncthreads();
            for (int g = 0; g < C::G; ++g) {  // deterministic order over the groups
                if (worker && grp == g) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int p = I * 4 + u;
                        if (p < D) {
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                const int q = J * 4 + v;
                                if (q <= p) {
                                    Kacc[tri(p, q)].x += (double)acc[u][v].x;
                                    Kacc[tri(p, q)].y += (double)acc[u][v].y;
                                }
                            }
                            if (diag) {
                                Kacc[NPK + p].x += (double)yacc[u].x;
                                Kacc[NPK + p].y += (double)yacc[u].y;
                            }
                        }
                    }
                }
                __syncthreads();
            }
            for (int q = tid; q < NPK + D; q += NTH) out[q] = from_d2<V>(Kacc[q]);
        }
    }
}

// ------------------------------------------------------------------------
// Row of slot s owned by a lane in the warp-level factorization: even slots
// take rows 32 s + lane, odd slots mirror them (32 s + 31 - lane), so the two
// rows of a lane have complementary lengths and the work per lane is balanced.
__device__ __forceinline__ int owned_row(int s, int lane) { return 32 * s + ((s & 1) ? 31 - lane : lane); }

// Warp-level Hermitian Cholesky (K = L L^H) of a D x D packed lower matrix
// in shared or global memory, right-looking and blocked by NBK columns:
//  (1) the NBK x NBK diagonal block is factored column by column;
//  (2) every panel row r below it, owned by one lane, is solved in registers:
//      L[r][j0..j1) = K[r][j0..j1) L_dd^{-H};
//  (3) the trailing matrix gets the rank-NBK update
//      L[r][q] -= sum_k L[r][j0+k] conj(L[q][j0+k]), the lane holding its
//      panel row in registers while all lanes read the same panel row q.
// The diagonal of L is real, so its imaginary slot stores 1 / L_cc for the
// triangular solves.  Returns false (warp-uniform) when a pivot is <= tol.
template <typename E, typename S, int NS>
__device__ bool warp_chol(E* Lm, int D, S tol, int lane)
{
    constexpr int NBK = 8;
    for (int j0 = 0; j0 < D; j0 += NBK) {
        const int j1 = min(j0 + NBK, D);
        // (1) diagonal block
        for (int c = j0; c < j1; ++c) {
            __syncwarp();
            const S d = Lm[tri(c, c)].x;
            if (!(d > tol)) return false;
            const S piv = sqrt(d), inv = S(1) / piv;
            __syncwarp();
            if (lane == 0) {
                E v;
                v.x = piv;
                v.y = inv;
                Lm[tri(c, c)] = v;
            }
            const int r = c + 1 + lane;
            if (r < j1) {
                E l = Lm[tri(r, c)];
                l.x *= inv;
                l.y *= inv;
                Lm[tri(r, c)] = l;
            }
            __syncwarp();
            if (r < j1) {
                const E a = Lm[tri(r, c)];
                for (int q = c + 1; q <= r; ++q) {
                    E cur = Lm[tri(r, q)];
                    csub_mul_conj(cur, a, Lm[tri(q, c)]);
                    Lm[tri(r, q)] = cur;
                }
            }
        }
        __syncwarp();
        if (j1 >= D) break;
        const int nb = j1 - j0;
        // (2) panel rows, solved in registers by their owner lanes
        E x[NS][NBK];
        if constexpr (sizeof(S) == 4) {
            // complex64: the same substitution with the terms as packed fused
            // multiply-adds (the trailing update's form below)
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int r = owned_row(s, lane);
                if (r >= j1 && r < D) {
                    E* rowp = Lm + tri(r, 0);
                    uint64_t p1[NBK], p2[NBK];
#pragma unroll
                    for (int cc = 0; cc < NBK; ++cc) {
                        x[s][cc] = E{};
                        p1[cc] = 0ull;
                        p2[cc] = 0ull;
                        if (cc < nb) {
                            const uint64_t* drow = reinterpret_cast<const uint64_t*>(Lm + tri(j0 + cc, 0) + j0);
                            const E e0 = rowp[j0 + cc];
                            uint64_t acc = c2pack(e0.x, e0.y), sw = 0ull;
#pragma unroll
                            for (int k = 0; k < cc; ++k) {
                                const uint64_t b = drow[k];
                                acc = c2fma(b, p1[k], acc);
                                sw = c2fma(b, p2[k], sw);
                            }
                            float ar, ai, si, sr;
                            c2unpack(acc, ar, ai);
                            c2unpack(sw, si, sr);
                            const S inv = Lm[tri(j0 + cc, j0 + cc)].y;
                            E v;
                            v.x = (ar + sr) * inv;
                            v.y = (ai + si) * inv;
                            x[s][cc] = v;
                            p1[cc] = c2pack(-v.x, v.x);
                            p2[cc] = c2pack(-v.y, -v.y);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < NBK; ++k)
                        if (k < nb) rowp[j0 + k] = x[s][k];
                }
            }
        } else {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int r = owned_row(s, lane);
            if (r >= j1 && r < D) {
                const E* rowp = Lm + tri(r, 0);
#pragma unroll
                for (int k = 0; k < NBK; ++k) x[s][k] = k < nb ? rowp[j0 + k] : E{};
#pragma unroll
                for (int cc = 0; cc < NBK; ++cc) {
                    if (cc < nb) {
                        const E* drow = Lm + tri(j0 + cc, 0);
#pragma unroll
                        for (int k = 0; k < cc; ++k) csub_mul_conj(x[s][cc], x[s][k], drow[j0 + k]);
                        const S inv = drow[j0 + cc].y;
                        x[s][cc].x *= inv;
                        x[s][cc].y *= inv;
                    }
                }
                E* roww = Lm + tri(r, 0);
#pragma unroll
                for (int k = 0; k < NBK; ++k)
                    if (k < nb) roww[j0 + k] = x[s][k];
            }
        }
        }
        __syncwarp();
        // (3) rank-NBK trailing update
        if constexpr (sizeof(S) == 4) {
            // complex64: L[r][q] -= sum_k x_k conj(l_k) (l = L[q][j0 + k]) as
            // two packed fused multiply-adds per term, with the factors of
            // x_k prepared once per row: l (.) (-x.re, x.re) goes into
            // (re, im) and l (.) (-x.im, -x.im) into a second accumulator
            // that holds (im, re)
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int r = owned_row(s, lane);
                if (r >= j1 && r < D) {
                    uint64_t p1[NBK], p2[NBK];
#pragma unroll
                    for (int k = 0; k < NBK; ++k) {
                        const float xr = k < nb ? x[s][k].x : 0.f, xi = k < nb ? x[s][k].y : 0.f;
                        p1[k] = c2pack(-xr, xr);
                        p2[k] = c2pack(-xi, -xi);
                    }
                    E* rowp = Lm + tri(r, 0);
                    auto finish = [&](uint64_t acc, uint64_t sw) {
                        float ar, ai, si, sr;
                        c2unpack(acc, ar, ai);
                        c2unpack(sw, si, sr);
                        E v;
                        v.x = ar + sr;
                        v.y = ai + si;
                        return v;
                    };
                    int q = j1;
                    for (; q + 1 <= r; q += 2) {
                        const uint64_t* qa = reinterpret_cast<const uint64_t*>(Lm + tri(q, 0) + j0);
                        const uint64_t* qb = reinterpret_cast<const uint64_t*>(Lm + tri(q + 1, 0) + j0);
                        const E ea = rowp[q], eb = rowp[q + 1];
                        uint64_t ca = c2pack(ea.x, ea.y), cb = c2pack(eb.x, eb.y), sa = 0ull, sb = 0ull;
                        uint64_t va[NBK], vb[NBK];
#pragma unroll
                        for (int k = 0; k < NBK; ++k)
                            if (k < nb) { va[k] = qa[k]; vb[k] = qb[k]; }
#pragma unroll
                        for (int k = 0; k < NBK; ++k)
                            if (k < nb) {
                                ca = c2fma(va[k], p1[k], ca);
                                sa = c2fma(va[k], p2[k], sa);
                                cb = c2fma(vb[k], p1[k], cb);
                                sb = c2fma(vb[k], p2[k], sb);
                            }
                        rowp[q] = finish(ca, sa);
                        rowp[q + 1] = finish(cb, sb);
                    }
                    if (q <= r) {
                        const uint64_t* qr = reinterpret_cast<const uint64_t*>(Lm + tri(q, 0) + j0);
                        const E e0 = rowp[q];
                        uint64_t c0 = c2pack(e0.x, e0.y), s0 = 0ull;
#pragma unroll
                        for (int k = 0; k < NBK; ++k)
                            if (k < nb) {
                                const uint64_t v = qr[k];
                                c0 = c2fma(v, p1[k], c0);
                                s0 = c2fma(v, p2[k], s0);
                            }
                        rowp[q] = finish(c0, s0);
                    }
                }
            }
        } else {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int r = owned_row(s, lane);
            if (r >= j1 && r < D) {
                E* rowp = Lm + tri(r, 0);
                // two columns per step: both elements and both panel rows are
                // loaded before either element is stored (independent chains)
                int q = j1;
                for (; q + 1 <= r; q += 2) {
                    const E* qa = Lm + tri(q, 0) + j0;
                    const E* qb = Lm + tri(q + 1, 0) + j0;
                    E ca = rowp[q], cb = rowp[q + 1];
                    E va[NBK], vb[NBK];
#pragma unroll
                    for (int k = 0; k < NBK; ++k)
                        if (k < nb) { va[k] = qa[k]; vb[k] = qb[k]; }
#pragma unroll
                    for (int k = 0; k < NBK; ++k)
                        if (k < nb) {
                            csub_mul_conj(ca, x[s][k], va[k]);
                            csub_mul_conj(cb, x[s][k], vb[k]);
                        }
                    rowp[q] = ca;
                    rowp[q + 1] = cb;
                }
                if (q <= r) {
                    const E* qrow = Lm + tri(q, 0) + j0;
                    E cur = rowp[q];
#pragma unroll
                    for (int k = 0; k < NBK; ++k)
                        if (k < nb) csub_mul_conj(cur, x[s][k], qrow[k]);
                    rowp[q] = cur;
                }
            }
        }
        }
    }
    __syncwarp();
    return true;
}

// Column-oriented triangular solves with the right-hand side spread over the
// lanes: row p lives in slot p / 32 of lane p % 32.  L z = b, then L^H x = z.
template <typename E, typename S, int NS>
__device__ __forceinline__ void warp_chol_solve(const E* Lm, int D, E (&bv)[NS], int lane)
{
#pragma unroll
    for (int slot = 0; slot < NS; ++slot) {
        for (int owner = 0; owner < 32; ++owner) {
            const int p = slot * 32 + owner;
            if (p >= D) break;
            E zp;
            zp.x = __shfl_sync(0xffffffffu, bv[slot].x, owner);
            zp.y = __shfl_sync(0xffffffffu, bv[slot].y, owner);
            const S inv = Lm[tri(p, p)].y;
            zp.x *= inv;
            zp.y *= inv;
            if (lane == owner) bv[slot] = zp;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int q = lane + 32 * s;
                if (q > p && q < D) {
                    const E l = Lm[tri(q, p)];
                    bv[s].x -= l.x * zp.x - l.y * zp.y;
                    bv[s].y -= l.x * zp.y + l.y * zp.x;
                }
            }
        }
    }
#pragma unroll
    for (int slot = NS - 1; slot >= 0; --slot) {
        for (int owner = 31; owner >= 0; --owner) {
            const int p = slot * 32 + owner;
            if (p >= D) continue;
            E xp;
            xp.x = __shfl_sync(0xffffffffu, bv[slot].x, owner);
            xp.y = __shfl_sync(0xffffffffu, bv[slot].y, owner);
            const S inv = Lm[tri(p, p)].y;
            xp.x *= inv;
            xp.y *= inv;
            if (lane == owner) bv[slot] = xp;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int q = lane + 32 * s;
                if (q < p) {
                    const E l = Lm[tri(p, q)];   // conj(l) * xp
                    bv[s].x -= l.x * xp.x + l.y * xp.y;
                    bv[s].y -= l.x * xp.y - l.y * xp.x;
                }
            }
        }
    }
}

// Left environment update of slice k: h_{m+1}(e) = h_m(e)^T Z^{m+1}(k) for the
// slice's entries (lanes over entries), scattered into order m+1.
template <typename T, int R>
__device__ __forceinline__ void slice_h_update(const typename cvec<T>::type* __restrict__ H,
                                               const typename cvec<T>::type* zt_s, const int32_t* __restrict__ nxt,
                                               typename cvec<T>::type* __restrict__ Hn, int s0, int s1, int lane)
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
    // two entries per lane and step: both loads are in flight together
    for (int p = s0 + lane; p < s1; p += 64) {
        const int p2 = p + 32;
        const bool two = p2 < s1;
        V h[R], g[R];
        load_row(p, h);
        if (two) load_row(p2, g);
        else
#pragma unroll
            for (int a = 0; a < R; ++a) g[a] = czero<V>();
        const size_t o = (size_t)nxt[p] * R;
        const size_t o2 = two ? (size_t)nxt[p2] * R : 0;
        V r1[R], r2[R];
#pragma unroll
        for (int c = 0; c < R; ++c) {
            V acc2 = czero<V>(), acc3 = czero<V>();
#pragma unroll
            for (int a = 0; a < R; ++a) {
                const V z = zt_s[a * R + c];
                cmac(acc2, h[a], z);
                cmac(acc3, g[a], z);
            }
            r1[c] = acc2;
            r2[c] = acc3;
        }
        store_row(o, r1);
        if (two) store_row(o2, r2);
    }
}

template <typename T, int R> struct SolveCfg {
    static constexpr int D = R * R;
    static constexpr int NPK = D * (D + 1) / 2;
    static constexpr int NS = (D + 31) / 32;
    static constexpr bool MIXED = sizeof(T) == 4;
    // per warp: factor (compute type, padded to 16 bytes), FP64 solution
    // vector, new slice (compute type)
    static constexpr size_t LBYTES = ((size_t)NPK * sizeof(typename cvec<T>::type) + 15) / 16 * 16;
    static constexpr size_t WCORE = (LBYTES + (size_t)D * sizeof(double2) +
                                     (size_t)D * sizeof(typename cvec<T>::type) + (size_t)D * sizeof(T) + 15) /
                                    16 * 16;
    // + one mbarrier per warp (the bulk copy of the record), padded to 16 bytes
    static constexpr size_t WBYTES = WCORE + 16;
    static constexpr int WPB0 = (int)((96 * 1024) / WBYTES);
    static constexpr int WPB = WPB0 < 1 ? 1 : (WPB0 > 4 ? 4 : WPB0);
    static constexpr size_t SMEM = WBYTES * WPB;
    // CTAs per SM the register budget of k_mid_solve targets (bounded by shared memory)
    static constexpr int MINB0 = (int)((227 * 1024) / SMEM);
    static constexpr int MINB = MINB0 < 1 ? 1 : (MINB0 > 3 ? 3 : MINB0);
};

// Middle level m, stage 2 (solve + left update): one warp per slice.
// Precision form (float): the slice's K block arrives in shared memory by one
// bulk copy; complex64 Cholesky of the Jacobi-equilibrated S (K + lambda I) S,
// complex64 solve, then up to three steps of iterative refinement: the
// residual y - (K + lambda I) s is formed in double-float arithmetic
// (TwoSum-compensated float pairs, rows spread over the lanes) against a
// solution kept as a double-float pair, and the correction goes through the
// complex64 factor.  If the factorization breaks down or the refinement does
// not contract, the slice goes on a list for the FP64 Cholesky of
// k_mid_fallback.  FP64 path (double): FP64 Cholesky directly.  The slice is
// written row-major in FP64 and the compute type; then
// h_{m+1}(e) = h_m(e)^T Z^{m+1}(k) for the slice's entries is scattered into
// order m+1.  A singular system keeps its old slice.
template <typename T, int R>
__global__ void __launch_bounds__(32 * SolveCfg<T, R>::WPB, SolveCfg<T, R>::MINB)
k_mid_solve(const typename cvec<T>::type* __restrict__ rec, const typename cvec<T>::type* __restrict__ H,
            const int32_t* __restrict__ seg, const int32_t* __restrict__ nxt,
            typename cvec<T>::type* __restrict__ Hn, double2* __restrict__ Zd,
            typename cvec<T>::type* __restrict__ Zt, double2* __restrict__ fb, double lambda_in, double ridge,
            unsigned long long* __restrict__ nsing, unsigned long long* __restrict__ nfb,
            unsigned long long* __restrict__ nsteps, int32_t* __restrict__ fblist, int S,
            unsigned long long* __restrict__ terr, int skip_copy)
{
    // nfb: slices handed to the FP64 fallback (length of fblist); nsteps: refinement steps;
    // terr: raised when the bulk copy of a record does not complete within the wait limit;
    // skip_copy (failure injection of the tests, bfc_inject_fault): the bulk copies are not
    // issued and the waits give up after a few tries
    typedef typename cvec<T>::type V;
    typedef SolveCfg<T, R> C;
    constexpr int D = C::D, NPK = C::NPK, NS = C::NS;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char* base = smem + (size_t)wib * C::WBYTES;
    V* Lm = (V*)base;
    double2* s_d = (double2*)(base + C::LBYTES);
    V* zt_s = (V*)(s_d + D);
    T* sc_s = (T*)(zt_s + D);  // Jacobi scaling of the complex64 factorization
    // The record's K block reaches shared memory by one bulk copy (the copy
    // engine, completion counted on a per-warp mbarrier) in the precision
    // form; the wait is bounded.
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(base + C::WCORE);
    constexpr uint32_t KBULK = (uint32_t)((NPK & ~1) * sizeof(V));   // a multiple of 16 bytes
    constexpr bool BULK = C::MIXED && KBULK >= 16;
    uint32_t phase = 0;
    // warp-uniform: bulk copies still in use (cleared for good when a wait
    // expires); pending: a copy that was issued and then given up on
    bool use_bulk = BULK;
    bool pending = false;
    uint32_t pending_phase = 0;
    const uint32_t wait_limit = skip_copy ? 64u : (1u << 22);
    if constexpr (BULK) {
        if (lane == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncwarp();
    }

    for (int k = blockIdx.x * C::WPB + wib; k < S; k += gridDim.x * C::WPB) {
        const V* K = rec + (size_t)k * (NPK + D);
        __syncwarp();
        bool have = false;
        if constexpr (BULK) {
            if (use_bulk) {
                // the record stride D (D + 3) / 2 is even for D = r^2, so every
                // record starts on a 16-byte boundary; the previous slice's
                // accesses to the factor area are ordered before the copy
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
                                 ::"r"(bar), "r"(KBULK) : "memory");
                    if (!skip_copy)
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     ::"r"((uint32_t)__cvta_generic_to_shared(Lm)), "l"(K), "r"(KBULK), "r"(bar)
                                     : "memory");
                }
                if ((NPK & 1) && lane == 0) Lm[NPK - 1] = K[NPK - 1];
                bool done = false;
                for (uint32_t it = 0; it < wait_limit && !done; ++it) {
                    uint32_t ok;
                    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                                 "selp.u32 %0, 1, 0, p;\n}\n"
                                 : "=r"(ok) : "r"(bar), "r"(phase) : "memory");
                    done = ok != 0;
                }
                // the phase completes once for all lanes: any lane that saw it
                // completed makes the copy valid for the warp
                done = __any_sync(0xffffffffu, done);
                if (done) {
                    have = true;
                } else {
                    // the copy did not complete: report it, issue no further
                    // copies on this barrier and load by plain loads from here
                    // on (the call's results are undefined)
                    if (lane == 0) atomicExch(terr, 1ull);
                    use_bulk = false;
                    pending = !skip_copy;
                    pending_phase = phase;
                }
                phase ^= 1u;
            }
        }
        if (!have) {
            if constexpr (C::MIXED) {
                const float4* src = reinterpret_cast<const float4*>(K);
                float4* dst = reinterpret_cast<float4*>(Lm);
#pragma unroll 4
                for (int q = lane; q < NPK / 2; q += 32) dst[q] = src[q];
                if ((NPK & 1) && lane == 0) Lm[NPK - 1] = K[NPK - 1];
            } else {
                for (int q = lane; q < NPK; q += 32) Lm[q] = K[q];
            }
        }
        __syncwarp();
        double tr = 0.0;
        for (int p = lane; p < D; p += 32) tr += (double)Lm[tri(p, p)].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        // lambda, raised to the ridge floor (relative to the mean diagonal) when set
        const double lambda = fmax(lambda_in, ridge * tr / D);
        const double tol = lambda > 0.0 ? 0.0 : 1e-14 * (tr + D * lambda);
        if constexpr (C::MIXED) {
            // equilibrate: factor S (K + lambda I) S with S = diag(K_pp + lambda)^(-1/2)
            for (int p = lane; p < D; p += 32) {
                const T dp = Lm[tri(p, p)].x + (T)lambda;
                sc_s[p] = dp > (T)0 ? rsqrt(dp) : (T)1;
            }
            __syncwarp();
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int r = owned_row(s, lane);
                if (r < D) {
                    V* rowp = Lm + tri(r, 0);
                    const T sr = sc_s[r];
                    for (int q = 0; q <= r; ++q) {
                        V v = rowp[q];
                        if (q == r) v.x += (T)lambda;
                        const T f = sr * sc_s[q];
                        v.x *= f;
                        v.y *= f;
                        rowp[q] = v;
                    }
                }
            }
        } else {
            for (int p = lane; p < D; p += 32) Lm[tri(p, p)].x += (T)lambda;
        }
        __syncwarp();
        double2 sv[NS];
        bool ok;
        if constexpr (C::MIXED) {
            bool conv = false;
            if (warp_chol<V, T, NS>(Lm, D, (T)tol, lane)) {
                V bv[NS];
                T scl[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int p = lane + 32 * s;
                    scl[s] = p < D ? sc_s[p] : (T)0;
                    bv[s] = p < D ? K[NPK + p] : czero<V>();
                    bv[s].x *= scl[s];
                    bv[s].y *= scl[s];
                }
                warp_chol_solve<V, T, NS>(Lm, D, bv, lane);
                // solution as a double-float pair (hi, lo) per component
                float2 sh[NS], sl[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    sh[s] = make_float2(bv[s].x * scl[s], bv[s].y * scl[s]);
                    sl[s] = make_float2(0.f, 0.f);
                }
                float4* s_df = reinterpret_cast<float4*>(s_d);  // {re_hi, im_hi, re_lo, im_lo} per row
                const float lamf = (float)lambda;
                float dmax = 0.f, smax = 0.f;
                for (int it = 0; it < 3; ++it) {
                    // residual r = y - (K + lambda I) s in double-float arithmetic, rows over the lanes
                    __syncwarp();
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const int p = lane + 32 * s;
                        if (p < D) s_df[p] = make_float4(sh[s].x, sh[s].y, sl[s].x, sl[s].y);
                    }
                    __syncwarp();
                    // one pass over q for all rows of the lane: s_q is read once
                    // for them, and K_pq comes from the stored lower triangle
                    // (conjugated above the diagonal), so no lane idles
                    // packed double-float accumulators: (re, im) of hi and of lo
                    uint64_t ahi[NS], alo[NS];
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const int p = lane + 32 * s;
                        ahi[s] = 0ull;
                        alo[s] = 0ull;
                        if (p < D) {
                            const V yp = K[NPK + p];
                            ahi[s] = c2pack(yp.x, yp.y);
                            df2_sub_cmul(ahi[s], alo[s], make_float2(lamf, 0.f), df2_prep(sh[s], sl[s]));
                        }
                    }
                    // K_pq for 8 columns are fetched (from L2) before their products
                    constexpr int QB = 8;
                    for (int q0 = 0; q0 < D; q0 += QB) {
                        V kv[NS][QB];
#pragma unroll
                        for (int i = 0; i < QB; ++i) {
                            const int q = q0 + i;
#pragma unroll
                            for (int s = 0; s < NS; ++s) {
                                const int p = lane + 32 * s;
                                kv[s][i] = czero<V>();
                                if (p < D && q < D) {
                                    const bool lo = q <= p;
                                    kv[s][i] = K[lo ? tri(p, q) : tri(q, p)];
                                    if (!lo) kv[s][i].y = -kv[s][i].y;
                                }
                            }
                        }
#pragma unroll
                        for (int i = 0; i < QB; ++i) {
                            const int q = q0 + i;
                            if (q < D) {
                                const float4 sq = s_df[q];
                                const DfS2 sp = df2_prep(make_float2(sq.x, sq.y), make_float2(sq.z, sq.w));
#pragma unroll
                                for (int s = 0; s < NS; ++s)
                                    if (lane + 32 * s < D) df2_sub_cmul(ahi[s], alo[s], kv[s][i], sp);
                            }
                        }
                    }
                    float rr[NS][2];
                    float rmax = 0.f;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        c2unpack(c2add(ahi[s], alo[s]), rr[s][0], rr[s][1]);
                        rmax = fmaxf(rmax, fmaxf(fabsf(rr[s][0]), fabsf(rr[s][1])));
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
                    const float sc = rmax > 0.f ? rmax : 1.f;
                    const float isc = 1.f / sc;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        bv[s].x = rr[s][0] * isc * scl[s];
                        bv[s].y = rr[s][1] * isc * scl[s];
                    }
                    warp_chol_solve<V, T, NS>(Lm, D, bv, lane);
                    dmax = 0.f;
                    smax = 0.f;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        const float dx = bv[s].x * scl[s] * sc, dy = bv[s].y * scl[s] * sc;
                        float t, e;
                        two_sum(sh[s].x, dx, t, e); sh[s].x = t; sl[s].x += e;
                        two_sum(sh[s].y, dy, t, e); sh[s].y = t; sl[s].y += e;
                        dmax = fmaxf(dmax, fmaxf(fabsf(dx), fabsf(dy)));
                        smax = fmaxf(smax, fmaxf(fabsf(sh[s].x), fabsf(sh[s].y)));
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
                        smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
                    }
                    if (lane == 0) atomicAdd(nsteps, 1ull);
                    // after a step with relative correction rho the remaining error is
                    // about rho^2: stop once that is below 1e-10
                    if (dmax <= 1e-5f * smax) break;
                }
#pragma unroll
                for (int s = 0; s < NS; ++s)
                    sv[s] = make_double2((double)sh[s].x + (double)sl[s].x, (double)sh[s].y + (double)sl[s].y);
                conv = dmax <= 1e-4 * smax;
            }
            ok = conv;
            if (!conv) {
                // solved afterwards in FP64 by k_mid_fallback (slice and its entries untouched here)
                if (lane == 0) fblist[atomicAdd(nfb, 1ull)] = k;
                continue;
            }
        } else {
            ok = warp_chol<V, T, NS>(Lm, D, (T)tol, lane);
            if (ok) {
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int p = lane + 32 * s;
                    sv[s] = p < D ? to_d2(K[NPK + p]) : make_double2(0.0, 0.0);
                }
                warp_chol_solve<V, T, NS>(Lm, D, sv, lane);
            }
        }
        if (!ok && lane == 0) atomicAdd(nsing, 1ull);
        __syncwarp();
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int p = lane + 32 * s;
            if (p < D) {
                if (ok) {
                    Zd[(size_t)k * D + p] = sv[s];
                    const V st = from_d2<V>(sv[s]);
                    Zt[(size_t)k * D + p] = st;
                    zt_s[p] = st;
                } else {
                    zt_s[p] = Zt[(size_t)k * D + p];
                }
            }
        }
        __syncwarp();
        // left environment update into the next order
        slice_h_update<T, R>(H, zt_s, nxt, Hn, seg[k], seg[k + 1], lane);
    }
    if (pending) {
        // a copy that was given up on may still land: wait for it (bounded)
        // before the warp's shared memory is released
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            uint32_t ok;
            asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                         "selp.u32 %0, 1, 0, p;\n}\n"
                         : "=r"(ok) : "r"(bar), "r"(pending_phase) : "memory");
            if (ok) break;
        }
    }
}

// FP64 fallback of the precision form: one warp per slice listed by
// k_mid_solve (complex64 factorization broke down or refinement did not
// contract): FP64 Cholesky of K + lambda I in the slice's FP64 record, solve,
// slice write (or keep the old slice and count it singular), left update.
template <typename T, int R>
__global__ void __launch_bounds__(32 * SolveCfg<T, R>::WPB)
k_mid_fallback(const typename cvec<T>::type* __restrict__ rec, const typename cvec<T>::type* __restrict__ H,
               const int32_t* __restrict__ seg, const int32_t* __restrict__ nxt,
               typename cvec<T>::type* __restrict__ Hn, double2* __restrict__ Zd,
               typename cvec<T>::type* __restrict__ Zt, double2* __restrict__ fb, double lambda_in, double ridge,
               unsigned long long* __restrict__ nsing, const unsigned long long* __restrict__ nfb,
               const int32_t* __restrict__ fblist, unsigned long long* __restrict__ nfb_sweep)
{
    typedef typename cvec<T>::type V;
    typedef SolveCfg<T, R> C;
    constexpr int D = C::D, NPK = C::NPK, NS = C::NS;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    V* zt_s = (V*)(smem + (size_t)wib * C::WBYTES);
    const long long count = (long long)*nfb;
    // the level's fallbacks join the sweep's count (one thread; nothing else
    // writes it while this kernel runs)
    if (blockIdx.x == 0 && threadIdx.x == 0) *nfb_sweep += (unsigned long long)count;
    for (long long idx = (long long)blockIdx.x * C::WPB + wib; idx < count; idx += (long long)gridDim.x * C::WPB) {
        const int k = fblist[idx];
        const V* K = rec + (size_t)k * (NPK + D);
        double tr = 0.0;
        for (int p = lane; p < D; p += 32) tr += (double)K[tri(p, p)].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        const double lambda = fmax(lambda_in, ridge * tr / D);
        const double tol = lambda > 0.0 ? 0.0 : 1e-14 * (tr + D * lambda);
        double2* Kd = fb + (size_t)k * NPK;
        __syncwarp();
        for (int q = lane; q < NPK; q += 32) Kd[q] = to_d2(K[q]);
        __syncwarp();
        for (int p = lane; p < D; p += 32) Kd[tri(p, p)].x += lambda;
        double2 sv[NS];
        const bool ok = warp_chol<double2, double, NS>(Kd, D, tol, lane);
        if (ok) {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int p = lane + 32 * s;
                sv[s] = p < D ? to_d2(K[NPK + p]) : make_double2(0.0, 0.0);
            }
            warp_chol_solve<double2, double, NS>(Kd, D, sv, lane);
        } else if (lane == 0) {
            atomicAdd(nsing, 1ull);
        }
        __syncwarp();
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int p = lane + 32 * s;
            if (p < D) {
                if (ok) {
                    Zd[(size_t)k * D + p] = sv[s];
                    const V st = from_d2<V>(sv[s]);
                    Zt[(size_t)k * D + p] = st;
                    zt_s[p] = st;
                } else {
                    zt_s[p] = Zt[(size_t)k * D + p];
                }
            }
        }
        __syncwarp();
        slice_h_update<T, R>(H, zt_s, nxt, Hn, seg[k], seg[k + 1], lane);
    }
}

// ------------------------------------------------------------------------
// Entry evaluation x = z1(i)^T Z^2(k_2) ... Z^{L+1}(k_{L+1}) zL(j)
// (Eq. (BF_tensor_rep)) for arbitrary pairs; optional residual statistics.
template <typename T, int R>
__device__ __forceinline__ typename cvec<T>::type
eval_one(int i, int j, const typename cvec<T>::type* __restrict__ z1,
         const typename cvec<T>::type* __restrict__ Z, const typename cvec<T>::type* __restrict__ zL,
         int L, int b, int64_t S)
{
    typedef typename cvec<T>::type V;
    V h[R];
#pragma unroll
    for (int a = 0; a < R; ++a) h[a] = z1[(size_t)i * R + a];
    const int pi = i / b, pj = j / b;
    for (int m = 1; m <= L; ++m) {
        const V* Zk = Z + ((size_t)(m - 1) * S + slice_of(pi, pj, m, L)) * R * R;
        V nh[R];
#pragma unroll
        for (int c = 0; c < R; ++c) {
            V acc = czero<V>();
#pragma unroll
            for (int a = 0; a < R; ++a) cmac(acc, h[a], Zk[a * R + c]);
            nh[c] = acc;
        }
#pragma unroll
        for (int c = 0; c < R; ++c) h[c] = nh[c];
    }
    V x = czero<V>();
#pragma unroll
    for (int c = 0; c < R; ++c) cmac(x, h[c], zL[(size_t)j * R + c]);
    return x;
}

template <typename T, int R>
__global__ void __launch_bounds__(256)
k_eval(const int32_t* __restrict__ ii, const int32_t* __restrict__ jj, int64_t M,
       const typename cvec<T>::type* __restrict__ z1, const typename cvec<T>::type* __restrict__ Z,
       const typename cvec<T>::type* __restrict__ zL, int L, int b, int64_t S,
       double2* __restrict__ out, const double2* __restrict__ tref, double* __restrict__ part)
{
    // A group of GS >= R lanes evaluates one entry: lane c keeps h_c and
    // forms column c of h^T Z^{m}(k), so the group reads each slice row as
    // one contiguous segment; h is passed around the group by shuffles.  The
    // sums run over a in the same order as in eval_one.
    typedef typename cvec<T>::type V;
    constexpr int GS = R <= 2 ? 2 : R <= 4 ? 4 : R <= 8 ? 8 : R <= 16 ? 16 : 32;
    static_assert(R <= 32, "rank above 32");
    constexpr int GPW = 32 / GS;
    const int lane = threadIdx.x & 31, c = lane % GS, g = lane / GS;
    const bool col = c < R;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // a group leader sums about a dozen entries in the compute type; the
    // reductions across lanes and warps run in FP64
    T numl = T(0), denl = T(0);
    for (int64_t base = warp0 * GPW; base < M; base += nwarps * GPW) {   // warp-uniform
        const int64_t e = base + g;
        const bool valid = e < M;
        const int i = valid ? ii[e] : 0, j = valid ? jj[e] : 0;   // entry 0's indices stand in for the tail
        V h = col ? z1[(size_t)i * R + c] : czero<V>();
        const int pi = i / b, pj = j / b;
        // the slice of every level depends only on (i, j): level m + 1's
        // column is fetched while level m is formed, so the L2 latency of the
        // gathers leaves the chain of dependent levels
        auto fetch = [&](int m, V* zc) {
            const V* Zk = Z + ((size_t)(m - 1) * S + slice_of(pi, pj, m, L)) * R * R;
#pragma unroll
            for (int a = 0; a < R; ++a) zc[a] = col ? Zk[a * R + c] : czero<V>();
        };
        V zcur[R], znext[R];
        if (L >= 1) fetch(1, zcur);
        for (int m = 1; m <= L; ++m) {
            if (m < L) fetch(m + 1, znext);
            V acc = czero<V>();
#pragma unroll
            for (int a = 0; a < R; ++a) {
                V ha;
                ha.x = __shfl_sync(0xffffffffu, h.x, a, GS);
                ha.y = __shfl_sync(0xffffffffu, h.y, a, GS);
                if (col) cmac(acc, ha, zcur[a]);
            }
            h = acc;
#pragma unroll
            for (int a = 0; a < R; ++a) zcur[a] = znext[a];
        }
        V x = czero<V>();
#pragma unroll
        for (int a = 0; a < R; ++a) {
            V ha;
            ha.x = __shfl_sync(0xffffffffu, h.x, a, GS);
            ha.y = __shfl_sync(0xffffffffu, h.y, a, GS);
            cmac(x, ha, zL[(size_t)j * R + a]);
        }
        if (valid && c == 0) {
            if (out) out[e] = to_d2(x);
            if (tref) {
                const double2 t = tref[e];
                const T tx = (T)t.x, ty = (T)t.y;
                const T dx = tx - x.x, dy = ty - x.y;
                numl += dx * dx + dy * dy;
                denl += tx * tx + ty * ty;
            }
        }
    }
    double num = (double)numl, den = (double)denl;
    if (part) {
        __shared__ double sn[8], sd[8];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            num += __shfl_xor_sync(0xffffffffu, num, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        if (lane == 0) { sn[w] = num; sd[w] = den; }
        __syncthreads();
        if (threadIdx.x == 0) {
            double a = 0.0, c = 0.0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { a += sn[q]; c += sd[q]; }
            part[2 * blockIdx.x] = a;
            part[2 * blockIdx.x + 1] = c;
        }
    }
}

// ------------------------------------------------------------------------
// Gradient (Eqs. (grad_butterfly_1), (grad_butterfly_l), (grad_butterfly_last)
// with z = x - t): the residual r_e is formed at the row level from the full
// right environment (x = z1(i)^T w_0) and carried with h along the orders.

// Sums of the row and column gradients: lane partials and the warp reduction
// in the compute type (a lane sums about two entries of a fiber, so float
// partials keep complex64 accuracy), FP64 in the FP64 path.
template <typename T> struct GradAcc {
    T x, y;
    __device__ __forceinline__ void zero() { x = T(0); y = T(0); }
    // += r conj(w)
    template <typename V> __device__ __forceinline__ void add_r_conj(V r, V w)
    {
        x += r.x * w.x + r.y * w.y;
        y += r.y * w.x - r.x * w.y;
    }
    __device__ __forceinline__ void warp_sum()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
        }
    }
    __device__ __forceinline__ double2 d2() const { return make_double2((double)x, (double)y); }
};

// Loads row p of an R-column complex array (16-byte moves in complex64 at
// even rank).
template <typename V, int R>
__device__ __forceinline__ void load_row_v(const V* __restrict__ A, size_t p, V (&v)[R])
{
    if constexpr (sizeof(V) == 8 && R % 2 == 0) {
        const float4* s4 = reinterpret_cast<const float4*>(A + p * R);
#pragma unroll
        for (int c = 0; c < R / 2; ++c) {
            const float4 x = s4[c];
            v[2 * c].x = x.x; v[2 * c].y = x.y;
            v[2 * c + 1].x = x.z; v[2 * c + 1].y = x.w;
        }
    } else {
#pragma unroll
        for (int c = 0; c < R; ++c) v[c] = A[p * R + c];
    }
}

// Rows: r = z1(i)^T w_0 - t, G1(i) = sum r conj(w_0); writes h_1 = z1(i) and r
// into order 1; per-fiber sum of |r|^2 into part[f].
template <typename T, int R>
__global__ void __launch_bounds__(256)
k_grad_rows(const typename cvec<T>::type* __restrict__ W0, const typename cvec<T>::type* __restrict__ tv,
            const int32_t* __restrict__ seg, int nfib, const typename cvec<T>::type* __restrict__ z1t,
            const int32_t* __restrict__ nxt, typename cvec<T>::type* __restrict__ Hn,
            typename cvec<T>::type* __restrict__ Rn, double2* __restrict__ G1, double* __restrict__ part)
{
    typedef typename cvec<T>::type V;
    constexpr bool VEC = sizeof(V) == 8 && R % 2 == 0;
    const int lane = threadIdx.x & 31;
    const int f = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (f >= nfib) return;
    const int s0 = seg[f], s1 = seg[f + 1];
    V z[R];
#pragma unroll
    for (int c = 0; c < R; ++c) z[c] = z1t[(size_t)f * R + c];
    GradAcc<T> g[R];
#pragma unroll
    for (int c = 0; c < R; ++c) g[c].zero();
    double fit = 0.0;
    for (int p = s0 + lane; p < s1; p += 32) {
        V w[R];
        load_row_v<V, R>(W0, (size_t)p, w);
        V x = czero<V>();
#pragma unroll
        for (int c = 0; c < R; ++c) cmac(x, z[c], w[c]);
        const V t = tv[p];
        V rr;
        rr.x = x.x - t.x;
        rr.y = x.y - t.y;
        fit += (double)rr.x * (double)rr.x + (double)rr.y * (double)rr.y;
#pragma unroll
        for (int c = 0; c < R; ++c) g[c].add_r_conj(rr, w[c]);
        const size_t o = (size_t)nxt[p];
        if constexpr (VEC) {
#pragma unroll
            for (int c = 0; c < R / 2; ++c)
                reinterpret_cast<float4*>(Hn + o * R)[c] = make_float4(z[2 * c].x, z[2 * c].y, z[2 * c + 1].x,
                                                                       z[2 * c + 1].y);
        } else {
#pragma unroll
            for (int c = 0; c < R; ++c) Hn[o * R + c] = z[c];
        }
        Rn[o] = rr;
    }
#pragma unroll
    for (int c = 0; c < R; ++c) g[c].warp_sum();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fit += __shfl_xor_sync(0xffffffffu, fit, o);
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < R; ++c) G1[(size_t)f * R + c] = g[c].d2();
        part[f] = fit;
    }
}

// Middle level m: G^{m+1}(k) = sum r conj(h_m (x) w_m); h_{m+1} = h_m^T Z(k); r carried.
// One CTA per slice at a time (persistent over slices), chunks of CH entries
// staged in shared memory as contiguous blocks (bulk copies in complex64 at
// even rank).  For D = R^2 <= 64 the 128
// threads split the gradient components (q = t mod 64) and the chunk's
// entries (two interleaved halves, t / 64); the halves are added at the end
// of the slice.  The carried h rows are read back from global memory (the
// chunk just loaded them, so they come from L1) and written as 16-byte
// vectors in complex64 at even rank.
template <typename T, int R>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 4)
k_grad_mid(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Wm,
           const typename cvec<T>::type* __restrict__ Rc, const int32_t* __restrict__ seg,
           const int32_t* __restrict__ nxt, const typename cvec<T>::type* __restrict__ Zt,
           typename cvec<T>::type* __restrict__ Hn, typename cvec<T>::type* __restrict__ Rn,
           double2* __restrict__ Gm, int S, unsigned long long* __restrict__ terr, int skip_copy)
{
    typedef typename cvec<T>::type V;
    constexpr int D = R * R;
    constexpr int CH = 128;
    constexpr int NG = D <= 64 ? 2 : 1;              // entry groups
    constexpr int NQ = NG == 2 ? 1 : (D + 127) / 128;  // components per thread
    constexpr bool VEC = sizeof(V) == 8 && R % 2 == 0;
    __shared__ V z_s[D];
    __shared__ __align__(16) V h_s[CH * R];
    __shared__ __align__(16) V w_s[CH * R];
    __shared__ V r_s[CH];
    __shared__ double2 g_s[NG == 2 ? 64 : 1];
    // complex64 at even rank: a chunk's h and w rows (contiguous, 16-byte
    // multiples) arrive by two bulk copies counted on one mbarrier (the wait
    // is bounded; on expiry *terr is raised, the results are undefined, and
    // the CTA issues no further copies: it loads by plain loads from then on).
    // skip_copy (failure injection of the tests, bfc_inject_fault): the copies
    // are not issued and the waits give up after a few tries.
    __shared__ __align__(8) unsigned long long cbar;
    const int tid = threadIdx.x;
    const int grp = NG == 2 ? tid >> 6 : 0;
    const int q0 = NG == 2 ? (tid & 63) : tid;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&cbar);
    uint32_t phase = 0;
    bool use_bulk = VEC;          // CTA-uniform
    bool pending = false;         // copies issued and then given up on
    uint32_t pending_phase = 0;
    const uint32_t wait_limit = skip_copy ? 64u : (1u << 22);
    if constexpr (VEC) {
        if (tid == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
    }
    for (int k = blockIdx.x; k < S; k += gridDim.x) {
        const int s0 = seg[k], s1 = seg[k + 1];
        __syncthreads();
        for (int q = tid; q < D; q += blockDim.x) z_s[q] = Zt[(size_t)k * D + q];
        double2 g[NQ];
#pragma unroll
        for (int u = 0; u < NQ; ++u) g[u] = make_double2(0.0, 0.0);
        for (int base = s0; base < s1; base += CH) {
            const int cnt = min(CH, s1 - base);
            bool have = false;
            if constexpr (VEC) {
                if (use_bulk) {
                    // every thread's reads of the previous chunk are ordered
                    // before the copy engine overwrites the buffers
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncthreads();
                    if (tid == 0) {
                        const uint32_t bytes = (uint32_t)(cnt * R * sizeof(V));
                        asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
                                     ::"r"(bar), "r"(2 * bytes) : "memory");
                        if (!skip_copy) {
                            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                         ::"r"((uint32_t)__cvta_generic_to_shared(h_s)), "l"(H + (size_t)base * R),
                                         "r"(bytes), "r"(bar) : "memory");
                            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                         ::"r"((uint32_t)__cvta_generic_to_shared(w_s)), "l"(Wm + (size_t)base * R),
                                         "r"(bytes), "r"(bar) : "memory");
                        }
                    }
                    for (int x = tid; x < cnt; x += blockDim.x) r_s[x] = Rc[base + x];
                    bool done = false;
                    for (uint32_t it = 0; it < wait_limit && !done; ++it) {
                        uint32_t ok;
                        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                                     "selp.u32 %0, 1, 0, p;\n}\n"
                                     : "=r"(ok) : "r"(bar), "r"(phase) : "memory");
                        done = ok != 0;
                    }
                    // the phase completes once for every thread: any thread
                    // that saw it complete makes the chunk valid for the CTA
                    done = __syncthreads_or(done) != 0;
                    if (done) {
                        have = true;
                    } else {
                        if (tid == 0) atomicExch(terr, 1ull);
                        use_bulk = false;
                        pending = !skip_copy;
                        pending_phase = phase;
                    }
                    phase ^= 1u;
                }
            }
            if (!have) {
                __syncthreads();
                for (int x = tid; x < cnt * R; x += blockDim.x) {
                    h_s[x] = H[(size_t)base * R + x];
                    w_s[x] = Wm[(size_t)base * R + x];
                }
                for (int x = tid; x < cnt; x += blockDim.x) r_s[x] = Rc[base + x];
            }
            __syncthreads();
            // gradient components owned by threads
#pragma unroll
            for (int u = 0; u < NQ; ++u) {
                const int q = q0 + 128 * u;
                if (q < D) {
                    const int pa = q / R, pc = q - pa * R;
                    V acc = czero<V>();
                    for (int e = grp; e < cnt; e += NG) {
                        const V a = cmul(h_s[e * R + pa], w_s[e * R + pc]);
                        cmacc(acc, a, r_s[e]);   // conj(a) r
                    }
                    g[u].x += (double)acc.x;
                    g[u].y += (double)acc.y;
                }
            }
            // carry h and r into the next order
            for (int e = tid; e < cnt; e += blockDim.x) {
                const size_t o = (size_t)nxt[base + e];
                const size_t src = (size_t)(base + e) * R;
                V hv[R];
                if constexpr (VEC) {
#pragma unroll
                    for (int c = 0; c < R / 2; ++c) {
                        const float4 v4 = reinterpret_cast<const float4*>(H + src)[c];
                        hv[2 * c].x = v4.x; hv[2 * c].y = v4.y;
                        hv[2 * c + 1].x = v4.z; hv[2 * c + 1].y = v4.w;
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < R; ++c) hv[c] = H[src + c];
                }
                // one pair of output columns at a time, stored at once (not
                // unrolled, so the slice's R x R values are not all held in
                // registers across entries)
#pragma unroll 1
                for (int c = 0; c < R; c += 2) {
                    V a0 = czero<V>(), a1 = czero<V>();
#pragma unroll
                    for (int a = 0; a < R; ++a) {
                        cmac(a0, hv[a], z_s[a * R + c]);
                        if (c + 1 < R) cmac(a1, hv[a], z_s[a * R + c + 1]);
                    }
                    if constexpr (VEC) {
                        reinterpret_cast<float4*>(Hn + o * R)[c / 2] = make_float4(a0.x, a0.y, a1.x, a1.y);
                    } else {
                        Hn[o * R + c] = a0;
                        if (c + 1 < R) Hn[o * R + c + 1] = a1;
                    }
                }
                Rn[o] = r_s[e];
            }
        }
        if constexpr (NG == 2) {
            // add the second entry group's sums to the first
            __syncthreads();
            if (grp == 1 && q0 < D) g_s[q0] = g[0];
            __syncthreads();
            if (grp == 0 && q0 < D) {
                const double2 o2 = g_s[q0];
                Gm[(size_t)k * D + q0] = make_double2(g[0].x + o2.x, g[0].y + o2.y);
            }
        } else {
#pragma unroll
            for (int u = 0; u < NQ; ++u) {
                const int q = q0 + 128 * u;
                if (q < D) Gm[(size_t)k * D + q] = g[u];
            }
        }
    }
    if (pending) {
        // copies that were given up on may still land: wait for them
        // (bounded) before the CTA's shared memory is released
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            uint32_t ok;
            asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n"
                         "selp.u32 %0, 1, 0, p;\n}\n"
                         : "=r"(ok) : "r"(bar), "r"(pending_phase) : "memory");
            if (ok) break;
        }
    }
}

// Columns: G^{L+2}(j) = sum r conj(h_{L+1}).
template <typename T, int R>
__global__ void __launch_bounds__(256)
k_grad_cols(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Rc,
            const int32_t* __restrict__ seg, int nfib, double2* __restrict__ GL)
{
    typedef typename cvec<T>::type V;
    const int lane = threadIdx.x & 31;
    const int f = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (f >= nfib) return;
    const int s0 = seg[f], s1 = seg[f + 1];
    GradAcc<T> g[R];
#pragma unroll
    for (int c = 0; c < R; ++c) g[c].zero();
    for (int p = s0 + lane; p < s1; p += 32) {
        const V rr = Rc[p];
        V h[R];
        load_row_v<V, R>(H, (size_t)p, h);
#pragma unroll
        for (int c = 0; c < R; ++c) g[c].add_r_conj(rr, h[c]);
    }
#pragma unroll
    for (int c = 0; c < R; ++c) g[c].warp_sum();
    if (lane == 0) {
#pragma unroll
        for (int c = 0; c < R; ++c) GL[(size_t)f * R + c] = g[c].d2();
    }
}

}  // namespace bfc
