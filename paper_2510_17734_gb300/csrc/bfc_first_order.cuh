// First-order butterfly completion (ADAM, Alg. 3/4; ADF, Alg. 5 with the
// App. A.3 orthogonalization sweeps) and the O(n log n) butterfly
// matrix-vector product (Eq. (butterfly-mat-vec)), templated on the compute
// type T (float: complex64 environments, double: FP64) and the rank R.
//
// The sweeps keep the ALS sweep's data layout: every training entry has a
// position in each level order l = 0..L+1, W[l] holds the right environments
// w_l in order l, the left environment h_l travels from order l-1 to order
// l through nxt, and so does the ADF residual.  Factor updates happen in
// FP64 on the master factors, followed by the compute-type copy.
#pragma once

#include "bfc_fo.h"
#include "bfc_internal.h"
#include "bfc_kernels.cuh"
#include "bfc_path.cuh"
#include "bfc_util.h"

namespace bfc {

// One Alg. 3 update of a complex parameter s (two reals) with gradient g and
// moments (Re, Im pairs) in FP64.
__device__ __forceinline__ double2 adam_step(double2 s, double2 g, double2* __restrict__ Mp,
                                             double2* __restrict__ Vp, const AdamHyper& h)
{
    double2 m = *Mp, v = *Vp;
    m.x = h.beta1 * m.x + (1.0 - h.beta1) * g.x;
    m.y = h.beta1 * m.y + (1.0 - h.beta1) * g.y;
    v.x = h.beta2 * v.x + (1.0 - h.beta2) * (g.x * g.x);
    v.y = h.beta2 * v.y + (1.0 - h.beta2) * (g.y * g.y);
    *Mp = m;
    *Vp = v;
    s.x -= h.alpha * (m.x * h.inv1) / (sqrt(v.x * h.inv2) + h.sigma);
    s.y -= h.alpha * (m.y * h.inv1) / (sqrt(v.y * h.inv2) + h.sigma);
    return s;
}

// The value lane c of a warp holds for a register array indexed by c.
template <typename A, int R> __device__ __forceinline__ A pick(const A (&arr)[R], int c)
{
    A out = arr[0];
#pragma unroll
    for (int q = 1; q < R; ++q)
        if (q == c) out = arr[q];
    return out;
}

// Entries base .. base + cnt of a level into shared memory: the rows of H as
// they are, the rows of W as r conj(w).  128 threads, contiguous loads.
template <typename T, int R>
__device__ __forceinline__ void stage_rows(const typename cvec<T>::type* __restrict__ H,
                                           const typename cvec<T>::type* __restrict__ Wm,
                                           const typename cvec<T>::type* __restrict__ Rc, int base, int cnt,
                                           typename cvec<T>::type* h_s, typename cvec<T>::type* w_s, int tid)
{
    typedef typename cvec<T>::type V;
    if constexpr (sizeof(V) == 8 && R % 2 == 0) {
        const float4* h4 = reinterpret_cast<const float4*>(H + (size_t)base * R);
        const float4* w4 = reinterpret_cast<const float4*>(Wm + (size_t)base * R);
        for (int x = tid; x < cnt * (R / 2); x += 128) {
            const float4 w = w4[x];
            const V r = Rc[base + x / (R / 2)];
            reinterpret_cast<float4*>(h_s)[x] = h4[x];
            reinterpret_cast<float4*>(w_s)[x] =
                make_float4(w.x * r.x + w.y * r.y, w.x * r.y - w.y * r.x, w.z * r.x + w.w * r.y, w.z * r.y - w.w * r.x);
        }
    } else if constexpr (sizeof(V) == 8) {
        // all loads of a thread's R values in flight together
        V h[R], w[R], r[R];
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int x = min(tid + 128 * u, cnt * R - 1);
            h[u] = H[(size_t)base * R + x];
            w[u] = Wm[(size_t)base * R + x];
            r[u] = Rc[base + x / R];
        }
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int x = tid + 128 * u;
            if (x < cnt * R) {
                V rw = czero<V>();
                cmacc(rw, w[u], r[u]);
                h_s[x] = h[u];
                w_s[x] = rw;
            }
        }
    } else {
        for (int x = tid; x < cnt * R; x += 128) {
            V rw = czero<V>();
            cmacc(rw, Wm[(size_t)base * R + x], Rc[base + x / R]);
            h_s[x] = H[(size_t)base * R + x];
            w_s[x] = rw;
        }
    }
}

// ------------------------------------------------------------------ ADAM

// Outer factor of Alg. 4 (rows: S^1 with design w_0; columns: S^{L+2} with
// design h_{L+1}), one warp per fiber: gradient sum (x - t) conj(a) +
// lambda s at the current fiber, the Alg. 3 update, then (rows) h_1 = the new
// fiber and the residual h_1^T w_0 - t into order 1 or (columns) the training
// residual partials with the new fiber.
template <typename T, int R, bool COLS>
__global__ void __launch_bounds__(256)
k_adam_outer(const typename cvec<T>::type* __restrict__ A, const typename cvec<T>::type* __restrict__ tv,
             const int32_t* __restrict__ seg, int nfib, double2* __restrict__ zd,
             typename cvec<T>::type* __restrict__ zt, double2* __restrict__ Mo, double2* __restrict__ Vo,
             AdamHyper hp, double lam, const int32_t* __restrict__ nxt, typename cvec<T>::type* __restrict__ Hn,
             typename cvec<T>::type* __restrict__ Rn, double* __restrict__ part)
{
    typedef typename cvec<T>::type V;
    const int lane = threadIdx.x & 31;
    const int f = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (f >= nfib) return;
    const int s0 = seg[f], s1 = seg[f + 1];
    V s[R];
#pragma unroll
    for (int c = 0; c < R; ++c) s[c] = zt[(size_t)f * R + c];
    GradAcc<T> g[R];
#pragma unroll
    for (int c = 0; c < R; ++c) g[c].zero();
    for (int p = s0 + lane; p < s1; p += 32) {
        V a[R];
        load_row_v<V, R>(A, (size_t)p, a);
        V x = czero<V>();
#pragma unroll
        for (int c = 0; c < R; ++c) cmac(x, s[c], a[c]);
        const V t = tv[p];
        V rr;
        rr.x = x.x - t.x;
        rr.y = x.y - t.y;
#pragma unroll
        for (int c = 0; c < R; ++c) g[c].add_r_conj(rr, a[c]);
    }
#pragma unroll
    for (int c = 0; c < R; ++c) g[c].warp_sum();
    if (lane < R) {
        const GradAcc<T> gc = pick<GradAcc<T>, R>(g, lane);
        const size_t q = (size_t)f * R + lane;
        const double2 sd = zd[q];
        const double2 gd = make_double2((double)gc.x + lam * sd.x, (double)gc.y + lam * sd.y);
        const double2 ns = adam_step(sd, gd, Mo + q, Vo + q, hp);
        zd[q] = ns;
        zt[q] = from_d2<V>(ns);
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < R; ++c) s[c] = zt[(size_t)f * R + c];
    if constexpr (!COLS) {
        for (int p = s0 + lane; p < s1; p += 32) {
            const size_t o = (size_t)nxt[p];
            V a[R];
            load_row_v<V, R>(A, (size_t)p, a);
            V x = czero<V>();
#pragma unroll
            for (int c = 0; c < R; ++c) cmac(x, s[c], a[c]);
            const V t = tv[p];
            x.x -= t.x;
            x.y -= t.y;
            store_row_v<V, R>(Hn, o, s);
            Rn[o] = x;
        }
    } else {
        double fit = 0.0, den = 0.0;
        for (int p = s0 + lane; p < s1; p += 32) {
            V a[R];
            load_row_v<V, R>(A, (size_t)p, a);
            V x = czero<V>();
#pragma unroll
            for (int c = 0; c < R; ++c) cmac(x, s[c], a[c]);
            const V t = tv[p];
            const double dx = (double)x.x - (double)t.x, dy = (double)x.y - (double)t.y;
            fit += dx * dx + dy * dy;
            den += (double)t.x * (double)t.x + (double)t.y * (double)t.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fit += __shfl_xor_sync(0xffffffffu, fit, o);
            den += __shfl_xor_sync(0xffffffffu, den, o);
        }
        if (lane == 0) {
            part[2 * f] = fit;
            part[2 * f + 1] = den;
        }
    }
}

// Middle factor of Alg. 4, one CTA per slice (grid-stride): the gradient sum
// r conj(h (x) w) + lambda Z with the carried residuals (SliceSums, chunks of
// entries staged with w already multiplied by r), the Alg. 3 update of the
// slice, then h_{m+1} = h_m^T Z(new) and the residual h_{m+1}^T w_m - t into
// order m+1 (r products instead of the r^2 of h_m^T Z w_m at the next level).
template <typename T, int R>
__global__ void __launch_bounds__(128)
k_adam_mid(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Wm,
           const typename cvec<T>::type* __restrict__ Rc, const typename cvec<T>::type* __restrict__ tv,
           const int32_t* __restrict__ seg, const int32_t* __restrict__ nxt, double2* __restrict__ Zd,
           typename cvec<T>::type* __restrict__ Zt, double2* __restrict__ Mo, double2* __restrict__ Vo, AdamHyper hp,
           double lam, typename cvec<T>::type* __restrict__ Hn, typename cvec<T>::type* __restrict__ Rn, int S)
{
    typedef typename cvec<T>::type V;
    typedef SliceSums<T, R, true> SS;
    constexpr int D = R * R;
    constexpr int CH = 128;
    constexpr size_t ROWS = (size_t)CH * R * sizeof(V) + 16;
    __shared__ __align__(16) unsigned char buf[2 * ROWS > SS::RED ? 2 * ROWS : SS::RED];
    __shared__ __align__(16) V z_s[D];
    V* h_s = (V*)buf;
    V* w_s = (V*)(buf + ROWS);
    const int tid = threadIdx.x;
    for (int k = blockIdx.x; k < S; k += gridDim.x) {
        const int s0 = seg[k], s1 = seg[k + 1];
        SS ss;
        ss.start(tid);
        for (int base = s0; base < s1; base += CH) {
            const int cnt = min(CH, s1 - base);
            __syncthreads();
            stage_rows<T, R>(H, Wm, Rc, base, cnt, h_s, w_s, tid);
            __syncthreads();
            ss.chunk(h_s, w_s, nullptr, cnt);
            if (ss.full(CH)) ss.reduce(buf, tid);
        }
        ss.finish(buf, tid, [&](int q, double2 g) {
            const size_t o = (size_t)k * D + q;
            const double2 sd = Zd[o];
            const double2 gd = make_double2(g.x + lam * sd.x, g.y + lam * sd.y);
            const double2 ns = adam_step(sd, gd, Mo + o, Vo + o, hp);
            Zd[o] = ns;
            const V st = from_d2<V>(ns);
            Zt[o] = st;
            z_s[q] = st;
        });
        __syncthreads();
        for (int p = s0 + tid; p < s1; p += blockDim.x) {
            V h[R], hn[R];
            load_row_v<V, R>(H, (size_t)p, h);
            const size_t o = (size_t)nxt[p];
            row_times_slice<V, R>(h, z_s, hn);
            store_row_v<V, R>(Hn, o, hn);
            if (Rn) {
                load_row_v<V, R>(Wm, (size_t)p, h);
                V x = czero<V>();
#pragma unroll
                for (int c = 0; c < R; ++c) cmac(x, hn[c], h[c]);
                const V t = tv[p];
                x.x -= t.x;
                x.y -= t.y;
                Rn[o] = x;
            }
        }
        __syncthreads();   // z_s is read to the end before the next slice's update
    }
}

// ------------------------------------------------------------------- ADF

// Outer factor of Alg. 5, one warp per fiber: the residual G (rows: t - x
// from the current fiber; columns: carried in order L+1), the direction
// N = sum G conj(a) - lambda s, the exact step
// alpha = ||N||^2 / (sum |a . N|^2 + lambda ||N||^2), s += alpha N, and the
// new residual G - alpha a . N: into order 1 (rows) or as training residual
// partials (columns).  Bound by the FP64 pipe (the direction, its products and
// their conversions), so the direction is formed with a lane per component and
// the residual and product of a lane's first KEEP entries (fibers of up to 64)
// stay in registers for the last pass: n = 16384, r = 8, 50 entries a fiber
// 0.49 -> 0.33 ms (rows), 0.51 -> 0.36 ms (columns) per launch.
template <typename T, int R, bool COLS>
__global__ void __launch_bounds__(256)
k_adf_outer(const typename cvec<T>::type* __restrict__ A, const typename cvec<T>::type* __restrict__ tv,
            const typename cvec<T>::type* __restrict__ Gin, const int32_t* __restrict__ seg, int nfib,
            double2* __restrict__ zd, typename cvec<T>::type* __restrict__ zt, double lam,
            const int32_t* __restrict__ nxt, typename cvec<T>::type* __restrict__ Gn, double* __restrict__ part)
{
    typedef typename cvec<T>::type V;
    const int lane = threadIdx.x & 31;
    const int f = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (f >= nfib) return;
    const int s0 = seg[f], s1 = seg[f + 1];
    constexpr int KEEP = 2;
    V s[R];
#pragma unroll
    for (int c = 0; c < R; ++c) s[c] = zt[(size_t)f * R + c];
    auto residual = [&](int p, const V (&a)[R]) {
        if constexpr (COLS) {
            return Gin[p];
        } else {
            V x = czero<V>();
#pragma unroll
            for (int c = 0; c < R; ++c) cmac(x, s[c], a[c]);
            const V t = tv[p];
            V g;
            g.x = t.x - x.x;
            g.y = t.y - x.y;
            return g;
        }
    };
    // body(p, k): the lane's k-th entry, k < KEEP with k known at compile time
    // (values kept in registers between the passes), then k = KEEP
    auto entries = [&](auto body) {
#pragma unroll
        for (int k = 0; k < KEEP; ++k)
            if (s0 + lane + 32 * k < s1) body(s0 + lane + 32 * k, k);
        for (int p = s0 + lane + 32 * KEEP; p < s1; p += 32) body(p, KEEP);
    };
    V gk[KEEP + 1];      // [KEEP]: scratch
    double2 zk[KEEP + 1];
    GradAcc<T> nacc[R];
#pragma unroll
    for (int c = 0; c < R; ++c) nacc[c].zero();
    entries([&](int p, int k) {
        V a[R];
        load_row_v<V, R>(A, (size_t)p, a);
        gk[k] = residual(p, a);
#pragma unroll
        for (int c = 0; c < R; ++c) nacc[c].add_r_conj(gk[k], a[c]);
    });
    // lane c: component c of the direction
    double2 sl = make_double2(0.0, 0.0), nl = sl;
    if (lane < R) sl = zd[(size_t)f * R + lane];
#pragma unroll
    for (int c = 0; c < R; ++c) {
        nacc[c].warp_sum();
        if (lane == c) nl = nacc[c].d2();
    }
    nl.x -= lam * sl.x;
    nl.y -= lam * sl.y;
    double nn = nl.x * nl.x + nl.y * nl.y;
    double2 N[R];
#pragma unroll
    for (int c = 0; c < R; ++c)
        N[c] = make_double2(__shfl_sync(0xffffffffu, nl.x, c), __shfl_sync(0xffffffffu, nl.y, c));
    auto product = [&](int p) {   // a . N
        V a[R];
        load_row_v<V, R>(A, (size_t)p, a);
        double zx = 0.0, zy = 0.0;
#pragma unroll
        for (int c = 0; c < R; ++c) {
            zx += (double)a[c].x * N[c].x - (double)a[c].y * N[c].y;
            zy += (double)a[c].x * N[c].y + (double)a[c].y * N[c].x;
        }
        return make_double2(zx, zy);
    };
    double zz = 0.0;
    entries([&](int p, int k) {
        zk[k] = product(p);
        zz += zk[k].x * zk[k].x + zk[k].y * zk[k].y;
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        zz += __shfl_xor_sync(0xffffffffu, zz, o);
        nn += __shfl_xor_sync(0xffffffffu, nn, o);
    }
    const double den = zz + lam * nn;
    const double alpha = den > 0.0 ? nn / den : 0.0;
    if (lane < R) {
        const double2 ns = make_double2(sl.x + alpha * nl.x, sl.y + alpha * nl.y);
        zd[(size_t)f * R + lane] = ns;
        zt[(size_t)f * R + lane] = from_d2<V>(ns);
    }
    double fit = 0.0, dent = 0.0;
    entries([&](int p, int k) {
        if (k == KEEP) {
            V a[R];
            load_row_v<V, R>(A, (size_t)p, a);
            gk[k] = residual(p, a);
            zk[k] = product(p);
        }
        const double gx = (double)gk[k].x - alpha * zk[k].x, gy = (double)gk[k].y - alpha * zk[k].y;
        if constexpr (COLS) {
            const V t = tv[p];
            fit += gx * gx + gy * gy;
            dent += (double)t.x * (double)t.x + (double)t.y * (double)t.y;
        } else {
            Gn[nxt[p]] = from_d2<V>(make_double2(gx, gy));
        }
    });
    if constexpr (COLS) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fit += __shfl_xor_sync(0xffffffffu, fit, o);
            dent += __shfl_xor_sync(0xffffffffu, dent, o);
        }
        if (lane == 0) {
            part[2 * f] = fit;
            part[2 * f + 1] = dent;
        }
    }
}

// Middle factor of Alg. 5, one CTA per slice (grid-stride): the direction
// N = sum G conj(h (x) w) - lambda Z (SliceSums), the exact step
// alpha = ||N||^2 / (sum |h^T N w|^2 + lambda ||N||^2), Z += alpha N,
// and the new residual G - alpha h^T N w into order m+1.  The products
// h^T N w of up to ZC entries of a slice are kept between the two uses.
template <typename T, int R>
__global__ void __launch_bounds__(128)
k_adf_mid(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Wm,
          const typename cvec<T>::type* __restrict__ Gin, const int32_t* __restrict__ seg,
          const int32_t* __restrict__ nxt, double2* __restrict__ Zd, typename cvec<T>::type* __restrict__ Zt,
          double lam, typename cvec<T>::type* __restrict__ Gn, int S)
{
    typedef typename cvec<T>::type V;
    typedef SliceSums<T, R, true> SS;
    constexpr int D = R * R;
    constexpr int CH = 128;
    constexpr size_t ROWS = (size_t)CH * R * sizeof(V) + 16;
    constexpr size_t BUF = 2 * ROWS > SS::RED ? 2 * ROWS : SS::RED;
    constexpr int ZC = (int)(BUF / sizeof(V));   // the chunk buffer is free by then
    __shared__ __align__(16) unsigned char buf[BUF];
    __shared__ double2 n_s[D];
    __shared__ V nt_s[D];   // the direction in the compute type, for the per-entry products
    __shared__ double red[4];
    __shared__ double alpha_s;
    V* h_s = (V*)buf;
    V* w_s = (V*)(buf + ROWS);
    V* zc = (V*)buf;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    auto block_sum = [&](double v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if (lane == 0) red[wid] = v;
        __syncthreads();
        return red[0] + red[1] + red[2] + red[3];
    };
    // z_e = h^T N w in the compute type (the entry's own precision)
    auto zval = [&](int p) {
        V h[R], w[R];
        load_row_v<V, R>(H, (size_t)p, h);
        load_row_v<V, R>(Wm, (size_t)p, w);
        V z = czero<V>();
#pragma unroll
        for (int a = 0; a < R; ++a) {
            V nw = czero<V>();   // (N w)_a
#pragma unroll
            for (int c = 0; c < R; ++c) cmac(nw, nt_s[a * R + c], w[c]);
            cmac(z, h[a], nw);
        }
        return z;
    };
    for (int k = blockIdx.x; k < S; k += gridDim.x) {
        const int s0 = seg[k], s1 = seg[k + 1];
        SS ss;
        ss.start(tid);
        for (int base = s0; base < s1; base += CH) {
            const int cnt = min(CH, s1 - base);
            __syncthreads();
            stage_rows<T, R>(H, Wm, Gin, base, cnt, h_s, w_s, tid);
            __syncthreads();
            ss.chunk(h_s, w_s, nullptr, cnt);
            if (ss.full(CH)) ss.reduce(buf, tid);
        }
        double nn = 0.0;
        ss.finish(buf, tid, [&](int q, double2 g) {
            const double2 sd = Zd[(size_t)k * D + q];
            const double2 nv = make_double2(g.x - lam * sd.x, g.y - lam * sd.y);
            n_s[q] = nv;
            nt_s[q] = from_d2<V>(nv);
            nn += nv.x * nv.x + nv.y * nv.y;
        });
        nn = block_sum(nn);   // its first barrier also publishes n_s and frees buf
        double zz = 0.0;
        for (int p = s0 + tid; p < s1; p += blockDim.x) {
            asm volatile("" ::: "memory");   // the direction stays in shared memory, not hoisted into registers
            const V z = zval(p);
            if (p - s0 < ZC) zc[p - s0] = z;
            const double2 zd = to_d2(z);
            zz += zd.x * zd.x + zd.y * zd.y;
        }
        zz = block_sum(zz);
        if (tid == 0) {
            const double den = zz + lam * nn;
            alpha_s = den > 0.0 ? nn / den : 0.0;
        }
        __syncthreads();
        const double alpha = alpha_s;
        for (int q = tid; q < D; q += blockDim.x) {
            const size_t o = (size_t)k * D + q;
            const double2 sd = Zd[o], nv = n_s[q];
            const double2 ns = make_double2(sd.x + alpha * nv.x, sd.y + alpha * nv.y);
            Zd[o] = ns;
            Zt[o] = from_d2<V>(ns);
        }
        for (int p = s0 + tid; p < s1; p += blockDim.x) {
            const double2 z = to_d2(p - s0 < ZC ? zc[p - s0] : zval(p));
            const V g = Gin[p];
            Gn[nxt[p]] = from_d2<V>(make_double2((double)g.x - alpha * z.x, (double)g.y - alpha * z.y));
        }
        __syncthreads();   // n_s and zc are read to the end before the next slice
    }
}

// h_{m+1}(e) = h_m(e)^T Z[m][k] for the entries of every slice k, into order
// m+1 (one CTA per slice, grid-stride).
template <typename T, int R>
__global__ void __launch_bounds__(128)
k_h_next(const typename cvec<T>::type* __restrict__ H, const int32_t* __restrict__ seg,
         const int32_t* __restrict__ nxt, const typename cvec<T>::type* __restrict__ Zt,
         typename cvec<T>::type* __restrict__ Hn, int S)
{
    typedef typename cvec<T>::type V;
    __shared__ __align__(16) V z_s[R * R];
    for (int k = blockIdx.x; k < S; k += gridDim.x) {
        const int s0 = seg[k], s1 = seg[k + 1];
        if (s0 == s1) continue;
        __syncthreads();
        for (int q = threadIdx.x; q < R * R; q += blockDim.x) z_s[q] = Zt[(size_t)k * R * R + q];
        __syncthreads();
        for (int p = s0 + threadIdx.x; p < s1; p += blockDim.x) {
            V h[R], hn[R];
            load_row_v<V, R>(H, (size_t)p, h);
            row_times_slice<V, R>(h, z_s, hn);
            store_row_v<V, R>(Hn, (size_t)nxt[p], hn);
        }
    }
}

// h_1(e) = z1(i) for the entries of every row fiber i, into order 1.
template <typename T, int R>
__global__ void __launch_bounds__(256)
k_h1_rows(const int32_t* __restrict__ seg, int nfib, const typename cvec<T>::type* __restrict__ zt,
          const int32_t* __restrict__ nxt, typename cvec<T>::type* __restrict__ Hn)
{
    typedef typename cvec<T>::type V;
    const int lane = threadIdx.x & 31;
    const int f = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (f >= nfib) return;
    V s[R];
#pragma unroll
    for (int c = 0; c < R; ++c) s[c] = zt[(size_t)f * R + c];
    for (int p = seg[f] + lane; p < seg[f + 1]; p += 32) store_row_v<V, R>(Hn, (size_t)nxt[p], s);
}

// ---------------------------------------------------------------- matvec

// Y[p][q] = sum over the leaf of zL(j)^T v_q(j), p = j / b (the contraction of
// S^{L+2} with the vectors over j_L); one thread per (p, q).
template <typename T, int R>
__global__ void k_mv_leaf(const typename cvec<T>::type* __restrict__ zL, const double2* __restrict__ Vin, int b,
                          int nvec, int npre, typename cvec<T>::type* __restrict__ Y)
{
    typedef typename cvec<T>::type V;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)npre * nvec) return;
    const int p = (int)(idx / nvec), q = (int)(idx - (int64_t)p * nvec);
    V acc[R];
#pragma unroll
    for (int c = 0; c < R; ++c) acc[c] = czero<V>();
    for (int l = 0; l < b; ++l) {
        const int64_t j = (int64_t)p * b + l;
        const V v = from_d2<V>(Vin[j * nvec + q]);
#pragma unroll
        for (int c = 0; c < R; ++c) cmac(acc[c], zL[j * R + c], v);
    }
#pragma unroll
    for (int c = 0; c < R; ++c) Y[idx * R + c] = acc[c];
}

// One pass over several levels.  Y_m[k] = Z[m][k] T_m[g(k)], where T_L[g] =
// Y_{L+1}[g] with g = the column bits of k (the leaf sums), and for m < L
// T_m[g] = Y_{m+1}[2g] + Y_{m+1}[2g + 1] (the sum over j_m) with g = k without
// its bit m (i_{L-m}).  With k = (row bits I, column bits J) a level turns the
// last column bit into a new last row bit, so s levels close on 2^s elements
// that share I's first bits and J's first bits, as a stage of an FFT does.  A
// block takes 16 elements (s = 4 bits x, level t of the pass works on bit t of
// x: the pair differing there is summed and replaced by the two products; fewer
// bits: several such groups) for VT vectors through up to four levels: the intermediates pass through memory
// four times at L = 12 instead of thirteen.  Thread = (pair, TV vectors 16
// apart): T in registers, Z read from shared memory for TV products each, the
// next level's 16 slices copied in meanwhile.  The first pass starts from the
// leaf sums of 8 column prefixes (level L has no sum), the last ends with the
// rows u(i) = z1(i)^T T_0[p_i].  Intermediates are laid out [k][c][q].
// n = 65536, r = 8, 64 vectors, complex64: 0.65 ms of kernels before (a thread
// per slice and vector, a pass per level), now 0.20 (with one group per block
// 0.22; 0.28 with 64 vectors per block, 2 blocks per SM, 0.24 with 16).
template <typename T, int R> struct MvCfg {
    static constexpr size_t VS = sizeof(typename cvec<T>::type);
    static constexpr int E = 16;                                   // elements of a block
    static constexpr int CAP = (int)(32768 / (E * R * VS));        // vectors in 32 KB
    static constexpr int VT = CAP >= 64 ? 64 : CAP >= 32 ? 32 : 16;
    static constexpr int TV = VT / 16;
    static constexpr size_t YB = (size_t)E * R * VT * VS;
    static constexpr size_t ZB = ((size_t)E * R * R * VS + 15) / 16 * 16;
    static constexpr size_t SMEM = YB + 2 * ZB;
    static_assert(SMEM <= 227 * 1024, "shared memory of a block");
};

struct MvPass {
    int L, M;       // levels of the network; first (highest) level of the pass
    int s, lv;      // element bits; levels (lv = s, or s - 1 in the last pass)
    int first, last;
    int b, nvec;
};

template <typename T, int R>
__global__ void __launch_bounds__(128)
k_mv_pass(MvPass ps, const typename cvec<T>::type* __restrict__ Z, const typename cvec<T>::type* __restrict__ zL,
          const typename cvec<T>::type* __restrict__ z1, const double2* __restrict__ Vin,
          const typename cvec<T>::type* __restrict__ Yin, typename cvec<T>::type* __restrict__ Yout,
          double2* __restrict__ U)
{
    typedef typename cvec<T>::type V;
    typedef MvCfg<T, R> C;
    constexpr int VT = C::VT, TV = C::TV, D = R * R;
    extern __shared__ __align__(16) unsigned char smem[];
    V* ys = (V*)smem;                                      // [x][c][q]
    const int s = ps.s, nel = 1 << s, npair = nel >> 1;
    // C::E >> s groups of 2^s elements; this thread's group, pair and lane
    const int tid = threadIdx.x, l = tid & 15;
    const int grp = (tid >> 4) / npair, bf = (tid >> 4) - grp * npair;
    const int nJ = ps.M + 1 - s;                           // column bits shared by a group
    const unsigned ngrp = 1u << (ps.L + 1 - s), grp0 = blockIdx.x * (unsigned)(C::E >> s);
    const bool active = grp0 + grp < ngrp;
    const int I0 = (int)((grp0 + grp) >> nJ), J0 = (int)((grp0 + grp) & ((1u << nJ) - 1));
    V* yg = ys + (size_t)grp * nel * R * C::VT;            // the group's elements
    const int q0 = blockIdx.y * VT, nq = min(VT, ps.nvec - q0);
    const int nt = (nq + 15) >> 4;                         // vectors of lane 0
    const size_t S = (size_t)2 << ps.L;
    // row bits I, then the first `cnt` bits of x
    auto row_bits = [&](int I, int x, int cnt) {
        for (int u = 0; u < cnt; ++u) I = I << 1 | ((x >> u) & 1);
        return I;
    };
    // the slices of level t of the pass into buffer t & 1
    auto stage = [&](int t) {
        const int m = ps.M - t;
        V* dst = (V*)(smem + C::YB + (size_t)(t & 1) * C::ZB);
        constexpr bool W16 = (D * C::VS) % 16 == 0;
        constexpr int PIECE = W16 ? 16 : 8, PP = (int)(D * C::VS / PIECE);
        for (int y = tid; y < C::E * PP; y += 128) {
            const int gx = y / PP, w = y - gx * PP, x = gx & (nel - 1);
            const unsigned g = grp0 + (unsigned)(gx >> s);
            if (g >= ngrp) break;
            const size_t k = ((size_t)row_bits((int)(g >> nJ), x, t + 1) << m) |
                             ((size_t)(g & ((1u << nJ) - 1)) << (s - 1 - t)) | (size_t)(x >> (t + 1));
            const unsigned char* src = (const unsigned char*)(Z + ((size_t)(m - 1) * S + k) * D) + (size_t)w * PIECE;
            unsigned char* d = (unsigned char*)(dst + (size_t)gx * D) + (size_t)w * PIECE;
            if constexpr (W16) cp_async16(d, src);
            else cp_async8(d, src);
        }
        cp_async_commit();
    };
    V tv[R][TV];
    // the pair's inputs of level t: their sum (the first level of all: one)
    auto load_pair = [&](int t, int e0, int e1) {
        const bool expand = ps.first && t == 0;
        if (expand) {
            // leaf sums of column prefix J
            const int J = (J0 << (s - 1)) | (e0 >> 1);
#pragma unroll
            for (int c = 0; c < R; ++c)
#pragma unroll
                for (int v = 0; v < TV; ++v) tv[c][v] = czero<V>();
            for (int r = 0; r < ps.b; ++r) {
                const size_t j = (size_t)J * ps.b + r;
                V z[R];
                load_row_v<V, R>(zL, j, z);
#pragma unroll
                for (int v = 0; v < TV; ++v)
                    if (l + 16 * v < nq) {
                        const V x = from_d2<V>(Vin[j * ps.nvec + q0 + l + 16 * v]);
#pragma unroll
                        for (int c = 0; c < R; ++c) cmac(tv[c][v], z[c], x);
                    }
            }
        } else if (t == 0) {
            const size_t k0 = ((size_t)I0 << (ps.M + 1)) | ((size_t)J0 << s);
            const V* a = Yin + (k0 + e0) * R * ps.nvec + q0 + l;
            const V* b = Yin + (k0 + e1) * R * ps.nvec + q0 + l;
#pragma unroll
            for (int c = 0; c < R; ++c)
#pragma unroll
                for (int v = 0; v < TV; ++v) {
                    tv[c][v] = czero<V>();
                    if (l + 16 * v < nq) {
                        const V x = a[(size_t)c * ps.nvec + 16 * v], y = b[(size_t)c * ps.nvec + 16 * v];
                        tv[c][v].x = x.x + y.x;
                        tv[c][v].y = x.y + y.y;
                    }
                }
        } else {
            const V* a = yg + (size_t)e0 * R * VT + l;
            const V* b = yg + (size_t)e1 * R * VT + l;
#pragma unroll
            for (int c = 0; c < R; ++c)
#pragma unroll
                for (int v = 0; v < TV; ++v) {
                    tv[c][v] = czero<V>();
                    if (v < nt) {
                        const V x = a[c * VT + 16 * v], y = b[c * VT + 16 * v];
                        tv[c][v].x = x.x + y.x;
                        tv[c][v].y = x.y + y.y;
                    }
                }
        }
    };
    if (ps.lv > 0) stage(0);
    for (int t = 0; t < ps.lv; ++t) {
        const int e0 = ((bf >> t) << (t + 1)) | (bf & ((1 << t) - 1)), e1 = e0 | 1 << t;
        // level 0 reads global memory: before the wait for its slices
        if (t == 0 && active) load_pair(0, e0, e1);
        cp_async_wait_all();
        __syncthreads();   // the level's slices and the elements of the level before; the other buffer is free
        if (t + 1 < ps.lv) stage(t + 1);
        if (!active) continue;
        if (t > 0) load_pair(t, e0, e1);
        const V* zt = (const V*)(smem + C::YB + (size_t)(t & 1) * C::ZB) + (size_t)grp * nel * D;
        const bool out = t + 1 == s;   // to global memory (not in the last pass)
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            const int x = i ? e1 : e0;
            const V* z = zt + (size_t)x * D;
            const size_t ko = out ? ((size_t)row_bits(I0, x, s) << nJ) | (size_t)J0 : 0;
#pragma unroll 1
            for (int a = 0; a < R; ++a) {
                V acc[TV], zr[R];
#pragma unroll
                for (int v = 0; v < TV; ++v) acc[v] = czero<V>();
                load_row_v<V, R>(z, (size_t)a, zr);
#pragma unroll
                for (int c = 0; c < R; ++c)
#pragma unroll
                    for (int v = 0; v < TV; ++v) cmac(acc[v], zr[c], tv[c][v]);
                if (out) {
#pragma unroll
                    for (int v = 0; v < TV; ++v)
                        if (l + 16 * v < nq) Yout[(ko * R + a) * ps.nvec + q0 + l + 16 * v] = acc[v];
                } else {
#pragma unroll
                    for (int v = 0; v < TV; ++v)
                        if (v < nt) yg[((size_t)x * R + a) * VT + l + 16 * v] = acc[v];
                }
            }
        }
    }
    if (ps.last) {
        // rows of the 2^(s-1) leaf prefixes of the block
        __syncthreads();
        if (!active) return;
        const int t = ps.lv;
        load_pair(t, bf, bf | 1 << t);   // bits 0 .. t - 1 of bf are the new row bits
        const size_t p = (size_t)row_bits(I0, bf, t);
        for (int r = 0; r < ps.b; ++r) {
            const size_t i = p * ps.b + r;
            V z[R];
            load_row_v<V, R>(z1, i, z);
#pragma unroll
            for (int v = 0; v < TV; ++v)
                if (l + 16 * v < nq) {
                    V acc = czero<V>();
#pragma unroll
                    for (int c = 0; c < R; ++c) cmac(acc, z[c], tv[c][v]);
                    U[i * ps.nvec + q0 + l + 16 * v] = to_d2(acc);
                }
        }
    }
}

// Level m of the contraction (m = L .. 1) by itself, one thread per (k, q) (the
// FP64 form for few vectors, see MvRule).  Intermediates are laid out [k][q][c].
template <typename T, int R>
__global__ void k_mv_level(const typename cvec<T>::type* __restrict__ Zm, const typename cvec<T>::type* __restrict__ Yin,
                           typename cvec<T>::type* __restrict__ Yout, int m, int L, int nvec, int S)
{
    typedef typename cvec<T>::type V;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (int64_t)S * nvec) return;
    const int k = (int)(idx / nvec), q = (int)(idx - (int64_t)k * nvec);
    V tv[R];
    if (m == L) {
        const int64_t g = k & ((1 << L) - 1);
#pragma unroll
        for (int c = 0; c < R; ++c) tv[c] = Yin[(g * nvec + q) * R + c];
    } else {
        const int64_t g = ((int64_t)(k >> (m + 1)) << m) | (k & ((1 << m) - 1));
#pragma unroll
        for (int c = 0; c < R; ++c) {
            const V a = Yin[((2 * g) * nvec + q) * R + c], b = Yin[((2 * g + 1) * nvec + q) * R + c];
            tv[c].x = a.x + b.x;
            tv[c].y = a.y + b.y;
        }
    }
    const V* Z = Zm + (size_t)k * R * R;
#pragma unroll
    for (int a = 0; a < R; ++a) {
        V acc = czero<V>();
#pragma unroll
        for (int c = 0; c < R; ++c) cmac(acc, Z[a * R + c], tv[c]);
        Yout[idx * R + a] = acc;
    }
}

// u_q(i) = z1(i)^T T_0[p_i], T_0[p] = Y_1[2p] + Y_1[2p + 1] (the sum over j_0)
// for L >= 1, or the leaf contraction for L = 0; one thread per (i, q).
template <typename T, int R>
__global__ void k_mv_root(const typename cvec<T>::type* __restrict__ z1, const typename cvec<T>::type* __restrict__ Y,
                          int b, int L, int nvec, int64_t n, double2* __restrict__ U)
{
    typedef typename cvec<T>::type V;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * nvec) return;
    const int64_t i = idx / nvec;
    const int q = (int)(idx - i * nvec);
    const int64_t p = i / b;
    V acc = czero<V>();
#pragma unroll
    for (int a = 0; a < R; ++a) {
        V t;
        if (L == 0) {
            t = Y[(int64_t)q * R + a];
        } else {
            const V x = Y[((2 * p) * nvec + q) * R + a], y = Y[((2 * p + 1) * nvec + q) * R + a];
            t.x = x.x + y.x;
            t.y = x.y + y.y;
        }
        cmac(acc, z1[i * R + a], t);
    }
    U[idx] = to_d2(acc);
}

// Whether the mat-vec takes passes over several levels (k_mv_pass; always in
// complex64) or goes level by level.  In FP64 the pipe counts a warp's
// instructions whatever its lanes do, so the 16 vector lanes of a pass have to
// be filled, and only ranks 5 .. 8 then gain.  us of kernels, levels / passes: n =
// 65536, L = 12, r = 8 1 vector 366 / 1110, 16 1109 / 1074, 17 1122 / 1706, 64
// 3600 / 3298; n = 4096, r = 8, 64 vectors 263 / 212, r = 4 121 / 135; n = 65536, r
// = 12, 64 vectors 7404 / 8107.
template <typename T, int R> struct MvRule {
    static constexpr bool ANY = sizeof(T) == 4 || (R >= 5 && R <= 8);
    static bool passes(int nvec) { return ANY && (sizeof(T) == 4 || 8 * nvec >= 7 * ((nvec + 15) / 16 * 16)); }
};

// --------------------------------------------------------------- drivers

template <typename T, int R> struct FirstOrder {
    typedef typename cvec<T>::type V;

    static unsigned grid_slices(int64_t S) { return (unsigned)(S < 152 * 16 ? S : 152 * 16); }

    // u = X(S) V (Eq. (butterfly-mat-vec)) for nvec vectors on the device:
    // Vd, Ud n x nvec complex128; Y0, Y1 scratch of 2^{L+1} nvec R values.
    static bfc_status matvec(Ctx* c, int nvec, const double2* Vd, double2* Ud, V* Y0, V* Y1)
    {
        const int L = c->L;
        const int64_t S = c->S;
        if (L == 0 || !MvRule<T, R>::passes(nvec)) {
            const int64_t npre = (int64_t)1 << L;
            {
                ProfScope ps(c, "mv_leaf");
                k_mv_leaf<T, R><<<nblocks(npre * nvec, 256), 256, 0, c->stream>>>((const V*)c->zLt, Vd, c->b, nvec,
                                                                                  (int)npre, Y0);
            }
            V* yin = Y0;
            V* yout = Y1;
            if constexpr (sizeof(T) == 8)
                for (int m = L; m >= 1; --m) {
                    ProfScope ps(c, "mv_level");
                    k_mv_level<T, R><<<nblocks(S * nvec, 256), 256, 0, c->stream>>>(
                        (const V*)c->Zt + (size_t)(m - 1) * S * R * R, yin, yout, m, L, nvec, (int)S);
                    std::swap(yin, yout);
                }
            {
                ProfScope ps(c, "mv_root");
                k_mv_root<T, R><<<nblocks(c->n * nvec, 256), 256, 0, c->stream>>>((const V*)c->z1t, yin, c->b, L, nvec,
                                                                                  c->n, Ud);
            }
            BFC_LAUNCH_CHECK(c, "matvec");
            return BFC_OK;
        }
        if constexpr (MvRule<T, R>::ANY) {
            typedef MvCfg<T, R> MC;
            BFC_CK(c, cudaFuncSetAttribute(k_mv_pass<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MC::SMEM));
            // the last pass takes up to 3 levels, the first up to 4, the others the
            // rest in even parts of at most 4
            const int nlast = std::min(3, L - 1), nfirst = std::min(4, L - nlast);
            int rest = L - nlast - nfirst, mids = (rest + 3) / 4;
            V* yin = nullptr;
            V* yout = Y0;
            auto pass = [&](int M, int s, int lv, int first, int last) {
                ProfScope ps(c, "mv_pass");
                const MvPass mp{L, M, s, lv, first, last, c->b, nvec};
                const unsigned groups = 1u << (L + 1 - s), per = (unsigned)(MC::E >> s);
                const dim3 grid((groups + per - 1) / per, (unsigned)((nvec + MC::VT - 1) / MC::VT));
                k_mv_pass<T, R><<<grid, 128, MC::SMEM, c->stream>>>(mp, (const V*)c->Zt, (const V*)c->zLt,
                                                                    (const V*)c->z1t, Vd, yin, yout, Ud);
                V* t = yin == nullptr ? Y1 : yin;
                yin = yout;
                yout = t;
            };
            int M = L;
            pass(M, nfirst, nfirst, 1, 0);
            M -= nfirst;
            for (; mids > 0; --mids) {
                const int s = (rest + mids - 1) / mids;
                pass(M, s, s, 0, 0);
                M -= s;
                rest -= s;
            }
            pass(M, nlast + 1, nlast, 0, 1);
        }
        BFC_LAUNCH_CHECK(c, "matvec");
        return BFC_OK;
    }

    // One outer iteration of Alg. 4 (right environments, then S^1, the middle
    // factors and S^{L+2} in order) plus the training residual partials.
    static bfc_status adam_iter(Ctx* c, const AdamHyper& hp, double2* M, double2* Vm)
    {
        const int64_t n = c->n, NR = c->N * R, S = c->S;
        const int L = c->L;
        const double lam = c->P.lambda;
        V* W = (V*)c->W;
        V* Hb[2] = {(V*)c->H[0], (V*)c->H[1]};
        V* Rb[2] = {(V*)c->Rres[0], (V*)c->Rres[1]};
        BFC_TRY((Path<T, R>::right_envs(c)));
        const size_t offZ = (size_t)n * R, offL = offZ + (size_t)L * S * R * R;
        {
            ProfScope ps(c, "adam_rows");
            k_adam_outer<T, R, false><<<nblocks(n, 8), 256, 0, c->stream>>>(
                W, (const V*)c->tval[0], c->seg[0], (int)n, c->z1d, (V*)c->z1t, M, Vm, hp, lam, c->nxt[0], Hb[0],
                Rb[0], nullptr);
        }
        for (int m = 1; m <= L; ++m) {
            ProfScope ps(c, "adam_mid");
            const size_t o = offZ + (size_t)(m - 1) * S * R * R;
            k_adam_mid<T, R><<<grid_slices(S), 128, 0, c->stream>>>(
                Hb[(m - 1) & 1], W + (size_t)m * NR, Rb[(m - 1) & 1], (const V*)c->tval[m], c->seg[m], c->nxt[m],
                c->Zd + (size_t)(m - 1) * S * R * R, (V*)c->Zt + (size_t)(m - 1) * S * R * R, M + o, Vm + o, hp, lam,
                Hb[m & 1], m < L ? Rb[m & 1] : nullptr, (int)S);
        }
        {
            ProfScope ps(c, "adam_cols");
            k_adam_outer<T, R, true><<<nblocks(n, 8), 256, 0, c->stream>>>(
                Hb[L & 1], (const V*)c->tval[L + 1], c->seg[L + 1], (int)n, c->zLd, (V*)c->zLt, M + offL,
                Vm + offL, hp, lam, nullptr, nullptr, nullptr, c->d_red);
        }
        BFC_LAUNCH_CHECK(c, "adam iteration");
        return BFC_OK;
    }

    // Compute-type copy of FP64 factor values [off, off + cnt).
    static void refresh(Ctx* c, size_t off, int64_t cnt)
    {
        if constexpr (sizeof(T) == 4) {
            ProfScope ps(c, "d2f");
            launch_d2f(c->z1d + off, (float2*)c->z1t + off, cnt, c->stream);
        }
    }

    // One iteration of Alg. 5: right-to-left orthogonalization (App. A.3),
    // right environments, then S^1, the middle factors and S^{L+2}, each with
    // the exact-step update and (but S^{L+2}) the QR of its bond groups with
    // R moved into the next factor; the training residual partials last.
    static bfc_status adf_iter(Ctx* c)
    {
        const int64_t n = c->n, NR = c->N * R, S = c->S;
        const int L = c->L;
        const double lam = c->P.lambda;
        const size_t offZ = (size_t)n * R, offL = offZ + (size_t)L * S * R * R, slz = (size_t)S * R * R;
        V* W = (V*)c->W;
        V* Hb[2] = {(V*)c->H[0], (V*)c->H[1]};
        V* Gb[2] = {(V*)c->Rres[0], (V*)c->Rres[1]};
        {
            ProfScope ps(c, "adf_orth", L + 1);
            cudaError_t e = launch_rl_orthogonalize(c->z1d, c->Zd, c->zLd, n, L, c->b, R, c->stream);
            if (e != cudaSuccess) return fail(c, BFC_ECUDA, std::string("orthogonalization: ") + cudaGetErrorString(e));
        }
        refresh(c, 0, c->Pn);
        BFC_TRY((Path<T, R>::right_envs(c)));
        {
            ProfScope ps(c, "adf_rows");
            k_adf_outer<T, R, false><<<nblocks(n, 8), 256, 0, c->stream>>>(
                W, (const V*)c->tval[0], nullptr, c->seg[0], (int)n, c->z1d, (V*)c->z1t, lam, c->nxt[0], Gb[0], nullptr);
        }
        {
            ProfScope ps(c, "adf_qr");
            cudaError_t e = launch_canon_level(c->z1d, c->Zd, c->zLd, n, L, c->b, R, 0, c->stream);
            if (e != cudaSuccess) return fail(c, BFC_ECUDA, std::string("QR: ") + cudaGetErrorString(e));
        }
        refresh(c, 0, (int64_t)n * R);
        refresh(c, L >= 1 ? offZ : offL, L >= 1 ? (int64_t)slz : (int64_t)n * R);
        if (L >= 1) {
            ProfScope ps(c, "adf_h");
            k_h1_rows<T, R><<<nblocks(n, 8), 256, 0, c->stream>>>(c->seg[0], (int)n, (const V*)c->z1t, c->nxt[0], Hb[0]);
        }
        for (int m = 1; m <= L; ++m) {
            V* hin = Hb[(m - 1) & 1];
            V* hout = Hb[m & 1];
            {
                ProfScope ps(c, "adf_mid");
                k_adf_mid<T, R><<<grid_slices(S), 128, 0, c->stream>>>(
                    hin, W + (size_t)m * NR, Gb[(m - 1) & 1], c->seg[m], c->nxt[m], c->Zd + (size_t)(m - 1) * slz,
                    (V*)c->Zt + (size_t)(m - 1) * slz, lam, Gb[m & 1], (int)S);
            }
            {
                ProfScope ps(c, "adf_qr");
                cudaError_t e = launch_canon_level(c->z1d, c->Zd, c->zLd, n, L, c->b, R, m, c->stream);
                if (e != cudaSuccess) return fail(c, BFC_ECUDA, std::string("QR: ") + cudaGetErrorString(e));
            }
            refresh(c, offZ + (size_t)(m - 1) * slz, (int64_t)slz);
            refresh(c, m < L ? offZ + (size_t)m * slz : offL, m < L ? (int64_t)slz : (int64_t)n * R);
            {
                ProfScope ps(c, "adf_h");
                k_h_next<T, R><<<grid_slices(S), 128, 0, c->stream>>>(
                    hin, c->seg[m], c->nxt[m], (const V*)c->Zt + (size_t)(m - 1) * slz, hout, (int)S);
            }
        }
        {
            ProfScope ps(c, "adf_cols");
            const V* hc = L == 0 ? nullptr : Hb[L & 1];
            if (L == 0) {
                // L = 0: the column design is z1(i) itself, in the column order
                k_h1_rows<T, R><<<nblocks(n, 8), 256, 0, c->stream>>>(c->seg[0], (int)n, (const V*)c->z1t,
                                                                      c->nxt[0], Hb[0]);
                hc = Hb[0];
            }
            k_adf_outer<T, R, true><<<nblocks(n, 8), 256, 0, c->stream>>>(
                hc, (const V*)c->tval[L + 1], Gb[L & 1], c->seg[L + 1], (int)n, c->zLd, (V*)c->zLt, lam, nullptr,
                nullptr, c->d_red);
        }
        BFC_LAUNCH_CHECK(c, "adf iteration");
        return BFC_OK;
    }
};

template <typename T, int R> struct FoEntry {
    static bfc_status matvec(Ctx* c, int nvec, const double2* Vd, double2* Ud, void* y0, void* y1)
    {
        return FirstOrder<T, R>::matvec(c, nvec, Vd, Ud, (typename cvec<T>::type*)y0, (typename cvec<T>::type*)y1);
    }
    static constexpr FoOps ops{&matvec, &FirstOrder<T, R>::adam_iter, &FirstOrder<T, R>::adf_iter};
};

}  // namespace bfc
