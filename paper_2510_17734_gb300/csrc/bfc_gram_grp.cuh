// Per-slice normal equations of one middle level, by groups of entries that
// share an environment (CUDA cores, rank R >= 2).
//
// Inside a slice k of S^{m+1}, the left environment h_m of an entry depends
// only on its row i (the column bits it passed, j_0 .. j_{m-2}, are fixed by
// the slice) and the right environment w_m only on its column j.  With the
// design a_e = h_e (x) w_e (a[a R + c] = h_a w_c),
//   K[(a,c),(a',c')] = sum_e conj(h_a w_c) h_a' w_c'
//                    = sum_g X_g[a][a'] Y_g[c][c'],
//   y[(a,c)]         = sum_g xv_g[a] yv_g[c],
// where a group g is the entries of one row (X = conj(h) h^T, xv = conj(h),
// Y = sum_e conj(w_e) w_e^T, yv = sum_e conj(w_e) t_e) or of one column
// (Y = conj(w) w^T, yv = conj(w), X = sum_e conj(h_e) h_e^T,
// xv = sum_e conj(h_e) t_e).  The slice's sums (Alg. 1, middle factors) are
// the same; the rank-one update per entry becomes one per group, which at
// the outer levels (few rows or few columns per slice) is many times fewer.
//
// Two kernels: k_group_sums forms one record [s | M | v] per group (s the
// shared vector, M and v the sums of the other side); k_mid_gram_grp streams
// a slice's records through shared memory and accumulates the Kronecker
// updates.  Layout: the level order keeps each group contiguous; gseg[k] is
// the first group of slice k, gstart[g] the first position of group g.  Work
// per slice as in k_mid_gram: T x T complex tiles of the lower triangle of K
// owned by threads, each inside one (a, a') block (GrpTile).  Precision form: a group's term can be a large part of the
// slice's sum (16 row groups at the first level), so every term is added
// with Kahan compensation, and the group sums are compensated across blocks
// of 16 entries; the error of K then matches the per-entry kernels' (the
// rounding of the stored complex64 record dominates both).  Same output
// record as k_mid_gram.
//
// Measured, all middle levels of a sweep, against the per-entry kernels that
// these levels ran before: n = 4096, L = 8, r = 12, 3.41 M entries, complex64
// 107.2 -> 2.9 ms (against k_mid_gram); n = 4096, L = 8, r = 6, 265 k entries,
// FP64 19.1 -> 2.8 ms (k_mid_gram, bound by the FP64 pipe at 1.25 TFLOP/s);
// n = 3072, L = 8, r = 5, 961 k entries, complex64 1.42 -> 0.66 ms (against
// k_mid_gram_tc).  Issue-bound; two groups per compensated step took 3.6 -> 2.9,
// 0.87 -> 0.66 and (n = 65536, r = 8) 1.70 -> 1.54 ms, the parallel reduction of
// the thread groups 34 -> 5 us a level at n = 256, r = 4 (32 slices).
#pragma once

#include "bfc_kernels.cuh"

namespace bfc {

template <typename V> __device__ __forceinline__ V make_conj(V a)
{
    a.y = -a.y;
    return a;
}

// 16-byte asynchronous global -> shared copy (L2 only) and its group waits.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem_src) : "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait_n()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gmem_src)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem_src) : "memory");
}

// Tile side of the grouped Gram's K tiles and the padded column count RP (a
// multiple of it): a tile then lies inside one (a, a') block of K, so it needs
// one value of the shared side and T x T of the other.  T = 4 where it divides
// R, else 3, 5 or 2; the primes 7 and 11 use T = 4 with one padded column
// (7 x 8 of 7 x 7, 11 x 12 of 11 x 11).
template <int R> struct GrpTile {
    static constexpr int T = R % 4 == 0 ? 4 : R % 3 == 0 ? 3 : R % 5 == 0 ? 5 : R == 2 ? 2 : 4;
    static constexpr int RP = (R + T - 1) / T * T;
};

// Group record [s | M | v] of rank R in values of type V, s and v padded to RP
// values, M to RP rows of RP values (padding is zero): s at 0, M[c][c'] at
// m(c, c'), v at VOFF.  The T x T blocks of M that the Gram tiles read at once
// should fall into distinct shared-memory banks: at R = 4 and 8 the rows
// c >= RP / 2 of M sit 64 bytes further on; at R = 7, 11 and 12 every block of
// four rows sits 16 bytes further than the last (its natural distance is a
// multiple of 128 bytes).
template <typename V, int R> struct GrpRec {
    static constexpr int T = GrpTile<R>::T, RP = GrpTile<R>::RP;
    static constexpr bool HALF = R == 4 || R == 8;
    static constexpr int PADV = HALF ? (int)(64 / sizeof(V)) : (T == 4 ? (int)(16 / sizeof(V)) : 0);
    static constexpr int PADS = HALF ? PADV : PADV * (RP / T);
    static constexpr int VOFF = RP + RP * RP + PADS;
    static constexpr int RS = ((VOFF + RP) * (int)sizeof(V) + 15) / 16 * 16 / (int)sizeof(V);
    __host__ __device__ static constexpr int m(int c, int cc)
    {
        return RP + c * RP + cc + (HALF ? (c >= RP / 2 ? PADV : 0) : (c / T) * PADV);
    }
};

// Shared-memory budget of k_group_sums: a block's entries (rows of the
// summed side and values) are staged when they fit.  CAP is the most a block
// stages (SMEM bytes); a launch sizes its dynamic shared memory for the
// level's largest block, at most CAP entries, so levels with small groups
// keep more blocks resident.
template <typename T, int R> struct GsumCfg {
    static constexpr int NTH = 128;
    static constexpr int GB = NTH / R;                    // groups per block
    static constexpr size_t VS = sizeof(typename cvec<T>::type);
    static constexpr int CAP = (int)(46080 / ((R + 1) * VS));   // staged entries per block
    static constexpr size_t SMEM = (size_t)CAP * (R + 1) * VS;
};

// Zeros into the padded values of a group record (lane of `lanes`).
template <typename V, int R> __device__ __forceinline__ void grp_zero_padding(V* o, int lane, int lanes)
{
    typedef GrpRec<V, R> RL;
    constexpr int RP = RL::RP;
    for (int q = lane; q < RP * RP; q += lanes)
        if (q / RP >= R || q % RP >= R) o[RL::m(q / RP, q % RP)] = czero<V>();
    for (int q = R + lane; q < RP; q += lanes) {
        o[q] = czero<V>();
        o[RL::VOFF + q] = czero<V>();
    }
}

// Group sums of one middle level, one thread per (group, row a): the shared
// vector s of the group (h of a row group, w of a column group, taken from
// its first entry), and over the group's entries the sums
//   M[a][a'] = sum_e conj(u_e[a]) u_e[a'],   v[a] = sum_e conj(u_e[a]) t_e
// of the other environment u (w, resp. h).  Record per group, compute type:
// [s (R) | M (R x R, row-major) | v (R)].  A block's groups are contiguous
// in the level order, and so are their entries: when they fit (cap <= CAP
// entries, the dynamic shared memory of the launch, sized for the level's
// largest block), the rows u_e and values t_e of all of them are copied to
// shared memory at once (cp.async), so their loads overlap; otherwise they
// are read from global memory.  In the precision form the sums run in complex64 over blocks of 16
// entries, Kahan-compensated across blocks.
template <typename T, int R>
__global__ void __launch_bounds__(GsumCfg<T, R>::NTH)
k_group_sums(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Wm,
             const typename cvec<T>::type* __restrict__ tv, const int32_t* __restrict__ gstart, int G, int by_col,
             typename cvec<T>::type* __restrict__ out, int cap)
{
    typedef typename cvec<T>::type V;
    typedef GsumCfg<T, R> C;
    typedef GrpRec<V, R> RL;
    constexpr int RS = RL::RS;
    extern __shared__ __align__(16) unsigned char smem[];
    V* su = (V*)smem;                          // [cap][R] rows
    V* st = su + (size_t)cap * R;              // [cap] values
    const V* Sv = by_col ? Wm : H;
    const V* Uv = by_col ? H : Wm;

    const int gb0 = blockIdx.x * C::GB;
    const int gb1 = min(gb0 + C::GB, G);
    const int E0 = gstart[gb0], E1 = gstart[gb1];
    const bool staged = E1 - E0 <= cap;
    if (staged) {
        // rows: (E1 - E0) R contiguous values, in 16-byte pieces; in 8-byte
        // ones in complex64 at odd rank, where a row can start between them
        if constexpr ((R * C::VS) % 16 == 0) {
            const int rpieces = (int)((size_t)(E1 - E0) * R * C::VS / 16);
            const unsigned char* usrc = (const unsigned char*)(Uv + (size_t)E0 * R);
            for (int q = threadIdx.x; q < rpieces; q += C::NTH)
                cp_async16((unsigned char*)su + 16 * (size_t)q, usrc + 16 * (size_t)q);
        } else {
            for (int q = threadIdx.x; q < (E1 - E0) * R; q += C::NTH) cp_async8(su + q, Uv + (size_t)E0 * R + q);
        }
        // values: one copy per entry (8 or 16 bytes)
        for (int q = threadIdx.x; q < E1 - E0; q += C::NTH) {
            if constexpr (sizeof(V) == 16)
                cp_async16(st + q, tv + E0 + q);
            else
                cp_async8(st + q, tv + E0 + q);
        }
        cp_async_commit();
        cp_async_wait_all();
    }
    __syncthreads();
    const int g = gb0 + (int)threadIdx.x / R, a = (int)threadIdx.x % R;
    if (g >= gb1) return;
    const int e0 = gstart[g], e1 = gstart[g + 1];
    // the block's entries in shared memory (staged) or global memory, indexed
    // from the block's first entry E0
    const V* ub = staged ? su : Uv + (size_t)E0 * R;
    const V* tb = staged ? st : tv + E0;
    V* o = out + (size_t)g * RS;
    o[a] = Sv[(size_t)e0 * R + a];
    if (RL::RP > R && a == 0) grp_zero_padding<V, R>(o, 0, 1);
    V ms[R], vs;
    float mc[R][2], vc[2];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        ms[q] = czero<V>();
        mc[q][0] = mc[q][1] = 0.f;
    }
    vs = czero<V>();
    vc[0] = vc[1] = 0.f;
    for (int eb = e0; eb < e1; eb += 16) {
        V mp[R], vp = czero<V>();
#pragma unroll
        for (int q = 0; q < R; ++q) mp[q] = czero<V>();
        const int ee = min(eb + 16, e1);
        for (int e = eb; e < ee; ++e) {
            V u[R];
            const V* row = ub + (size_t)(e - E0) * R;
#pragma unroll
            for (int q = 0; q < R; ++q) u[q] = row[q];
            const V ua = row[a];   // one more load instead of a select chain
#pragma unroll
            for (int q = 0; q < R; ++q) cmacc(mp[q], ua, u[q]);
            cmacc(vp, ua, tb[e - E0]);
        }
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                kahan(ms[q].x, mc[q][0], mp[q].x);
                kahan(ms[q].y, mc[q][1], mp[q].y);
            }
            kahan(vs.x, vc[0], vp.x);
            kahan(vs.y, vc[1], vp.y);
        } else {
#pragma unroll
            for (int q = 0; q < R; ++q) {
                ms[q].x += mp[q].x;
                ms[q].y += mp[q].y;
            }
            vs.x += vp.x;
            vs.y += vp.y;
        }
    }
#pragma unroll
    for (int q = 0; q < R; ++q) {
        V m = ms[q];
        if constexpr (sizeof(T) == 4) {
            m.x -= mc[q][0];
            m.y -= mc[q][1];
        }
        o[RL::m(a, q)] = m;
    }
    if constexpr (sizeof(T) == 4) {
        vs.x -= vc[0];
        vs.y -= vc[1];
    }
    o[RL::VOFF + a] = vs;
}

// Group sums of a level with many entries per group: one warp per group
// (warp_sums: the lower triangle of M and v, chunks of 32 entries), the upper
// triangle of M by conjugation.  Same record as k_group_sums, whose block
// holds 128 / R groups: with hundreds of entries in each, few threads would
// walk long lists.
template <typename T, int R>
__global__ void __launch_bounds__(128)
k_group_sums_warp(const typename cvec<T>::type* __restrict__ H, const typename cvec<T>::type* __restrict__ Wm,
                  const typename cvec<T>::type* __restrict__ tv, const int32_t* __restrict__ gstart, int G, int by_col,
                  typename cvec<T>::type* __restrict__ out)
{
    typedef typename cvec<T>::type V;
    typedef GrpRec<V, R> RL;
    __shared__ __align__(16) V a_s[4][32 * R + 2];
    __shared__ V t_s[4][32];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int g = blockIdx.x * 4 + wib;
    if (g >= G) return;   // whole warp leaves; only warp-level barriers below
    const V* Sv = by_col ? Wm : H;
    const V* Uv = by_col ? H : Wm;
    const int e0 = gstart[g];
    V* o = out + (size_t)g * RL::RS;
    if (lane < R) o[lane] = Sv[(size_t)e0 * R + lane];
    if (RL::RP > R) grp_zero_padding<V, R>(o, lane, 32);
    warp_sums<T, R, sizeof(T) == 4>(Uv, tv, e0, gstart[g + 1], a_s[wib], t_s[wib], lane, [&](int, int p, int q, V s, V c) {
        if constexpr (sizeof(T) == 4) {
            s.x = __fsub_rn(s.x, c.x);
            s.y = __fsub_rn(s.y, c.y);
        }
        if (q < 0) {
            o[RL::VOFF + p] = s;
        } else {
            o[RL::m(p, q)] = s;
            if (p != q) o[RL::m(q, p)] = make_conj(s);
        }
    });
}

// acc += x * y.  Precision form: (s, c) is a Kahan pair per component and
// the product enters with one rounding per component (the carried
// compensation is subtracted inside the fused multiply-adds); FP64: plain
// fused multiply-adds.
__device__ __forceinline__ void grp_acc(float2& s, float2& c, float2 x, float2 y)
{
    const float yr = __fmaf_rn(x.x, y.x, __fmaf_rn(-x.y, y.y, -c.x));
    const float yi = __fmaf_rn(x.x, y.y, __fmaf_rn(x.y, y.x, -c.y));
    float t = __fadd_rn(s.x, yr);
    c.x = __fsub_rn(__fsub_rn(t, s.x), yr);
    s.x = t;
    t = __fadd_rn(s.y, yi);
    c.y = __fsub_rn(__fsub_rn(t, s.y), yi);
    s.y = t;
}
__device__ __forceinline__ void grp_acc(double2& s, double2&, double2 x, double2 y) { cmac(s, x, y); }

// (s, nc) += x y + x' y' with packed operands: X1 = (x.re, x.re), X2 = (x.im,
// x.im), Y = (y.re, y.im), Yr = i y = (-y.im, y.re), so x y = X1 Y + X2 Yr.  s
// is the Kahan sum and nc its negated compensation (the value is s + nc); the
// compensation enters inside the fused multiply-adds.  Two groups per step: the
// products' roundings, two per group and component, are as many as with one
// step per group, the three additions of the step are shared.
__device__ __forceinline__ void grp_acc2(uint64_t& s, uint64_t& nc, uint64_t X1, uint64_t X2, uint64_t Y, uint64_t Yr,
                                         uint64_t W1, uint64_t W2, uint64_t Z, uint64_t Zr)
{
    const uint64_t q = c2fma(X1, Y, c2fma(X2, Yr, c2fma(W1, Z, c2fma(W2, Zr, nc))));   // x y + x' y' - c
    const uint64_t t = c2add(s, q);
    nc = c2sub(q, c2sub(t, s));
    s = t;
}

template <typename T, int R> struct GrpCfg {
    static_assert(R >= 2, "grouped Gram needs R >= 2");
    static constexpr int TT = GrpTile<R>::T, RP = GrpTile<R>::RP;
    static constexpr int D = R * R;
    static constexpr int NB = R * RP / TT;                 // tile rows over p' = a RP + c
    static constexpr int NT = NB * (NB + 1) / 2;           // T x T tiles of the lower triangle
    // groups per chunk
    static constexpr int CG = (sizeof(T) == 4 ? 32 : 16) / (R >= 11 ? 2 : 1);
    // blocks that share a slice's tiles (ranks 9, 11, 12: 378 to 666 tiles): in
    // one block of 666 threads a thread has 80 registers, too few for its sums
    static constexpr int NSPLIT = NT > 224 ? (NT + 191) / 192 : 1;
    static constexpr int NTB = (NT + NSPLIT - 1) / NSPLIT; // tiles of a block
    static constexpr int GT = (160 / NTB) < 1 ? 1 : (160 / NTB);
    static constexpr int G = NSPLIT > 1 ? 1 : (GT > CG ? CG : GT);   // thread groups over the chunk's groups
    static constexpr int NW = NTB * G;                     // tile threads
    static constexpr int NTH = ((NW + 31) / 32) * 32;
    // the right-hand side on the threads past the tiles when there are
    // enough of them (R = 8: 24 threads, 3 entries of y each), else on the
    // diagonal tiles
    static constexpr int NY = NTH - NW;
    static constexpr bool YSPARE = G == 1 && NSPLIT == 1 && NY >= 8 && (D + NY - 1) / NY <= TT;
    static constexpr int YPT = YSPARE ? (D + NY - 1) / NY : 0;
    static constexpr int NST = 3;                          // ring stages
    static constexpr int NPK = D * (D + 1) / 2;
    typedef GrpRec<typename cvec<T>::type, R> RL;
    static constexpr int RS = RL::RS;                      // group record [s | M | v]
    static constexpr size_t VS = sizeof(typename cvec<T>::type);
    static constexpr int PIECES = (int)(RS * VS / 16);     // 16-byte pieces per record
    static_assert(RS * VS % 16 == 0, "records must be whole 16-byte pieces");
    static constexpr size_t STAGE = (size_t)CG * RS * VS;
    static constexpr size_t RING = NST * STAGE;
    static constexpr size_t KBYTES = G > 1 ? (size_t)G * (NPK + D) * VS : 0;
    static constexpr size_t SMEM = RING > KBYTES ? RING : KBYTES;
    static_assert(SMEM <= 227 * 1024, "shared memory of a block");
    // blocks per SM the registers are budgeted for: a tile's sums (and, in the
    // precision form, compensations) take 4 T^2 registers, plus about 64 (25
    // outputs at T = 5, 104 registers at T = 3 and 4 in complex64)
    static constexpr int REGS = 4 * TT * TT + 68;
    static constexpr int MINB0 = 65536 / (NTH * REGS);
    static constexpr int MINB1 = sizeof(T) == 4 ? 3 : 2;
    static constexpr int MINB = MINB0 < 1 ? 1 : (MINB0 > MINB1 ? MINB1 : MINB0);
};

// T consecutive values: 16-byte loads where T and the alignment allow.
template <typename V, int TT> __device__ __forceinline__ void load_t(V (&d)[TT], const V* p)
{
    if constexpr (TT == 4) {
        load4(d, p);
    } else {
#pragma unroll
        for (int u = 0; u < TT; ++u) d[u] = p[u];
    }
}

// Per-slice normal equations from the group records of k_group_sums (NSPLIT
// blocks per slice; the grid is a multiple of NSPLIT, grid-stride).  grec starts
// with group gbase of the level, the first of the S slices.  Chunks of CG records stream through an
// NST-stage shared-memory ring by 16-byte cp.async copies; per group, the
// shared side's outer product is formed in registers (conj(s_a) s_a' for row
// groups; conj(s_c) s_c' for column groups) and multiplied with the other
// side's sums M, each product added to the tile's accumulators (compensated
// per group in the precision form: a group's term can be a large part of
// the slice's sum).
template <typename T, int R, int BY_COL>
__global__ void __launch_bounds__(GrpCfg<T, R>::NTH, GrpCfg<T, R>::MINB)
k_mid_gram_grp(const typename cvec<T>::type* __restrict__ grec, const int32_t* __restrict__ gseg, int gbase,
               T* __restrict__ rec, int S)
{
    typedef typename cvec<T>::type V;
    typedef GrpCfg<T, R> C;
    typedef Rec<T, R> RC;
    constexpr int D = C::D, NPK = C::NPK, CG = C::CG, NTH = C::NTH, RS = C::RS, NST = C::NST;
    constexpr int TT = C::TT, RP = C::RP;
    extern __shared__ __align__(16) unsigned char smem[];
    typedef typename C::RL RL;
    V* ring = (V*)smem;                           // [NST][CG][RS]
    V* red = (V*)smem;                            // thread-group reduction (G > 1), after the ring

    const int tid = threadIdx.x;
    const int part = C::NSPLIT > 1 ? blockIdx.x % C::NSPLIT : 0;   // this block's share of the tiles
    const bool worker = tid < C::NW && part * C::NTB + tid < C::NT * C::G;
    const bool ythread = C::YSPARE && !worker;
    const int grp = worker ? tid / C::NTB : 0, tile = worker ? part * C::NTB + tid - grp * C::NTB : 0;
    int I = 0;
    while ((I + 1) * (I + 2) / 2 <= tile) ++I;
    const int J = tile - I * (I + 1) / 2;
    const bool diag = !C::YSPARE && (I == J);
    // row T I + u of the padded index a RP + c is the pair a = aI, c = cI + u
    // (T divides RP); columns likewise
    const int aI = (TT * I) / RP, cI = (TT * I) % RP, aJ = (TT * J) / RP, cJ = (TT * J) % RP;
    // right-hand side entries p = yb + NY x of a spare thread
    const int yb = tid - C::NW;

    // records [gfirst, gfirst + cnt) into ring stage st
    auto issue = [&](int st, int gfirst, int cnt) {
        const unsigned char* src = (const unsigned char*)(grec + (size_t)gfirst * RS);
        unsigned char* dst = (unsigned char*)(ring + (size_t)st * CG * RS);
        const int pieces = cnt * C::PIECES;
        for (int q = tid; q < pieces; q += NTH) cp_async16(dst + 16 * (size_t)q, src + 16 * (size_t)q);
    };

    for (int k = blockIdx.x / C::NSPLIT; k < S; k += gridDim.x / C::NSPLIT) {
        const int g0 = gseg[k] - gbase, g1 = gseg[k + 1] - gbase;
        const int nch = (g1 - g0 + CG - 1) / CG;
        // tiles: s_/c_ (Kahan pairs); right-hand side: ys/yc (diagonal tiles
        // or spare threads)
        V s_[TT][TT], c_[TT][TT], ys[TT], yc[TT];
        uint64_t s2[TT][TT], n2[TT][TT];   // complex64 tiles: packed Kahan sums, negated compensations
#pragma unroll
        for (int u = 0; u < TT; ++u) {
            ys[u] = czero<V>();
            yc[u] = czero<V>();
#pragma unroll
            for (int v = 0; v < TT; ++v) {
                s_[u][v] = czero<V>();
                c_[u][v] = czero<V>();
                s2[u][v] = 0ull;
                n2[u][v] = 0ull;
            }
        }
        __syncthreads();  // previous slice done with the ring and the reduction
#pragma unroll
        for (int c = 0; c < NST - 1; ++c) {
            if (c < nch) issue(c, g0 + c * CG, min(CG, g1 - g0 - c * CG));
            cp_async_commit();
        }
        for (int c = 0; c < nch; ++c) {
            cp_async_wait_n<NST - 2>();   // this thread's copies of chunk c landed
            __syncthreads();              // everyone's; stage (c - 1) mod NST is free
            const int cn = c + NST - 1;
            if (cn < nch) issue(cn % NST, g0 + cn * CG, min(CG, g1 - g0 - cn * CG));
            cp_async_commit();
            const V* buf = ring + (size_t)(c % NST) * CG * RS;
            const int cnt = min(CG, g1 - g0 - c * CG);
            if constexpr (sizeof(T) == 4) {
              if (worker) {
                for (int gi = grp; gi < cnt; gi += 2 * C::G) {
                    const V* gr = buf + gi * RS;
                    // the second group of the step; past the end the first one
                    // again with a zero factor
                    const bool two = gi + C::G < cnt;
                    const V* gs = two ? gr + C::G * RS : gr;
                    if constexpr (!BY_COL) {
                        // X = conj(h) h^T from s = h; Y = M (sums of the w side)
                        const V x = cmul(make_conj(gr[aI]), gr[aJ]);
                        V w = cmul(make_conj(gs[aI]), gs[aJ]);
                        if (!two) w = czero<V>();
                        const uint64_t X1 = c2pack(x.x, x.x), X2 = c2pack(x.y, x.y);
                        const uint64_t W1 = c2pack(w.x, w.x), W2 = c2pack(w.y, w.y);
#pragma unroll
                        for (int u = 0; u < TT; ++u) {
                            V yr[TT], zr[TT];
                            load_t<V, TT>(yr, gr + RL::m(cI + u, cJ));
                            load_t<V, TT>(zr, gs + RL::m(cI + u, cJ));
#pragma unroll
                            for (int v = 0; v < TT; ++v)
                                grp_acc2(s2[u][v], n2[u][v], X1, X2, c2pack(yr[v].x, yr[v].y),
                                         c2pack(-yr[v].y, yr[v].x), W1, W2, c2pack(zr[v].x, zr[v].y),
                                         c2pack(-zr[v].y, zr[v].x));
                        }
                        if (diag) {
#pragma unroll
                            for (int u = 0; u < TT; ++u) {
                                grp_acc(ys[u], yc[u], make_conj(gr[aI]), gr[RL::VOFF + cI + u]);
                                if (two) grp_acc(ys[u], yc[u], make_conj(gs[aI]), gs[RL::VOFF + cI + u]);
                            }
                        }
                    } else {
                        // X = M (sums of the h side); Y = conj(w) w^T from s = w:
                        // term (u, v) = (conj(s_cI+u) x) s_cJ+v
                        const V x = gr[RL::m(aI, aJ)];
                        V w = gs[RL::m(aI, aJ)];
                        if (!two) w = czero<V>();
                        V sj[TT], tj[TT];
                        load_t<V, TT>(sj, gr + cJ);
                        load_t<V, TT>(tj, gs + cJ);
#pragma unroll
                        for (int u = 0; u < TT; ++u) {
                            const V si = gr[cI + u], ti = gs[cI + u];
                            const V xa = cmul(make_conj(si), x), wa = cmul(make_conj(ti), w);
                            const uint64_t X1 = c2pack(xa.x, xa.x), X2 = c2pack(xa.y, xa.y);
                            const uint64_t W1 = c2pack(wa.x, wa.x), W2 = c2pack(wa.y, wa.y);
#pragma unroll
                            for (int v = 0; v < TT; ++v)
                                grp_acc2(s2[u][v], n2[u][v], X1, X2, c2pack(sj[v].x, sj[v].y),
                                         c2pack(-sj[v].y, sj[v].x), W1, W2, c2pack(tj[v].x, tj[v].y),
                                         c2pack(-tj[v].y, tj[v].x));
                            if (diag) {
                                grp_acc(ys[u], yc[u], gr[RL::VOFF + aI], make_conj(si));
                                if (two) grp_acc(ys[u], yc[u], gs[RL::VOFF + aI], make_conj(ti));
                            }
                        }
                    }
                }
              }
            } else if (worker) {
                for (int gi = grp; gi < cnt; gi += C::G) {
                    const V* gr = buf + gi * RS;
                    if constexpr (!BY_COL) {
                        // X = conj(h) h^T from s = h; Y = M (sums of the w side)
                        const V x = cmul(make_conj(gr[aI]), gr[aJ]);
#pragma unroll
                        for (int u = 0; u < TT; ++u) {
                            V yr[TT];
                            load_t<V, TT>(yr, gr + RL::m(cI + u, cJ));
#pragma unroll
                            for (int v = 0; v < TT; ++v) grp_acc(s_[u][v], c_[u][v], x, yr[v]);
                        }
                        if (diag) {
                            const V xv = make_conj(gr[aI]);
#pragma unroll
                            for (int u = 0; u < TT; ++u) grp_acc(ys[u], yc[u], xv, gr[RL::VOFF + cI + u]);
                        }
                    } else {
                        // X = M (sums of the h side); Y = conj(w) w^T from s = w
                        const V x = gr[RL::m(aI, aJ)];
                        V sj[TT], si[TT];
                        load_t<V, TT>(sj, gr + cJ);
                        load_t<V, TT>(si, gr + cI);
#pragma unroll
                        for (int v = 0; v < TT; ++v) sj[v] = cmul(x, sj[v]);
#pragma unroll
                        for (int u = 0; u < TT; ++u) {
                            const V a = make_conj(si[u]);
#pragma unroll
                            for (int v = 0; v < TT; ++v) grp_acc(s_[u][v], c_[u][v], a, sj[v]);
                        }
                        if (diag) {
                            const V xv = gr[RL::VOFF + aI];
#pragma unroll
                            for (int u = 0; u < TT; ++u) grp_acc(ys[u], yc[u], xv, make_conj(si[u]));
                        }
                    }
                }
            }
            if (ythread) {
                // y[(a, c)] += xv[a] yv[c] for p = yb + NY x
                for (int gi = 0; gi < cnt; ++gi) {
                    const V* gr = buf + gi * RS;
#pragma unroll
                    for (int x = 0; x < C::YPT; ++x) {
                        const int p = yb + C::NY * x;
                        if (p < D) {
                            const int a = p / R, cc = p - (p / R) * R;
                            const V xv = BY_COL ? gr[RL::VOFF + a] : make_conj(gr[a]);
                            const V yv = BY_COL ? make_conj(gr[cc]) : gr[RL::VOFF + cc];
                            grp_acc(ys[x], yc[x], xv, yv);
                        }
                    }
                }
            }
        }
        cp_async_wait_n<0>();
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int u = 0; u < TT; ++u) {
#pragma unroll
                for (int v = 0; v < TT; ++v) {
                    c2unpack(c2add(s2[u][v], n2[u][v]), s_[u][v].x, s_[u][v].y);
                }
                ys[u].x = __fsub_rn(ys[u].x, yc[u].x);
                ys[u].y = __fsub_rn(ys[u].y, yc[u].y);
            }
        }
        T* out = rec + (size_t)k * RC::SIZE;
        if constexpr (C::G == 1) {
            if (worker) {
#pragma unroll
                for (int u = 0; u < TT; ++u) {
                    const int p = aI * R + cI + u;
                    if (RP > R && cI + u >= R) continue;   // padding
#pragma unroll
                    for (int v = 0; v < TT; ++v) {
                        const int q = aJ * R + cJ + v;
                        if (q <= p && (RP == R || cJ + v < R)) RC::put(out, p, q, s_[u][v]);
                    }
                    if (diag) RC::put_y(out, p, ys[u]);
                }
            } else if (ythread) {
#pragma unroll
                for (int x = 0; x < C::YPT; ++x) {
                    const int p = yb + C::NY * x;
                    if (p < D) RC::put_y(out, p, ys[x]);
                }
            }
        } else {
            static_assert(C::G == 1 || !C::YSPARE, "the thread-group reduction takes y from the diagonal tiles");
            // every thread group's sums side by side (the ring is done with),
            // then a thread per element adds them in FP64, in order
            __syncthreads();
            if (worker) {
                V* rg = red + (size_t)grp * (NPK + D);
#pragma unroll
                for (int u = 0; u < TT; ++u) {
                    const int p = aI * R + cI + u;
                    if (RP > R && cI + u >= R) continue;   // padding
#pragma unroll
                    for (int v = 0; v < TT; ++v) {
                        const int q = aJ * R + cJ + v;
                        if (q <= p && (RP == R || cJ + v < R)) rg[tri(p, q)] = s_[u][v];
                    }
                    if (diag) rg[NPK + p] = ys[u];
                }
            }
            __syncthreads();
            for (int x = tid; x < D * D + D; x += NTH) {
                const int p = x / D, q = x - p * D;
                if (p < D && q > p) continue;
                const V* src = red + (p < D ? tri(p, q) : NPK + q);
                double2 v = make_double2(0.0, 0.0);
#pragma unroll 4
                for (int g = 0; g < C::G; ++g) {
                    const V t = src[(size_t)g * (NPK + D)];
                    v.x += (double)t.x;
                    v.y += (double)t.y;
                }
                if (p < D) RC::put(out, p, q, v);
                else RC::put_y(out, q, v);
            }
        }
    }
}

}  // namespace bfc
