// Gauge fixing of the butterfly factors by left orthogonalization, in FP64
// on the master factors.  Eq. (BF_tensor_rep) is unchanged when an
// invertible r x r matrix G is inserted on a bond between two factors
// (X -> X G, Y -> G^{-1} Y).  Level by level, from S^1 to S^{L+1}, the
// matrix of every bond group is factored M = Q R (R with a real positive
// diagonal, so the factorization is unique) and replaced by Q, and R
// multiplies the factors on the other side of the bond:
//  * level 0, leaf block p of rows i: M = z1[p b .. p b + b - 1] (b x r),
//    R multiplies the slices 2p and 2p + 1 of S^2;
//  * level m = 1 .. L, bond (A, B) with k_{m+1} = ((A << 1 | a) << m) | B:
//    M = [Z[m][k(a = 0)]; Z[m][k(a = 1)]] (2r x r), R multiplies the slices
//    (A << (m + 1)) | (B << 1 | c), c = 0, 1, of S^{m+2} (m < L) or the
//    columns zL[j] of leaf block p_j = B (m = L).
// Classical Gram-Schmidt applied twice per column (orthogonal to rounding
// level), a half or a whole warp per bond group, the group's matrix in shared
// memory; leaf blocks of more than 32 rows: a warp on global memory.
#include "bfc_internal.h"

namespace bfc {

namespace {

__device__ __forceinline__ double2 d2(double x, double y) { return make_double2(x, y); }

// M (nrows x R, rows contiguous) = Q R in place, one warp, rows over the lanes.
template <int R>
__device__ void warp_qr(double2* M, int64_t nrows, double2 (*Rm)[R], int lane)
{
    for (int x = lane; x < R * R; x += 32) Rm[x / R][x % R] = d2(0.0, 0.0);
    __syncwarp();
    for (int j = 0; j < R; ++j) {
        for (int pass = 0; pass < 2; ++pass) {
            for (int i = 0; i < j; ++i) {
                double cx = 0.0, cy = 0.0;   // c = Q_i^H v
                for (int64_t q = lane; q < nrows; q += 32) {
                    const double2 qi = M[q * R + i], v = M[q * R + j];
                    cx += qi.x * v.x + qi.y * v.y;
                    cy += qi.x * v.y - qi.y * v.x;
                }
                for (int o = 16; o > 0; o >>= 1) {
                    cx += __shfl_xor_sync(0xffffffffu, cx, o);
                    cy += __shfl_xor_sync(0xffffffffu, cy, o);
                }
                __syncwarp();
                for (int64_t q = lane; q < nrows; q += 32) {
                    double2* rw = M + q * R;
                    const double2 qi = rw[i];
                    double2 v = rw[j];
                    v.x -= cx * qi.x - cy * qi.y;
                    v.y -= cx * qi.y + cy * qi.x;
                    rw[j] = v;
                }
                if (lane == 0) {
                    Rm[i][j].x += cx;
                    Rm[i][j].y += cy;
                }
                __syncwarp();
            }
        }
        double s = 0.0;
        for (int64_t q = lane; q < nrows; q += 32) {
            const double2 v = M[q * R + j];
            s += v.x * v.x + v.y * v.y;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const double nrm = sqrt(s);
        const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
        __syncwarp();
        for (int64_t q = lane; q < nrows; q += 32) {
            double2* rw = M + q * R;
            rw[j].x *= inv;
            rw[j].y *= inv;
        }
        if (lane == 0) Rm[j][j] = d2(nrm, 0.0);
        __syncwarp();
    }
}

// Lanes per bond group of a middle level: its 2R rows (and the 2R rows or
// columns of the neighbours that R multiplies) fit the lanes one to one.
template <int R>
struct QrCfg {
    static constexpr int GS = R <= 8 ? 16 : 32, GPW = 32 / GS;
    static constexpr int ROWS = 32, LD = ROWS + 1;   // odd: lanes on different columns of one row hit different banks
};

// The matrix A[column][row] (nrows <= 32 rows) = Q R in place by GS lanes (gl).
// The projections of a column on all columns before it are taken at once: the
// dot products with lanes over columns x parts of the rows, the update with a
// lane per row.
template <int R>
__device__ __forceinline__ void group_qr(double2 (*A)[QrCfg<R>::LD], double2 (*Rm)[R], double2* cs, int nrows, int gl)
{
    constexpr int GS = QrCfg<R>::GS, KR = QrCfg<R>::ROWS / GS;
    for (int x = gl; x < R * R; x += GS) Rm[x / R][x % R] = d2(0.0, 0.0);
    __syncwarp();
    int w = 1;   // power of two >= j
#pragma unroll 1
    for (int j = 0; j < R; ++j) {
        double2 v[KR];
#pragma unroll
        for (int k = 0; k < KR; ++k) v[k] = gl + k * GS < nrows ? A[j][gl + k * GS] : d2(0.0, 0.0);
        if (j > w) w *= 2;
        if (j > 0) {
            const int i = gl & (w - 1), part = gl / w, parts = GS / w;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                double xx = 0.0, yy = 0.0, xy = 0.0, yx = 0.0;   // c = Q_i^H v
                if (i < j)
#pragma unroll 4
                    for (int q = part; q < nrows; q += parts) {
                        const double2 a = A[i][q], b = A[j][q];
                        xx = fma(a.x, b.x, xx);
                        yy = fma(a.y, b.y, yy);
                        xy = fma(a.x, b.y, xy);
                        yx = fma(a.y, b.x, yx);
                    }
                double cx = xx + yy, cy = xy - yx;
                for (int o = w; o < GS; o <<= 1) {
                    cx += __shfl_xor_sync(0xffffffffu, cx, o);
                    cy += __shfl_xor_sync(0xffffffffu, cy, o);
                }
                if (part == 0 && i < j) {
                    cs[i] = d2(cx, cy);
                    Rm[i][j].x += cx;
                    Rm[i][j].y += cy;
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < KR; ++k) {
                    const int q = gl + k * GS;
                    if (q < nrows) {
                        double px = 0.0, py = 0.0;   // Q c, two chains beside v's two
#pragma unroll 2
                        for (int l = 0; l < j; ++l) {
                            const double2 c = cs[l], a = A[l][q];
                            v[k].x = fma(-c.x, a.x, v[k].x);
                            v[k].y = fma(-c.x, a.y, v[k].y);
                            px = fma(c.y, a.y, px);
                            py = fma(c.y, a.x, py);
                        }
                        v[k].x += px;
                        v[k].y -= py;
                        A[j][q] = v[k];
                    }
                }
                __syncwarp();
            }
        }
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < KR; ++k) s += v[k].x * v[k].x + v[k].y * v[k].y;
        for (int o = 1; o < GS; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const double nrm = sqrt(s);
        const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
#pragma unroll
        for (int k = 0; k < KR; ++k)
            if (gl + k * GS < nrows) A[j][gl + k * GS] = d2(v[k].x * inv, v[k].y * inv);
        if (gl == 0) Rm[j][j] = d2(nrm, 0.0);
        __syncwarp();
    }
}

// One row or column of r values (element k at p[k * ld]) that R multiplies:
// out[a] = sum_{k >= a} R[a][k] in[k], with conj(R) if CJ.
template <int R>
struct Line {
    double2 v[R];
    __device__ __forceinline__ void load(const double2* p, int ld)
    {
#pragma unroll
        for (int k = 0; k < R; ++k) v[k] = p[(size_t)k * ld];
    }
    template <bool CJ>
    __device__ __forceinline__ void times(const double2 (*Rm)[R], double2* p, int ld) const
    {
#pragma unroll
        for (int a = 0; a < R; ++a) {
            double sx = 0.0, sy = 0.0;
#pragma unroll
            for (int k = a; k < R; ++k) {
                double2 x = Rm[a][k];
                if (CJ) x.y = -x.y;
                sx += x.x * v[k].x - x.y * v[k].y;
                sy += x.x * v[k].y + x.y * v[k].x;
            }
            p[(size_t)a * ld] = d2(sx, sy);
            asm volatile("" ::: "memory");   // R stays in shared memory (hoisted loads spill at r >= 10)
        }
    }
};

template <int R, bool CJ>
__device__ void rows_times(double2* rows, int64_t count, const double2 (*Rm)[R], int gl, int step)
{
    for (int64_t q = gl; q < count; q += step) {
        Line<R> t;
        t.load(rows + (size_t)q * R, 1);
        t.template times<CJ>(Rm, rows + (size_t)q * R, 1);
    }
}

// Orthogonalization of one level, from the left (RL = 0, the levels above) or
// from the right (RL = 1):
//  * level L + 1, leaf block p of columns j: M = zL[p b .. p b + b - 1]
//    (b x r) = Q R, zL := Q and R^T right-multiplies the slices
//    (i_0 << L) | p of S^{L+1} (for L = 0: every row z1[i]);
//  * level m = L .. 1, group g: the two slices k = 2g, 2g + 1 of S^{m+1}
//    (differing in j_{m-1}, bit 0) form [Z0 | Z1] = R^H Q^H, computed as the
//    QR of the stacked conjugate transposes [Z0^H; Z1^H] (2r x r); Z_b :=
//    (half b of Q)^H, and R^H right-multiplies the two slices of S^m that
//    share the bond, ((g >> (m-1)) << m) | (c << (m-1)) | (g mod 2^(m-1)),
//    or, for m = 1, the rows z1[i] of leaf block p_i = g.
// Bound: the FP64 pipe (a warp instruction takes it for about 16 cycles however
// many lanes are active), so groups of up to 16 rows share a warp, and the dot
// products use as many lanes as the columns so far allow.  One warp per CTA
// spreads the groups over all SMs.  The lines that R multiplies are loaded
// before the factorization.  n = 16384, L = 10, r = 8 (1024 groups of 16 x 8,
// most launches): 51 us per launch; 168 us (from the right) and 130 us (from
// the left) with a warp per group on global memory, one projection at a time.
template <int R, bool RL>
__global__ void __launch_bounds__(32)
k_qr_level(double2* __restrict__ z1, double2* __restrict__ Z, double2* __restrict__ zL, int64_t n, int L, int b,
           int level, int ngroups)
{
    typedef QrCfg<R> C;
    constexpr int GS = C::GS;
    __shared__ double2 As[C::GPW][R][C::LD];
    __shared__ double2 Rs[C::GPW][R][R];
    __shared__ double2 cs[C::GPW][R];
    const int h = threadIdx.x / GS, gl = threadIdx.x % GS;
    const int g = blockIdx.x * C::GPW + h;
    const bool live = g < ngroups;   // a dead half runs along on zeros
    const int64_t S = (int64_t)1 << (L + 1);
    auto slice = [&](int m, int64_t k) { return Z + ((size_t)(m - 1) * S + k) * R * R; };   // Z[m][k], m = 1..L
    const bool leaf = level == (RL ? L + 1 : 0);
    const int nrows = leaf ? b : 2 * R;
    const int A = RL ? 0 : g >> level, B = RL ? 0 : g & ((1 << level) - 1);
    double2 (*M)[C::LD] = As[h];

    double2 *s0 = nullptr, *s1 = nullptr;   // the group's rows, or its two slices
    if (leaf) {
        s0 = (RL ? zL : z1) + (size_t)g * b * R;
    } else if (RL) {
        s0 = slice(level, 2 * (int64_t)g);
        s1 = s0 + R * R;
    } else {
        s0 = slice(level, ((int64_t)(A << 1) << level) | B);
        s1 = slice(level, ((int64_t)(A << 1 | 1) << level) | B);
    }
    auto at = [&](int x) -> double2* { return leaf || x < R * R ? s0 + x : s1 + (x - R * R); };
    // element x of the group: its place in M; from the right the slices enter conjugate-transposed
    auto put = [&](int x) -> double2& {
        if (!RL || leaf) return M[x % R][x / R];
        const int t = x % (R * R);
        return M[t / R][t % R + (x < R * R ? 0 : R)];
    };
    const double cj = RL && !leaf ? -1.0 : 1.0;
    for (int x = gl; x < nrows * R; x += GS) {
        const double2 v = live ? *at(x) : d2(0.0, 0.0);
        put(x) = d2(v.x, cj * v.y);
    }
    // the lines of the two neighbour slices, or the rows of a leaf block
    const bool rows = RL ? (leaf ? L == 0 : level == 1) : (leaf ? L == 0 : level == L);
    double2* rowp = nullptr;
    int64_t nr = 0;
    Line<R> t;
    double2* line = nullptr;
    if (rows) {
        rowp = (RL ? z1 : zL) + (L == 0 ? 0 : (size_t)(RL ? g : B) * b * R);
        nr = L == 0 ? n : b;
    } else if (live && gl < 2 * R) {
        const int c = gl / R, x = gl % R;
        if (RL) {
            const int m = level;
            line = (leaf ? slice(L, ((int64_t)c << L) | g)
                         : slice(m - 1, ((int64_t)(g >> (m - 1)) << m) | ((int64_t)c << (m - 1)) |
                                            (g & ((1 << (m - 1)) - 1)))) + x * R;
        } else {
            line = slice(level + 1, leaf ? 2 * (int64_t)g + c : ((int64_t)A << (level + 1)) | (B << 1 | c)) + x;
        }
        t.load(line, RL ? 1 : R);
    }
    __syncwarp();
    group_qr<R>(M, Rs[h], cs[h], nrows, gl);
    if (!live) return;
    for (int x = gl; x < nrows * R; x += GS) {
        const double2 v = put(x);
        *at(x) = d2(v.x, cj * v.y);
    }
    if (rows) {
        if (RL && !leaf) rows_times<R, true>(rowp, nr, Rs[h], gl, GS);
        else rows_times<R, false>(rowp, nr, Rs[h], gl, GS);
    } else if (line) {
        if (RL && !leaf) t.template times<true>(Rs[h], line, 1);
        else t.template times<false>(Rs[h], line, RL ? 1 : R);
    }
}

// The leaf level of k_qr_level for blocks of any number of rows (b).
template <int R, bool RL>
__global__ void __launch_bounds__(128)
k_qr_leaf(double2* __restrict__ z1, double2* __restrict__ Z, double2* __restrict__ zL, int64_t n, int L, int b,
          int ngroups)
{
    __shared__ double2 Rs[4][R][R];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * 4 + w;
    if (g >= ngroups) return;
    warp_qr<R>((RL ? zL : z1) + (size_t)g * b * R, b, Rs[w], lane);
    if (L == 0) {
        rows_times<R, false>(RL ? z1 : zL, n, Rs[w], lane, 32);
    } else if (lane < 2 * R) {
        const int64_t S = (int64_t)1 << (L + 1);
        const int c = lane / R, x = lane % R;
        const int64_t k = RL ? ((int64_t)c << L) | g : 2 * (int64_t)g + c;
        double2* line = Z + ((size_t)(RL ? L - 1 : 0) * S + k) * R * R + (RL ? x * R : x);
        Line<R> t;
        t.load(line, RL ? 1 : R);
        t.template times<false>(Rs[w], line, RL ? 1 : R);
    }
}

// One level; leaf blocks of up to 32 rows and every middle level (2r <= 24
// rows) fit the shared-memory kernel.
template <int R, bool RL>
cudaError_t qr_one(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, int level, cudaStream_t st)
{
    const bool leaf = level == (RL ? L + 1 : 0);
    const int bb = L == 0 ? (int)n : b;
    const int g = !leaf ? 1 << L : L == 0 ? 1 : (int)(n / b);
    if (leaf && bb > QrCfg<R>::ROWS)
        k_qr_leaf<R, RL><<<(g + 3) / 4, 128, 0, st>>>(z1, Z, zL, n, L, bb, g);
    else
        k_qr_level<R, RL><<<(g + QrCfg<R>::GPW - 1) / QrCfg<R>::GPW, 32, 0, st>>>(z1, Z, zL, n, L, bb, level, g);
    return cudaGetLastError();
}

template <int R>
cudaError_t rl_all(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, cudaStream_t st)
{
    for (int m = L + 1; m >= 1; --m) {
        const cudaError_t e = qr_one<R, true>(z1, Z, zL, n, L, b, m, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int R>
cudaError_t canon_one(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, int level, cudaStream_t st)
{
    return qr_one<R, false>(z1, Z, zL, n, L, b, level, st);
}

template <int R>
cudaError_t canon_all(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, cudaStream_t st)
{
    for (int m = 0; m <= L; ++m) {
        const cudaError_t e = qr_one<R, false>(z1, Z, zL, n, L, b, m, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

#define BFC_GAUGE_DISPATCH(FN, ...)                 \
    switch (r) {                                    \
    case 1: return FN<1>(__VA_ARGS__);              \
    case 2: return FN<2>(__VA_ARGS__);              \
    case 3: return FN<3>(__VA_ARGS__);              \
    case 4: return FN<4>(__VA_ARGS__);              \
    case 5: return FN<5>(__VA_ARGS__);              \
    case 6: return FN<6>(__VA_ARGS__);              \
    case 7: return FN<7>(__VA_ARGS__);              \
    case 8: return FN<8>(__VA_ARGS__);              \
    case 9: return FN<9>(__VA_ARGS__);              \
    case 10: return FN<10>(__VA_ARGS__);            \
    case 11: return FN<11>(__VA_ARGS__);            \
    case 12: return FN<12>(__VA_ARGS__);            \
    default: return cudaErrorInvalidValue;          \
    }

cudaError_t launch_canonicalize(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, int r, cudaStream_t st)
{
    BFC_GAUGE_DISPATCH(canon_all, z1, Z, zL, n, L, b, st)
}

cudaError_t launch_canon_level(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, int r, int level,
                               cudaStream_t st)
{
    BFC_GAUGE_DISPATCH(canon_one, z1, Z, zL, n, L, b, level, st)
}

cudaError_t launch_rl_orthogonalize(double2* z1, double2* Z, double2* zL, int64_t n, int L, int b, int r,
                                    cudaStream_t st)
{
    BFC_GAUGE_DISPATCH(rl_all, z1, Z, zL, n, L, b, st)
}

}  // namespace bfc
