// helm_dense.cu - exact solve of one coarse multigrid level by its dense inverse.
//
// Below the grid levels the shifted-Laplace cycle needs an (approximate) solve
// of a small coarse system M_d e = f. With few right-hand sides, running the
// levels under d as a multigrid cycle inside one block is a chain of dozens of
// dependent shared-memory passes on one SM. Instead the level d whose node
// count is at most kDenseMaxPoints is solved exactly: its Galerkin matrix M_d
// (complex symmetric, 9-point) is inverted once per distinct (model, frequency)
// when the solve starts, and every cycle applies the inverse with one
// matrix-vector kernel spread over the GPU.
//
// The inversion eliminates the grid's rows (or columns) block by block, without
// pivoting. That is safe here: M_d = G_d - (b1 - j b2) (h omega)^2 K_d with G_d and K_d
// real symmetric positive definite (Galerkin products P^T G P and P^T K P of the 5-point or
// flux-form Laplacian and of diag(m^2)), so for b2 != 0 the imaginary part of
// x^H M_d x is b2 (h omega)^2 x^H K_d x != 0 for every x != 0: the field of
// values of M_d, and of every principal block and every Schur complement the
// elimination forms, excludes 0, and no pivot can vanish. A non-finite or
// vanishing pivot is still checked and reported, and the solver then uses the
// multigrid tail in place of the dense solve.
#include <algorithm>

#include "helm_internal.h"
#include "helm_solver.h"

namespace helm {

namespace {

// G and K of entry (i, j) of the level's shifted-Laplace matrix G - hw (b1 - j b2) K: the
// coefficient of u_j in (M u)_i. Stored forward entries: east (1,0), north (0,1), north-east (1,1) and
// north-west (-1,1) at the node they start from; the reverse direction reads the
// entry stored at the other node (M is symmetric).
__device__ __forceinline__ double2 gal_raw(const double* __restrict__ gk, size_t n, int nx, int i, int j) {
    const int ix = i % nx, iz = i / nx, jx = j % nx, jz = j / nx;
    const int dx = jx - ix, dz = jz - iz;
    int ent, at;
    if (dx == 0 && dz == 0) { ent = 0; at = i; }
    else if (dz == 0) { ent = 1; at = dx > 0 ? i : j; }
    else if (dx == 0) { ent = 2; at = dz > 0 ? i : j; }
    else if (dx == dz) { ent = 3; at = dx > 0 ? i : j; }
    else { ent = 4; at = dz > 0 ? i : j; }
    return make_double2(__ldg(gk + (size_t)ent * n + at), __ldg(gk + (size_t)(5 + ent) * n + at));
}

// Block-tridiagonal inversion. Ordered by the grid's rows (or columns), M_d is block
// tridiagonal with nb blocks of w x w nodes, tridiagonal couplings U_k between
// consecutive blocks, and symmetric. With the Schur complements of elimination from
// the first block down and from the last block up,
//   Delta_0 = A_0,          Delta_{k+1} = A_{k+1} - U_k^T Delta_k^-1 U_k,
//   Sigma_{nb-1} = A_{nb-1}, Sigma_{k-1} = A_{k-1} - U_{k-1} Sigma_k^-1 U_{k-1}^T,
// the inverse G has G_jj = (Delta_j + Sigma_j - A_j)^-1 and G_ij = -Delta_i^-1 U_i G_{i+1,j}
// for i < j; G_ji = G_ij^T. That is n^2 w operations in place of n^3, and its serial
// part is n pivots of a w x w matrix held in one block's registers (one block barrier
// each), in place of n / 8 strip steps with a grid barrier each. On the 1024-node
// level of a 1041 x 1041 grid (complex64) the three launches take 242 us where a strip
// elimination of the whole matrix took 2843 us; on 690 nodes in complex128, bound by the
// FP64 rate and latency of the two SMs that run the chains, 2.0 ms instead of 8.2 ms. Its
// error in complex64 is that of the strip elimination (2-norm, five levels of 441 to 1024
// nodes: 1.8e-7 .. 2.7e-7 against 2.0e-7 .. 2.7e-7).
//
// No workspace: until the last launch the block upper triangle of minv holds
// W_i = Delta_i^-1 U_i (i < nb - 1), Delta_1 .. Delta_{nb-1} and Sigma_0 .. Sigma_{nb-2},
// 3 (nb - 1) blocks, which fit there for nb >= 6; k_dense_columns writes the block
// lower triangle and the diagonal, and k_dense_mirror overwrites the upper one.
struct TriShape {
    int nx, nz, w, nb, alongx;   // alongx: a block is a column of the grid (x fixed), else a row
    __device__ __forceinline__ int node(int k, int p) const { return alongx ? p * nx + k : k * nx + p; }
    __device__ __forceinline__ int block(int i) const { return alongx ? i % nx : i / nx; }
    // element (p, q) of block (ab.x, ab.y) as an index into minv
    __device__ __forceinline__ unsigned at(int2 ab, int p, int q) const {
        return (unsigned)node(ab.x, p) * (unsigned)(nx * nz) + (unsigned)node(ab.y, q);
    }
    // scratch block t: the pairs (a, b), a < b, row by row
    __device__ __forceinline__ int2 scratch(int t) const {
        int a = 0, len = nb - 1;
        while (t >= len) { t -= len; ++a; --len; }
        return make_int2(a, a + 1 + t);
    }
};
constexpr int kTriMinBlocks = 6;
constexpr int kTriMaxW = 36;      // shared tiles of the widest instance (48 KB limit in complex128)
constexpr int kTriThreads = 256;  // 16 x 16, each thread RT x RT elements of the w x w matrix
constexpr int kTriCols = 8;       // columns of a block column per block of k_dense_columns

// 1 / det of a pivot block; false if it vanishes or is not finite. Float: |det|^2 inverted by one
// Newton step x + x (1 - d x) on the approximate reciprocal; an IEEE divide behind its range
// test costs every step (284 against 226 us for the 1024-node level), and so does scaling each
// determinant (271 us). The range left, |det| within 1e-18 .. 3e18, is that of pivots within nine
// decimal orders of 1, and the matrix is scaled for it (tri_scale). Double: the divide (Newton
// steps from a float seed measured the same).
__device__ __forceinline__ bool pivot_inv(cx<float> det, cx<float>& inv) {
    const float d = det.re * det.re + det.im * det.im;
    float x = __fdividef(1.0f, d);
    x = fmaf(x, fmaf(-d, x, 1.0f), x);
    inv = cx<float>(det.re * x, -det.im * x);
    return d > 1e-37f && d < 1e37f;
}
__device__ __forceinline__ bool pivot_inv(cx<double> det, cx<double>& inv) {
    const double d = det.re * det.re + det.im * det.im, id = 1.0 / d;
    inv = cx<double>(det.re * id, -det.im * id);
    return d > 0.0 && isfinite(d);
}
// The power of two that brings the level's first diagonal entry near 1: the matrix is inverted
// scaled by it (exactly), so the frequency's magnitude does not eat the pivots' range.
__device__ __forceinline__ double tri_scale(const double* __restrict__ gk, size_t n, double hb1, double hb2) {
    const double g = __ldg(gk), q = __ldg(gk + 5 * n);
    const double v = fmax(fabs(g - hb1 * q), fabs(hb2 * q));
    return v > 0.0 && isfinite(v) ? exp2(-(double)ilogb(v)) : 1.0;
}

// In-place Gauss-Jordan inversion of a w x w matrix by 2 x 2 pivot blocks without pivoting
// (see the head of this file; half the barriers of single pivots): thread (ti, tj) =
// (tid / 16, tid % 16) holds elements (ti + 16 r, tj + 16 c). Two consecutive pivot rows
// belong to one warp: it takes the pivot block by shuffle, inverts it (one division per
// block; a division by every thread would cost the step more than its update in
// complex128), multiplies the two rows by the inverse and publishes them with the
// inverse in the pivot's place; the threads of the two pivot columns publish those and
// clear them, so that one formula a - c0 r0 - c1 r1 updates every other row. Two buffers
// in turn: one barrier a step. An odd w is padded with a unit diagonal element.
// Returns false (in some thread) if a pivot block was singular or not finite.
template <typename T, int RT>
__device__ __forceinline__ bool gj_invert(cx<T> (&a)[RT][RT], int w, int ti, int tj, cx<T> (*srow)[2][16 * RT],
                                          cx<T> (*scol)[2][16 * RT]) {
    bool ok = true;
    if (w & 1)
#pragma unroll
        for (int r = 0; r < RT; ++r)
            if (ti + 16 * r == w && tj == ti) a[r][r] = cx<T>(1, 0);
    const int half = ti & 1;
#pragma unroll
    for (int kr = 0; kr < RT; ++kr) {
        for (int kk = 0; kk < 16; kk += 2) {
            const int k = 16 * kr + kk, buf = (k >> 1) & 1;
            if (k >= w) break;
            if ((ti & ~1) == kk) {   // the warp of the pivot rows (uniform)
                auto from = [&](int src) {
                    return cx<T>(__shfl_sync(0xffffffffu, a[kr][kr].re, src), __shfl_sync(0xffffffffu, a[kr][kr].im, src));
                };
                const cx<T> p00 = from(kk), p01 = from(kk + 1), p10 = from(16 + kk), p11 = from(17 + kk);
                const cx<T> det = p00 * p11 - p01 * p10;
                cx<T> di;
                ok = pivot_inv(det, di) && ok;
                // this half-warp's row of the inverse: row 0 is (p11, -p01) / det, row 1 (-p10, p00) / det
                const cx<T> q0 = half ? cx<T>(-p10.re, -p10.im) : p11, q1 = half ? p00 : cx<T>(-p01.re, -p01.im);
                const cx<T> i0 = di * q0, i1 = di * q1;
#pragma unroll
                for (int c = 0; c < RT; ++c) {
                    const cx<T> own = a[kr][c];
                    const cx<T> oth(__shfl_xor_sync(0xffffffffu, own.re, 16), __shfl_xor_sync(0xffffffffu, own.im, 16));
                    cx<T> v = i0 * (half ? oth : own) + i1 * (half ? own : oth);
                    if (c == kr && tj == kk) v = i0;
                    if (c == kr && tj == kk + 1) v = i1;
                    srow[buf][half][tj + 16 * c] = v;
                }
            }
            if ((tj & ~1) == kk)
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    scol[buf][tj & 1][ti + 16 * r] = a[r][kr];
                    a[r][kr] = cx<T>(0, 0);
                }
            __syncthreads();
            cx<T> r0[RT], r1[RT];
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                r0[c] = srow[buf][0][tj + 16 * c];
                r1[c] = srow[buf][1][tj + 16 * c];
            }
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                if ((ti & ~1) + 16 * r >= w) break;   // a warp without rows of the matrix (uniform)
                const cx<T> c0 = scol[buf][0][ti + 16 * r], c1 = scol[buf][1][ti + 16 * r];
                const bool prow = r == kr && (ti & ~1) == kk;
#pragma unroll
                for (int c = 0; c < RT; ++c) {
                    const cx<T> v = a[r][c] - c0 * r0[c] - c1 * r1[c];
                    a[r][c] = prow ? (half ? r1[c] : r0[c]) : v;
                }
            }
        }
    }
    return ok;
}

// Block x = 0 runs the elimination downwards, x = 1 upwards; blockIdx.y is the slot.
// Each step: invert the block's Schur complement X, W = X C with C the (tridiagonal)
// coupling to the next block, next complement A - C^T W. The next step's entries of C
// and A are loaded before the inversion, which hides their latency.
template <typename T, int RT>
__global__ void __launch_bounds__(kTriThreads) k_dense_chain(TriShape sh, const double* __restrict__ gkall,
                                                             size_t gkstride, const double* __restrict__ w2s,
                                                             const int* __restrict__ mods, double b1, double b2,
                                                             T* __restrict__ minv, int* err) {
    constexpr int WM = 16 * RT, WS = WM < kTriMaxW ? WM : kTriMaxW;
    __shared__ cx<T> srow[2][2][WM], scol[2][2][WM];
    __shared__ cx<T> Xs[WS][WS + 1];         // X, then W
    __shared__ cx<T> Cs[3][WM], As[3][WM];   // [d][q]: entry (q + d - 1, q)
    const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
    const int w = sh.w, nb = sh.nb, n = sh.nx * sh.nz;
    const bool up = blockIdx.x == 1;
    const double hw = w2s[blockIdx.y], hb1 = hw * b1, hb2 = hw * b2;
    const double* gk = gkall + (size_t)mods[blockIdx.y] * gkstride;
    T* out = minv + 2 * (size_t)n * n * blockIdx.y;
    const double sc = tri_scale(gk, (size_t)n, hb1, hb2);
    auto form = [&](double2 e) { return cx<T>((T)(sc * (e.x - hb1 * e.y)), (T)(sc * (hb2 * e.y))); };
    auto raw = [&](int kr, int r, int kc, int q) -> double2 {
        if (r < 0 || r >= w) return make_double2(0.0, 0.0);
        return gal_raw(gk, (size_t)n, sh.nx, sh.node(kr, r), sh.node(kc, q));
    };
    cx<T> a[RT][RT];
    const int k0 = up ? nb - 1 : 0;
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < RT; ++c) {
            const int i = ti + 16 * r, j = tj + 16 * c;
            a[r][c] = (i < w && j < w && i - j <= 1 && j - i <= 1) ? form(raw(k0, i, k0, j)) : cx<T>(0, 0);
        }
    const int ed = tid / WM, eq = tid - ed * WM;   // this thread's entry of C and A (tid < 3 WM <= 144)
    bool ok = true;
    for (int s = 0; s < nb - 1; ++s) {
        const int k = up ? nb - 1 - s : s, kn = up ? k - 1 : k + 1;
        double2 ce = make_double2(0.0, 0.0), ae = ce;
        if (ed < 3 && eq < w) {
            ce = raw(k, eq + ed - 1, kn, eq);
            ae = raw(kn, eq + ed - 1, kn, eq);
        }
        ok = gj_invert<T, RT>(a, w, ti, tj, srow, scol) && ok;
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                const int i = ti + 16 * r, j = tj + 16 * c;
                if (i < w && j < w) Xs[i][j] = a[r][c];
            }
        if (ed < 3) { Cs[ed][eq] = form(ce); As[ed][eq] = form(ae); }
        __syncthreads();
        const int2 bw = sh.scratch(s);
        // W = X C
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                const int i = ti + 16 * r, j = tj + 16 * c;
                cx<T> v(0, 0);
                if (i < w && j < w) {
                    v = Xs[i][j] * Cs[1][j];
                    if (j > 0) v = v + Xs[i][j - 1] * Cs[0][j];
                    if (j + 1 < w) v = v + Xs[i][j + 1] * Cs[2][j];
                    if (!up) stc(out, sh.at(bw, i, j), v);
                }
                a[r][c] = v;
            }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                const int i = ti + 16 * r, j = tj + 16 * c;
                if (i < w && j < w) Xs[i][j] = a[r][c];
            }
        __syncthreads();
        // next Schur complement A - C^T W, kept and published (Delta_{s+1}; Sigma_{nb-2-s})
        const int2 bs = sh.scratch(up ? 2 * (nb - 1) + kn : (nb - 1) + s);
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < RT; ++c) {
                const int i = ti + 16 * r, j = tj + 16 * c;
                cx<T> v(0, 0);
                if (i < w && j < w) {
                    const int d = i - j + 1;
                    if (d >= 0 && d <= 2) v = As[d][j];
                    v = v - Cs[1][i] * Xs[i][j];
                    if (i > 0) v = v - Cs[0][i] * Xs[i - 1][j];
                    if (i + 1 < w) v = v - Cs[2][i] * Xs[i + 1][j];
                    stc(out, sh.at(bs, i, j), v);
                }
                a[r][c] = v;
            }
        __syncthreads();   // Xs, Cs and As are rewritten by the next step
    }
    if (!ok) atomicExch(err, 2);
}

// Block column j = blockIdx.x, its columns c0 .. c0 + kTriCols - 1 (blockIdx.y),
// slot blockIdx.z: G_jj from the two Schur complements (inverted in every block of the
// column: w pivots are cheaper than another launch), then G_ij = -W_i G_{i+1,j} for
// i = j - 1 .. 0 in shared memory, the next W_i on its way while this one is used.
// G_ij is written as G_ji = G_ij^T, in the block lower triangle.
template <typename T, int RT>
__global__ void __launch_bounds__(kTriThreads) k_dense_columns(TriShape sh, const double* __restrict__ gkall,
                                                               size_t gkstride, const double* __restrict__ w2s,
                                                               const int* __restrict__ mods, double b1, double b2,
                                                               T* minv, int* err) {
    constexpr int WM = 16 * RT, WS = WM < kTriMaxW ? WM : kTriMaxW;
    constexpr int NP = (WS * WS + kTriThreads - 1) / kTriThreads, NY = WS * kTriCols;
    __shared__ cx<T> srow[2][2][WM], scol[2][2][WM];
    __shared__ cx<T> Wb[WS][WS + 1];
    __shared__ cx<T> Y[2][WS][kTriCols + 1];
    const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
    const int w = sh.w, nb = sh.nb, n = sh.nx * sh.nz;
    // the long chains first: a block column's work grows with j
    const int j = nb - 1 - blockIdx.x, c0 = blockIdx.y * kTriCols, cw = min(kTriCols, w - c0);
    const double hw = w2s[blockIdx.z];
    const double* gk = gkall + (size_t)mods[blockIdx.z] * gkstride;
    const double sc = tri_scale(gk, (size_t)n, hw * b1, hw * b2);
    T* out = minv + 2 * (size_t)n * n * blockIdx.z;
    const int2 bd = j > 0 ? sh.scratch((nb - 1) + j - 1) : make_int2(0, 0);
    const int2 bu = j < nb - 1 ? sh.scratch(2 * (nb - 1) + j) : make_int2(0, 0);
    cx<T> a[RT][RT];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < RT; ++c) {
            const int p = ti + 16 * r, q = tj + 16 * c;
            cx<T> v(0, 0);
            if (p < w && q < w) {
                if (j > 0) v = ldcc(out, sh.at(bd, p, q));
                if (j < nb - 1) v = v + ldcc(out, sh.at(bu, p, q));
                if (j > 0 && j < nb - 1 && p - q <= 1 && q - p <= 1) {
                    const double2 e = gal_raw(gk, (size_t)n, sh.nx, sh.node(j, p), sh.node(j, q));
                    v = v - cx<T>((T)(sc * (e.x - hw * b1 * e.y)), (T)(sc * (hw * b2 * e.y)));
                }
            }
            a[r][c] = v;
        }
    cx<T> wn[NP];   // the next W_i, in flight
    auto fetch = [&](int i) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int e = tid + k * kTriThreads, p = e / WS, q = e - p * WS;
            wn[k] = (i >= 0 && p < w && q < w) ? ldcc(out, sh.at(make_int2(0, i + 1), p, q)) : cx<T>(0, 0);
        }
    };
    fetch(j - 1);
    if (!gj_invert<T, RT>(a, w, ti, tj, srow, scol)) atomicExch(err, 2);
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < RT; ++c) {
            a[r][c] = (T)sc * a[r][c];   // the inverse of the unscaled matrix
            const int p = ti + 16 * r, q = tj + 16 * c - c0;
            if (p < w && q >= 0 && q < kTriCols) {
                Y[0][p][q] = a[r][c];
                if (q < cw) stc(out, sh.at(make_int2(j, j), p, q + c0), a[r][c]);
            }
        }
    int cur = 0;
    for (int i = j - 1; i >= 0; --i, cur ^= 1) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int e = tid + k * kTriThreads;
            if (e < WS * WS) Wb[e / WS][e % WS] = wn[k];
        }
        __syncthreads();
        fetch(i - 1);
#pragma unroll
        for (int k = 0; k < (NY + kTriThreads - 1) / kTriThreads; ++k) {
            const int e = tid + k * kTriThreads, p = e / kTriCols, q = e % kTriCols;
            if (e < NY && p < w) {
                cx<T> s0(0, 0), s1(0, 0);
                int r = 0;
                for (; r + 1 < w; r += 2) {
                    s0 = s0 + Wb[p][r] * Y[cur][r][q];
                    s1 = s1 + Wb[p][r + 1] * Y[cur][r + 1][q];
                }
                if (r < w) s0 = s0 + Wb[p][r] * Y[cur][r][q];
                const cx<T> v(-(s0.re + s1.re), -(s0.im + s1.im));
                Y[cur ^ 1][p][q] = v;
                if (q < cw) stc(out, sh.at(make_int2(j, i), q + c0, p), v);
            }
        }
        __syncthreads();
    }
}

// minv[r][c] = minv[c][r] for the elements of the block upper triangle (block of r
// before block of c): tiles of 32 x 32, read along rows and written along rows.
template <typename T>
__global__ void __launch_bounds__(256) k_dense_mirror(TriShape sh, T* minv) {
    __shared__ cx<T> t[32][33];
    const int n = sh.nx * sh.nz;
    T* out = minv + 2 * (size_t)n * n * blockIdx.z;
    const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;   // the tile that is written
    if (!sh.alongx && sh.block(r0) >= sh.block(min(c0 + 31, n - 1))) return;   // wholly on or below the diagonal
    for (int y = ly; y < 32; y += 8) {
        const int r = c0 + y, c = r0 + lx;   // read the transposed tile; only its lower elements are used
        if (r < n && c < n && sh.block(c) < sh.block(r)) t[y][lx] = ldcc(out, (size_t)r * n + c);
    }
    __syncthreads();
    for (int y = ly; y < 32; y += 8) {
        const int r = r0 + y, c = c0 + lx;
        if (r < n && c < n && sh.block(r) < sh.block(c)) stc(out, (size_t)r * n + c, t[lx][y]);
    }
}

__global__ void k_order() {}

// e_b (+)= M_d^-1 f_b for the right-hand sides of one group (consecutive RHS of
// one slot, group g = [grp[g], grp[g+1])); one warp per row of the inverse, the
// row held in registers (NR complex values per lane) and reused for
// every right-hand side of the group, whose vectors are staged in shared memory.
// Warps per block: as many rows as give every SM a block, at most 8. In FP64 the multiplications bound
// it (a quarter of an SM does one lane in two clocks): 690 rows, two right-hand sides, 41 us in 87 blocks of
// 8 rows with products and sums apart, 23 us in 138 blocks of 5 with fused ones, 16 us with the whole row and
// four values of f in flight per thread; complex64, 966 rows, four right-hand sides, 13.4 -> 12.1 us.
template <typename T, int NR>
__global__ void __launch_bounds__(256) k_coarse_dense(int n, const T* __restrict__ minv, const int* __restrict__ slot,
                                                      const int* __restrict__ grp, int maxg, const T* f, T* e,
                                                      int accumulate, const RhsState* st) {
    extern __shared__ __align__(16) unsigned char cd_smem[];
    cx<T>* fs = reinterpret_cast<cx<T>*>(cd_smem);   // [group][n]
    pdl_trigger_for<T>();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.x * (blockDim.x >> 5) + warp;
    const int g = blockIdx.y;
    const int b0 = grp[g], b1 = grp[g + 1];
    const T* Mr = minv + 2 * ((size_t)slot[b0] * n * n + (size_t)min(row, n - 1) * n);
    static_assert(32 * NR >= kDenseMaxPoints, "a row of the inverse in one warp's registers");
    cx<T> rv[NR];
    // this warp's row is ordered before any early launch (launch_order): load it ahead of the wait
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int j = lane + 32 * k;
        rv[k] = j < n ? ldc(Mr, j) : cx<T>(0, 0);
    }
    pdl_wait();
    const int nb = b1 - b0;
    for (int idx = threadIdx.x; idx < nb * n; idx += 4 * blockDim.x) {   // four loads in flight
        cx<T> q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = idx + k * blockDim.x;
            q[k] = i < nb * n ? ldcc(f, (size_t)b0 * n + i) : cx<T>(0, 0);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = idx + k * blockDim.x;
            if (i < nb * n) fs[i] = q[k];
        }
    }
    __syncthreads();
    if (row >= n) return;
    T are[8], aim[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) { are[r] = T(0); aim[r] = T(0); }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        if (r >= nb) break;
        const cx<T>* fv = fs + (size_t)r * n;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const int j = lane + 32 * k;
            if (j < n) {
                const cx<T> v = fv[j];
                are[r] = fma(-rv[k].im, v.im, fma(rv[k].re, v.re, are[r]));
                aim[r] = fma(rv[k].im, v.re, fma(rv[k].re, v.im, aim[r]));
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        if (r >= nb) break;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            are[r] += __shfl_xor_sync(0xffffffffu, are[r], o);
            aim[r] += __shfl_xor_sync(0xffffffffu, aim[r], o);
        }
        const int b = b0 + r;
        if (lane == 0 && rhs_active(st, b)) {
            cx<T> v(are[r], aim[r]);
            if (accumulate) v = v + ldcc(e, (size_t)b * n + row);
            stc(e, (size_t)b * n + row, v);
        }
    }
    (void)maxg;
}

}  // namespace

// Whether an nx x nz level can be inverted: its blocks (the shorter side) fit the
// register tiles and the block upper triangle holds the scratch blocks. Every level of
// a hierarchy with at most kDenseMaxPoints nodes does (the shorter side is at most 34, and a
// level left by halving a grid of more than 128 nodes has at least 6 on its longer side).
bool dense_invert_fits(int nx, int nz) {
    return nx * nz <= kDenseMaxPoints && std::min(nx, nz) <= kTriMaxW && std::max(nx, nz) >= kTriMinBlocks;
}

void launch_order(cudaStream_t s) {
    k_order<<<1, 32, 0, s>>>();
    count_launches(1);
}

template <typename T, int RT>
static void dense_invert_rt(const TriShape& sh, const double* gk, size_t gks, const double* w2s, const int* mods,
                            int nslots, double b1, double b2, T* minv, int* err, cudaStream_t s) {
    const int n = sh.nx * sh.nz, nt = (n + 31) / 32;
    k_dense_chain<T, RT><<<dim3(2, nslots), kTriThreads, 0, s>>>(sh, gk, gks, w2s, mods, b1, b2, minv, err);
    k_dense_columns<T, RT><<<dim3(sh.nb, (sh.w + kTriCols - 1) / kTriCols, nslots), kTriThreads, 0, s>>>(
        sh, gk, gks, w2s, mods, b1, b2, minv, err);
    k_dense_mirror<T><<<dim3(nt, nt, nslots), 256, 0, s>>>(sh, minv);
    count_launches(3);
}

// Inverts M_d of every slot (distinct model and (h omega)^2) into minv
// [nslots][n][n] in the kernel's precision; err: one int, 0 on success, 2 on a
// vanishing or non-finite pivot. No synchronisation.
// Blocks run along the shorter side of the grid: the serial part is n pivots in either
// case, and a pivot's work grows with the square of the block.
template <typename T>
cudaError_t launch_dense_invert(const LevelDev& Ld, const double* w2s, const int* mods, int nslots, double b1,
                                double b2, T* minv, int* err, cudaStream_t s, bool order) {
    cudaError_t e = cudaMemsetAsync(err, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    const double n = (double)Ld.nx * Ld.nz;
    ProfScope prof(PK_DENSE_INVERT, Ld.nx, Ld.nz, n * n * nslots * 2.0 * sizeof(T), s);
    TriShape sh;
    sh.nx = Ld.nx;
    sh.nz = Ld.nz;
    sh.alongx = Ld.nx > Ld.nz;
    sh.w = std::min(Ld.nx, Ld.nz);
    sh.nb = std::max(Ld.nx, Ld.nz);
    const double* gk = static_cast<const double*>(Ld.gk);
    if (sh.w <= 16) dense_invert_rt<T, 1>(sh, gk, Ld.gkstride, w2s, mods, nslots, b1, b2, minv, err, s);
    else if (sh.w <= 32) dense_invert_rt<T, 2>(sh, gk, Ld.gkstride, w2s, mods, nslots, b1, b2, minv, err, s);
    else dense_invert_rt<T, 3>(sh, gk, Ld.gkstride, w2s, mods, nslots, b1, b2, minv, err, s);
    if (order) launch_order(s);
    return cudaGetLastError();
}
template cudaError_t launch_dense_invert<float>(const LevelDev&, const double*, const int*, int, double, double,
                                                float*, int*, cudaStream_t, bool);
template cudaError_t launch_dense_invert<double>(const LevelDev&, const double*, const int*, int, double, double,
                                                 double*, int*, cudaStream_t, bool);

template <typename T>
void launch_coarse_dense(int n, const T* minv, const int* slot, const int* grp, int ngroups, int maxg, const T* f,
                         T* e, int accumulate, const RhsState* st, cudaStream_t s) {
    constexpr int NR = (kDenseMaxPoints + 31) / 32;   // a row fits the registers, so that all of it is loaded ahead
    // the inverse of each group's slot once per group, f read and e written (and read when accumulating)
    ProfScope prof(PK_COARSE_DENSE, n, 1,
                   ((double)n * n * ngroups + (double)n * (2 + accumulate) * ngroups * maxg) * 2.0 * sizeof(T), s);
    const size_t smem = (size_t)maxg * n * sizeof(T) * 2;
    static const bool attr = [] {
        cudaFuncSetAttribute(k_coarse_dense<T, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        return true;
    }();
    (void)attr;
    const int warps = std::min(8, std::max(1, (int)(((size_t)n * ngroups + 151) / 152)));
    launch_pdl(k_coarse_dense<T, NR>, dim3((n + warps - 1) / warps, ngroups), dim3(32 * warps), smem, s, n, minv, slot, grp, maxg, f, e,
               accumulate, st);
}
template void launch_coarse_dense<float>(int, const float*, const int*, const int*, int, int, const float*, float*,
                                         int, const RhsState*, cudaStream_t);
template void launch_coarse_dense<double>(int, const double*, const int*, const int*, int, int, const double*,
                                          double*, int, const RhsState*, cudaStream_t);

}  // namespace helm
