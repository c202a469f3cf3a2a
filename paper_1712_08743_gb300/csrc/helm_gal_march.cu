// helm_gal_march.cu - Galerkin multigrid levels for large batches (complex64): each
// warp marches down the rows of one right-hand side with every field in registers.
//
// With many right-hand sides the one-tile-per-block kernels of helm_gal_tiles.cuh are
// bound by shared memory: each of their 9-point evaluations reads nine staged complex
// coefficients and nine values (144 bytes), and forming a right-hand side's coefficients
// in shared memory costs as much again (ncu, 220 x 120 nodes, 160 right-hand sides:
// the load/store pipe 83 % busy, DRAM at 5 %). Here lane j of a warp owns the fine
// columns 2I and 2I + 1 of coarse column I = I0 + j (the odd one is the coarse node's
// column); the warp walks down the rows, holding u of two rows and the partly summed
// residual of the next one. Each stored coefficient is read once per warp and used
// for both nodes it couples: row z's coefficients finish row z (its own row and the row
// below it) and start row z + 1 (their transposes). Neighbours across a lane boundary,
// fields and coefficients, come by shuffle. The warps of a block take consecutive
// right-hand sides of one tile, so that the model's coefficients come from L1 after the
// first of them.
//
// Where the density is constant, G is the same 9-point stencil at every node off the
// grid's border (LevelDev::g0): such warps read only K, 20 of the 40 bytes per node.
//
// Measured per launch in the batched 441 x 241 solve (320 right-hand sides, converged ones
// leaving as it goes; 220 x 120 nodes, then 110 x 60), tile kernels that staged the real
// coefficients for four right-hand sides per block -> these: restriction 101 -> 42 us and
// 34 -> 17 us, with a coarse correction 35 -> 18 us, prolongation 89 -> 44 us and 31 -> 17 us.
// They are now bound by issue and the load pipe (odd row lengths keep loads at 8 bytes).
#include <algorithm>

#include "helm_gal_tiles.cuh"
#include "helm_internal.h"

namespace helm {

namespace {

enum GalMode : int { GM_RESTRICT = 0, GM_CORRECT = 1, GM_PROLONG = 2 };

constexpr int kGmWarps = 4;    // right-hand sides (one per warp) of a tile in a block
constexpr int kGmBlocks = 3;   // resident blocks asked of the compiler: 170 registers, no spills; 4 and 5
                               // blocks measured 44 -> 48 and 119 us (level 1 prolongation), 8 warps 57 us
constexpr int kGmCols = 30;    // coarse columns a warp writes (lanes 1 .. 30)

__device__ __forceinline__ cx<float> up1(cx<float> a) {
    return cx<float>(__shfl_up_sync(0xffffffffu, a.re, 1), __shfl_up_sync(0xffffffffu, a.im, 1));
}
__device__ __forceinline__ cx<float> dn1(cx<float> a) {
    return cx<float>(__shfl_down_sync(0xffffffffu, a.re, 1), __shfl_down_sync(0xffffffffu, a.im, 1));
}

// One row of a lane's two columns as loaded: right-hand side, K and (LOADG) G entries
// (centre, east, north, north-east, north-west).
template <bool LOADG>
struct GmRow {
    cx<float> f0, f1;
    float k0[5], k1[5];
    float g0[LOADG ? 5 : 1], g1[LOADG ? 5 : 1];
};
// ... and as computed: u, the residual's start, wj D^-1
struct GmVal {
    cx<float> u0, u1, uw, ue;   // own columns, the neighbours at 2I - 1 and 2I + 2
    cx<float> d0, d1;           // prolongation: wj D^-1
};

// The march over fine rows. Restriction: coarse rows [A0, A1) are written. Prolongation: fine
// rows [A0, A1), A0 even. LOADG: G is read (a density level, or a warp that touches the
// border); EDGE: rows or columns outside the grid occur.
template <int MODE, bool LOADG, bool EDGE>
__device__ __forceinline__ void gal_march(const LevelDev& Lf, const LevelDev& Lc, int I, int lane, int A0, int A1,
                                          float hb1, float hb2, float wj, const float* __restrict__ fb,
                                          const float* __restrict__ gk, const float* __restrict__ eb,
                                          float* __restrict__ ob, int accumulate) {
    const int nx = Lf.nx, nz = Lf.nz, cnx = Lc.nx, cnz = Lc.nz;
    const int n = nx * nz;
    const int c0 = 2 * I;
    const float omw = 1.0f - wj;
    const bool in0 = !EDGE || (c0 >= 0 && c0 < nx), in1 = !EDGE || (c0 + 1 >= 0 && c0 + 1 < nx);
    const float gcc = Lf.g0[0], gce = Lf.g0[1], gca = Lf.g0[2];

    auto ld = [&](int z) {
        GmRow<LOADG> r;
        const bool zin = !EDGE || (z >= 0 && z < nz);
        const bool a = zin && in0, b = zin && in1;
        const int i = z * nx + c0;
        r.f0 = a ? ldc(fb, i) : cx<float>(0, 0);
        r.f1 = b ? ldc(fb, i + 1) : cx<float>(0, 0);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const float* K = gk + (size_t)(5 + k) * n;
            r.k0[k] = a ? __ldg(K + i) : 0.0f;
            r.k1[k] = b ? __ldg(K + i + 1) : 0.0f;
            if constexpr (LOADG) {
                const float* G = gk + (size_t)k * n;
                // outside the grid the centre is 1: D^-1 stays finite where u is set to zero
                r.g0[k] = a ? __ldg(G + i) : (k == 0 ? 1.0f : 0.0f);
                r.g1[k] = b ? __ldg(G + i + 1) : (k == 0 ? 1.0f : 0.0f);
            }
        }
        return r;
    };
    auto coef = [&](float g, float q) { return cx<float>(g - hb1 * q, hb2 * q); };
    auto gof = [&](const GmRow<LOADG>& r, int col, int k) -> float {
        if constexpr (LOADG) return col ? r.g1[k] : r.g0[k];
        else return k == 0 ? gcc : (k < 3 ? gce : gca);
    };
    const bool ein = !EDGE || (I >= 0 && I < cnx);
    auto erow = [&](int K) -> cx<float> {
        if constexpr (MODE == GM_RESTRICT) return cx<float>(0, 0);
        const bool ok = ein && (!EDGE || (K >= 0 && K < cnz));
        return ok ? ldc(eb, (size_t)K * cnx + I) : cx<float>(0, 0);
    };
    // u of row z and the start of its residual: (1 - wj) f (- D P e) or f; ev: P e's coarse row
    auto prep = [&](int z, const GmRow<LOADG>& r, cx<float> ev, GmVal& v, cx<float>& s0, cx<float>& s1) {
        const cx<float> D0 = coef(gof(r, 0, 0), r.k0[0]), D1 = coef(gof(r, 1, 0), r.k1[0]);
        auto winv = [&](cx<float> D) {
            const float sc = wj * rcp_fast(D.re * D.re + D.im * D.im);
            return cx<float>(sc * D.re, -sc * D.im);
        };
        const cx<float> w0 = winv(D0), w1 = winv(D1);
        v.u0 = w0 * r.f0;
        v.u1 = w1 * r.f1;
        if constexpr (MODE == GM_PROLONG) {
            s0 = r.f0;
            s1 = r.f1;
            v.d0 = w0;
            v.d1 = w1;
        } else {
            s0 = omw * r.f0;
            s1 = omw * r.f1;
        }
        if constexpr (MODE != GM_RESTRICT) {
            const cx<float> p0 = 0.5f * (up1(ev) + ev);   // column 2I: the mean of e(I - 1) and e(I)
            v.u0 = v.u0 + p0;
            v.u1 = v.u1 + ev;
            if constexpr (MODE == GM_CORRECT) {
                s0 = s0 - D0 * p0;
                s1 = s1 - D1 * ev;
            }
        }
        if constexpr (EDGE) {
            const bool zin = z >= 0 && z < nz;
            if (!(zin && in0)) v.u0 = cx<float>(0, 0);
            if (!(zin && in1)) v.u1 = cx<float>(0, 0);
        }
        v.uw = up1(v.u1);
        v.ue = dn1(v.u0);
    };
    // with row z's coefficients: finishes row z's residual (o0, o1) and starts row z + 1's (s0, s1)
    auto couple = [&](const GmRow<LOADG>& r, const GmVal& u, const GmVal& v, cx<float>& o0, cx<float>& o1,
                      cx<float>& s0, cx<float>& s1) {
        // east at 2I - 1, north-east at 2I - 1, north-west at 2I + 2
        const float kew = __shfl_up_sync(0xffffffffu, r.k1[1], 1), kaw = __shfl_up_sync(0xffffffffu, r.k1[3], 1);
        const float kbe = __shfl_down_sync(0xffffffffu, r.k0[4], 1);
        float gew = gce, gaw = gca, gbe = gca;
        if constexpr (LOADG) {
            gew = __shfl_up_sync(0xffffffffu, r.g1[1], 1);
            gaw = __shfl_up_sync(0xffffffffu, r.g1[3], 1);
            gbe = __shfl_down_sync(0xffffffffu, r.g0[4], 1);
        }
        const cx<float> E0 = coef(gof(r, 0, 1), r.k0[1]), E1 = coef(gof(r, 1, 1), r.k1[1]), EW = coef(gew, kew);
        const cx<float> N0 = coef(gof(r, 0, 2), r.k0[2]), N1 = coef(gof(r, 1, 2), r.k1[2]);
        const cx<float> A0c = coef(gof(r, 0, 3), r.k0[3]), A1c = coef(gof(r, 1, 3), r.k1[3]), AW = coef(gaw, kaw);
        const cx<float> B0 = coef(gof(r, 0, 4), r.k0[4]), B1 = coef(gof(r, 1, 4), r.k1[4]), BE = coef(gbe, kbe);
        o0 = o0 - E0 * u.u1 - EW * u.uw - N0 * v.u0 - A0c * v.u1 - B0 * v.uw;
        o1 = o1 - E1 * u.ue - E0 * u.u0 - N1 * v.u1 - A1c * v.ue - B1 * v.u0;
        s0 = s0 - N0 * u.u0 - AW * u.uw - B1 * u.u1;
        s1 = s1 - N1 * u.u1 - A0c * u.u0 - BE * u.ue;
    };

    if constexpr (MODE != GM_PROLONG) {
        // restriction: r on rows 2 A0 .. 2 A1, u on one row more at each end
        const bool wr = lane >= 1 && lane <= kGmCols && I < cnx;
        auto hsum = [&](int z, cx<float> r0, cx<float> r1) -> cx<float> {
            if constexpr (EDGE) {
                const bool zin = z < nz;
                if (!(zin && in0)) r0 = cx<float>(0, 0);
                if (!(zin && in1)) r1 = cx<float>(0, 0);
            }
            return (r0 + dn1(r0)) + 2.0f * r1;   // r(2I) + 2 r(2I + 1) + r(2I + 2)
        };
        const int zf = 2 * A0 - 1;
        GmRow<LOADG> R0 = ld(zf), R1 = ld(zf + 1), R2 = ld(zf + 2);
        cx<float> e0 = erow(A0 - 1), e1 = erow(A0);   // of coarse rows A0 - 1, A0
        GmVal ua, ub;
        cx<float> t0, t1, o0, o1, s0, s1;
        prep(zf, R0, e0, ua, t0, t1);
        prep(zf + 1, R1, 0.5f * (e0 + e1), ub, o0, o1);
        couple(R0, ua, ub, t0, t1, o0, o1);
        cx<float> acc(0, 0);
        // at the top of step K: ub is u of row 2K, R1 its coefficients, (o0, o1) its residual
        // started; R2 is row 2K + 1, loaded; e1 is e of coarse row K
        for (int K = A0; K < A1; ++K) {
            const GmRow<LOADG> R3 = ld(2 * K + 2);
            const cx<float> e2 = erow(K + 1);
            prep(2 * K + 1, R2, e1, ua, s0, s1);
            couple(R1, ub, ua, o0, o1, s0, s1);
            const cx<float> h0 = hsum(2 * K, o0, o1);
            if (K > A0) {
                const cx<float> q = acc + h0;
                if (wr) stc(ob, (size_t)(K - 1) * cnx + I, 0.25f * q);
            }
            acc = h0;
            const GmRow<LOADG> R4 = ld(2 * K + 3);
            prep(2 * K + 2, R3, 0.5f * (e1 + e2), ub, o0, o1);
            couple(R2, ua, ub, s0, s1, o0, o1);
            acc = acc + 2.0f * hsum(2 * K + 1, s0, s1);
            R1 = R3;
            R2 = R4;
            e1 = e2;
        }
        // the last row, 2 A1
        prep(2 * A1 + 1, R2, e1, ua, s0, s1);
        couple(R1, ub, ua, o0, o1, s0, s1);
        const cx<float> q = acc + hsum(2 * A1, o0, o1);
        if (wr) stc(ob, (size_t)(A1 - 1) * cnx + I, 0.25f * q);
    } else {
        // prolongation: u2 on rows A0 - 1 .. A1, u3 on rows A0 .. A1 - 1
        const bool outl = lane >= 1 && lane <= kGmCols;
        const bool w0 = outl && in0, w1 = outl && in1;
        auto emit = [&](int z, const GmVal& u, cx<float> o0, cx<float> o1, cx<float> p0, cx<float> p1) {
            if (EDGE && z >= A1) return;
            const int i = z * nx + c0;
            cx<float> q0 = omw * u.u0 + u.d0 * o0, q1 = omw * u.u1 + u.d1 * o1;
            if (accumulate) { q0 = p0 + q0; q1 = p1 + q1; }
            if (w0) stc(ob, i, q0);
            if (w1) stc(ob, i + 1, q1);
        };
        auto ldo = [&](int z, cx<float>& p0, cx<float>& p1) {
            const bool ok = accumulate && z < A1;
            const int i = z * nx + c0;
            p0 = ok && w0 ? ldcc(ob, i) : cx<float>(0, 0);
            p1 = ok && w1 ? ldcc(ob, i + 1) : cx<float>(0, 0);
        };
        const int k0 = A0 / 2;
        GmRow<LOADG> R0 = ld(A0 - 1), R1 = ld(A0), R2 = ld(A0 + 1);
        cx<float> e0 = erow(k0 - 1), e1 = erow(k0);
        GmVal ua, ub;
        cx<float> t0, t1, o0, o1, s0, s1, p0, p1, p2, p3;
        ldo(A0, p0, p1);
        prep(A0 - 1, R0, e0, ua, t0, t1);
        prep(A0, R1, 0.5f * (e0 + e1), ub, o0, o1);
        couple(R0, ua, ub, t0, t1, o0, o1);
        for (int z = A0; z < A1; z += 2) {
            // ub is u2 of row z, R1 its coefficients; R2 is row z + 1, loaded; e1 is e of row z / 2
            const GmRow<LOADG> R3 = ld(z + 2);
            const cx<float> e2 = erow(z / 2 + 1);
            ldo(z + 1, p2, p3);
            prep(z + 1, R2, e1, ua, s0, s1);
            couple(R1, ub, ua, o0, o1, s0, s1);
            emit(z, ub, o0, o1, p0, p1);
            const GmRow<LOADG> R4 = ld(z + 3);
            ldo(z + 2, p0, p1);
            prep(z + 2, R3, 0.5f * (e1 + e2), ub, o0, o1);
            couple(R2, ua, ub, s0, s1, o0, o1);
            emit(z + 1, ua, s0, s1, p2, p3);
            R1 = R3;
            R2 = R4;
            e1 = e2;
        }
    }
}

template <int MODE>
__global__ void __launch_bounds__(32 * kGmWarps, kGmBlocks) k_gal_march(LevelDev Lf, LevelDev Lc, const float* __restrict__ hwv,
                                                            float b1, float b2, float wj,
                                                            const float* __restrict__ f,
                                                            const float* __restrict__ ec, float* __restrict__ out,
                                                            const RhsState* st, int accumulate, int rows, int nrhs) {
    pdl_trigger();
    pdl_wait();
    const int b = blockIdx.z * kGmWarps + (threadIdx.x >> 5);
    if (b >= nrhs || !rhs_active(st, b)) return;   // uniform in the warp; no block barrier below
    const int lane = threadIdx.x & 31;
    const int Ib = blockIdx.x * kGmCols - 1;   // coarse column of lane 0
    const int nx = Lf.nx, nz = Lf.nz;
    const size_t nf = (size_t)nx * nz, nc = (size_t)Lc.nx * Lc.nz;
    const float hw = hwv[b];
    const float* fb = f + 2 * nf * b;
    const float* gk = static_cast<const float*>(Lf.gk) + (size_t)b * Lf.gkstride;
    const float* eb = MODE == GM_RESTRICT ? nullptr : ec + 2 * nc * b;
    float* ob = out + 2 * (MODE == GM_PROLONG ? nf : nc) * b;
    const int A0 = blockIdx.y * rows, A1 = min(A0 + rows, MODE == GM_PROLONG ? nz : Lc.nz);
    // fine rows and columns the warp touches (rows loaded ahead included); inside the border?
    const int zlo = MODE == GM_PROLONG ? A0 - 1 : 2 * A0 - 1, zhi = MODE == GM_PROLONG ? A1 + 3 : 2 * A1 + 1;
    const int klo = MODE == GM_PROLONG ? A0 / 2 - 1 : A0 - 1, khi = MODE == GM_PROLONG ? (A1 + 1) / 2 + 1 : A1;
    const bool edge = 2 * Ib < 1 || 2 * Ib + 63 > nx - 2 || zlo < 1 || zhi > nz - 2 ||
                      (MODE != GM_RESTRICT && (Ib + 31 >= Lc.nx || klo < 0 || khi >= Lc.nz)) ||
                      (MODE == GM_PROLONG && (A1 & 1));
    if (edge)
        gal_march<MODE, true, true>(Lf, Lc, Ib + lane, lane, A0, A1, hw * b1, hw * b2, wj, fb, gk, eb, ob, accumulate);
    else if (Lf.gconst)
        gal_march<MODE, false, false>(Lf, Lc, Ib + lane, lane, A0, A1, hw * b1, hw * b2, wj, fb, gk, eb, ob, accumulate);
    else
        gal_march<MODE, true, false>(Lf, Lc, Ib + lane, lane, A0, A1, hw * b1, hw * b2, wj, fb, gk, eb, ob, accumulate);
}

// Rows per warp (coarse rows of a restriction, fine rows of a prolongation): long segments
// repeat fewer rows at their ends (16 and 32 measured best among 8 .. 64 at 128 and 320
// right-hand sides), shorter ones keep 24 warps per SM in small batches.
int gm_rows(int cols, int rows, int nrhs, int longest, int least) {
    int zs = longest;
    while (zs > least && (size_t)cols * ((rows + zs - 1) / zs) * nrhs < 152u * 24u) zs /= 2;
    return zs;
}

}  // namespace

void launch_gal_march_restrict(bool correct, const LevelDev& Lf, const LevelDev& Lc, const float* hw, double b1,
                               double b2, double wj, const float* f, const float* ec, float* fc, const RhsState* st,
                               int nrhs, cudaStream_t s) {
    const int cols = (Lc.nx + kGmCols - 1) / kGmCols;
    const int rows = gm_rows(cols, Lc.nz, nrhs, 16, 4);
    const dim3 grd(cols, (Lc.nz + rows - 1) / rows, (nrhs + kGmWarps - 1) / kGmWarps);
    if (correct)
        launch_pdl(k_gal_march<GM_CORRECT>, grd, dim3(32 * kGmWarps), 0, s, Lf, Lc, hw, (float)b1, (float)b2,
                   (float)wj, f, ec, fc, st, 0, rows, nrhs);
    else
        launch_pdl(k_gal_march<GM_RESTRICT>, grd, dim3(32 * kGmWarps), 0, s, Lf, Lc, hw, (float)b1, (float)b2,
                   (float)wj, f, ec, fc, st, 0, rows, nrhs);
}

void launch_gal_march_prolong(const LevelDev& Lf, const LevelDev& Lc, const float* hw, double b1, double b2,
                              double wj, const float* f, const float* ec, float* out, const RhsState* st, int nrhs,
                              cudaStream_t s, int accumulate) {
    const int cols = (Lf.nx + 2 * kGmCols - 1) / (2 * kGmCols);
    const int rows = gm_rows(cols, Lf.nz, nrhs, 32, 8);
    const dim3 grd(cols, (Lf.nz + rows - 1) / rows, (nrhs + kGmWarps - 1) / kGmWarps);
    launch_pdl(k_gal_march<GM_PROLONG>, grd, dim3(32 * kGmWarps), 0, s, Lf, Lc, hw, (float)b1, (float)b2, (float)wj,
               f, ec, out, st, accumulate, rows, nrhs);
}

}  // namespace helm
