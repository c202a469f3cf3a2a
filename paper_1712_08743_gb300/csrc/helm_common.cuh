// helm_common.cuh - device helpers shared by the Helmholtz kernels: complex
// arithmetic on float2/double2, the damping profile of the absorbing layer,
// per-right-hand-side solver state and deterministic block reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace helm {

// ----------------------------------------------------------------- complex
template <typename T> struct C2;
template <> struct C2<float> { using type = float2; };
template <> struct C2<double> { using type = double2; };

template <typename T> struct cx {
    T re, im;
    __host__ __device__ cx() {}
    __host__ __device__ cx(T r, T i) : re(r), im(i) {}
};
template <typename T> __device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <typename T> __device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return {a.re - b.re, a.im - b.im}; }
template <typename T> __device__ __forceinline__ cx<T> operator*(cx<T> a, cx<T> b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename T> __device__ __forceinline__ cx<T> operator*(T s, cx<T> a) { return {s * a.re, s * a.im}; }
// Sums and real multiples of complex values for kernels that are bound by the issue of
// instructions: in FP32 both parts go through one packed instruction (two rounded
// operations each, the same results as the scalar pair). Complex products stay scalar:
// packed, they need the parts of one factor swapped and cost as many instructions.
template <typename T> __device__ __forceinline__ cx<T> padd(cx<T> a, cx<T> b) { return a + b; }
template <> __device__ __forceinline__ cx<float> padd(cx<float> a, cx<float> b) {
    const float2 r = __fadd2_rn(make_float2(a.re, a.im), make_float2(b.re, b.im));
    return {r.x, r.y};
}
template <typename T> __device__ __forceinline__ cx<T> pfma(T s, cx<T> a, cx<T> c) {   // s a + c
    return {s * a.re + c.re, s * a.im + c.im};
}
template <> __device__ __forceinline__ cx<float> pfma(float s, cx<float> a, cx<float> c) {
    const float2 r = __ffma2_rn(make_float2(s, s), make_float2(a.re, a.im), make_float2(c.re, c.im));
    return {r.x, r.y};
}
template <typename T> __device__ __forceinline__ cx<T> cfma(cx<T> a, cx<T> b, cx<T> c) {   // a b + c
    return {(c.re + a.re * b.re) - a.im * b.im, (c.im + a.re * b.im) + a.im * b.re};
}
template <typename T> __device__ __forceinline__ cx<T> conjx(cx<T> a) { return {a.re, -a.im}; }
// Reciprocal of |b|^2 in complex division: the FP32 smoother and preconditioner
// use the hardware approximate reciprocal (max 1 ulp), FP64 keeps the IEEE divide. The form that
// takes subnormal arguments for zero is one instruction, without scaling around it (|b|^2 of a
// diagonal is 0 or far above 2^-126): 1 to 4 % of the finest smoothers' time.
__device__ __forceinline__ float rcp_fast(float d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    return r;
}
__device__ __forceinline__ double rcp_fast(double d) { return 1.0 / d; }
template <typename T> __device__ __forceinline__ cx<T> cdiv(cx<T> a, cx<T> b) {
    T d = b.re * b.re + b.im * b.im;
    T inv = rcp_fast(d);
    return {(a.re * b.re + a.im * b.im) * inv, (a.im * b.re - a.re * b.im) * inv};
}

// 8- or 16-byte vector loads/stores of one complex value.
__device__ __forceinline__ cx<float> ldc(const float* p, size_t i) {
    float2 v = __ldg(reinterpret_cast<const float2*>(p) + i);
    return {v.x, v.y};
}
__device__ __forceinline__ cx<double> ldc(const double* p, size_t i) {
    double2 v = __ldg(reinterpret_cast<const double2*>(p) + i);
    return {v.x, v.y};
}
// plain (coherent) loads, for buffers written earlier in the same kernel chain
__device__ __forceinline__ cx<float> ldcc(const float* p, size_t i) {
    float2 v = reinterpret_cast<const float2*>(p)[i];
    return {v.x, v.y};
}
__device__ __forceinline__ cx<double> ldcc(const double* p, size_t i) {
    double2 v = reinterpret_cast<const double2*>(p)[i];
    return {v.x, v.y};
}
__device__ __forceinline__ void stc(float* p, size_t i, cx<float> a) {
    reinterpret_cast<float2*>(p)[i] = make_float2(a.re, a.im);
}
__device__ __forceinline__ void stc(double* p, size_t i, cx<double> a) {
    reinterpret_cast<double2*>(p)[i] = make_double2(a.re, a.im);
}

// ------------------------------------------------------------ damping layer
// alpha of Eq. 2 at padded node (ix, iz): alpha_max (d / npml)^2 with d the
// node distance into the layer, the larger of the two axes in corners.
// Same profile from the integer layer depth, with acoef = alpha_max / npml^2
// precomputed on the host: no division on the device, in the kernel's precision.
__device__ __forceinline__ int layer_depth(int ix, int iz, int nx, int nz, int npml) {
    const int dx = max(npml - ix, ix - (nx - 1 - npml));
    const int dz = max(npml - iz, iz - (nz - 1 - npml));
    return max(max(dx, dz), 0);
}
template <typename T>
__device__ __forceinline__ T layer_alpha_t(int ix, int iz, int nx, int nz, int npml, T acoef) {
    const int d = layer_depth(ix, iz, nx, nz, npml);
    return acoef * (T)(d * d);
}
inline double layer_coef(int npml, double alpha_max) { return npml > 0 ? alpha_max / ((double)npml * npml) : 0.0; }

// ------------------------------------------------------- solver state per RHS
enum RhsFlag : int { FLAG_RUNNING = 0, FLAG_CONVERGED = 1, FLAG_BREAKDOWN = 2, FLAG_MAXIT = 3 };

struct RhsState {
    // Krylov scalars (BiCGSTAB); complex values as (re, im)
    double rho[2], alpha[2], omega[2], beta[2];
    double bnorm2;       // ||b||^2 of the inner system
    double rnorm2;       // ||r||^2 of the recursive residual
    double tol_rel;      // inner relative tolerance on ||r|| / ||b||
    double relres;       // outer FP64 relative residual
    double fnorm2;       // ||f||^2 of the outer system
    int active;          // 1 while this RHS iterates
    int iters;           // inner iterations, summed over outer steps
    int flag;            // RhsFlag of the last inner solve
    int outer_active;    // 1 while the outer refinement continues
    int max_it;
    int kfg;             // FGMRES: Arnoldi steps of the current cycle
    int reorth;          // FGMRES: 1 if the current column takes a second Gram-Schmidt pass
    unsigned int counter[4];  // last-block election counters, one per reduction site
};

// A right-hand side takes part in a kernel while its state says so (no state: always).
__device__ __forceinline__ bool rhs_active(const RhsState* st, int b) { return st == nullptr || st[b].active; }

// ------------------------------------------------ programmatic dependent launch
// Kernels of the iteration chain let the next kernel start launching at once
// (its blocks then wait in pdl_wait until this grid has completed and its
// writes are visible), so launch latency and prologues that read only
// immutable model data overlap the previous kernel. Without a programmatic
// dependency both instructions return immediately.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The FP64 kernels of the chain start the next one at their end. An FP64 instruction holds a quarter of an
// SM for 64 cycles, so a kernel takes as long as its busiest quarter; blocks that arrive while the kernel
// before is still running are placed where that one leaves room instead of one per SM, and
// the chain of a 241 x 191 solve took 45 ms in place of 24 (with the trigger in the smallest kernels
// alone 28).
template <typename T> __device__ __forceinline__ void pdl_trigger_for() {
    if constexpr (sizeof(T) == 4) pdl_trigger();
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// -------------------------------------------------------------- reductions
__device__ __forceinline__ int lin_tid() { return threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z); }
__device__ __forceinline__ int lin_nthreads() { return blockDim.x * blockDim.y * blockDim.z; }

template <int NV>
__device__ __forceinline__ void warp_sum(double (&v)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
}

// Block-wide sum of NV doubles (blocks of whole warps); result valid in
// linear thread 0. Deterministic order.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sh /* >= 32*NV */) {
    warp_sum<NV>(v);
    const int tid = lin_tid();
    const int lane = tid & 31, warp = tid >> 5;
    const int nwarps = (lin_nthreads() + 31) >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k * 32 + warp] = v[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = (lane < nwarps) ? sh[k * 32 + lane] : 0.0;
        warp_sum<NV>(v);
    }
}

// Block-wide sum of per-thread partials held in the kernel's precision A: the
// warp stage runs in A, only warp totals are widened to double (so an FP32
// kernel issues almost no FP64 instructions). Result in linear thread 0.
template <int NV, typename A>
__device__ __forceinline__ void block_sum_t(const A (&v)[NV], double (&o)[NV], double* sh /* >= 32*NV */) {
    A w[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        w[k] = v[k];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) w[k] += __shfl_xor_sync(0xffffffffu, w[k], d);
    }
    const int tid = lin_tid();
    const int lane = tid & 31, warp = tid >> 5;
    const int nwarps = (lin_nthreads() + 31) >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k * 32 + warp] = (double)w[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) o[k] = 0.0;
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) o[k] = (lane < nwarps) ? sh[k * 32 + lane] : 0.0;
        warp_sum<NV>(o);
    }
}

// Sums per-thread partials in precision A over the blocks of a right-hand side; true in the block that
// ends last, with the totals in tot of its thread 0. Order fixed. An FP64 addition holds a quarter of an
// SM for 64 cycles whatever lanes take part, and this is the end of a short kernel: the warp totals
// are added by one lane per value, side by side, and the last block's partials by the warps that share
// a value, so that five to eight additions follow one another where shuffles of all values took 15 to 30
// (end of a BiCGSTAB vector update on 19881 nodes: 10.4 -> 9.3 us for the kernel).
template <int NV, typename A>
__device__ __forceinline__ bool last_block_reduce_t(const A (&v)[NV], double (&tot)[NV], double* sh /* >= 32*NV */,
                                                    double* partials, int nblk, int blk, unsigned int* counter) {
    __shared__ int s_last_t;
    const int tid = lin_tid(), lane = tid & 31, warp = tid >> 5;
    const int nw = (lin_nthreads() + 31) >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        A w = v[k];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) w += __shfl_xor_sync(0xffffffffu, w, d);
        if (lane == 0) sh[k * 32 + warp] = (double)w;
    }
    __syncthreads();
    if (warp == 0) {
        if (lane < NV) {
            double a = 0.0, c = 0.0;
            for (int q = 0; q < nw; q += 2) {
                a += sh[lane * 32 + q];
                if (q + 1 < nw) c += sh[lane * 32 + q + 1];
            }
            partials[(size_t)lane * nblk + blk] = a + c;
            __threadfence();
        }
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            s_last_t = atomicAdd(counter, 1u) == (unsigned int)(nblk - 1);
        }
    }
    __syncthreads();
    if (!s_last_t) return false;
    __threadfence();
    const int parts = nw >= NV ? nw / NV : 1;
    for (int q = warp; q < NV * parts; q += nw) {
        const int k = q % NV, part = q / NV;
        const double* pk = partials + (size_t)k * nblk;
        double a = 0.0;
        for (int x = part * 32 + lane; x < nblk; x += parts * 32 * 4) {
            double t[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) t[m] = x + m * parts * 32 < nblk ? __ldcg(pk + x + m * parts * 32) : 0.0;
            a += (t[0] + t[1]) + (t[2] + t[3]);
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
        if (lane == 0) sh[k * 32 + part] = a;
    }
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            tot[k] = sh[k * 32];
            for (int m = 1; m < parts; ++m) tot[k] += sh[k * 32 + m];
        }
        *counter = 0u;
    }
    return true;
}

}  // namespace helm
