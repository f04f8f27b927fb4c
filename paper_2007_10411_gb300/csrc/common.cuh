// Device-side definitions shared by the kernels of libjfnk (sm_103a).
//
// Vectors are field-major planes [field][z][x] (x fastest), n = nf * npt
// entries.  Krylov vectors live in scaled units (every field divided by its
// scale U, U, Theta, P); the state and the Newton residual are float64 and
// unscaled.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/jfnk.h"

namespace jfnk {

constexpr int KMAX = 32;          // largest restart length the kernels are built for
constexpr int NTHREADS = 256;     // threads per block of every streaming kernel
constexpr int MAX_STREAM_BLOCKS = 2 * 152;  // streaming grid: two CTAs per SM
constexpr int MAX_DOT_BLOCKS = 3 * 152;     // Arnoldi passes A and C: three CTAs per SM
constexpr int MAX_REDUCE_BLOCKS = 8192;     // multi-dot grids grow so a thread sums <= 64 vectors' worth
constexpr int MAX_PC_SWEEPS = 64;

// The float32 kernels' copies of the constants of Geo.  A float64 -> float32
// conversion in a kernel runs at the FP64 pipe's rate (64 cycles per warp
// instruction and sub-partition): a dozen per thread cost several microseconds
// of a 20 us launch.
struct GeoF {
    float inv_dx, inv_dy, inv_dz, wx1, wx2, wy1, wy2, wz1, wz2, ex, ey, ez;
    float theta0, beta, pbar, gth, gamma_p, K_M, K_H, cs2, inv_Pr;
    float dd_cm, dd_cM, dd_cl, dd_delta, dd_ah, dd_az;
    float two_over_dt, schur_cdiv, schur_cgrad, half_dt;
};

// Geometry and physics constants, passed by value to the stencil kernels.
struct Geo {
    GeoF f32;
    int dim, nx, ny, nz, npt, nf;     // 2-D: ny = 1, nf = 4 (u, w, theta, p); 3-D: nf = 5 (u, v, w, theta, p)
    double inv_dy;
    int pb[5], pt[5];                 // mirror parity per field at bottom / top (+1 / -1)
    double inv_dx, inv_dz;
    double theta0, beta, pbar, g, gamma_p, heat_coef;   // heat_coef = 1/(rho0 cp dz)
    int smag;                         // eddy coefficients from the strain (Smagorinsky or Deardorff)
    int sgs;                          // 0 constant K, 1 Smagorinsky, 2 Deardorff (anisotropic)
    double K_M, K_H, cs2;             // cs2 = (Cs Delta)^2
    // Deardorff closure in terms of s = sqrt(2 S:S): K_m = dd_cm s, K_M = dd_cM s,
    // K_h = K_m (1 + dd_ah l), K_H = K_M (1 + dd_az l), l = min(dd_delta, dd_cl s)
    // (dd_cl < 0: l = dd_delta)
    double dd_cm, dd_cM, dd_cl, dd_delta, dd_ah, dd_az;
    // derivative weights with 1/h folded in: D f = w1 (f_{+1} - f_{-1}) + w2 (f_{+2} - f_{-2})
    double wx1, wx2, wy1, wy2, wz1, wz2;
    // D f = w (1 + e) (...): what rounding took from the weights, e the relative difference
    // of 2/3 times 1/h (each rounded) from w1, and of -1/12 times 1/h from w2 = -w1/8; here
    // (not in GeoF) that of y and z less that of x, the common factor being harmless
    // and an operation of the FP64 pipe.  The divergence of a nearly solenoidal flow is a
    // small part of its terms, so what the rounding of one axis's weight adds against the
    // others counts in full, and the pressure equation multiplies it by gamma_p pbar.
    double ey, ez;
    double gth;                       // g / theta0
    double inv_Pr;
    double two_over_dt;
    double scale[5], inv_scale[5];
    const double* heat;               // surface flux H(x) or nullptr
    int tile_jv, tile_pc;             // tile shapes of the float32 Jv / preconditioner kernels
    int pc_schur;                     // preconditioner: 0 field-block, 1 acoustic Schur complement (2-D)
    // acoustic Schur complement constants (host-computed): Helmholtz coefficient
    // a = gamma_p pbar theta0 dt/2, c_div = gamma_p pbar (dt/2) s_u/s_p,
    // c_grad = theta0 s_p/s_u, dt/2
    double helm_a, schur_cdiv, schur_cgrad, half_dt;
    void* s3;                         // 3-D: scratch of the split stencil passes (stencil3d_scratch_bytes)
};

// Constant `name` of Geo in the kernel's type T.
template <typename T>
__device__ __forceinline__ T geo_const(double d, float f) {
    if constexpr (sizeof(T) == sizeof(double)) return d;
    else return f;
}
#define GC(name) geo_const<T>(G.name, G.f32.name)

// D applied twice, from the first differences g_k = x_{k+1} - x_k of a line:
// sum_s c_s x_s (c_s = sum_{a+b=s} w_a w_b: -65/72, 1/9, 4/9, -1/9, 1/144 for |s| = 0 .. 4,
// which add up to zero) = sum_{k=0..3} C_k (g_k - g_{-1-k}) with C_k = sum_{s>k} c_s.
constexpr double HELM_DIFF[4] = {65.0 / 144.0, 49.0 / 144.0, -15.0 / 144.0, 1.0 / 144.0};

constexpr int NUM_TILE_SHAPES = 4;

// Solver control block in device memory.  Written by the "last block" of the
// reduction kernels, read by later kernels and, after a stream sync, by the host.
struct Ctl {
    int done;            // current GMRES cycle finished: later cycle kernels return at once
    int converged;       // |g_{j+1}| <= target (or lucky breakdown)
    int breakdown;
    int nan;
    int k;               // columns in the finished cycle
    int iters;           // Krylov iterations in this Newton solve
    int m;               // restart length
    int ncap;            // training pairs recorded for the learned preconditioner
    int eps_part;        // ||z||^2 of the last preconditioner apply is pending at the head of the
                         // partial buffer, and the Jacobian-product kernel forms eps from it:
                         // > 0: that many float-float partials (float32 2-D field blocks);
                         // < 0: minus that many float64 partials (float32 2-D Schur complement);
                         // 0: eps_jv holds the step.  Every writer of eps_jv clears it.
    int pad_;
    double beta0;        // ||b|| of the Newton system
    double target;       // eta * beta0
    double res2;         // ||W R||^2 of the last residual evaluation
    double unorm2;       // ||W u||^2 of the same state
    double eps_num, inv_eps_num;     // sqrt(eps_mach (1 + ||W u||)) of that state, and its reciprocal
    double eps_mach;     // unit roundoff of the stencil precision
    double eps_jv;       // finite-difference step of the next Jacobian-vector product (put_eps)
    double kmax;         // max eddy coefficient K_M (preconditioner bounds)
    double gstart;       // ||r|| at the start of the current GMRES cycle
    double gres;         // rotated residual |g_{j+1}| after the latest Arnoldi step
    double scratch[8];   // misc reductions (||x||^2, ||r||^2, ...)
    double h1[KMAX + 1];      // first-projection coefficients (pass B block 0, for the Hessenberg column)
    double Hbar[KMAX + 1][KMAX];     // Hessenberg as built (row, col)
    double Rt[KMAX][KMAX];           // rotated upper-triangular factor
    double cs[KMAX], sn[KMAX];
    double g[KMAX + 1];
    double y[KMAX];
    double zscale[KMAX];      // direction k of the cycle enters the update as zscale[k] y_k z_k
                              // (1 unless the lagged second projection normalised w_k on the fly)
    // Chebyshev coefficients per field block and sweep: 1/theta_c, rho_k rho_{k-1}, 2 rho_k / delta
    double cheb[6][MAX_PC_SWEEPS][3];   // slot 5: pressure Helmholtz of the Schur complement
    float chebf[6][MAX_PC_SWEEPS][3];   // the same in float32
    unsigned int counter[8];         // last-block counters, one per kernel family
    double scale[5], inv_scale[5];   // field scales (Geo::scale) and their reciprocals, set once
    // eps_jv scale_f and its reciprocal, formed once with the step instead of by every block
    // of a Jacobian product (a float64 division is some 25 issues of 64 cycles)
    double ev[5], cf[5];
    float evf[5], cff[5];
};

// A finite-difference step e that is not pending (eps_part) and its reciprocal:
// called by threads 0 .. 4 of one block (thread f forms field f's values).
__device__ __forceinline__ void put_eps(Ctl* ctl, double e, double ie) {
    const int f = threadIdx.x;
    if (f == 0) {
        ctl->eps_jv = e;
        ctl->eps_part = 0;
    }
    if (f < 5) {
        const double v = e * ctl->scale[f], r = ie * ctl->inv_scale[f];
        ctl->ev[f] = v;
        ctl->cf[f] = r;
        ctl->evf[f] = (float)v;
        ctl->cff[f] = (float)r;
    }
}


template <typename T>
__device__ __forceinline__ T cheb_coef(const Ctl* ctl, int f, int k, int i) {
    if constexpr (sizeof(T) == sizeof(double)) return ctl->cheb[f][k][i];
    else return ctl->chebf[f][k][i];
}

// Programmatic dependent launch.  Kernels of the Arnoldi step are launched
// with launch_pdl: the next kernel may be scheduled before this one has
// finished, so every such kernel calls pdl_wait() before its first global read
// (it returns once the preceding grid has completed and its writes are
// visible) and pdl_trigger() once its main loop is done (only the reduction
// tail remains), letting the successor's launch overlap that tail.  Both are
// no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

enum CounterSlot { CNT_STENCIL = 0, CNT_UPDATE, CNT_RESTART, CNT_PC, CNT_EDDY, CNT_MISC };

// -x by the sign bit (an FP64 multiplication by -1, predicated off or not, costs the FP64 pipe)
__device__ __forceinline__ float flip(float x) { return __int_as_float(__float_as_int(x) ^ 0x80000000); }
__device__ __forceinline__ double flip(double x) {
    return __hiloint2double(__double2hiint(x) ^ 0x80000000, __double2loint(x));
}

// Square root for kernels bound by the FP64 pipe (64 cycles per warp
// instruction): Goldschmidt's iteration (Markstein, "IA-64 and Elementary
// Functions", 2000) from the hardware's 20-bit reciprocal square root estimate,
// seven FP64 operations: one coupled step takes g ~ sqrt(x), h ~ 1/(2 sqrt(x))
// to ~39 bits, the residual step g + h (x - g^2) rounds the result (within one
// unit in the last place).  Zero, subnormal, negative and non-finite operands go to sqrt().
__device__ __forceinline__ double root(double x) {
    const int hi = __double2hiint(x);
    if (hi < 0x00100000 || hi >= 0x7ff00000) return sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double g = __dmul_rn(x, y), h = __dmul_rn(0.5, y);
    const double r = __fma_rn(-g, h, 0.5);
    g = __fma_rn(g, r, g);
    h = __fma_rn(h, r, h);
    return __fma_rn(__fma_rn(-g, g, x), h, g);
}
__device__ __forceinline__ float root(float x) { return sqrtf(x); }

// sqrt(x) and 1 / sqrt(x) of a positive x by the same iteration, two coupled
// steps (relative error of a few 2^-53): about ten dependent operations where a
// square root and a division take nearly a hundred, each a 64-cycle issue for
// every block that waits on it.  Zero (and negative) give 0 and 0, infinity gives
// infinity and 0, NaN gives NaN twice: a norm that is not a number stays visible.
__device__ __forceinline__ void root_pair(double x, double& g, double& ig) {
    const int hi = __double2hiint(x);
    if (hi < 0x00100000 || hi >= 0x7ff00000) {
        g = x > 0.0 ? sqrt(x) : (x <= 0.0 ? 0.0 : x);
        ig = g > 0.0 ? 1.0 / g : g;
        return;
    }
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double h = __dmul_rn(0.5, y);
    g = __dmul_rn(x, y);
    double r = __fma_rn(-g, h, 0.5);
    g = __fma_rn(g, r, g);
    h = __fma_rn(h, r, h);
    r = __fma_rn(-g, h, 0.5);
    h = __fma_rn(h, r, h);
    g = __fma_rn(__fma_rn(-g, g, x), h, g);
    ig = h + h;
}

// A flux K D phi - (u_j / 2) phi, kd - hp with one rounded product.  float32: the
// product of the velocities, the larger term, enters unrounded (F of a mixed handle
// errs by 1.7e-6 instead of 2.4e-6 at 1024 x 512).  float64: that product is rounded
// first, as a plain evaluation of D(u phi) rounds it, so that F differs from such an
// evaluation by the rounding of the sum alone.
__device__ __forceinline__ float flux_sum(float k, float d, float h, float p) { return __fmaf_rn(-h, p, __fmul_rn(k, d)); }
__device__ __forceinline__ double flux_sum(double k, double d, double h, double p) {
    return __fma_rn(k, d, -__dmul_rn(h, p));
}

// ---------------------------------------------------------------- reductions
// c + a . b.  float32: the four products meet each other first, so that the running
// sum is rounded once a vector instead of once an element.  float64: one chain of
// fused multiply-adds, because an addition occupies the FP64 pipe for as long as a
// fused multiply-add (two roundings of the running sum a vector instead of one, at
// 2^-53 each; the passes would take a quarter longer with a separate addition).
__device__ __forceinline__ float dotacc(float4 a, float4 b, float c) {
    return c + fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
}
__device__ __forceinline__ double dotacc(double2 a, double2 b, double c) { return fma(a.y, b.y, fma(a.x, b.x, c)); }
__device__ __forceinline__ float dotacc(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double dotacc(double a, double b, double c) { return fma(a, b, c); }

// Sum NV thread-local values over the block and store them, as float64, at
// part[k * stride + blk] (k < nv).  Deterministic (fixed shuffle tree).  The
// tree runs in the type of the thread values: float32 kernels reduce their
// float32 partials in float32 within a block (GB300's float64 rate is a small
// fraction of its float32 rate) and switch to float64 across blocks.
template <int NV, typename TA>
__device__ __forceinline__ void block_partials(const TA (&v)[NV], int nv, double* part,
                                               int stride, int blk) {
    __shared__ TA red[NV][NTHREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        if (k < nv) {
            TA s = v[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) red[k][warp] = s;
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) s += (double)red[k][w];
        part[(size_t)k * stride + blk] = s;
        __threadfence();          // publish before the block's arrival is counted
    }
}

// Maximum that propagates NaN (fmax drops a NaN operand): a NaN in any value
// makes the reduced maximum NaN, so a diagnostic cannot report finite extrema
// for a state that holds NaN.
__device__ __forceinline__ double max_nan(double a, double b) { return (a > b || a != a) ? a : b; }

template <int NV>
__device__ __forceinline__ void block_partials_max(const double (&v)[NV], int nv, double* part,
                                                   int stride, int blk) {
    __shared__ double red[NV][NTHREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        if (k < nv) {
            double s = v[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s = max_nan(s, __shfl_down_sync(0xffffffffu, s, o));
            if (lane == 0) red[k][warp] = s;
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nv; k += blockDim.x) {
        double s = red[k][0];
        for (int w = 1; w < nw; ++w) s = max_nan(s, red[k][w]);
        part[(size_t)k * stride + blk] = s;
        __threadfence();          // publish before the block's arrival is counted
    }
}

// Double-float addition of unevaluated float32 pairs (x = hi, y = lo): TwoSum
// of the high parts (Knuth, TAOCP vol. 2), low parts added, renormalised
// (Dekker 1971).  ~2^-44 relative rounding on the float32 pipes.
__device__ __forceinline__ float2 ff_add(float2 a, float2 b) {
    const float s = a.x + b.x;
    const float bb = s - a.x;
    const float e = (a.x - (s - bb)) + (b.x - bb);
    const float lo = e + (a.y + b.y);
    const float hi = s + lo;
    return make_float2(hi, lo - (hi - s));
}

// One float-float partial of a block's float32 values: fixed shuffle tree per
// warp, warps added in order by thread 0, stored at p[blk].
__device__ __forceinline__ void block_partial_ff(float v, float2* p, int blk) {
    __shared__ float red[NTHREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float2 t = make_float2(red[0], 0.f);
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) t = ff_add(t, make_float2(red[w], 0.f));
        p[blk] = t;
    }
}

// The state's norms from a residual evaluation: tot[0] = ||W R||^2, tot[1] = ||W u||^2.
__device__ __forceinline__ void put_norms(Ctl* ctl, const double* tot) {
    ctl->res2 = tot[0];
    ctl->unorm2 = tot[1];
    ctl->nan = !(isfinite(tot[0]) && isfinite(tot[1]));
    const double num = sqrt(ctl->eps_mach * (1.0 + sqrt(tot[1])));
    ctl->eps_num = num;
    ctl->inv_eps_num = 1.0 / num;
}

// eps = eps_num / ||z||, by threads 0 .. 4 of one block.
__device__ __forceinline__ void put_eps_norm2(Ctl* ctl, double zn2) {
    double zn, izn;
    root_pair(zn2, zn, izn);
    put_eps(ctl, ctl->eps_num * izn, zn * ctl->inv_eps_num);
}

// Finite-difference step of a Jacobian product and its reciprocal: eps_jv, or,
// when ctl->eps_part is not 0, eps = eps_num / ||z|| with ||z||^2 summed from the
// pending partials.  The first four warps add them (a float64 addition takes a
// sub-partition's pipe for 64 cycles; more warps would queue for it), across the
// warps in float64, in one fixed order: every block of the launch, whatever its
// size, obtains bitwise the same value.  (0.7 us of jv2d's 22.9 at 1024 x 512 against
// float-float sums across all warps.)  Called by all threads of a block of at
// least 128.
__device__ __forceinline__ double2 pending_eps(const Ctl* ctl, const double* part) {
    constexpr int NT = 128;
    __shared__ double wsum[NT / 32];
    __shared__ double2 eps_s;
    const int np = ctl->eps_part;
    const double num = ctl->eps_num, inum = ctl->inv_eps_num;
    if (np != 0) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (np > 0 && threadIdx.x < NT) {
            const float2* p = reinterpret_cast<const float2*>(part);
            float2 s = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int b = threadIdx.x; b < np; b += NT) s = ff_add(s, __ldcg(p + b));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                s = ff_add(s, make_float2(__shfl_down_sync(0xffffffffu, s.x, o), __shfl_down_sync(0xffffffffu, s.y, o)));
            if (lane == 0) wsum[warp] = (double)s.x + (double)s.y;
        } else if (threadIdx.x < NT) {
            double s = 0.0;
#pragma unroll 8
            for (int b = threadIdx.x; b < -np; b += NT) s += __ldcg(part + b);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if (lane == 0) wsum[warp] = s;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = wsum[0];
            for (int w = 1; w < NT / 32; ++w) t += wsum[w];
            double zn, izn;
            root_pair(t, zn, izn);
            eps_s = make_double2(num * izn, zn * inum);
        }
    } else if (threadIdx.x == 0) {
        const double e = ctl->eps_jv;
        eps_s = make_double2(e, e != 0.0 ? 1.0 / e : 0.0);
    }
    __syncthreads();
    return eps_s;
}

// True in exactly one block: the last one to arrive.  The threads that wrote
// the block's partial sums fenced them (block_partials); the barrier orders
// those fences before thread 0's arrival.  Counters wrap to zero by
// themselves (atomicInc limit), so no reset is needed between launches.
__device__ __forceinline__ bool arrive_last(unsigned int* counter, unsigned int total) {
    __shared__ bool am_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();      // cumulative: orders the block's fenced partials before the count
        unsigned int t = atomicInc(counter, total - 1);
        am_last = (t == total - 1);
    }
    __syncthreads();
    if (am_last) __threadfence();
    return am_last;
}

// In the last block: out[k] = sum over blocks of part[k * nblk + b], in a fixed
// order (deterministic).  Loads are issued four at a time into independent
// accumulators so that a lane never waits on one L2 round trip per partial;
// a single value is reduced by the whole block, several values warp by warp.
template <bool MAXOP>
__device__ __forceinline__ double combine(double a, double b) { return MAXOP ? max_nan(a, b) : a + b; }

template <bool MAXOP>
__device__ __forceinline__ double strided_reduce(const double* p, int n, int start, int stride) {
    const double id = MAXOP ? -1.0e300 : 0.0;
    double s0 = id, s1 = id, s2 = id, s3 = id;
    int b = start;
    for (; b + 3 * stride < n; b += 4 * stride) {
        const double v0 = __ldcg(p + b), v1 = __ldcg(p + b + stride);
        const double v2 = __ldcg(p + b + 2 * stride), v3 = __ldcg(p + b + 3 * stride);
        s0 = combine<MAXOP>(s0, v0);
        s1 = combine<MAXOP>(s1, v1);
        s2 = combine<MAXOP>(s2, v2);
        s3 = combine<MAXOP>(s3, v3);
    }
    for (; b < n; b += stride) s0 = combine<MAXOP>(s0, __ldcg(p + b));
    return combine<MAXOP>(combine<MAXOP>(s0, s1), combine<MAXOP>(s2, s3));
}

template <bool MAXOP>
__device__ __forceinline__ double warp_reduce(double s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = combine<MAXOP>(s, __shfl_down_sync(0xffffffffu, s, o));
    return s;
}

template <bool MAXOP>
__device__ __forceinline__ void final_reduce(const double* part, int nblk, int nv, double* out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    if (nv == 1) {
        __shared__ double red[NTHREADS / 32];
        const double s = warp_reduce<MAXOP>(strided_reduce<MAXOP>(part, nblk, threadIdx.x, blockDim.x));
        if (lane == 0) red[warp] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = red[0];
            for (int w = 1; w < nw; ++w) t = combine<MAXOP>(t, red[w]);
            out[0] = t;
        }
        __syncthreads();
        return;
    }
    for (int k = warp; k < nv; k += nw) {
        const double s = warp_reduce<MAXOP>(strided_reduce<MAXOP>(part + (size_t)k * nblk, nblk, lane, 32));
        if (lane == 0) out[k] = s;
    }
    __syncthreads();
}

__device__ __forceinline__ void final_sums(const double* part, int nblk, int nv, double* out) {
    final_reduce<false>(part, nblk, nv, out);
}

__device__ __forceinline__ void final_maxes(const double* part, int nblk, int nv, double* out) {
    final_reduce<true>(part, nblk, nv, out);
}

}  // namespace jfnk
