// 2-D stencil kernels of libjfnk: F(u), R(u), the Jacobian-vector product,
// the Smagorinsky eddy field, the field-block Chebyshev preconditioner and
// the budgets.
//
// Discretisation (Hossain & Alam):
//   * Deslauriers-Dubuc collocation derivative of order p = 2 (Section 2.3):
//     the 4-point interpolating scheme gives phi'(+-1) = -+2/3, phi'(+-2) = +-1/12,
//     i.e. D f_j = [2/3 (f_{j+1} - f_{j-1}) - 1/12 (f_{j+2} - f_{j-2})] / h.
//   * skew-symmetric convection C(u)phi = 1/2 D_j(u_j phi) + 1/2 u_j D_j phi (Section 2.2)
//     for every field;
//   * Eqs. ch2_28-ch2_30 with Laplacian-form eddy diffusion sum_j D_j(K D_j phi),
//     constant K_M, K_H (Table 1) or Smagorinsky nu = (Cs Delta)^2 sqrt(2 S:S),
//     K_M = nu, K_H = nu / Pr (Section 2.4);
//   * x periodic, z cell-centred with mirror ghosts (w odd, theta and p even,
//     u even for free slip / odd for no slip); the eddy field is mirrored even.
//
// Tiling: one CTA computes a TX x TZ tile of output points.  The fields are
// staged with a halo of 2r = 4 points in shared memory (periodic / mirror
// index mapping, coalesced along x); every flux that D differentiates is
// formed once at the points and on the arms it is read from, and then
// differentiated.  Nothing but the inputs and the outputs touches HBM: the
// eddy viscosity and the derivatives live only on the chip.
#include <math.h>

#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace jfnk {

constexpr int R = 2;          // derivative radius for p = 2
constexpr int HALO = 2 * R;   // input halo (derivative applied twice)

// Explicitly rounded product and fused multiply-add: expressions written with
// them round the same way in every instantiation (tile shape) of a kernel.
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

// Source row / sign of a ghost-extended z index.  side: 0 interior, 1 bottom, 2 top.
__device__ __forceinline__ int mirror_z(int gz, int nz, int& side) {
    side = 0;
    if (gz < 0) { side = 1; return -1 - gz; }
    if (gz >= nz) { side = 2; return 2 * nz - 1 - gz; }
    return gz;
}

__device__ __forceinline__ int wrap_x(int gx, int nx) {
    if ((unsigned)gx < (unsigned)nx) return gx;        // interior: no division
    int r = gx % nx;
    return r < 0 ? r + nx : r;
}

// Ghost row (side 1 bottom, 2 top) of a field that is odd at that wall.
__device__ __forceinline__ bool odd_ghost(const Geo& G, int f, int side) {
    return (side == 1 && G.pb[f] < 0) || (side == 2 && G.pt[f] < 0);
}

template <typename T> struct Vec16;
template <> struct Vec16<float> {
    using type = float4;
    static constexpr int W = 4;
    __device__ static float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ static float4 fma(float a, float4 x, float4 y) {
        return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
    }
    __device__ static float4 neg(float4 x) { return make_float4(flip(x.x), flip(x.y), flip(x.z), flip(x.w)); }
};
template <> struct Vec16<double> {
    using type = double2;
    static constexpr int W = 2;
    __device__ static double2 zero() { return make_double2(0.0, 0.0); }
    __device__ static double2 fma(double a, double2 x, double2 y) {
        return make_double2(::fma(a, x.x, y.x), ::fma(a, x.y, y.y));
    }
    __device__ static double2 neg(double2 x) { return make_double2(flip(x.x), flip(x.y)); }
};

// Every row of every plane of the arrays starts on a 16-byte boundary: planes are
// nx * nz elements apart, and the base may be the caller's array, which need only
// be aligned to its element (8 bytes).
template <typename T>
static bool rows_aligned(const Geo& G, const T* a, const T* b = nullptr) {
    return G.nx % Vec16<T>::W == 0 && ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
}

// Stage 1: s[f][SZ][SX] <- (LOADMODE 0) u, (1) u + ev*v for fields f0 .. f0+NF-1,
// ghost-extended (periodic x, signed mirror z).  aligned: the
// host's rows_aligned(u, v); a tile whose x-range [x0 - HALO, x0 - HALO + SX)
// lies inside the grid then loads its rows as 16-byte vectors.
template <typename T, int LOADMODE, int NF = 4>
__device__ __forceinline__ void load_fields(T* s, const T* __restrict__ u, const T* __restrict__ v,
                                            const T (&ev)[4], const Geo& G, int aligned, int x0, int z0,
                                            int SX, int SZ, int f0 = 0) {
    using VT = typename Vec16<T>::type;
    constexpr int VW = Vec16<T>::W;
    if (aligned && x0 - HALO >= 0 && x0 - HALO + SX <= G.nx) {
        const int nch = SX / VW;
        const int total = nch * SZ;
        for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
            const int iz = idx / nch, c = idx - iz * nch;
            const int gz = z0 + iz - HALO;
            int side;
            const int sz = mirror_z(gz, G.nz, side);
            const bool ok = sz >= 0 && sz < G.nz;
            const size_t off = (size_t)sz * G.nx + (x0 - HALO + c * VW);
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                const int f = f0 + q;
                VT val = Vec16<T>::zero();
                if (ok) {
                    const size_t o = (size_t)f * G.npt + off;
                    if (LOADMODE == 0) val = *reinterpret_cast<const VT*>(u + o);
                    else
                        val = Vec16<T>::fma(ev[f], *reinterpret_cast<const VT*>(v + o),
                                            *reinterpret_cast<const VT*>(u + o));
                    if (odd_ghost(G, f, side)) val = Vec16<T>::neg(val);
                }
                *reinterpret_cast<VT*>(s + (q * SZ + iz) * SX + c * VW) = val;
            }
        }
        return;
    }
    const int total = SX * SZ;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int iz = idx / SX, ix = idx - iz * SX;
        const int gz = z0 + iz - HALO, gx = x0 + ix - HALO;
        int side;
        const int sz = mirror_z(gz, G.nz, side);
        const int sx = wrap_x(gx, G.nx);
        const bool ok = sz >= 0 && sz < G.nz;
        const size_t off = (size_t)sz * G.nx + sx;
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            const int f = f0 + q;
            T val = T(0);
            if (ok) {
                const size_t o = (size_t)f * G.npt + off;
                if (LOADMODE == 0) val = u[o];
                else val = rfma(ev[f], v[o], u[o]);
                if (odd_ghost(G, f, side)) val = flip(val);
            }
            s[(q * SZ + iz) * SX + ix] = val;
        }
    }
}

// Deardorff heat factor s (1 + a l(s)), l = min(Delta, c_l s) (c_l < 0: l = Delta).
template <typename T>
__device__ __forceinline__ T dd_heat(T s, T a, const Geo& G) {
    const T cls = rmul(GC(dd_cl), s);
    const T l = GC(dd_cl) < T(0) ? GC(dd_delta) : (cls < GC(dd_delta) ? cls : GC(dd_delta));
    return rmul(s, rfma(a, l, T(1)));
}

template <typename T>
__device__ __forceinline__ T smag_nu(T ux, T uz, T wx, T wz, T cs2) {
    const T s13 = T(0.5) * (uz + wx);
    const T ss = ux * ux + wz * wz + T(2) * s13 * s13;
    return cs2 * sqrt(T(2) * ss);
}

// ============================================================================
// F, 2u/dt + F, residual and plain forward-difference Jv
//
// Compute-once tiles.  Every term of F that is differentiated along an axis
// is one flux, formed once per point,
//   X_phi = K D_x phi - 1/2 u phi,   Z_phi = K D_z phi - 1/2 w phi   (K = 0 for p),
// so that F_phi = D_x X_phi + D_z Z_phi + S_phi with the point-wise part
//   S_phi = -1/2 (u D_x phi + w D_z phi) + pressure gradient, buoyancy, ...
// Phase 1 stages the four fields of a TX x TZ tile with a halo of 4; phase 2
// forms both fluxes and S at the tile's points, X alone on two columns either
// side and Z alone on two rows above and below (the arms); phase 3, one item
// per point and field, differentiates the fluxes and writes the mode's output.
//
// Bound (float64): the FP64 pipe, 2 FMA per clock and SM, that is 64 cycles
// per warp instruction and sub-partition, so only the number of FP64
// operations counts: about 130 a point (32 first derivatives, 17 eddy
// coefficient, 14 fluxes, 18 point-wise, 32 flux derivatives, 16 output and
// norms) and 45 per arm point, against about 255 for the form that rebuilt
// the products at every tap and formed all derivatives on the whole halo.
// One F(u) at 1024 x 512, Smagorinsky: 236 -> 144 us; at 128 x 64: 31 -> 8 us.
// ============================================================================
// The strain magnitude sqrt(2 S:S) from the velocity gradients.
template <typename T>
__device__ __forceinline__ T flux_strain(T ux, T uz, T wx, T wz) {
    const T a = uz + wx;                            // 2 S:S = 2 (ux^2 + wz^2) + (uz + wx)^2
    const T d = rfma(ux, ux, rmul(wz, wz));
    return root(rfma(a, a, d + d));
}

// D f = w1 (f_{+1} - f_{-1}) + w2 (f_{+2} - f_{-2})
template <typename T>
__device__ __forceinline__ T wd(const T* s, int i, int st, T w1, T w2) {
    return rfma(w1, s[i + st] - s[i - st], rmul(w2, s[i + 2 * st] - s[i - 2 * st]));
}

struct FluxShape {
    int lx, lz;                                     // TX = 1 << lx, TZ = 1 << lz
    __host__ __device__ int tx() const { return 1 << lx; }
    __host__ __device__ int tz() const { return 1 << lz; }
    __host__ __device__ int cn() const { return 1 << (lx + lz); }
    __host__ __device__ int sx() const { return tx() + 2 * HALO; }
    __host__ __device__ int plane() const { return sx() * (tz() + 2 * HALO); }
    __host__ __device__ int xn() const { return (tx() + 2 * R) * tz(); }       // X flux of one field
    __host__ __device__ int zn() const { return tx() * (tz() + 2 * R); }       // Z flux of one field
    __host__ __device__ int ppt() const { return cn() / NTHREADS; }            // 0: phase 3 per point and field
    __host__ __device__ int elems() const { return 4 * (plane() + xn() + zn() + (ppt() ? 0 : cn())); }
};

// Tile row whose eddy value a flux point in tile row iz takes: its mirror
// image in the two ghost rows next to a wall (K is mirrored even), else itself.
__device__ __forceinline__ int flux_eddy_row(int iz, int z0, int nz) {
    const int gz = z0 + iz;
    if (gz < 0) return (-1 - gz) - z0;
    if (gz >= nz) return (2 * nz - 1 - gz) - z0;
    return iz;
}

// Phase 2 at one point.  i: staged index; is: staged index of the point whose
// eddy coefficient it takes.  XF / ZF: form the X / Z fluxes; both: a tile
// point, which also gets its point-wise part.
template <typename T, int SMAG, bool XF, bool ZF>
__device__ __forceinline__ void flux_point(const Geo& G, const FluxShape& sh, const T* __restrict__ s, int i, int is,
                                           T* __restrict__ X, T* __restrict__ Z, T (&S)[4]) {
    const int PL = sh.plane(), SX = sh.sx(), XN = sh.xn(), ZN = sh.zn();
    const T wx1 = GC(wx1), wx2 = GC(wx2), wz1 = GC(wz1), wz2 = GC(wz2);
    const T *U = s, *W = s + PL, *H = s + 2 * PL, *P = s + 3 * PL;
    T ux = T(0), uz = T(0), wx = T(0), wz = T(0), tx = T(0), tz = T(0);
    if (XF || SMAG) { ux = wd(U, i, 1, wx1, wx2); wx = wd(W, i, 1, wx1, wx2); }
    if (ZF || SMAG) { uz = wd(U, i, SX, wz1, wz2); wz = wd(W, i, SX, wz1, wz2); }
    if (XF) tx = wd(H, i, 1, wx1, wx2);
    if (ZF) tz = wd(H, i, SX, wz1, wz2);
    T kx = GC(K_M), kz = GC(K_M), kxh = GC(K_H), kzh = GC(K_H);
    if (SMAG) {
        const T st = is == i ? flux_strain(ux, uz, wx, wz)
                             : flux_strain(wd(U, is, 1, wx1, wx2), wd(U, is, SX, wz1, wz2),
                                           wd(W, is, 1, wx1, wx2), wd(W, is, SX, wz1, wz2));
        if (SMAG == 2) {       // Deardorff: K_m along x, K_M along z, heat with its own factors
            kx = rmul(GC(dd_cm), st);
            kz = rmul(GC(dd_cM), st);
            if (XF) kxh = rmul(GC(dd_cm), dd_heat(st, GC(dd_ah), G));
            if (ZF) kzh = rmul(GC(dd_cM), dd_heat(st, GC(dd_az), G));
        } else {
            kx = kz = rmul(GC(cs2), st);
            kxh = kzh = rmul(kx, GC(inv_Pr));
        }
    }
    const T hu = rmul(T(0.5), U[i]), hw = rmul(T(0.5), W[i]);
    // K D phi - 1/2 u_j phi: see flux_sum
    if (XF) {
        X[0] = flux_sum(kx, ux, hu, U[i]);
        X[XN] = flux_sum(kx, wx, hu, W[i]);
        X[2 * XN] = flux_sum(kxh, tx, hu, H[i]);
        X[3 * XN] = -rmul(hu, P[i]);
    }
    if (ZF) {
        Z[0] = flux_sum(kz, uz, hw, U[i]);
        Z[ZN] = flux_sum(kz, wz, hw, W[i]);
        Z[2 * ZN] = flux_sum(kzh, tz, hw, H[i]);
        Z[3 * ZN] = -rmul(hw, P[i]);
    }
    if (XF && ZF) {
        const T px = wd(P, i, 1, wx1, wx2), pz = wd(P, i, SX, wz1, wz2);
        const T th0 = GC(theta0);
        T div = rfma(GC(ez), wz, ux + wz);
        if constexpr (sizeof(T) == sizeof(float)) div = rfma(G.f32.ex, ux, div);
        S[0] = rfma(-hu, ux, rfma(-hw, uz, -rmul(th0, px)));
        S[1] = rfma(-hu, wx, rfma(-hw, wz, rfma(GC(gth), H[i], -rmul(th0, pz))));
        S[2] = rfma(-hu, tx, rfma(-hw, tz, -rmul(GC(beta), W[i])));
        S[3] = rfma(-hu, px, rfma(-hw, pz, -rmul(rmul(GC(gamma_p), GC(pbar) + P[i]), div)));
    }
}

// Derivative of the fluxes of field fl at tile point (tx, tz) plus S.
template <typename T>
__device__ __forceinline__ T flux_div(const Geo& G, const FluxShape& sh, const T* X, const T* Z, int fl, int tz, int tx,
                                      T S) {
    const int PXW = sh.tx() + 2 * R, TX = sh.tx();
    const T* x = X + fl * sh.xn() + tz * PXW + tx + R;
    const T* z = Z + fl * sh.zn() + (tz + R) * TX + tx;
    return rfma(GC(wx1), x[1] - x[-1],
                rfma(GC(wx2), x[2] - x[-2],
                     rfma(GC(wz1), z[TX] - z[-TX], rfma(GC(wz2), z[2 * TX] - z[-2 * TX], S))));
}

// The mode's output at point o of field fl from F (ar, au: sums of R^2 and u^2
// of the field in its own units).
template <typename T>
__device__ __forceinline__ void flux_out(const Geo& G, int mode, int fl, T Fv, double uo, size_t o,
                                         const T* __restrict__ v, const T* __restrict__ Fu,
                                         const double* __restrict__ f, T* __restrict__ out, T* __restrict__ out2,
                                         double cf, double& ar, double& au) {
    const double Fd = (double)Fv;
    if (mode == MODE_F) {
        out[o] = Fv;
    } else if (mode == MODE_JV) {   // w_hat = 2 v_hat/dt - (F(u + eps V) - F(u)) / (eps scale)
        const double diff = Fd - (double)Fu[o];
        out[o] = T(G.two_over_dt * (double)v[o] - diff * cf);
    } else if (mode == MODE_RHS) {
        out[o] = T(G.two_over_dt * uo + Fd);
    } else {
        double Rv;
        if (mode == MODE_RHSRES) {
            // at u = u^n the residual 2u/dt - F(u) - f with f = 2u/dt + F(u) is -2 F(u)
            out[o] = T(G.two_over_dt * uo + Fd);
            Rv = -2.0 * Fd;
            out2[o] = T(Rv);
        } else {
            Rv = G.two_over_dt * uo - Fd - f[o];
            out[o] = T(Rv);
            if (out2 != nullptr) out2[o] = Fv;
        }
        ar = fma(Rv, Rv, ar);
        au = fma(uo, uo, au);
    }
}

// PPT > 0: TX * TZ = PPT * NTHREADS; a thread keeps the point-wise parts of its
// PPT points in registers and finishes them itself.  PPT = 0 (tiles of fewer
// points than threads): the point-wise parts go through shared memory and phase
// 3 runs one item per point and field, which spreads a small tile over the
// sub-partitions' FP64 pipes.
template <typename T, int SMAG, int PPT>
__global__ void __launch_bounds__(NTHREADS)
flux2d(Geo G, int mode, FluxShape sh, int aligned, const T* __restrict__ u, const T* __restrict__ v, const T* __restrict__ Fu,
       const double* __restrict__ f, T* __restrict__ out, T* __restrict__ out2, double* __restrict__ part, Ctl* ctl,
       int check_done) {
    pdl_wait();
    if (mode == MODE_JV && check_done && ctl->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int TX = sh.tx(), TZ = sh.tz(), CN = sh.cn(), SX = sh.sx(), PXW = TX + 2 * R;
    T* s1 = reinterpret_cast<T*>(smem_raw);         // [4][SZ][SX]
    T* X = s1 + 4 * sh.plane();                     // [4][TZ][TX + 4]
    T* Z = X + 4 * sh.xn();                         // [4][TZ + 4][TX]
    T* Ss = Z + 4 * sh.zn();                        // [4][TZ][TX] (PPT = 0)
    const int x0 = blockIdx.x << sh.lx, z0 = blockIdx.y << sh.lz;
    T ev[4] = {T(0), T(0), T(0), T(0)};
    if (mode == MODE_JV) {
#pragma unroll
        for (int q = 0; q < 4; ++q) ev[q] = T(ctl->ev[q]);
        load_fields<T, 1>(s1, u, v, ev, G, aligned, x0, z0, SX, TZ + 2 * HALO);
    } else {
        load_fields<T, 0>(s1, u, v, ev, G, aligned, x0, z0, SX, TZ + 2 * HALO);
    }
    __syncthreads();
    T S[PPT > 0 ? PPT : 1][4];
    auto point = [&](int w, T (&Sw)[4]) {           // a tile point
        const int iz = w >> sh.lx, ix = w & (TX - 1);
        if (z0 + iz > G.nz + 1 || x0 + ix > G.nx + 1) return;        // feeds no output
        const int i = (iz + HALO) * SX + ix + HALO;
        const int is = SMAG ? (flux_eddy_row(iz, z0, G.nz) + HALO) * SX + ix + HALO : i;
        flux_point<T, SMAG, true, true>(G, sh, s1, i, is, X + iz * PXW + ix + R, Z + (iz + R) * TX + ix, Sw);
    };
    if (PPT > 0) {
#pragma unroll
        for (int k = 0; k < PPT; ++k) point(threadIdx.x + k * NTHREADS, S[k]);
    } else if (threadIdx.x < CN) {
        point(threadIdx.x, S[0]);
#pragma unroll
        for (int q = 0; q < 4; ++q) Ss[q * CN + threadIdx.x] = S[0][q];
    }
    // the arms; a small tile gives them to the warps that have no tile point
    for (int a = PPT > 0 ? threadIdx.x : (threadIdx.x + NTHREADS - CN) % NTHREADS; a < 4 * (TX + TZ); a += NTHREADS) {
        const bool zarm = a < 4 * TX;
        const int b = a - 4 * TX, r = zarm ? a >> sh.lx : b & 3;
        const int ix = zarm ? a & (TX - 1) : (r < 2 ? r - 2 : TX + r - 2);
        const int iz = zarm ? (r < 2 ? r - 2 : TZ + r - 2) : b >> 2;
        if (z0 + iz > G.nz + 1 || x0 + ix > G.nx + 1) continue;
        const int i = (iz + HALO) * SX + ix + HALO;
        const int is = SMAG ? (flux_eddy_row(iz, z0, G.nz) + HALO) * SX + ix + HALO : i;
        T none[4];
        if (zarm) flux_point<T, SMAG, false, true>(G, sh, s1, i, is, X, Z + (iz + R) * TX + ix, none);
        else flux_point<T, SMAG, true, false>(G, sh, s1, i, is, X + iz * PXW + ix + R, Z, none);
    }
    __syncthreads();
    double acc[2] = {0.0, 0.0};
    auto finish = [&](int fl, int pt, T Sv, double& ar, double& au) {
        const int tz = pt >> sh.lx, tx = pt & (TX - 1);
        const int gz = z0 + tz, gx = x0 + tx;
        if (gz >= G.nz || gx >= G.nx) return;
        T Fv = flux_div(G, sh, X, Z, fl, tz, tx, Sv);
        if (fl == 2 && gz == 0 && G.heat != nullptr) Fv += T(G.heat[gx] * G.heat_coef);
        const double uo = (double)s1[fl * sh.plane() + (tz + HALO) * SX + tx + HALO];
        flux_out(G, mode, fl, Fv, uo, (size_t)fl * G.npt + (size_t)gz * G.nx + gx, v, Fu, f, out, out2,
                 mode == MODE_JV ? ctl->cf[fl] : 0.0, ar, au);
    };
    if (PPT > 0) {
#pragma unroll
        for (int fl = 0; fl < 4; ++fl) {
            double ar = 0.0, au = 0.0;
#pragma unroll
            for (int k = 0; k < PPT; ++k) finish(fl, threadIdx.x + k * NTHREADS, S[k][fl], ar, au);
            const double i2 = G.inv_scale[fl] * G.inv_scale[fl];
            acc[0] = fma(ar, i2, acc[0]);
            acc[1] = fma(au, i2, acc[1]);
        }
    } else {
        for (int w = threadIdx.x; w < 4 * CN; w += NTHREADS) {
            const int fl = w >> (sh.lx + sh.lz), pt = w & (CN - 1);
            double ar = 0.0, au = 0.0;
            finish(fl, pt, Ss[w], ar, au);
            const double i2 = G.inv_scale[fl] * G.inv_scale[fl];
            acc[0] = fma(ar, i2, acc[0]);
            acc[1] = fma(au, i2, acc[1]);
        }
    }
    pdl_trigger();
    if (mode == MODE_RES || mode == MODE_RHSRES) {
        const int nblk = gridDim.x * gridDim.y;
        const int blk = blockIdx.y * gridDim.x + blockIdx.x;
        block_partials<2>(acc, 2, part, nblk, blk);
        if (arrive_last(&ctl->counter[CNT_STENCIL], nblk)) {
            __shared__ double tot[2];
            final_sums(part, nblk, 2, tot);
            if (threadIdx.x == 0) {
                put_norms(ctl, tot);
            }
        }
    }
}

// ============================================================================
// Asynchronous tile staging (cp.async, sm_80 and later): the copies of the
// next tile land in shared memory while the current tile is computed.
// 16-byte chunks for rows inside the grid, element copies at the periodic x
// seam; a source size of 0 zero-fills (rows beyond one mirror reflection).
// ============================================================================
__device__ __forceinline__ void cpa16(void* dst, const void* src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(src_bytes) : "memory");
}
template <int B>
__device__ __forceinline__ void cpa_elem(void* dst, const void* src, int src_bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(B), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Grid of a kernel with one CTA per tile: tile columns along x, tile rows along y
// and, past the 65 535 that y holds (heights above 8 x 65 535 points), along z too.
// The last rows may then lie past the wall; they feed no output.
static dim3 tile_grid(int cols, int rows) {
    constexpr int MAX_Y = 65535;
    const int nz = (rows + MAX_Y - 1) / MAX_Y;
    return dim3(cols, (rows + nz - 1) / nz, nz);
}
__device__ __forceinline__ int tile_row() { return blockIdx.z * gridDim.y + blockIdx.y; }

// Row vectors: a thread of the float32 sweeps and of the Schur-complement kernels
// owns W consecutive points along x (16 bytes where nx allows it).
template <typename T, int W> struct RowVec { using type = typename Vec16<T>::type; };
template <typename T> struct RowVec<T, 1> { using type = T; };
template <> struct RowVec<float, 2> { using type = float2; };
template <typename T, int W>
__device__ __forceinline__ void rload(const T* p, T (&v)[W]) {
    *reinterpret_cast<typename RowVec<T, W>::type*>(v) = *reinterpret_cast<const typename RowVec<T, W>::type*>(p);
}
template <typename T, int W>
__device__ __forceinline__ void rstore(T* p, const T (&v)[W]) {
    *reinterpret_cast<typename RowVec<T, W>::type*>(p) = *reinterpret_cast<const typename RowVec<T, W>::type*>(v);
}

// Asynchronous copy of W elements (16, 8 or 4 bytes) into shared memory.
template <typename T, int W>
__device__ __forceinline__ void cpa_vec(T* dst, const T* src) {
    if constexpr (W * sizeof(T) == 16) cpa16(dst, src, 16);
    else cpa_elem<W * (int)sizeof(T)>(dst, src, W * (int)sizeof(T));
}

// ============================================================================
// Mixed-path Jv in 2-D (float32): the forward difference F(u + eps V) - F(u)
// formed term by term, free of cancellation.  With a = u, b = eps V (per field
// eps scale_f) and the midpoint m = a + b/2 of the two states,
//   convection  a'_j phi' - a_j phi = m_j b_phi + b_j m_phi,
//   diffusion   K' D phi' - K D phi = Km D b_phi + dK D m_phi,
//               Km = (K + K')/2, dK = K' - K in cancellation-free form,
//   pressure    (pbar + p') div' - (pbar + p) div = (pbar + m_p) div b + b_p div m,
// so each flux difference X_phi = Km D_x b + dK D_x m - 1/2 (m_u b_phi + b_u m_phi)
// (Z_phi alike) is formed once per point and
//   dF_phi = D_x X_phi + D_z Z_phi + S_phi.
// Phase 1 stages u and the raw direction v of a TX x TZ tile with a halo of 4
// (cp.async; D(b) = eps D(v) is scaled in registers).  Phase 2 forms, for W
// consecutive points per thread, both fluxes and the point-wise part S (kept in
// registers), and on the arms X (two columns either side) or Z (two rows above
// and below) alone.  Phase 3 differentiates the fluxes and writes Jv.
// The arithmetic is explicitly rounded, so a flux formed in a tile and the same
// flux formed in a neighbour's arm are bitwise equal and every tile shape gives
// the same result for the same step eps.  The eddy coefficient of a point in a ghost row is that of
// its mirror image.
//
// Bound: issue and shared-memory latency.  The form with one point per thread,
// diffusive and convective fluxes apart and products about a: 22 us at
// 1024 x 512 and 7.4 us at 250 x 119; this form 17.5 and 5.3 us.
// ============================================================================
// The strain magnitude s = sqrt(2 S:S) at a, at a' = a + b, and their
// difference ds = s' - s in cancellation-free form, from the velocity
// gradients of a (ux, uz, wx, wz) and of b.
__device__ __forceinline__ void jv_strain(float aux, float auz, float awx, float awz, float bux, float buz,
                                          float bwx, float bwz, float& sa, float& sp, float& ds) {
    const float a13 = __fmul_rn(0.5f, __fadd_rn(auz, awx)), b13 = __fmul_rn(0.5f, __fadd_rn(buz, bwx));
    const float ssa = __fmaf_rn(aux, aux, __fmaf_rn(awz, awz, __fmul_rn(2.f, __fmul_rn(a13, a13))));
    // S':S' - S:S = (2 S + S_b) : S_b
    const float dss = __fmaf_rn(__fmaf_rn(2.f, aux, bux), bux,
                                __fmaf_rn(__fmaf_rn(2.f, awz, bwz), bwz,
                                          __fmul_rn(2.f, __fmul_rn(__fmaf_rn(2.f, a13, b13), b13))));
    // square roots and the quotient by the special-function unit (x rsqrt(x), a / b via
    // the approximate reciprocal): a few ulp, deterministic
    const float s1 = __fmul_rn(2.f, ssa);
    sa = s1 > 0.f ? __fmul_rn(s1, rsqrtf(s1)) : 0.f;
    const float s2 = __fmul_rn(2.f, __fadd_rn(ssa, dss));
    sp = s2 > 0.f ? __fmul_rn(s2, rsqrtf(s2)) : 0.f;
    // s' - s = 2 (S':S' - S:S) / (s' + s)
    const float den = __fadd_rn(sa, sp);
    ds = den > 0.f ? __fdividef(__fmul_rn(2.f, dss), den) : 0.f;
}

// Deardorff heat factor g(s) = s (1 + a l(s)), l = min(Delta, c_l s), at s and
// its difference g(s') - g(s) = ds (1 + a l') + a s (l' - l), with l' - l = c_l ds
// where neither side is capped (0 where both are; direct where they straddle).
__device__ __forceinline__ void jv_heat(const Geo& G, float sa, float sp, float ds, float a, float& g, float& dg) {
    const float cl = G.f32.dd_cl, dlt = G.f32.dd_delta;
    float la = dlt, lp = dlt, dl = 0.f;
    if (cl >= 0.f) {
        const float ta = __fmul_rn(cl, sa), tp = __fmul_rn(cl, sp);
        la = ta < dlt ? ta : dlt;
        lp = tp < dlt ? tp : dlt;
        if (ta < dlt && tp < dlt) dl = __fmul_rn(cl, ds);
        else if (ta < dlt || tp < dlt) dl = __fsub_rn(lp, la);
    }
    g = __fmul_rn(sa, __fmaf_rn(a, la, 1.f));
    dg = __fmaf_rn(ds, __fmaf_rn(a, lp, 1.f), __fmul_rn(__fmul_rn(a, sa), dl));
}

template <int W, int NT>
struct JvShape {
    static constexpr int NXT = W == 4 ? 16 : 32, TX = NXT * W, TZ = NT / NXT;
    static constexpr int SX = TX + 2 * HALO, SZ = TZ + 2 * HALO, PLANE = SX * SZ;
    static constexpr int XN = TZ * SX;                 // X flux of one field (rows padded like the staged ones)
    static constexpr int ZN = (TZ + 2 * R) * TX;       // Z flux of one field
    static constexpr int ZARM = 2 * R * NXT, XARM = 2 * R * TZ;      // arm items: W points, one point
    static constexpr size_t smem = sizeof(float) * (size_t)(8 * PLANE + 4 * XN + 4 * ZN);
};

// D_x / D_z of the W points at staged index i of a plane
template <int W>
__device__ __forceinline__ void jv_dx(const float* __restrict__ s, int i, float w1, float w2, float (&d)[W]) {
    float e[W + 4];
    if constexpr (W == 1) {
#pragma unroll
        for (int k = 0; k < 5; ++k) e[k] = s[i + k - 2];
    } else {
#pragma unroll
        for (int k = 0; k < W + 4; k += 2) {
            const float2 v = *reinterpret_cast<const float2*>(s + i - 2 + k);
            e[k] = v.x;
            e[k + 1] = v.y;
        }
    }
#pragma unroll
    for (int k = 0; k < W; ++k)
        d[k] = __fmaf_rn(w1, __fsub_rn(e[k + 3], e[k + 1]), __fmul_rn(w2, __fsub_rn(e[k + 4], e[k])));
}
template <int W>
__device__ __forceinline__ void jv_dz(const float* __restrict__ s, int i, int st, float w1, float w2, float (&d)[W]) {
    float a[W], b[W], c[W], e[W];
    rload<float, W>(s + i - 2 * st, a);
    rload<float, W>(s + i - st, b);
    rload<float, W>(s + i + st, c);
    rload<float, W>(s + i + 2 * st, e);
#pragma unroll
    for (int k = 0; k < W; ++k)
        d[k] = __fmaf_rn(w1, __fsub_rn(c[k], b[k]), __fmul_rn(w2, __fsub_rn(e[k], a[k])));
}

// Phase 2 at W points (staged index i; is: the index whose eddy coefficient they
// take).  XF / ZF: form the X / Z fluxes; both: tile points with their part S.
template <int W, int SMAG, bool XF, bool ZF, int SX, int PLANE, int XN, int ZN>
__device__ __forceinline__ void jv_points(const Geo& G, const float (&ev)[4], const float* __restrict__ st, int i, int is,
                                          float* __restrict__ X, float* __restrict__ Z, float (&S)[4][W]) {
    constexpr bool CEN = XF && ZF;
    const float wx1 = G.f32.wx1, wx2 = G.f32.wx2, wz1 = G.f32.wz1, wz2 = G.f32.wz2;
    const float* U = st;                     // u planes 0..3
    const float* V = st + 4 * PLANE;         // raw v planes 0..3
    // velocity gradients of a and b (b by its eps)
    float ax[2][W], az[2][W], bx[2][W], bz[2][W];
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        if (XF || SMAG) {
            jv_dx<W>(U + f * PLANE, i, wx1, wx2, ax[f]);
            jv_dx<W>(V + f * PLANE, i, wx1, wx2, bx[f]);
        }
        if (ZF || SMAG) {
            jv_dz<W>(U + f * PLANE, i, SX, wz1, wz2, az[f]);
            jv_dz<W>(V + f * PLANE, i, SX, wz1, wz2, bz[f]);
        }
#pragma unroll
        for (int k = 0; k < W; ++k) {
            if (XF || SMAG) bx[f][k] = __fmul_rn(ev[f], bx[f][k]);
            if (ZF || SMAG) bz[f][k] = __fmul_rn(ev[f], bz[f][k]);
        }
    }
    // exchange coefficients: midpoint and difference, momentum [0] and heat [1], along x and z
    float kx[2][W], dkx[2][W], kz[2][W], dkz[2][W];
    if (SMAG) {
        float sa[W], sp[W], ds[W];
        if (is == i) {
#pragma unroll
            for (int k = 0; k < W; ++k)
                jv_strain(ax[0][k], az[0][k], ax[1][k], az[1][k], bx[0][k], bz[0][k], bx[1][k], bz[1][k], sa[k], sp[k], ds[k]);
        } else {
            float cx[2][W], cz[2][W], ex[2][W], ez[2][W];
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                jv_dx<W>(U + f * PLANE, is, wx1, wx2, cx[f]);
                jv_dz<W>(U + f * PLANE, is, SX, wz1, wz2, cz[f]);
                jv_dx<W>(V + f * PLANE, is, wx1, wx2, ex[f]);
                jv_dz<W>(V + f * PLANE, is, SX, wz1, wz2, ez[f]);
            }
#pragma unroll
            for (int k = 0; k < W; ++k)
                jv_strain(cx[0][k], cz[0][k], cx[1][k], cz[1][k], __fmul_rn(ev[0], ex[0][k]), __fmul_rn(ev[0], ez[0][k]),
                          __fmul_rn(ev[1], ex[1][k]), __fmul_rn(ev[1], ez[1][k]), sa[k], sp[k], ds[k]);
        }
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const float sm = __fmaf_rn(0.5f, ds[k], sa[k]);
            if (SMAG == 2) {
                const float cm = G.f32.dd_cm, cM = G.f32.dd_cM;
                kx[0][k] = __fmul_rn(cm, sm);
                dkx[0][k] = __fmul_rn(cm, ds[k]);
                kz[0][k] = __fmul_rn(cM, sm);
                dkz[0][k] = __fmul_rn(cM, ds[k]);
                float g, dg;
                if (XF) {
                    jv_heat(G, sa[k], sp[k], ds[k], G.f32.dd_ah, g, dg);
                    kx[1][k] = __fmul_rn(cm, __fmaf_rn(0.5f, dg, g));
                    dkx[1][k] = __fmul_rn(cm, dg);
                }
                if (ZF) {
                    jv_heat(G, sa[k], sp[k], ds[k], G.f32.dd_az, g, dg);
                    kz[1][k] = __fmul_rn(cM, __fmaf_rn(0.5f, dg, g));
                    dkz[1][k] = __fmul_rn(cM, dg);
                }
            } else {
                kx[0][k] = kz[0][k] = __fmul_rn(G.f32.cs2, sm);
                dkx[0][k] = dkz[0][k] = __fmul_rn(G.f32.cs2, ds[k]);
                kx[1][k] = kz[1][k] = __fmul_rn(kx[0][k], G.f32.inv_Pr);
                dkx[1][k] = dkz[1][k] = __fmul_rn(dkx[0][k], G.f32.inv_Pr);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < W; ++k) {
            kx[0][k] = kz[0][k] = G.f32.K_M;
            kx[1][k] = kz[1][k] = G.f32.K_H;
            dkx[0][k] = dkx[1][k] = dkz[0][k] = dkz[1][k] = 0.f;
        }
    }
    // half the advecting velocities, midpoint and b
    float mu[W], bu[W], mw[W], bw[W];
    {
        float a[W], v[W];
        rload<float, W>(U + i, a);
        rload<float, W>(V + i, v);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const float b = __fmul_rn(ev[0], v[k]);
            bu[k] = __fmul_rn(0.5f, b);
            mu[k] = __fmul_rn(0.5f, __fadd_rn(a[k], bu[k]));
        }
        rload<float, W>(U + PLANE + i, a);
        rload<float, W>(V + PLANE + i, v);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const float b = __fmul_rn(ev[1], v[k]);
            bw[k] = __fmul_rn(0.5f, b);
            mw[k] = __fmul_rn(0.5f, __fadd_rn(a[k], bw[k]));
        }
    }
    float divb[W], divm[W];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        float a[W], v[W], dax[W], daz[W], dbx[W], dbz[W];
        rload<float, W>(U + f * PLANE + i, a);
        rload<float, W>(V + f * PLANE + i, v);
        const bool needx = XF && (f < 3 || CEN), needz = ZF && (f < 3 || CEN);
        if (f < 2) {
#pragma unroll
            for (int k = 0; k < W; ++k) {
                dax[k] = ax[f][k];
                daz[k] = az[f][k];
                dbx[k] = bx[f][k];
                dbz[k] = bz[f][k];
            }
        } else {
            if (needx) {
                jv_dx<W>(U + f * PLANE, i, wx1, wx2, dax);
                jv_dx<W>(V + f * PLANE, i, wx1, wx2, dbx);
            }
            if (needz) {
                jv_dz<W>(U + f * PLANE, i, SX, wz1, wz2, daz);
                jv_dz<W>(V + f * PLANE, i, SX, wz1, wz2, dbz);
            }
#pragma unroll
            for (int k = 0; k < W; ++k) {
                if (needx) dbx[k] = __fmul_rn(ev[f], dbx[k]);
                if (needz) dbz[k] = __fmul_rn(ev[f], dbz[k]);
            }
        }
        float Xv[W], Zv[W];
        const int h = f == 2 ? 1 : 0;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const float b = __fmul_rn(ev[f], v[k]), m = __fmaf_rn(0.5f, b, a[k]);
            float dmx = 0.f, dmz = 0.f;
            if (needx) dmx = __fmaf_rn(0.5f, dbx[k], dax[k]);
            if (needz) dmz = __fmaf_rn(0.5f, dbz[k], daz[k]);
            if (XF) {
                float x = -__fmaf_rn(mu[k], b, __fmul_rn(bu[k], m));
                if (f < 3) {
                    x = __fmaf_rn(kx[h][k], dbx[k], x);
                    if (SMAG) x = __fmaf_rn(dkx[h][k], dmx, x);
                }
                Xv[k] = x;
            }
            if (ZF) {
                float z = -__fmaf_rn(mw[k], b, __fmul_rn(bw[k], m));
                if (f < 3) {
                    z = __fmaf_rn(kz[h][k], dbz[k], z);
                    if (SMAG) z = __fmaf_rn(dkz[h][k], dmz, z);
                }
                Zv[k] = z;
            }
            if (CEN) {
                float s = -__fmaf_rn(mu[k], dbx[k], __fmaf_rn(bu[k], dmx, __fmaf_rn(mw[k], dbz[k], __fmul_rn(bw[k], dmz))));
                if (f == 0) { divb[k] = dbx[k]; divm[k] = dmx; }
                if (f == 1) {
                    divb[k] = __fadd_rn(divb[k], dbz[k]);
                    divm[k] = __fadd_rn(divm[k], dmz);
                    S[2][k] = -__fmul_rn(G.f32.beta, b);
                }
                if (f == 2) {
                    s = __fadd_rn(s, S[2][k]);
                    S[1][k] = __fmaf_rn(G.f32.gth, b, S[1][k]);
                }
                if (f == 3) {
                    S[0][k] = __fmaf_rn(-G.f32.theta0, dbx[k], S[0][k]);
                    S[1][k] = __fmaf_rn(-G.f32.theta0, dbz[k], S[1][k]);
                    s = __fmaf_rn(-G.f32.gamma_p, __fmaf_rn(__fadd_rn(G.f32.pbar, m), divb[k], __fmul_rn(b, divm[k])), s);
                }
                S[f][k] = s;
            }
        }
        if (XF) rstore<float, W>(X + f * XN, Xv);
        if (ZF) rstore<float, W>(Z + f * ZN, Zv);
    }
}

template <int W, int NT, int SMAG>
__global__ void __launch_bounds__(NT, 512 / NT)
jv2d(Geo G, const float* __restrict__ u, const float* __restrict__ v, float* __restrict__ out,
     const double* part, Ctl* ctl, int check_done) {
    using SH = JvShape<W, NT>;
    constexpr int TX = SH::TX, TZ = SH::TZ, SX = SH::SX, SZ = SH::SZ, PLANE = SH::PLANE, XN = SH::XN, ZN = SH::ZN;
    constexpr int RV = SX / W;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* st = reinterpret_cast<float*>(smem_raw);      // u (planes 0-3) and raw v (planes 4-7)
    float* X = st + 8 * PLANE;                           // [4][TZ][SX], tile column 0 at HALO
    float* Z = X + 4 * XN;                               // [4][TZ + 4][TX]
    pdl_wait();
    const int done = check_done ? ctl->done : 0;
    const int x0 = blockIdx.x * TX, z0 = tile_row() * TZ;
    const size_t np = (size_t)G.npt;
    if (done || z0 >= G.nz) return;
    for (int j = threadIdx.x; j < SZ * RV; j += NT) {
        const int iz = j / RV, ix = (j % RV) * W;
        int side;
        // rows beyond one reflection feed no output
        const int sz = min(max(mirror_z(z0 + iz - HALO, G.nz, side), 0), G.nz - 1);
        const size_t o = (size_t)sz * G.nx + wrap_x(x0 + ix - HALO, G.nx);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            cpa_vec<float, W>(st + f * PLANE + iz * SX + ix, u + f * np + o);
            cpa_vec<float, W>(st + (4 + f) * PLANE + iz * SX + ix, v + f * np + o);
        }
    }
    cpa_commit();
    // the step, while the copies are in flight
    const double2 eps = pending_eps(ctl, part);
    __shared__ float evs[4], cfs[4];
    if (threadIdx.x < 4) {
        evs[threadIdx.x] = (float)(eps.x * G.scale[threadIdx.x]);
        cfs[threadIdx.x] = (float)(eps.y * G.inv_scale[threadIdx.x]);
    }
    cpa_wait<0>();
    __syncthreads();
    float ev[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) ev[f] = evs[f];
    if (z0 - HALO < 0 || z0 + TZ + HALO > G.nz) {        // ghost rows: signs of the odd fields
        for (int j = threadIdx.x; j < PLANE; j += NT) {
            int side;
            mirror_z(z0 + j / SX - HALO, G.nz, side);
#pragma unroll
            for (int f = 0; f < 4; ++f)
                if (odd_ghost(G, f, side)) {
                    st[f * PLANE + j] = flip(st[f * PLANE + j]);
                    st[(4 + f) * PLANE + j] = flip(st[(4 + f) * PLANE + j]);
                }
        }
        __syncthreads();
    }
    auto eddy_index = [&](int iz, int ix) {              // staged index of the point whose eddy value (iz, ix) takes
        return (flux_eddy_row(iz, z0, G.nz) + HALO) * SX + ix + HALO;
    };
    const int tx = (threadIdx.x % SH::NXT) * W, tz = threadIdx.x / SH::NXT;
    float S[4][W];
    if (x0 + tx <= G.nx + 1 && z0 + tz <= G.nz + 1) {    // else it feeds no output
        const int i = (tz + HALO) * SX + tx + HALO;
        jv_points<W, SMAG, true, true, SX, PLANE, XN, ZN>(G, ev, st, i, SMAG ? eddy_index(tz, tx) : i,
                                                          X + tz * SX + tx + HALO, Z + (tz + R) * TX + tx, S);
    }
    // the arms: Z of rows -2, -1, TZ, TZ+1 (W points an item), X of columns -2, -1, TX, TX+1
    for (int w = threadIdx.x; w < SH::ZARM + SH::XARM; w += NT) {
        if (w < SH::ZARM) {
            const int a = w / SH::NXT, ix = (w % SH::NXT) * W, iz = a < 2 ? a - 2 : TZ + a - 2;
            if (x0 + ix > G.nx + 1 || z0 + iz > G.nz + 1) continue;
            const int i = (iz + HALO) * SX + ix + HALO;
            float none[4][W];
            jv_points<W, SMAG, false, true, SX, PLANE, XN, ZN>(G, ev, st, i, SMAG ? eddy_index(iz, ix) : i, X,
                                                               Z + (iz + R) * TX + ix, none);
        } else {
            const int a = (w - SH::ZARM) & 3, iz = (w - SH::ZARM) >> 2, ix = a < 2 ? a - 2 : TX + a - 2;
            if (x0 + ix > G.nx + 1 || z0 + iz > G.nz + 1) continue;
            const int i = (iz + HALO) * SX + ix + HALO;
            float none[4][1];
            jv_points<1, SMAG, true, false, SX, PLANE, XN, ZN>(G, ev, st, i, SMAG ? eddy_index(iz, ix) : i,
                                                               X + iz * SX + ix + HALO, Z, none);
        }
    }
    __syncthreads();
    if (x0 + tx < G.nx && z0 + tz < G.nz) {
        const float wx1 = G.f32.wx1, wx2 = G.f32.wx2, wz1 = G.f32.wz1, wz2 = G.f32.wz2;
        const size_t o = (size_t)(z0 + tz) * G.nx + x0 + tx;
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            float dx[W], dz[W], vc[W], r[W];
            jv_dx<W>(X + f * XN, tz * SX + tx + HALO, wx1, wx2, dx);
            jv_dz<W>(Z + f * ZN, (tz + R) * TX + tx, TX, wz1, wz2, dz);
            rload<float, W>(st + (4 + f) * PLANE + (tz + HALO) * SX + tx + HALO, vc);
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const float dF = __fadd_rn(S[f][k], __fadd_rn(dx[k], dz[k]));
                r[k] = __fmaf_rn(G.f32.two_over_dt, vc[k], __fmul_rn(-cfs[f], dF));
            }
            rstore<float, W>(out + f * np + o, r);
        }
    }
    pdl_trigger();
}

// ============================================================================
// Smagorinsky eddy field nu(u) at every point (preconditioner input) + max
// ============================================================================
template <typename T>
__global__ void __launch_bounds__(NTHREADS)
eddy2d(Geo G, const T* __restrict__ u, T* __restrict__ nu, double* part, Ctl* ctl) {
    T mxT = T(0);
    const T idx_ = GC(inv_dx), idz_ = GC(inv_dz);
    const T cs2 = G.sgs == 2 ? T(1) : GC(cs2);     // Deardorff: the strain s (coefficients follow from it)
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < G.npt; p += gridDim.x * blockDim.x) {
        const int z = p / G.nx, x = p - z * G.nx;
        T ux = T(0), uz = T(0), wx = T(0), wz = T(0);
#pragma unroll
        for (int l = 1; l <= 2; ++l) {
            const T c = l == 1 ? T(2.0 / 3.0) : T(-1.0 / 12.0);
            const int xp = wrap_x(x + l, G.nx), xm = wrap_x(x - l, G.nx);
            int sp_, sm_;
            const int zp = mirror_z(z + l, G.nz, sp_), zm = mirror_z(z - l, G.nz, sm_);
            const T sgu_p = sp_ == 2 ? T(G.pt[0]) : T(1), sgu_m = sm_ == 1 ? T(G.pb[0]) : T(1);
            const T sgw_p = sp_ == 2 ? T(G.pt[1]) : T(1), sgw_m = sm_ == 1 ? T(G.pb[1]) : T(1);
            const T* U = u;
            const T* W = u + G.npt;
            ux += c * (U[z * G.nx + xp] - U[z * G.nx + xm]);
            wx += c * (W[z * G.nx + xp] - W[z * G.nx + xm]);
            uz += c * (sgu_p * U[zp * G.nx + x] - sgu_m * U[zm * G.nx + x]);
            wz += c * (sgw_p * W[zp * G.nx + x] - sgw_m * W[zm * G.nx + x]);
        }
        const T v_ = smag_nu(ux * idx_, uz * idz_, wx * idx_, wz * idz_, cs2);
        nu[p] = v_;
        mxT = v_ > mxT ? v_ : mxT;
    }
    double mx[1] = {(double)mxT};
    block_partials_max<1>(mx, 1, part, gridDim.x, blockIdx.x);
    if (arrive_last(&ctl->counter[CNT_EDDY], gridDim.x)) {
        __shared__ double tot[1];
        final_maxes(part, gridDim.x, 1, tot);
        if (threadIdx.x == 0) ctl->kmax = tot[0];
    }
}

// ============================================================================
// Field-block Chebyshev preconditioner (Section 2.5.2): for u, w, theta the
// block A_f = (2/dt) I - sum_j D_j(K D_j .) with K frozen at the current
// iterate; the p block is (2/dt) I.  Spectrum bounds from Gershgorin:
// [2/dt, 2/dt + (3/2)^2 K_max (1/dx^2 + 1/dz^2)] ((3/2) = sum_l |phi'(l)|).
// Sweep k (k = 1 .. s-1) of the Chebyshev semi-iteration (Saad, Alg. 12.1):
//   res = r - A x_k;  d_k = rho_k rho_{k-1} d_{k-1} + (2 rho_k / delta) res;
//   x_{k+1} = x_k + d_k,   with x_1 = d_0 = r / theta_c.
// ============================================================================
// Coefficients of every sweep of every block, computed once per Newton
// iteration from the (frozen) eddy maximum: 1/theta_c, rho_k rho_{k-1} and
// 2 rho_k / delta, with rho_0 = 1/sigma, sigma = theta_c/delta.  One thread per
// block (slot 5: the pressure Helmholtz operator of the acoustic Schur
// complement, H = (2/dt) I - a sum_j D_j D_j, a = gamma_p pbar theta0 dt / 2);
// the recurrence is a serial chain of one division a sweep.  One thread doing
// all slots with three divisions a sweep took 85 us at 32 sweeps.
__global__ void pc_setup(Geo G, int sweeps, Ctl* ctl) {
    const int f = threadIdx.x;
    if (f > 5 || (f >= G.nf && f != 5)) return;
    const int fth = G.nf - 2, fp = G.nf - 1;         // theta and p
    const double h2 = G.inv_dx * G.inv_dx + G.inv_dz * G.inv_dz + (G.dim == 3 ? G.inv_dy * G.inv_dy : 0.0);
    // Deardorff: ctl->kmax is the largest strain s; every coefficient grows with s
    const double smax = ctl->kmax;
    const double lmax = G.dd_cl < 0.0 ? G.dd_delta : fmin(G.dd_delta, G.dd_cl * smax);
    const double hh2 = G.inv_dx * G.inv_dx + (G.dim == 3 ? G.inv_dy * G.inv_dy : 0.0);
    double kh2 = 0.0;        // sum_j max K_j / h_j^2
    if (f == 5) {
        kh2 = G.helm_a * h2;
    } else if (f != fp) {
        if (G.sgs == 2) {
            const double fh = f == fth ? 1.0 + G.dd_ah * lmax : 1.0;
            const double fz = f == fth ? 1.0 + G.dd_az * lmax : 1.0;
            kh2 = G.dd_cm * smax * fh * hh2 + G.dd_cM * smax * fz * G.inv_dz * G.inv_dz;
        } else {
            kh2 = (G.smag ? ctl->kmax * (f == fth ? G.inv_Pr : 1.0) : (f == fth ? G.K_H : G.K_M)) * h2;
        }
    }
    const double lo = G.two_over_dt, hi = lo + 2.25 * kh2;
    const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo);
    const bool degenerate = delta <= 1e-14 * theta;
    const double sigma = degenerate ? 1.0 : theta / delta, ith = 1.0 / theta;
    const double two_over_delta = degenerate ? 0.0 : 2.0 / delta;
    auto put = [&](int k, double c1, double c2) {
        ctl->cheb[f][k][0] = ith;
        ctl->cheb[f][k][1] = c1;
        ctl->cheb[f][k][2] = c2;
        ctl->chebf[f][k][0] = (float)ith;
        ctl->chebf[f][k][1] = (float)c1;
        ctl->chebf[f][k][2] = (float)c2;
    };
    double rho = 1.0 / sigma;
    put(0, 0.0, 0.0);
    for (int k = 1; k < sweeps && k < MAX_PC_SWEEPS; ++k) {
        const double rho_new = 1.0 / (2.0 * sigma - rho);
        put(k, degenerate ? 0.0 : rho_new * rho, rho_new * two_over_delta);
        rho = rho_new;
    }
}

// ----------------------------------------------------------------------------
// Field-block sweep, float32: one CTA sweeps all fields of a TX x TZ tile.  The
// three diffused fields (halo 4) and the eddy field (halo 2) are copied to
// shared memory at once, so a launch waits for memory once and meets one
// barrier; a thread owns W consecutive points along x and forms every flux its D
// reads itself (8 along x, 4 rows along z): twice the arithmetic of exchanging
// them, but no second phase.  first / last: roles of the sweep (both with
// pc_sweeps = 2); p is written by the last sweep.  Explicitly rounded, so every
// tile shape computes the same bits.
//
// Bound: latency of the one load phase and issue (19 MB a launch at
// 1024 x 512, 2.8 us).  One field per CTA with three barriers and the fluxes in
// shared memory took 19-20 us there and 7.1-7.8 us at 250 x 119; this form 11.2 and 4.4 us (with
// the overlap of the launches before it).  1024 threads an SM need 64 registers a
// thread, at which the 16-byte rows spill 80 bytes (Deardorff 136); 72 registers and
// three CTAs per SM, with the first field's loads hoisted over the loop, took 12.0 us.
// ----------------------------------------------------------------------------
template <int W> struct PcRow { static constexpr int NXT = W == 4 ? 16 : 32; };   // threads along x

template <int W, int NT, int SMAG>
__global__ void __launch_bounds__(NT, 1024 / NT)
cheb2d(Geo G, int k, int first, int last, const float* __restrict__ r, const float* __restrict__ zin,
       const float* __restrict__ din, float* __restrict__ zout, float* __restrict__ dout, const float* __restrict__ nu,
       double* part, Ctl* ctl, int check_done) {
    using T = float;
    constexpr int NXT = PcRow<W>::NXT, TX = NXT * W, TZ = NT / NXT;
    constexpr int SX = TX + 2 * HALO, SZ = TZ + 2 * HALO, KZ = TZ + 2 * R, RV = SX / W;
    __shared__ __align__(16) T zs[3][SZ * SX];
    __shared__ __align__(16) T ks[SMAG ? KZ * SX : 4];
    pdl_wait();
    const int done = check_done ? ctl->done : 0;
    const int x0 = blockIdx.x * TX, z0 = tile_row() * TZ;
    const T* src = first ? r : zin;
    const size_t np = (size_t)G.npt;
    // storage row of global row gz (rows beyond one reflection feed no output)
    auto row = [&](int gz) {
        int side;
        return min(max(mirror_z(gz, G.nz, side), 0), G.nz - 1) * G.nx;
    };
    for (int j = threadIdx.x; j < SZ * RV; j += NT) {
        const int iz = j / RV, ix = (j % RV) * W;
        const int o = row(z0 + iz - HALO) + wrap_x(x0 + ix - HALO, G.nx);
#pragma unroll
        for (int f = 0; f < 3; ++f) cpa_vec<T, W>(&zs[f][iz * SX + ix], src + f * np + o);
        if (SMAG && iz >= R && iz < SZ - R) cpa_vec<T, W>(&ks[(iz - R) * SX + ix], nu + o);
    }
    cpa_commit();
    const int tx = (threadIdx.x % NXT) * W, tz = threadIdx.x / NXT;
    const int gx = x0 + tx, gz = z0 + tz;
    const bool inside = gx < G.nx && gz < G.nz;
    const size_t own = inside ? (size_t)gz * G.nx + gx : 0;
    T pv[W];
    if (inside && !done && last) rload<T, W>(r + 3 * np + own, pv);
    cpa_wait<0>();
    if (done) return;
    __syncthreads();
    if (z0 - HALO < 0 || z0 + TZ + HALO > G.nz) {      // ghost rows: signs of the odd fields
        for (int j = threadIdx.x; j < SZ * SX; j += NT) {
            int side;
            mirror_z(z0 + j / SX - HALO, G.nz, side);
#pragma unroll
            for (int f = 0; f < 3; ++f)
                if (odd_ghost(G, f, side)) zs[f][j] = flip(zs[f][j]);
        }
        __syncthreads();
    }
    T acc[1] = {T(0)};
    if (inside) {
        const T wx1 = G.f32.wx1, wx2 = G.f32.wx2, wz1 = G.f32.wz1, wz2 = G.f32.wz2;
        const int me = (tz + HALO) * SX + tx + HALO, mk = (tz + R) * SX + tx + HALO;
#pragma unroll 1
        for (int f = 0; f < 3; ++f) {
            const T ith = cheb_coef<T>(ctl, f, k, 0), a1 = cheb_coef<T>(ctl, f, k, 1), a2 = cheb_coef<T>(ctl, f, k, 2);
            const T* p = zs[f];
            // what the fluxes leave out: c_m, c_M (Deardorff), 1/Pr of theta, the constant K, 1/theta_c of x_1 = r / theta_c
            const T ks_ = SMAG == 2 ? T(1) : SMAG ? (f == 2 ? G.f32.inv_Pr : T(1)) : (f == 2 ? G.f32.K_H : G.f32.K_M);
            T rv[W], dv[W], xk[W], e[W + 8], difx[W], difz[W];
            if (!first) {
                rload<T, W>(r + f * np + own, rv);
                rload<T, W>(din + f * np + own, dv);
            }
            if constexpr (W == 1) {
#pragma unroll
                for (int i = 0; i < 9; ++i) e[i] = p[me - 4 + i];
            } else {
#pragma unroll
                for (int i = 0; i < W + 8; i += W) {
                    T v[W];
                    rload<T, W>(p + me - 4 + i, v);
#pragma unroll
                    for (int j = 0; j < W; ++j) e[i + j] = v[j];
                }
            }
            {
                T fx[W + 4], kx[W + 4];                 // kx: eddy values on the x arm
                if (SMAG) {
#pragma unroll
                    for (int i = 0; i < W + 4; i += 2) {
                        if constexpr (W == 1) {
                            kx[i] = ks[mk - 2 + i];
                            if (i + 1 < W + 4) kx[i + 1] = ks[mk - 1 + i];
                        } else {
                            const float2 v = *reinterpret_cast<const float2*>(&ks[mk - 2 + i]);
                            kx[i] = v.x;
                            kx[i + 1] = v.y;
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < W + 4; ++i) {
                    const T d = rfma(wx1, e[i + 3] - e[i + 1], rmul(wx2, e[i + 4] - e[i]));
                    const T c = SMAG == 2 ? (f == 2 ? dd_heat(kx[i], G.f32.dd_ah, G) : kx[i]) : kx[i];
                    fx[i] = SMAG ? rmul(c, d) : d;
                }
#pragma unroll
                for (int i = 0; i < W; ++i) difx[i] = rfma(wx1, fx[i + 3] - fx[i + 1], rmul(wx2, fx[i + 4] - fx[i]));
            }
            {
                T v[9][W], fz[4][W], kz[4][W];          // kz: eddy values on the z arm
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    if (q != 4) rload<T, W>(p + me + (q - 4) * SX, v[q]);
                if (SMAG) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) rload<T, W>(&ks[mk + (q < 2 ? q - 2 : q - 1) * SX], kz[q]);
                }
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    v[4][i] = e[4 + i];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int c = q < 2 ? q + 2 : q + 3;             // rows -2, -1, 1, 2
                        const T d = rfma(wz1, v[c + 1][i] - v[c - 1][i], rmul(wz2, v[c + 2][i] - v[c - 2][i]));
                        const T kq = SMAG == 2 ? (f == 2 ? dd_heat(kz[q][i], G.f32.dd_az, G) : kz[q][i]) : kz[q][i];
                        fz[q][i] = SMAG ? rmul(kq, d) : d;
                    }
                    difz[i] = rfma(wz1, fz[2][i] - fz[1][i], rmul(wz2, fz[3][i] - fz[0][i]));
                }
            }
            T xo[W], dk[W];
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const T sum = SMAG == 2 ? rfma(G.f32.dd_cm, difx[i], rmul(G.f32.dd_cM, difz[i])) : rmul(ks_, __fadd_rn(difx[i], difz[i]));
                xk[i] = first ? rmul(ith, e[4 + i]) : e[4 + i];
                const T rr = first ? e[4 + i] : rv[i];
                const T res = __fsub_rn(rr, rfma(G.f32.two_over_dt, xk[i], -(first ? rmul(ith, sum) : sum)));
                dk[i] = rfma(a1, first ? xk[i] : dv[i], rmul(a2, res));
                xo[i] = __fadd_rn(xk[i], dk[i]);
                if (last) acc[0] = rfma(xo[i], xo[i], acc[0]);
            }
            rstore<T, W>(zout + f * np + own, xo);
            if (!last) rstore<T, W>(dout + f * np + own, dk);
        }
        if (last) {                                     // p block: (2/dt) I, exact in one step
            const T ith = cheb_coef<T>(ctl, 3, k, 0);
#pragma unroll
            for (int i = 0; i < W; ++i) {
                pv[i] = rmul(pv[i], ith);
                acc[0] = rfma(pv[i], pv[i], acc[0]);
            }
            rstore<T, W>(zout + 3 * np + own, pv);
        }
    }
    pdl_trigger();
    if (last) {
        // ||z||^2 stays pending, one float-float partial per block: the Jacobian
        // product that follows adds them (pending_eps), so this launch ends without
        // an arrival count and a serial tail
        const int blk = tile_row() * gridDim.x + blockIdx.x;
        block_partial_ff(acc[0], reinterpret_cast<float2*>(part), blk);
        if (blk == 0 && threadIdx.x == 0) ctl->eps_part = gridDim.x * gridDim.y * gridDim.z;
    }
}

// ----------------------------------------------------------------------------
// Field-block sweep, float64: one CTA = one field of one tile (blockIdx.z: u, w,
// theta, and p for the last sweep).  The fluxes K D_x x (tile rows, two columns
// either side) and K D_z x (tile columns, two rows either side) are formed once
// in shared memory, then differentiated.
// Bound: the FP64 pipe, about 28 operations a point and field plus the arms (37
// and the products rebuilt at every tap before), so the tile follows the grid as
// flux2d's does: 160 -> 115 us at 1024 x 512.
// ----------------------------------------------------------------------------
template <int SMAG>
__global__ void __launch_bounds__(NTHREADS)
cheb2d_f64(Geo G, int k, int first, int last, FluxShape sh, int aligned, const double* __restrict__ r,
           const double* __restrict__ zin, const double* __restrict__ din, double* __restrict__ zout,
           double* __restrict__ dout, const double* __restrict__ nu, double* part, Ctl* ctl, int check_done) {
    using T = double;
    pdl_wait();
    if (check_done && ctl->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int TX = sh.tx(), TZ = sh.tz(), CN = sh.cn(), SX = sh.sx(), PXW = TX + 2 * R;
    T* zs = reinterpret_cast<T*>(smem_raw);             // [SZ][SX] iterate (r for a first sweep)
    T* X = zs + sh.plane();                             // [TZ][TX + 4] K D_x
    T* Z = X + sh.xn();                                 // [TZ + 4][TX] K D_z
    const int fld = blockIdx.z, x0 = blockIdx.x << sh.lx, z0 = blockIdx.y << sh.lz;
    const T ith = ctl->cheb[fld][k][0], a1 = ctl->cheb[fld][k][1], a2 = ctl->cheb[fld][k][2];
    const size_t fo = (size_t)fld * G.npt;
    double acc[1] = {0.0};
    if (fld == 3) {
        for (int w = threadIdx.x; w < CN; w += NTHREADS) {      // p block: (2/dt) I, exact in one step
            const int gx = x0 + (w & (TX - 1)), gz = z0 + (w >> sh.lx);
            if (gx >= G.nx || gz >= G.nz) continue;
            const size_t o = fo + (size_t)gz * G.nx + gx;
            const T zv = r[o] * ith;
            zout[o] = zv;
            acc[0] = fma(zv, zv, acc[0]);
        }
    } else {
        const T none[4] = {0.0, 0.0, 0.0, 0.0};
        load_fields<T, 0, 1>(zs, first ? r : zin, nullptr, none, G, aligned, x0, z0, SX, TZ + 2 * HALO, fld);
        __syncthreads();
        // eddy coefficient of the point at tile (ix, iz), its constant factors left to the end
        auto coef = [&](int ix, int iz, bool zarm) -> T {
            int side;
            const int sz = min(max(mirror_z(z0 + iz, G.nz, side), 0), G.nz - 1);
            const T v = nu[(size_t)sz * G.nx + wrap_x(x0 + ix, G.nx)];
            return SMAG == 2 && fld == 2 ? dd_heat(v, zarm ? G.dd_az : G.dd_ah, G) : v;
        };
        for (int w = threadIdx.x; w < TZ * PXW; w += NTHREADS) {
            const int iz = w / PXW, ix = w - iz * PXW - R;
            const T d = wd(zs, (iz + HALO) * SX + ix + HALO, 1, G.wx1, G.wx2);
            X[w] = SMAG ? coef(ix, iz, false) * d : d;
        }
        for (int w = threadIdx.x; w < TX * (TZ + 2 * R); w += NTHREADS) {
            const int iz = (w >> sh.lx) - R, ix = w & (TX - 1);
            const T d = wd(zs, (iz + HALO) * SX + ix + HALO, SX, G.wz1, G.wz2);
            Z[w] = SMAG ? coef(ix, iz, true) * d : d;
        }
        __syncthreads();
        // factors the fluxes leave out, with 1/theta_c of x_1 = r / theta_c
        const T one = first ? ith : 1.0;
        const T kf = SMAG == 2 ? 1.0 : SMAG ? (fld == 2 ? G.inv_Pr : 1.0) : (fld == 2 ? G.K_H : G.K_M);
        const T cx = (SMAG == 2 ? G.dd_cm : kf) * one, cz = (SMAG == 2 ? G.dd_cM : kf) * one;
        const T wx1 = cx * G.wx1, wx2 = cx * G.wx2, wz1 = cz * G.wz1, wz2 = cz * G.wz2;
        for (int w = threadIdx.x; w < CN; w += NTHREADS) {
            const int tz = w >> sh.lx, tx = w & (TX - 1);
            const int gx = x0 + tx, gz = z0 + tz;
            if (gx >= G.nx || gz >= G.nz) continue;
            const size_t o = fo + (size_t)gz * G.nx + gx;
            const T* x = X + tz * PXW + tx + R;
            const T* z = Z + (tz + R) * TX + tx;
            const T xv = zs[(tz + HALO) * SX + tx + HALO];
            const T xk = first ? ith * xv : xv, rv = first ? xv : r[o];
            const T dif = fma(wx1, x[1] - x[-1], fma(wx2, x[2] - x[-2], fma(wz1, z[TX] - z[-TX], wz2 * (z[2 * TX] - z[-2 * TX]))));
            const T res = fma(-G.two_over_dt, xk, rv) + dif;
            const T dk = fma(a1, first ? xk : din[o], a2 * res);
            const T xn = xk + dk;
            zout[o] = xn;
            if (!last) dout[o] = dk;
            else acc[0] = fma(xn, xn, acc[0]);
        }
    }
    pdl_trigger();
    if (last) {
        const int nblk = gridDim.x * gridDim.y * gridDim.z;
        const int blk = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        block_partials<1, T>(acc, 1, part, nblk, blk);
        if (arrive_last(&ctl->counter[CNT_PC], nblk)) {
            __shared__ double tot[1];
            final_sums(part, nblk, 1, tot);
            if (threadIdx.x < 5) put_eps_norm2(ctl, tot[0]);
        }
    }
}

// p = 1 sweep count: z = r / theta_c for every field (point-wise), + eps from ||z||
template <typename T, int SMAG>
__global__ void __launch_bounds__(NTHREADS)
pc_diag(Geo G, const T* __restrict__ r, T* __restrict__ z, size_t n, double* part, Ctl* ctl,
        int check_done) {
    if (check_done && ctl->done) return;
    T acc[1] = {T(0)};
    T inv_th[5];
    for (int f = 0; f < G.nf; ++f) inv_th[f] = cheb_coef<T>(ctl, f, 0, 0);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int f = (int)(i / G.npt);
        const T zv = r[i] * inv_th[f];
        z[i] = zv;
        acc[0] += zv * zv;
    }
    block_partials<1, T>(acc, 1, part, gridDim.x, blockIdx.x);
    if (arrive_last(&ctl->counter[CNT_PC], gridDim.x)) {
        __shared__ double tot[1];
        final_sums(part, gridDim.x, 1, tot);
        if (threadIdx.x < 5) put_eps_norm2(ctl, tot[0]);
    }
}

// ============================================================================
// Acoustic Schur-complement preconditioner (2-D, scaled units).  Keeping only
// (2/dt) I and the pressure gradient / divergence couplings of Eqs.
// ch2_28-ch2_30 (linearised about pbar) -- the fast terms the semi-implicit
// scheme that Section 2.5 follows eliminates -- the velocities drop out:
//   H dp = v_p - c_div (D_x v_u + D_z v_w),   H = (2/dt) I - a sum_j D_j D_j,
//   z_u = (dt/2)(v_u - c_grad D_x dp),   z_w = (dt/2)(v_w - c_grad D_z dp),
// with c_div = gamma_p pbar (dt/2) s_u / s_p, c_grad = theta0 s_p / s_u and
// a = gamma_p pbar theta0 dt / 2.  H is inverted approximately by Chebyshev
// sweeps on its Gershgorin interval (coefficients ctl->cheb[5], pc_setup);
// theta gets r_theta / theta_c of its field block.
// ============================================================================
// D_x at W points of a periodic row (gx and nx multiples of W)
template <typename T, int W>
__device__ __forceinline__ void row_dx(const T* __restrict__ row, int gx, int nx, T w1, T w2, T (&d)[W]) {
    T e[W + 4];
    if constexpr (W == 1) {
#pragma unroll
        for (int k = 0; k < 5; ++k) e[k] = row[wrap_x(gx + k - 2, nx)];
    } else {
        T l[W], c[W], r[W];
        rload<T, W>(row + wrap_x(gx - W, nx), l);
        rload<T, W>(row + gx, c);
        rload<T, W>(row + wrap_x(gx + W, nx), r);
        e[0] = l[W - 2];
        e[1] = l[W - 1];
#pragma unroll
        for (int k = 0; k < W; ++k) e[2 + k] = c[k];
        e[W + 2] = r[0];
        e[W + 3] = r[1];
    }
#pragma unroll
    for (int i = 0; i < W; ++i) d[i] = rfma(w1, e[i + 3] - e[i + 1], rmul(w2, e[i + 4] - e[i]));
}

// D_z at W points of row gz of a plane (field parity fld, one mirror reflection)
template <typename T, int W>
__device__ __forceinline__ void row_dz(const T* __restrict__ f, const Geo& G, int gz, int gx, int fld, T w1, T w2, T (&d)[W]) {
    T a[4][W];
    constexpr int s[4] = {-2, -1, 1, 2};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        int side;
        const int sz = mirror_z(gz + s[k], G.nz, side);
        rload<T, W>(f + (size_t)sz * G.nx + gx, a[k]);
        if (odd_ghost(G, fld, side)) {
#pragma unroll
            for (int i = 0; i < W; ++i) a[k][i] = flip(a[k][i]);
        }
    }
#pragma unroll
    for (int i = 0; i < W; ++i) d[i] = rfma(w1, a[2][i] - a[1][i], rmul(w2, a[3][i] - a[0][i]));
}

// rhs = v_p - c_div (D_x v_u + D_z v_w)
template <typename T, int W>
__global__ void __launch_bounds__(NTHREADS)
schur_rhs2d(Geo G, const T* __restrict__ r, T* __restrict__ rhs, Ctl* ctl, int check_done) {
    pdl_wait();
    if (check_done && ctl->done) return;
    const unsigned nv = G.npt / W, nxv = G.nx / W;
    for (unsigned q = blockIdx.x * NTHREADS + threadIdx.x; q < nv; q += gridDim.x * NTHREADS) {
        const int gz = q / nxv, gx = (q - gz * nxv) * W;
        const size_t p = (size_t)q * W;
        T dx[W], dz[W], c[W];
        row_dx<T, W>(r + p - gx, gx, G.nx, GC(wx1), GC(wx2), dx);
        row_dz<T, W>(r + G.npt, G, gz, gx, 1, GC(wz1), GC(wz2), dz);
        rload<T, W>(r + (size_t)3 * G.npt + p, c);
#pragma unroll
        for (int i = 0; i < W; ++i) c[i] -= GC(schur_cdiv) * (dx[i] + dz[i]);
        rstore<T, W>(rhs + p, c);
    }
    pdl_trigger();
}

// ----------------------------------------------------------------------------
// S Chebyshev sweeps k .. k+S-1 for H x = rhs on one plane per launch (temporal
// blocking).  x_k of a TX x TZ tile is staged with a halo of 4 S (periodic x,
// even mirror in z; the mirrored ghost rows give the mirrored result, so ghosts
// are swept like other points); sweep s runs on the tile plus a ring of
// 4 (S - 1 - s) points.  Points are handled in groups of W along x; the groups are
// ordered tile first, then ring by ring, and dealt to the threads in that order: a
// thread keeps rhs and d of its groups in registers through all sweeps.
// float32: from one of two x buffers into the other, one barrier a sweep.  H is
// applied as the composite stencil of D taken twice, so no first derivative is
// exchanged, and in the first differences of x (HELM_DIFF), as D of D x is: x itself,
// times coefficients of which the sum is zero, cancels, and lost up to 40 times as
// much (p after 32 sweeps at 1024 x 512: relative error 4.7e-6, now 1.2e-7 as with D
// taken twice; 1 % of a launch).
// float64: D_x x and D_z x are exchanged, then differentiated again: the FP64 pipe
// counts operations, 20 a point and the arms against 33 in first differences (a Schur
// step at 1024 x 256: 12.2 against 19.0 ms).
// Needs nz >= 4 S (one reflection).
//
// Bound: a launch's fixed costs (staging latency, barriers) and issue; a plane
// is 2 MB at 1024 x 512 and stays in L2.  Per pair of sweeps the former kernel
// (D exchanged through shared memory, five barriers, no overlap of launches)
// took 11.7 us at 1024 x 512; four sweeps take 10.9 us here.
// ----------------------------------------------------------------------------
template <typename T>
struct Helm2C {
    T c0, cx[4], cz[4];             // res = rhs + c0 x + sum_k c_k (g_k - g_{-1-k}), g_k = x_{k+1} - x_k along each axis
                                    // (float64: cx, cz 0 and 1, the outer D's weights times a)
};
constexpr int HELM_THREADS = 512;
constexpr int HELM_TX = 64, HELM_TZ = 32;

template <typename T, int W, int S>
__global__ void __launch_bounds__(HELM_THREADS)
helm2d(Geo G, Helm2C<T> C, int k, int first, int last, const T* __restrict__ rhs, const T* __restrict__ xin,
       const T* __restrict__ din, T* __restrict__ xout, T* __restrict__ dout, Ctl* ctl, int check_done) {
    constexpr int TX = HELM_TX, TZ = HELM_TZ;
    constexpr int H0 = HALO * S, SX = TX + 2 * H0, SZ = TZ + 2 * H0;
    constexpr int CORE = TX * TZ / W;
    constexpr int ALL = (TX + 2 * HALO * (S - 1)) * (TZ + 2 * HALO * (S - 1)) / W;      // groups of sweep 0
    constexpr int NS = (ALL + HELM_THREADS - 1) / HELM_THREADS;
    static_assert(CORE % HELM_THREADS == 0, "whole slots of tile groups");
    constexpr int CS = CORE / HELM_THREADS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* xb = reinterpret_cast<T*>(smem_raw);         // [2][SZ][SX]; float64: x, D_x x, D_z x
    constexpr bool TWICE = sizeof(T) == sizeof(double);
    static_assert(!TWICE || W == 1, "float64: single points");
    pdl_wait();
    if (check_done && ctl->done) return;
    const int x0 = blockIdx.x * TX, z0 = blockIdx.y * TZ;
    const T ith = cheb_coef<T>(ctl, 5, k, 0);
    // storage row of global row gz (rows beyond one reflection feed no output)
    auto row = [&](int gz) {
        int side;
        return min(max(mirror_z(gz, G.nz, side), 0), G.nz - 1) * G.nx;
    };
    int off[NS], ring[NS], pos[NS];
    T rv[NS][W], dv[NS][W];
#pragma unroll
    for (int q = 0; q < NS; ++q) {
        int j = threadIdx.x + q * HELM_THREADS;
        int iz, ix, h = 0;
        if (q < CS) {
            iz = j / (TX / W);
            ix = (j % (TX / W)) * W;
        } else {
            j -= CORE;
            h = S;                                  // no group
            iz = ix = 0;
#pragma unroll
            for (int t = 1; t < S; ++t) {           // ring t: 4 rows above and below, then the two sides
                const int gw = (TX + 2 * HALO * t) / W, rows = 2 * HALO * gw;
                const int side_w = 2 * HALO / W, n = rows + (TZ + 2 * HALO * (t - 1)) * side_w;
                if (h == S && j < n) {
                    h = t;
                    if (j < rows) {
                        const int r = j / gw;
                        iz = r < HALO ? r - HALO * t : TZ + HALO * (t - 1) + r - HALO;
                        ix = (j % gw) * W - HALO * t;
                    } else {
                        const int c = (j - rows) % side_w;
                        iz = (j - rows) / side_w - HALO * (t - 1);
                        ix = c < side_w / 2 ? c * W - HALO * t : TX + HALO * (t - 1) + (c - side_w / 2) * W;
                    }
                }
                if (h == S) j -= n;
            }
        }
        ring[q] = h;
        off[q] = (iz + H0) * SX + ix + H0;
        pos[q] = row(z0 + iz) + wrap_x(x0 + ix, G.nx);
        if (h < S) {
            rload<T, W>(rhs + pos[q], rv[q]);
            if (first) {
#pragma unroll
                for (int i = 0; i < W; ++i) dv[q][i] = ith * rv[q][i];
            } else {
                rload<T, W>(din + pos[q], dv[q]);
            }
        }
    }
    {
        const T* src = first ? rhs : xin;
        const T sc = first ? ith : T(1);
        for (int j = threadIdx.x; j < SX * SZ / W; j += HELM_THREADS) {
            const int iz = j / (SX / W), ix = (j % (SX / W)) * W;
            T v[W];
            rload<T, W>(src + row(z0 + iz - H0) + wrap_x(x0 + ix - H0, G.nx), v);
#pragma unroll
            for (int i = 0; i < W; ++i) v[i] *= sc;
            rstore<T, W>(xb + j * W, v);
        }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const T* xa = TWICE ? xb : xb + (s & 1) * SX * SZ;
        T* xn = TWICE ? xb : xb + ((s + 1) & 1) * SX * SZ;
        [[maybe_unused]] T *gx = xb + SX * SZ, *gz = gx + SX * SZ;      // float64: D_x x, D_z x where this sweep reads them
        const T a1 = cheb_coef<T>(ctl, 5, k + s, 1), a2 = cheb_coef<T>(ctl, 5, k + s, 2);
        if constexpr (TWICE) {
            const int h = HALO * (S - 1 - s), RX = TX + 2 * h, RZ = TZ + 2 * h, o = (H0 - h) * SX + H0 - h;
            for (int j = threadIdx.x; j < RZ * (RX + 2 * R); j += HELM_THREADS) {
                const int i = o + j / (RX + 2 * R) * SX + j % (RX + 2 * R) - R;
                gx[i] = wd(xa, i, 1, GC(wx1), GC(wx2));
            }
            for (int j = threadIdx.x; j < (RZ + 2 * R) * RX; j += HELM_THREADS) {
                const int i = o + (j / RX - R) * SX + j % RX;
                gz[i] = wd(xa, i, SX, GC(wz1), GC(wz2));
            }
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            if (ring[q] > S - 1 - s) continue;
            const T* p = xa + off[q];
            T xo[W];
            if constexpr (TWICE) {
                const T *x = gx + off[q], *z = gz + off[q];
                const T xk = *p;
                const T r = rfma(C.c0, xk, rv[q][0]) + rfma(C.cx[0], x[1] - x[-1], rfma(C.cx[1], x[2] - x[-2],
                            rfma(C.cz[0], z[SX] - z[-SX], rmul(C.cz[1], z[2 * SX] - z[-2 * SX]))));
                dv[q][0] = rfma(a1, dv[q][0], rmul(a2, r));
                xo[0] = xk + dv[q][0];
            } else {
                T e[W + 2 * HALO], r[W];
#pragma unroll
                for (int i = 0; i < W + 2 * HALO; i += W) {
                    T v[W];
                    rload<T, W>(p - HALO + i, v);
#pragma unroll
                    for (int j = 0; j < W; ++j) e[i + j] = v[j];
                }
                T g[W + 2 * HALO - 1];                      // first differences along the row
#pragma unroll
                for (int i = 0; i < W + 2 * HALO - 1; ++i) g[i] = e[i + 1] - e[i];
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    r[i] = rv[q][i] + C.c0 * e[HALO + i];
#pragma unroll
                    for (int l = 0; l < HALO; ++l) r[i] += C.cx[l] * (g[HALO + i + l] - g[HALO - 1 + i - l]);
                }
                T pa[W], pb[W];
#pragma unroll
                for (int i = 0; i < W; ++i) pa[i] = pb[i] = e[HALO + i];
#pragma unroll
                for (int l = 1; l <= HALO; ++l) {
                    T a[W], b[W];
                    rload<T, W>(p + l * SX, a);
                    rload<T, W>(p - l * SX, b);
#pragma unroll
                    for (int i = 0; i < W; ++i) {
                        r[i] += C.cz[l - 1] * ((a[i] - pa[i]) - (pb[i] - b[i]));
                        pa[i] = a[i];
                        pb[i] = b[i];
                    }
                }
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    dv[q][i] = a1 * dv[q][i] + a2 * r[i];
                    xo[i] = e[HALO + i] + dv[q][i];
                }
            }
            if (s + 1 < S) {
                rstore<T, W>(xn + off[q], xo);
            } else {
                const int j = threadIdx.x + q * HELM_THREADS;
                if (x0 + (j % (TX / W)) * W < G.nx && z0 + j / (TX / W) < G.nz) {
                    rstore<T, W>(xout + pos[q], xo);
                    if (!last) rstore<T, W>(dout + pos[q], dv[q]);
                }
            }
        }
        if (s + 1 < S) __syncthreads();
    }
    pdl_trigger();
}

// z_u, z_w from the pressure solution (already in plane 3 of z), z_theta, and
// the finite-difference step eps from ||z|| (float32: pending, as float64 partials).
template <typename T, int W>
__global__ void __launch_bounds__(NTHREADS)
schur_back2d(Geo G, const T* __restrict__ r, T* __restrict__ z, double* part, Ctl* ctl, int check_done) {
    pdl_wait();
    if (check_done && ctl->done) return;
    const T cgrad = GC(schur_cgrad), hdt = GC(half_dt);
    const T ith_t = cheb_coef<T>(ctl, 2, 0, 0);
    const size_t np = (size_t)G.npt;
    const T* dp = z + 3 * np;
    T acc[1] = {T(0)};
    const unsigned nv = G.npt / W, nxv = G.nx / W;
    for (unsigned q = blockIdx.x * NTHREADS + threadIdx.x; q < nv; q += gridDim.x * NTHREADS) {
        const int gz = q / nxv, gx = (q - gz * nxv) * W;
        const size_t p = (size_t)q * W;
        T dx[W], dz[W], ru[W], rw[W], rt[W], zp[W];
        row_dx<T, W>(dp + p - gx, gx, G.nx, GC(wx1), GC(wx2), dx);
        row_dz<T, W>(dp, G, gz, gx, 3, GC(wz1), GC(wz2), dz);
        rload<T, W>(r + p, ru);
        rload<T, W>(r + np + p, rw);
        rload<T, W>(r + 2 * np + p, rt);
        rload<T, W>(dp + p, zp);
#pragma unroll
        for (int i = 0; i < W; ++i) {
            ru[i] = hdt * (ru[i] - cgrad * dx[i]);
            rw[i] = hdt * (rw[i] - cgrad * dz[i]);
            rt[i] *= ith_t;
            acc[0] += ru[i] * ru[i] + rw[i] * rw[i] + rt[i] * rt[i] + zp[i] * zp[i];
        }
        rstore<T, W>(z + p, ru);
        rstore<T, W>(z + np + p, rw);
        rstore<T, W>(z + 2 * np + p, rt);
    }
    pdl_trigger();
    block_partials<1, T>(acc, 1, part, gridDim.x, blockIdx.x);
    if constexpr (sizeof(T) == sizeof(float)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->eps_part = -(int)gridDim.x;      // float64 partials
    } else {
        if (arrive_last(&ctl->counter[CNT_PC], gridDim.x)) {
            __shared__ double tot[1];
            final_sums(part, gridDim.x, 1, tot);
            if (threadIdx.x < 5) put_eps_norm2(ctl, tot[0]);
        }
    }
}

// ============================================================================
// Budgets: E_k = 1/2 sum (u^2 + w^2) dV, E_p = sum (lz - z) theta dV (Section 3.1.3),
// sum theta dV, sum div(u) dV, max / min of every field.
// ============================================================================
__global__ void __launch_bounds__(NTHREADS)
budgets2d(Geo G, const double* __restrict__ u, double dV, double dz, double lz, double* part,
          Ctl* ctl, double* out) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    double mx[8];
    for (int f = 0; f < 4; ++f) { mx[f] = -1e300; mx[4 + f] = -1e300; }
    const double* U = u;
    const double* W = u + G.npt;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < G.npt; p += gridDim.x * blockDim.x) {
        const int z = p / G.nx, x = p - z * G.nx;
        const double zc = (z + 0.5) * dz;
        s[0] += 0.5 * (U[p] * U[p] + W[p] * W[p]);
        s[1] += (lz - zc) * u[2 * G.npt + p];
        s[2] += u[2 * G.npt + p];
        double ux = 0.0, wz = 0.0;
        for (int l = 1; l <= 2; ++l) {
            const double c = l == 1 ? 2.0 / 3.0 : -1.0 / 12.0;
            ux += c * (U[z * G.nx + wrap_x(x + l, G.nx)] - U[z * G.nx + wrap_x(x - l, G.nx)]);
            int sp_, sm_;
            const int zp = mirror_z(z + l, G.nz, sp_), zm = mirror_z(z - l, G.nz, sm_);
            const double gp = sp_ == 2 ? G.pt[1] : 1.0, gm = sm_ == 1 ? G.pb[1] : 1.0;
            wz += c * (gp * W[zp * G.nx + x] - gm * W[zm * G.nx + x]);
        }
        s[3] += ux * G.inv_dx + wz * G.inv_dz;
        for (int f = 0; f < 4; ++f) {
            const double v = u[(size_t)f * G.npt + p];
            mx[f] = max_nan(mx[f], v);
            mx[4 + f] = max_nan(mx[4 + f], -v);
        }
    }
    double* pmax = part + 4 * gridDim.x;
    block_partials<4>(s, 4, part, gridDim.x, blockIdx.x);
    block_partials_max<8>(mx, 8, pmax, gridDim.x, blockIdx.x);
    if (arrive_last(&ctl->counter[CNT_MISC], gridDim.x)) {
        __shared__ double tot[12];
        final_sums(part, gridDim.x, 4, tot);
        final_maxes(pmax, gridDim.x, 8, tot + 4);
        if (threadIdx.x == 0) {
            for (int i = 0; i < 4; ++i) out[i] = tot[i] * dV;
            for (int f = 0; f < 4; ++f) { out[4 + f] = tot[4 + f]; out[8 + f] = -tot[8 + f]; }
        }
    }
}

// ============================================================================
// launchers
// ============================================================================
template <typename K>
static cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Tile of flux2d for a grid: the shape with the least FP64 time, counted in
// operations per sub-partition: phase 2 (81 a tile point, 45 an arm point, no
// less than one warp's 81) and phase 3 (12 a point and field), times the
// rounds of tiles over the SMs.  Large grids take 32 x 16 (arms 14 % of the
// work); where 32 x 16 leaves SMs idle (128 x 64: 16 tiles for 152 SMs) the
// smallest tile that still fits one round spreads the points over all of them.
// F(u) per tile 8x8 / 16x8 / 16x16 / 32x16: 8 / 12 / 16 / 27 us at 128 x 64,
// 18 / 16 / 16 / 27 at 250 x 119, - / - / 152 / 142 at 1024 x 512.
static FluxShape flux_shape(const Geo& G) {
    constexpr int SMS = 152;
    constexpr FluxShape cand[] = {{3, 3}, {4, 3}, {4, 4}, {5, 4}};
    FluxShape best = cand[3];
    double least = 1e300;
    for (const FluxShape& c : cand) {
        if ((G.nz + c.tz() - 1) >> c.lz > 65535 && &c != &cand[3]) continue;      // more rows than gridDim.y holds
        const long long tiles = (long long)((G.nx + c.tx() - 1) >> c.lx) * ((G.nz + c.tz() - 1) >> c.lz);
        const double cw = c.cn() / 32.0, aw = 4.0 * (c.tx() + c.tz()) / 32.0;
        const double cost = (double)((tiles + SMS - 1) / SMS) *
                            (std::max(81.0, (81.0 * cw + 45.0 * aw) / 4.0) + std::max(12.0, 12.0 * cw));
        if (cost <= least) {      // on a tie the larger tile: fewer arm points
            if (cost < least || tiles > 2 * SMS) best = c;
            least = cost;
        }
    }
    return best;
}

template <typename T, int SMAG, int PPT>
static cudaError_t launch_flux_t(const FluxShape& sh, int mode, const Geo& G, const T* u, const T* v, const T* Fu,
                                 const double* f, T* out, T* out2, double* part, Ctl* ctl, int check_done,
                                 cudaStream_t s) {
    static std::atomic<bool> configured{false};   // set once; concurrent first calls are harmless
    if (!configured) {
        const FluxShape big{5, 4};
        cudaError_t e = set_smem(flux2d<T, SMAG, PPT>, big.elems() * sizeof(T));
        if (e != cudaSuccess) return e;
        configured = true;
    }
    const size_t sm = sh.elems() * sizeof(T);
    dim3 grid((G.nx + sh.tx() - 1) >> sh.lx, (G.nz + sh.tz() - 1) >> sh.lz);
    const int aligned = rows_aligned(G, u, mode == MODE_JV ? v : nullptr);
    if (mode == MODE_JV)
        return launch_pdl(flux2d<T, SMAG, PPT>, grid, NTHREADS, sm, s, G, mode, sh, aligned, u, v, Fu, f, out, out2, part,
                          ctl, check_done);
    flux2d<T, SMAG, PPT><<<grid, NTHREADS, sm, s>>>(G, mode, sh, aligned, u, v, Fu, f, out, out2, part, ctl, check_done);
    return cudaGetLastError();
}

template <typename T, int SMAG>
static cudaError_t launch_flux(int mode, const Geo& G, const T* u, const T* v, const T* Fu, const double* f, T* out,
                               T* out2, double* part, Ctl* ctl, int check_done, cudaStream_t s) {
    const FluxShape sh = flux_shape(G);
    switch (sh.ppt()) {
        case 2: return launch_flux_t<T, SMAG, 2>(sh, mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
        case 1: return launch_flux_t<T, SMAG, 1>(sh, mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
        default: return launch_flux_t<T, SMAG, 0>(sh, mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
    }
}

template <typename T>
cudaError_t launch_stencil(int mode, const Geo& G, const T* u, const T* v, const T* Fu,
                           const double* f, T* out, T* out2, double* part, Ctl* ctl,
                           int check_done, cudaStream_t s) {
    if (G.dim == 3) return launch_stencil3d<T>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
    if (mode < MODE_F || mode > MODE_RHSRES) return cudaErrorInvalidValue;
    return G.sgs == 2 ? launch_flux<T, 2>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s)
         : G.smag     ? launch_flux<T, 1>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s)
                      : launch_flux<T, 0>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
}
template cudaError_t launch_stencil<float>(int, const Geo&, const float*, const float*, const float*,
                                           const double*, float*, float*, double*, Ctl*, int, cudaStream_t);
template cudaError_t launch_stencil<double>(int, const Geo&, const double*, const double*, const double*,
                                            const double*, double*, double*, double*, Ctl*, int, cudaStream_t);

template <int W, int NT, int SMAG>
static cudaError_t launch_jv_t(const Geo& G, const float* u, const float* v, float* out, const double* part, Ctl* ctl,
                               int check_done, cudaStream_t s) {
    using SH = JvShape<W, NT>;
    static std::atomic<bool> configured{false};   // set once; concurrent first calls are harmless
    if (!configured) {
        const cudaError_t e = set_smem(jv2d<W, NT, SMAG>, SH::smem);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    return launch_pdl(jv2d<W, NT, SMAG>, tile_grid((G.nx + SH::TX - 1) / SH::TX, (G.nz + SH::TZ - 1) / SH::TZ), dim3(NT),
                      SH::smem, s, G, u, v, out, part, ctl, check_done);
}

// Rows of 16-byte, 8-byte or single-element vectors as nx allows (u and v are
// workspace vectors: their planes start multiples of npt elements in); 256 threads
// a CTA (a step with 256 / 128 at 1024 x 512: 52.9 / 57.1 ms, at 250 x 119: 3.91 / 4.01
// ms: a smaller tile has more arms), 128 for the autotuner and jfnk_set_tiles
// (tile index 2).
int jv2d_threads(const Geo& G, int tile) { return G.dim == 3 ? 0 : (tile == 2 ? 128 : 256); }

template <int SMAG>
static cudaError_t launch_jv(const Geo& G, const float* u, const float* v, float* out, const double* part, Ctl* ctl,
                             int check_done, cudaStream_t s) {
    const bool small = jv2d_threads(G, G.tile_jv) == 128;
#define JF_JV(W) (small ? launch_jv_t<W, 128, SMAG>(G, u, v, out, part, ctl, check_done, s) \
                        : launch_jv_t<W, 256, SMAG>(G, u, v, out, part, ctl, check_done, s))
    return G.nx % 4 == 0 ? JF_JV(4) : G.nx % 2 == 0 ? JF_JV(2) : JF_JV(1);
#undef JF_JV
}

cudaError_t launch_jv_diff(const Geo& G, const float* u, const float* v, float* out, double* part, Ctl* ctl,
                           int check_done, cudaStream_t s) {
    if (G.dim == 3) return launch_jv_diff3d(G, u, v, out, ctl, check_done, s);
    if (G.sgs == 2) return launch_jv<2>(G, u, v, out, part, ctl, check_done, s);
    return G.smag ? launch_jv<1>(G, u, v, out, part, ctl, check_done, s)
                  : launch_jv<0>(G, u, v, out, part, ctl, check_done, s);
}

static int stream_blocks(size_t n) {
    size_t b = (n + NTHREADS - 1) / NTHREADS;
    return (int)(b < (size_t)MAX_STREAM_BLOCKS ? (b > 0 ? b : 1) : MAX_STREAM_BLOCKS);
}

template <typename T>
cudaError_t launch_eddy(const Geo& G, const T* u, T* nu, double* part, Ctl* ctl, cudaStream_t s) {
    if (G.dim == 3) return launch_eddy3d<T>(G, u, nu, part, ctl, s);
    eddy2d<T><<<stream_blocks(G.npt), NTHREADS, 0, s>>>(G, u, nu, part, ctl);
    return cudaGetLastError();
}
template cudaError_t launch_eddy<float>(const Geo&, const float*, float*, double*, Ctl*, cudaStream_t);
template cudaError_t launch_eddy<double>(const Geo&, const double*, double*, double*, Ctl*, cudaStream_t);

template <typename T, int SMAG>
static cudaError_t launch_pc_diag(const Geo& G, const T* r, T* z, double* part, Ctl* ctl, int check_done, cudaStream_t s,
                                  long long* launches) {
    const size_t n = (size_t)G.nf * G.npt;
    pc_diag<T, SMAG><<<stream_blocks(n), NTHREADS, 0, s>>>(G, r, z, n, part, ctl, check_done);
    if (launches) ++*launches;
    return cudaGetLastError();
}

template <int W, int NT, int SMAG>
static cudaError_t launch_precond_w(const Geo& G, int sweeps, const float* r, float* z, float* za, float* zb, float* da,
                                    float* db, const float* nu, double* part, Ctl* ctl, int check_done,
                                    cudaStream_t s, long long* launches) {
    constexpr int TX = PcRow<W>::NXT * W, TZ = NT / PcRow<W>::NXT;
    const dim3 grid = tile_grid((G.nx + TX - 1) / TX, (G.nz + TZ - 1) / TZ);
    const float* zin = nullptr;
    const float* din = nullptr;
    float* zbuf[2] = {za, zb};
    float* dbuf[2] = {da, db};
    for (int k = 1; k <= sweeps - 1; ++k) {
        const int first = k == 1, last = k == sweeps - 1;
        float* zo = last ? z : zbuf[k & 1];
        float* dO = dbuf[k & 1];
        const cudaError_t e = launch_pdl(cheb2d<W, NT, SMAG>, grid, dim3(NT), 0, s, G, k, first, last, r, zin, din, zo, dO,
                                         nu, part, ctl, check_done);
        if (launches) ++*launches;
        if (e != cudaSuccess) return e;
        zin = zo;
        din = dO;
    }
    return cudaSuccess;
}

// Rows of 16-byte, 8-byte or single-element vectors as nx allows (r and z of the
// batched and per-call paths are workspace vectors: their planes start multiples
// of npt elements in); 256, 128 or 64 threads a CTA by Geo::tile_pc, by the grid
// for tile_pc = 0: 256 where that leaves no SM without a CTA, else 128, so that the
// CTAs reach more SMs (a step at 1024 x 512 with 256 / 128 / 64: 52.9 / 53.6 / 55.5 ms;
// at 250 x 119, below the line, 3.83 / 3.81 / 3.90 ms: 256 and 128 differ by less than
// runs do).  64 is for the autotuner and jfnk_set_tiles.
int cheb2d_threads(const Geo& G, int tile) {
    constexpr int SMS = 152;
    if (G.dim == 3 || G.pc_schur) return 0;
    if (tile != 0) return tile == 1 ? 256 : (tile == 2 ? 128 : 64);
    const int w = G.nx % 4 == 0 ? 4 : (G.nx % 2 == 0 ? 2 : 1);
    return (long long)((G.nx + w - 1) / w) * G.nz >= 256LL * SMS ? 256 : 128;       // threads with a point
}

template <int SMAG>
static cudaError_t launch_precond_f32(const Geo& G, int sweeps, const float* r, float* z, float* za, float* zb, float* da,
                                      float* db, const float* nu, double* part, Ctl* ctl, int check_done,
                                      cudaStream_t s, long long* launches) {
    const int w = G.nx % 4 == 0 ? 4 : (G.nx % 2 == 0 ? 2 : 1);
    const int nt = cheb2d_threads(G, G.tile_pc);
#define JF_PC(W, NT) launch_precond_w<W, NT, SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches)
#define JF_PCW(W) (nt == 256 ? JF_PC(W, 256) : nt == 128 ? JF_PC(W, 128) : JF_PC(W, 64))
    return w == 4 ? JF_PCW(4) : w == 2 ? JF_PCW(2) : JF_PCW(1);
#undef JF_PCW
#undef JF_PC
}

template <int SMAG>
static cudaError_t launch_precond_f64(const Geo& G, int sweeps, const double* r, double* z, double* za, double* zb,
                                      double* da, double* db, const double* nu, double* part, Ctl* ctl, int check_done,
                                      cudaStream_t s, long long* launches) {
    const FluxShape sh = flux_shape(G);
    const size_t sm = (sh.plane() + sh.xn() + sh.zn()) * sizeof(double);     // 17 KB at most
    dim3 grid((G.nx + sh.tx() - 1) >> sh.lx, (G.nz + sh.tz() - 1) >> sh.lz, 3);
    const double* zin = nullptr;
    const double* din = nullptr;
    double* zbuf[2] = {za, zb};
    double* dbuf[2] = {da, db};
    for (int k = 1; k <= sweeps - 1; ++k) {
        const int first = k == 1, last = k == sweeps - 1;
        double* zo = last ? z : zbuf[k & 1];
        double* dO = dbuf[k & 1];
        grid.z = last ? 4 : 3;            // the p block is written by the last sweep only
        const cudaError_t e = launch_pdl(cheb2d_f64<SMAG>, grid, dim3(NTHREADS), sm, s, G, k, first, last, sh,
                                         (int)rows_aligned(G, first ? r : zin), r, zin, din, zo, dO, nu, part, ctl, check_done);
        if (launches) ++*launches;
        if (e != cudaSuccess) return e;
        zin = zo;
        din = dO;
    }
    return cudaSuccess;
}

template <typename T, int SMAG>
static cudaError_t launch_precond_block(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                                        const T* nu, double* part, Ctl* ctl, int check_done, cudaStream_t s,
                                        long long* launches) {
    if (sweeps <= 1) return launch_pc_diag<T, SMAG>(G, r, z, part, ctl, check_done, s, launches);
    if constexpr (sizeof(T) == sizeof(double))
        return launch_precond_f64<SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
    else
        return launch_precond_f32<SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
}

template <typename T, int W, int S>
static cudaError_t launch_helm2d(const Geo& G, const Helm2C<T>& C, int k, int first, int last, const T* rhs, const T* xin,
                                 const T* din, T* xout, T* dout, Ctl* ctl, int check_done, cudaStream_t s) {
    constexpr int TX = HELM_TX, TZ = HELM_TZ;
    constexpr int PLANES = sizeof(T) == sizeof(double) ? 3 : S > 1 ? 2 : 1;
    constexpr size_t sm = sizeof(T) * PLANES * (size_t)(TX + 2 * HALO * S) * (TZ + 2 * HALO * S);
    static std::atomic<bool> configured{false};   // set once; concurrent first calls are harmless
    if (!configured) {
        const cudaError_t e = set_smem(helm2d<T, W, S>, sm);
        if (e != cudaSuccess) return e;
        configured = true;
    }
    return launch_pdl(helm2d<T, W, S>, dim3((G.nx + TX - 1) / TX, (G.nz + TZ - 1) / TZ), dim3(HELM_THREADS), sm, s, G, C,
                      k, first, last, rhs, xin, din, xout, dout, ctl, check_done);
}

// Helmholtz sweeps of one launch with `left` still to do: at most four where the
// rows are float32 vectors (a sweep's ring is then cheap next to a launch), two
// otherwise (float64: the rings cost the FP64 pipe; single points: three times the
// loads), within one reflection of nz.
int schur2d_sweeps(const Geo& G, size_t elem, bool vec, int left) {
    return std::min(std::min(elem == sizeof(float) && vec ? 4 : 2, G.nz / HALO), left);
}

// Acoustic Schur complement: rhs (plane 0 of da), sweeps - 1 Helmholtz
// sweeps (iterates in plane 0 of za / zb, directions in planes 0 / 1 of db,
// the last one into plane 3 of z), then the back-substitution.
template <typename T, int W>
static cudaError_t launch_schur_w(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                                  double* part, Ctl* ctl, int check_done, cudaStream_t s, long long* launches) {
    constexpr int SMS = 152;
    const size_t np = (size_t)G.npt;
    const int nb = (int)std::min<size_t>((np / W + NTHREADS - 1) / NTHREADS, 4 * SMS);
    T* rhs = da;
    cudaError_t e = launch_pdl(schur_rhs2d<T, W>, dim3(nb), dim3(NTHREADS), 0, s, G, r, rhs, ctl, check_done);
    if (e != cudaSuccess) return e;
    if (launches) ++*launches;
    Helm2C<T> C;
    const double ax = G.helm_a * G.inv_dx * G.inv_dx, az = G.helm_a * G.inv_dz * G.inv_dz;
    C.c0 = T(-G.two_over_dt);
    for (int l = 0; l < 4; ++l) {
        C.cx[l] = T(HELM_DIFF[l] * ax);
        C.cz[l] = T(HELM_DIFF[l] * az);
    }
    constexpr bool TWICE = sizeof(T) == sizeof(double);      // D applied twice by single points
    constexpr int WH = TWICE ? 1 : W;
    if (TWICE) {
        C.cx[0] = T(G.helm_a * G.wx1);
        C.cx[1] = T(G.helm_a * G.wx2);
        C.cz[0] = T(G.helm_a * G.wz1);
        C.cz[1] = T(G.helm_a * G.wz2);
    }
    T* xbuf[2] = {za, zb};
    T* dbuf[2] = {db, db + np};
    const T* xin = nullptr;
    const T* din = nullptr;
    int cur = 1;                              // buffer pair the next output goes to
    for (int k = 1; k <= sweeps - 1;) {
        const int n = schur2d_sweeps(G, sizeof(T), W > 1, sweeps - k);
        const int first = k == 1, last = k + n == sweeps;
        T* xo = last ? z + 3 * np : xbuf[cur];
        T* dO = dbuf[cur];
        const T* rh = rhs;
        if constexpr (sizeof(T) == sizeof(float) && W > 1) {
            if (n == 4) e = launch_helm2d<T, WH, 4>(G, C, k, first, last, rh, xin, din, xo, dO, ctl, check_done, s);
            if (n == 3) e = launch_helm2d<T, WH, 3>(G, C, k, first, last, rh, xin, din, xo, dO, ctl, check_done, s);
        }
        if (n == 2) e = launch_helm2d<T, WH, 2>(G, C, k, first, last, rh, xin, din, xo, dO, ctl, check_done, s);
        if (n == 1) e = launch_helm2d<T, WH, 1>(G, C, k, first, last, rh, xin, din, xo, dO, ctl, check_done, s);
        if (e != cudaSuccess) return e;
        if (launches) ++*launches;
        xin = xo;
        din = dO;
        cur ^= 1;
        k += n;
    }
    e = launch_pdl(schur_back2d<T, W>, dim3(nb), dim3(NTHREADS), 0, s, G, r, z, part, ctl, check_done);
    if (launches) ++*launches;
    return e;
}

template <typename T>
static cudaError_t launch_schur(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                                double* part, Ctl* ctl, int check_done, cudaStream_t s, long long* launches) {
    // 16-byte rows: the workspace planes start multiples of npt elements in; r and z of
    // the per-call entry may be the caller's (8-byte aligned) float64 arrays
    constexpr int W = 16 / sizeof(T);
    const bool vec = G.nx % W == 0 && ((reinterpret_cast<uintptr_t>(r) | reinterpret_cast<uintptr_t>(z)) & 15) == 0;
    return vec ? launch_schur_w<T, W>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches)
               : launch_schur_w<T, 1>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches);
}

template <typename T>
cudaError_t launch_precond(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                           const T* nu, double* part, Ctl* ctl, int check_done, cudaStream_t s,
                           long long* launches) {
    if (G.pc_schur && G.dim == 2 && sweeps > 1)
        return launch_schur<T>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches);
    if (G.dim == 3 && sweeps > 1)
        return launch_precond3d<T>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
    if (G.sgs == 2)
        return launch_precond_block<T, 2>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
    return G.smag ? launch_precond_block<T, 1>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches)
                  : launch_precond_block<T, 0>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
}
template cudaError_t launch_precond<float>(const Geo&, int, const float*, float*, float*, float*, float*,
                                           float*, const float*, double*, Ctl*, int, cudaStream_t, long long*);
template cudaError_t launch_precond<double>(const Geo&, int, const double*, double*, double*, double*,
                                            double*, double*, const double*, double*, Ctl*, int, cudaStream_t,
                                            long long*);

cudaError_t launch_pc_setup(const Geo& G, int sweeps, Ctl* ctl, cudaStream_t s) {
    pc_setup<<<1, 32, 0, s>>>(G, sweeps, ctl);
    return cudaGetLastError();
}

cudaError_t launch_budgets(const Geo& G, const double* u, double dx, double dz, double lz,
                           double* part, Ctl* ctl, double* out, cudaStream_t s) {
    if (G.dim == 3) return launch_budgets3d(G, u, dx * dz / G.inv_dy, dz, lz, part, ctl, out, s);
    budgets2d<<<stream_blocks(G.npt), NTHREADS, 0, s>>>(G, u, dx * dz, dz, lz, part, ctl, out);
    return cudaGetLastError();
}

}  // namespace jfnk
