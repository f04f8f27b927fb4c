// 3-D stencil kernels of libjfnk: F(u), R(u), the Jacobian-vector products,
// the eddy field, the field-block Chebyshev preconditioner, the acoustic
// Schur complement and the budgets, for fields (u, v, w, theta, p) on
// [z][y][x] (x, y periodic; z cell-centred with signed mirror ghosts: w odd,
// theta and p even, u and v even for free slip / odd for no slip; the eddy
// field is mirrored even).
//
// Same discretisation as the 2-D kernels (Deslauriers-Dubuc p = 2 derivative,
// Section 2.3; skew-symmetric convection of every field, Section 2.2;
// Eqs. ch2_28-ch2_30 with Laplacian-form eddy diffusion, Section 2.4), with
// the filter width Delta = (dx dy dz)^(1/3) and the full 3x3 strain.
//
// Every term of F is a sum over the three axes of a one-dimensional stencil
// once the eddy coefficient is known at each point (convection flux and
// advective form along j, D_j(K D_j phi), the pressure gradient and the
// divergence of the pressure equation), plus point-wise terms.  The operator
// is therefore evaluated in three passes that each stage only what their axis
// needs:
//   strain  |S| (and, for the difference-form Jacobian product, |S(a+b)| - |S(a)|
//           without cancellation) at every point: a plane tile with a halo of
//           r = 2 in x, y in shared memory, z neighbours in registers;
//   plane   the x and y terms and the point-wise ones for a tile of one plane:
//           every flux formed once, then differentiated; writes the partial sum;
//   column  the z terms, one column per thread marching in z with its values and
//           fluxes in registers, then the partial sum of the plane pass is added
//           and the mode's output (F, 2u/dt + F, the residual with its norms, or
//           the Jacobian product) written.
// Loads are coalesced along x in every pass; the halos are re-read from L2.
//
// Difference form (float32 Jacobian product): with a = u and b = eps v every
// term of F(a + b) - F(a) is written as a difference about the midpoint
// m = a + b/2 (products m_j b_phi + b_j m_phi, Km D b + dK D m), so no O(1)
// quantity is cancelled in float32.  The other modes evaluate F(b) for
// b = u, or b = u + eps v for the plain forward difference.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace jfnk {
namespace d3 {

constexpr int R = 2;
constexpr int HALO = 2 * R;
constexpr int MODE_F = 0, MODE_RHS = 1, MODE_RES = 2, MODE_JV = 3, MODE_RHSRES = 4;

// D f from the four neighbours f(-2), f(-1), f(+1), f(+2)
template <typename T>
__device__ __forceinline__ T d5(T m2, T m1, T p1, T p2, T ih) {
    return (T(2.0 / 3.0) * (p1 - m1) - T(1.0 / 12.0) * (p2 - m2)) * ih;
}

__device__ __forceinline__ int mirror(int gz, int nz, int& side) {
    side = 0;
    if (gz < 0) { side = 1; return -1 - gz; }
    if (gz >= nz) { side = 2; return 2 * nz - 1 - gz; }
    return gz;
}
__device__ __forceinline__ int wrap(int g, int n) {
    if ((unsigned)g < (unsigned)n) return g;
    int r = g % n;
    return r < 0 ? r + n : r;
}
// even mirror of a row of the eddy field (-1: beyond one reflection, never read)
__device__ __forceinline__ int eddy_row(int gz, int nz) {
    if (gz >= 0 && gz < nz) return gz;
    if (gz < 0) return -1 - gz < nz ? -1 - gz : -1;
    return 2 * nz - 1 - gz >= 0 ? 2 * nz - 1 - gz : -1;
}

// Deardorff coefficient along an arm (Section 2.4, Eq. KmM) from the strain s:
// momentum c s with c = K_m / s along x and y, K_M / s along z; heat times
// 1 + a l(s), a = 2 / sqrt(dx dy) horizontally, 2 / dz vertically.
template <typename T>
__device__ __forceinline__ T dd3_coef(T s, bool zarm, bool heat, const Geo& G) {
    const T c = T(zarm ? G.dd_cM : G.dd_cm);
    if (!heat) return c * s;
    const T cls = GC(dd_cl) * s;
    const T l = GC(dd_cl) < T(0) ? GC(dd_delta) : (cls < GC(dd_delta) ? cls : GC(dd_delta));
    return c * (s * (T(1) + T(zarm ? G.dd_az : G.dd_ah) * l));
}

// Coefficient pair (K(a), K(a + b) - K(a)) of one field at an arm point from
// na = |S(a)| and ds = |S(a + b)| - |S(a)| (na = 0: the coefficient K(b) of
// the one-state modes in the second slot).  SMAG 1: Smagorinsky (the caller
// applies 1/Pr for theta); SMAG 2: Deardorff, the arm's direction and the
// field (momentum / heat) picking the coefficient.
template <typename T, int SMAG>
__device__ __forceinline__ void kpair(const Geo& G, T na, T ds, bool zarm, bool heat, T& k, T& dk) {
    if (SMAG == 1) {
        const T c = GC(cs2);
        k = c * na;
        dk = c * ds;
        return;
    }
    const T c = T(zarm ? G.dd_cM : G.dd_cm);
    if (!heat) {
        k = c * na;
        dk = c * ds;
        return;
    }
    // heat: g(s) = c s (1 + a l(s)); g(s') - g(s) = ds (1 + a l') + a s (l' - l),
    // l' - l = c_l ds while both are below the cap
    const T a = T(zarm ? G.dd_az : G.dd_ah);
    const T dl_cap = GC(dd_delta);
    T la = dl_cap, lp = dl_cap, dl = T(0);
    if (GC(dd_cl) >= T(0)) {
        const T ta = GC(dd_cl) * na, tq = GC(dd_cl) * (na + ds);
        la = ta < dl_cap ? ta : dl_cap;
        lp = tq < dl_cap ? tq : dl_cap;
        if (ta < dl_cap && tq < dl_cap) dl = GC(dd_cl) * ds;
        else if (ta < dl_cap || tq < dl_cap) dl = lp - la;
    }
    k = c * (na * (T(1) + a * la));
    dk = c * (ds * (T(1) + a * lp) + a * na * dl);
}

// ------------------------------------------------------------------ states
// KIND of a pass: one state b = u (ONE) or b = u + eps v (SHIFT, the float64
// forward difference), or the difference F(a + b) - F(a) with a = u, b = eps v
// (PAIR).  PAIR works with the midpoint m = a + b/2, for which every
// product of the two states is
//   a'_j phi' - a_j phi = m_j b_phi + b_j m_phi,   K' D phi' - K D phi = Km D b + dK D m
// (Km = (K + K')/2, dK = K' - K): exact, free of cancellation, and two
// multiplications each.
constexpr int ONE = 0, SHIFT = 1, PAIR = 2;

template <typename T, int KIND>
__device__ __forceinline__ void load_mb(const T* __restrict__ u, const T* __restrict__ v, T ev, size_t o, T& m, T& b) {
    if constexpr (KIND == PAIR) {
        b = ev * v[o];
        m = u[o] + T(0.5) * b;
    } else if constexpr (KIND == SHIFT) {
        b = u[o] + ev * v[o];
    } else {
        b = u[o];
    }
}

// Exchange coefficients of an arm, momentum and heat: K(b) in dk (one state) or
// (Km, dK) from na = |S(a)|, ds = |S(a + b)| - |S(a)|.
template <typename T, int KIND, int SMAG>
__device__ __forceinline__ void coefs(const Geo& G, T na, T ds, bool zarm, T (&km)[2], T (&dk)[2]) {
    if constexpr (SMAG == 0) {
        km[0] = dk[0] = GC(K_M);
        km[1] = dk[1] = GC(K_H);
    } else if constexpr (SMAG == 1) {
        km[0] = KIND == PAIR ? GC(cs2) * (na + T(0.5) * ds) : T(0);
        dk[0] = GC(cs2) * ds;
        km[1] = KIND == PAIR ? km[0] * GC(inv_Pr) : T(0);
        dk[1] = dk[0] * GC(inv_Pr);
    } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            kpair<T, SMAG>(G, na, ds, zarm, h == 1, km[h], dk[h]);
            if (KIND == PAIR) km[h] += T(0.5) * dk[h];
        }
    }
}

// Flux along one axis of a diffused field (heat: h = 1), K D phi - 1/2 u_j phi:
// mj, bj half the velocity along the axis, m, b the field, dm, db its derivative.
template <typename T, int KIND, int SMAG>
__device__ __forceinline__ T flux_of(T km, T dk, T mj, T bj, T m, T b, T dm, T db) {
    if constexpr (KIND == PAIR) {
        T x = -(mj * b) - bj * m;
        x += km * db;
        return SMAG ? x + dk * dm : x;
    } else {
        return flux_sum(dk, db, bj, b);
    }
}
// The same for p, which is not diffused.
template <typename T, int KIND>
__device__ __forceinline__ T flux_p(T mj, T bj, T m, T b) {
    return KIND == PAIR ? -(mj * b) - bj * m : -(bj * b);
}
// The advective form -1/2 u_j D_j phi, added to s.
template <typename T, int KIND>
__device__ __forceinline__ T advect(T s, T mj, T bj, T dm, T db) {
    return KIND == PAIR ? s - mj * db - bj * dm : s - bj * db;
}

// -gamma_p (pbar + p) times a part of the divergence, added to the small terms s:
// p the state's (midpoint's) pressure, div the part (of b), divm the same of m, lost
// what the rounded weights left out of div.  The parts of the three axes nearly cancel
// each other; gamma_p (pbar + p) is the same factor in both passes, and the large
// product is rounded once, last.  (What the weights lost: 1 % of a float64 F.)
template <typename T, int KIND>
__device__ __forceinline__ T pressure_part(const Geo& G, T s, T p, T b, T div, T divm, T lost) {
    const T g = GC(gamma_p) * (GC(pbar) + p);
    if (KIND == PAIR) s = fma(-GC(gamma_p), b * divm, s);
    return fma(-g, div, fma(-g, lost, s));
}

// Asynchronous copy of one element into shared memory.
template <typename T>
__device__ __forceinline__ void cpa1(T* dst, const T* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"((int)sizeof(T)) : "memory");
}

// eps_f = eps_jv * scale_f and 1 / eps_f (Jacobian-product modes)
template <typename T>
__device__ __forceinline__ T eps_field(const Ctl* ctl, int f) {
    if constexpr (sizeof(T) == sizeof(float)) return ctl->evf[f];
    else return ctl->ev[f];
}
template <typename T>
__device__ __forceinline__ T inv_eps_field(const Ctl* ctl, int f) {
    if constexpr (sizeof(T) == sizeof(float)) return ctl->cff[f];
    else return ctl->cf[f];
}

// ------------------------------------------------------------------ tiles
constexpr int KX = 32, KY = 8;                 // strain tile
static_assert(KX * KY == NTHREADS, "one output per thread");

// The strain pass's states: a = u, b = eps v (PAIR), else b alone.
template <typename T, int KIND>
__device__ __forceinline__ void load_ab(const T* __restrict__ u, const T* __restrict__ v, T ev, size_t o, T& a, T& b) {
    a = KIND == PAIR ? u[o] : T(0);
    b = KIND == PAIR ? ev * v[o] : (KIND == SHIFT ? u[o] + ev * v[o] : u[o]);
}

// ============================================================================
// Strain pass: s = sqrt(2 S:S) of b (one-state modes) or, for the difference
// form, sa = |S(a)| and ds = |S(a + b)| - |S(a)| = (S':S' - S:S) * 2 / (s + s')
// at every point.  EDDY: the eddy field of u instead (nu = cs2 s, Deardorff:
// s itself), with its maximum.  One CTA marches up a KX x KY column of SZB
// planes: each thread keeps its point's velocity components at z-2 .. z+2 in
// registers (one new plane per step); the plane itself is staged with a halo
// of r = 2 in x and y for the horizontal derivatives.
// ============================================================================
constexpr int SZB = 16;      // planes per CTA of the strain pass

template <typename T, int KIND, int EDDY>
__global__ void __launch_bounds__(NTHREADS)
strain3d(Geo G, const T* __restrict__ u, const T* __restrict__ v, T* __restrict__ s0, T* __restrict__ s1,
         double* part, Ctl* ctl, int check_done) {
    constexpr bool TWO = KIND == PAIR;            // a = u, b = eps v
    constexpr int SX = KX + 2 * R, SY = KY + 2 * R, SP = SX * SY;
    constexpr int NA = TWO ? 6 : 3;               // (b u, b v, b w) [, (a u, a v, a w)]
    constexpr int XS = (SP + NTHREADS - 1) / NTHREADS;
    if (KIND != ONE && check_done && ctl->done) return;
    __shared__ T st[NA][SP];
    const int x0 = blockIdx.x * KX, y0 = blockIdx.y * KY;
    const int z0 = blockIdx.z * SZB, z1 = min(z0 + SZB, G.nz);
    T ev[3] = {T(0), T(0), T(0)};
    if (KIND != ONE) {
#pragma unroll
        for (int f = 0; f < 3; ++f) ev[f] = eps_field<T>(ctl, f);
    }
    const size_t nxy = (size_t)G.ny * G.nx;
    int xoff[XS];
#pragma unroll
    for (int q = 0; q < XS; ++q) {
        const int idx = threadIdx.x + q * NTHREADS;
        xoff[q] = idx < SP ? wrap(y0 + idx / SX - R, G.ny) * G.nx + wrap(x0 + idx % SX - R, G.nx) : -1;
    }
    const int tx = threadIdx.x % KX, ty = threadIdx.x / KX;
    const int gx = x0 + tx, gy = y0 + ty;
    const bool inside = gx < G.nx && gy < G.ny;
    const size_t own = inside ? (size_t)gy * G.nx + gx : 0;
    // the column's components at z-2 .. z+2 (mirror ghosts with each component's parity)
    T wb[3][5], wa[3][5];
    auto col = [&](int z, int f, T& a, T& b) {
        int side;
        const int sz = mirror(z, G.nz, side);
        load_ab<T, KIND>(u, v, ev[f], (size_t)f * G.npt + (size_t)sz * nxy + own, a, b);
        if ((side == 1 && G.pb[f] < 0) || (side == 2 && G.pt[f] < 0)) {
            a = flip(a);
            b = flip(b);
        }
    };
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int f = 0; f < 3; ++f) col(z0 - 2 + q, f, wa[f][q], wb[f][q]);
    // the next plane's staged values and the column's plane above them are loaded
    // one step ahead, so that their latency overlaps the current plane
    T na[XS][3], nb[XS][3], ca[3], cb[3];
    auto fetch = [&](int z) {
#pragma unroll
        for (int q = 0; q < XS; ++q)
#pragma unroll
            for (int f = 0; f < 3; ++f)
                if (xoff[q] >= 0)
                    load_ab<T, KIND>(u, v, ev[f], (size_t)f * G.npt + (size_t)z * nxy + xoff[q], na[q][f], nb[q][f]);
#pragma unroll
        for (int f = 0; f < 3; ++f) col(z + 2, f, ca[f], cb[f]);
    };
    fetch(z0);
    T mx = T(0);
    for (int z = z0; z < z1; ++z) {
        const size_t pz = (size_t)z * nxy;
#pragma unroll
        for (int q = 0; q < XS; ++q) {
            if (xoff[q] < 0) continue;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                st[f][threadIdx.x + q * NTHREADS] = nb[q][f];
                if (TWO) st[3 + f][threadIdx.x + q * NTHREADS] = na[q][f];
            }
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            wa[f][4] = ca[f];
            wb[f][4] = cb[f];
        }
        __syncthreads();
        if (z + 1 < z1) fetch(z + 1);
        if (inside) {
            const int c = (ty + R) * SX + tx + R;
            auto D = [&](const T* s, int st_, T w1, T w2) {
                return w1 * (s[c + st_] - s[c - st_]) + w2 * (s[c + 2 * st_] - s[c - 2 * st_]);
            };
            T gB[3][3], gA[3][3];
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                gB[f][0] = D(st[f], 1, GC(wx1), GC(wx2));
                gB[f][1] = D(st[f], SX, GC(wy1), GC(wy2));
                gB[f][2] = GC(wz1) * (wb[f][3] - wb[f][1]) + GC(wz2) * (wb[f][4] - wb[f][0]);
                if (TWO) {
                    gA[f][0] = D(st[3 + f], 1, GC(wx1), GC(wx2));
                    gA[f][1] = D(st[3 + f], SX, GC(wy1), GC(wy2));
                    gA[f][2] = GC(wz1) * (wa[f][3] - wa[f][1]) + GC(wz2) * (wa[f][4] - wa[f][0]);
                }
            }
            // 2 S:S = 2 sum g_ii^2 + sum_{i<j} (g_ij + g_ji)^2
            T sym[3], syma[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int j = (i + 1) % 3;
                sym[i] = gB[i][j] + gB[j][i];
                if (TWO) syma[i] = gA[i][j] + gA[j][i];
            }
            const size_t p = pz + own;
            if (TWO) {
                T dA = T(0), oA = T(0), dD = T(0), oD = T(0);     // diagonal and off-diagonal sums of S:S, S':S' - S:S
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    dA += gA[i][i] * gA[i][i];
                    dD += (T(2) * gA[i][i] + gB[i][i]) * gB[i][i];
                    oA += syma[i] * syma[i];
                    oD += (T(2) * syma[i] + sym[i]) * sym[i];
                }
                const T sa = T(2) * dA + oA, ds = T(2) * dD + oD;     // 2 S:S and its difference
                const T na_ = root(sa);
                const T tp = sa + ds;
                const T den = na_ + root(tp > T(0) ? tp : T(0));
                s0[p] = na_;
                s1[p] = den > T(0) ? ds / den : T(0);
            } else {
                const T dB = gB[0][0] * gB[0][0] + gB[1][1] * gB[1][1] + gB[2][2] * gB[2][2];
                const T sv = root(sym[0] * sym[0] + (sym[1] * sym[1] + (sym[2] * sym[2] + (dB + dB))));
                if (EDDY) {
                    const T val = G.sgs == 2 ? sv : GC(cs2) * sv;
                    s1[p] = val;
                    mx = val > mx ? val : mx;
                } else {
                    s1[p] = sv;
                }
            }
        }
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                wb[f][q] = wb[f][q + 1];
                wa[f][q] = wa[f][q + 1];
            }
        __syncthreads();      // the next plane overwrites the staged one
    }
    if (EDDY) {
        double m1[1] = {(double)mx};
        const int nblk = gridDim.x * gridDim.y * gridDim.z;
        const int blk = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        block_partials_max<1>(m1, 1, part, nblk, blk);
        if (arrive_last(&ctl->counter[CNT_EDDY], nblk)) {
            __shared__ double tot[1];
            final_maxes(part, nblk, 1, tot);
            if (threadIdx.x == 0) ctl->kmax = tot[0];
        }
    }
}

// The difference form's strain pass in float32, two points along x per thread: no
// shared memory and no barrier.  A thread reads its row's neighbours (x -+ 2, y -+ 1,
// y -+ 2) as 8-byte pairs through the L1 and keeps its columns' z-2 .. z+2 in
// registers; eps v enters as eps D(v).  For an even nx; strain3d above otherwise,
// and in float64, where the FP64 pipe bounds the pass.
// Bound: load latency and issue (134 MB, 20 us at 256 x 256 x 64): 67 -> 54 us there.
__global__ void __launch_bounds__(NTHREADS, 2)
strain3d_pairs(Geo G, const float* __restrict__ u, const float* __restrict__ v, float* __restrict__ s0,
               float* __restrict__ s1, const Ctl* ctl, int check_done) {
    if (check_done && ctl->done) return;
    const int gx = (blockIdx.x * KX + threadIdx.x % KX) * 2, gy = blockIdx.y * KY + threadIdx.x / KX;
    if (gx >= G.nx || gy >= G.ny) return;
    const int z0 = blockIdx.z * SZB, z1 = min(z0 + SZB, G.nz);
    const int nxy = G.ny * G.nx, own = gy * G.nx + gx;
    const int xl = gy * G.nx + wrap(gx - 2, G.nx), xr = gy * G.nx + wrap(gx + 2, G.nx);
    int yo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) yo[q] = wrap(gy + (q < 2 ? q - 2 : q - 1), G.ny) * G.nx + gx;
    float ev[3];
#pragma unroll
    for (int f = 0; f < 3; ++f) ev[f] = eps_field<float>(ctl, f);
    auto pair = [&](int st, int f, int z, int o) {
        return __ldg(reinterpret_cast<const float2*>((st ? v : u) + (size_t)f * G.npt + (size_t)z * nxy + o));
    };
    // mirror ghosts with each component's parity
    auto col = [&](int st, int f, int z) {
        int side;
        const int sz = mirror(z, G.nz, side);
        const float2 a = pair(st, f, sz, own);
        const bool odd = (side == 1 && G.pb[f] < 0) || (side == 2 && G.pt[f] < 0);
        return odd ? make_float2(flip(a.x), flip(a.y)) : a;
    };
    const float wx1 = G.f32.wx1, wx2 = G.f32.wx2, wy1 = G.f32.wy1, wy2 = G.f32.wy2, wz1 = G.f32.wz1, wz2 = G.f32.wz2;
    float2 w[2][3][5];
#pragma unroll
    for (int st = 0; st < 2; ++st)
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int q = 0; q < 4; ++q) w[st][f][q] = col(st, f, z0 - 2 + q);
    for (int z = z0; z < z1; ++z) {
        float g[2][3][3][2];      // [u, eps v][component][axis][point]
#pragma unroll
        for (int st = 0; st < 2; ++st)
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                w[st][f][4] = col(st, f, z + 2);
                const float2 l = pair(st, f, z, xl), r = pair(st, f, z, xr);
                const float2 d2 = pair(st, f, z, yo[0]), d1 = pair(st, f, z, yo[1]);
                const float2 u1 = pair(st, f, z, yo[2]), u2 = pair(st, f, z, yo[3]);
                const float2(&c)[5] = w[st][f];
                g[st][f][0][0] = wx1 * (c[2].y - l.y) + wx2 * (r.x - l.x);
                g[st][f][0][1] = wx1 * (r.x - c[2].x) + wx2 * (r.y - l.y);
                g[st][f][1][0] = wy1 * (u1.x - d1.x) + wy2 * (u2.x - d2.x);
                g[st][f][1][1] = wy1 * (u1.y - d1.y) + wy2 * (u2.y - d2.y);
                g[st][f][2][0] = wz1 * (c[3].x - c[1].x) + wz2 * (c[4].x - c[0].x);
                g[st][f][2][1] = wz1 * (c[3].y - c[1].y) + wz2 * (c[4].y - c[0].y);
                if (st)
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        g[1][f][d][0] *= ev[f];
                        g[1][f][d][1] *= ev[f];
                    }
            }
        float sa[2], ds[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float dA = 0.f, oA = 0.f, dD = 0.f, oD = 0.f;     // diagonal and off-diagonal sums of S:S, S':S' - S:S
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int j = (i + 1) % 3;
                const float a = g[0][i][i][e], b = g[1][i][i][e];
                const float ao = g[0][i][j][e] + g[0][j][i][e], bo = g[1][i][j][e] + g[1][j][i][e];
                dA += a * a;
                dD += (2.f * a + b) * b;
                oA += ao * ao;
                oD += (2.f * ao + bo) * bo;
            }
            const float q = 2.f * dA + oA, d = 2.f * dD + oD, t = q + d;     // 2 S:S and its difference
            sa[e] = root(q);
            const float den = sa[e] + root(t > 0.f ? t : 0.f);
            ds[e] = den > 0.f ? d / den : 0.f;
        }
        const size_t p = (size_t)z * nxy + own;
        *reinterpret_cast<float2*>(s0 + p) = make_float2(sa[0], sa[1]);
        *reinterpret_cast<float2*>(s1 + p) = make_float2(ds[0], ds[1]);
#pragma unroll
        for (int st = 0; st < 2; ++st)
#pragma unroll
            for (int f = 0; f < 3; ++f)
#pragma unroll
                for (int q = 0; q < 4; ++q) w[st][f][q] = w[st][f][q + 1];
    }
}

// ============================================================================
// Plane pass: x and y terms of every field and the point-wise terms, for a
// PX x PYT tile of plane z = blockIdx.z; writes their sum to P.  The fluxes
// X_phi, Y_phi are formed once per point and on the arms they are read from
// (two columns / rows either side), then differentiated; a thread keeps the
// point-wise parts of its points in registers.
//
// Bound: float64 the FP64 pipe (about 115 operations a point and 25 per arm
// point; the form that rebuilt the products at every tap took about 280),
// float32 shared-memory bandwidth (about 180 words a point, 300 before).
// Difference-form product at 256 x 256 x 64: 224 -> 115 us; float64 F at
// 256 x 256 x 128: 3.72 -> 2.19 ms.
// ============================================================================
constexpr int PX = 32;
template <typename T> struct PlaneT;
template <> struct PlaneT<float>  { static constexpr int PY = 16; };
template <> struct PlaneT<double> { static constexpr int PY = 8; };

template <typename T, int KIND, int SMAG>
struct PlaneShape {
    static constexpr int PY = PlaneT<T>::PY, SX = PX + 2 * HALO, SY = PY + 2 * HALO, SP = SX * SY;
    static constexpr int NS = KIND == PAIR ? 2 : 1;      // states staged: b [, m]
    static constexpr int XW = PX + 2 * R, XN = XW * PY, YN = PX * (PY + 2 * R);
    static constexpr int PPT = PX * PY / NTHREADS;
    static constexpr size_t smem = sizeof(T) * (size_t)(NS * 5 * SP + 5 * XN + 5 * YN);
    static_assert(PPT * NTHREADS == PX * PY && 4 * (PX + PY) <= NTHREADS, "thread mapping");
};

// Fluxes at one point (staged index c) along x (XF) and y (YF); both: a tile
// point, whose point-wise part goes to S.
template <typename T, int KIND, int SMAG, bool XF, bool YF>
__device__ __forceinline__ void plane_point(const Geo& G, const T* __restrict__ st, int c, T na, T ds,
                                            T* __restrict__ X, T* __restrict__ Y, T (&S)[5]) {
    using SH = PlaneShape<T, KIND, SMAG>;
    constexpr int SP = SH::SP, SX = SH::SX, XN = SH::XN, YN = SH::YN;
    const T* B = st;
    const T* M = st + 5 * SP;
    const T wx1 = GC(wx1), wx2 = GC(wx2), wy1 = GC(wy1), wy2 = GC(wy2);
    auto D = [&](const T* f, int s, T w1, T w2) { return w1 * (f[c + s] - f[c - s]) + w2 * (f[c + 2 * s] - f[c - 2 * s]); };
    T km[2], dk[2];
    coefs<T, KIND, SMAG>(G, na, ds, false, km, dk);
    const T bu = T(0.5) * B[c], bv = T(0.5) * B[SP + c];
    const T mu = KIND == PAIR ? T(0.5) * M[c] : T(0), mv = KIND == PAIR ? T(0.5) * M[SP + c] : T(0);
    T divb = T(0), divm = T(0), dive = T(0);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        const T b = B[f * SP + c], m = KIND == PAIR ? M[f * SP + c] : T(0);
        T dbx = T(0), dby = T(0), dmx = T(0), dmy = T(0), s = T(0);
        if (XF && (f < 4 || YF)) {
            dbx = D(B + f * SP, 1, wx1, wx2);
            if (KIND == PAIR) dmx = D(M + f * SP, 1, wx1, wx2);
        }
        if (YF && (f < 4 || XF)) {
            dby = D(B + f * SP, SX, wy1, wy2);
            if (KIND == PAIR) dmy = D(M + f * SP, SX, wy1, wy2);
        }
        const int h = f == 3 ? 1 : 0;
        if (XF) X[f * XN] = f < 4 ? flux_of<T, KIND, SMAG>(km[h], dk[h], mu, bu, m, b, dmx, dbx) : flux_p<T, KIND>(mu, bu, m, b);
        if (YF) Y[f * YN] = f < 4 ? flux_of<T, KIND, SMAG>(km[h], dk[h], mv, bv, m, b, dmy, dby) : flux_p<T, KIND>(mv, bv, m, b);
        if (XF && YF) {
            // the small advective terms first: the large linear ones are rounded once
            s = advect<T, KIND>(s, mu, bu, dmx, dbx);
            s = advect<T, KIND>(s, mv, bv, dmy, dby);
            if (f == 0) { divb = dbx; divm = dmx; if constexpr (sizeof(T) == sizeof(float)) dive = G.f32.ex * dbx; }
            if (f == 1) { divb += dby; divm += dmy; dive = fma(GC(ey), dby, dive); }
            if (f == 2) s += GC(gth) * B[3 * SP + c];
            if (f == 3) s -= GC(beta) * B[2 * SP + c];
            if (f == 4) {       // pressure equation, x and y parts of the divergence; gradient of p
                // (what the weights lost, Geo::ey, with the small terms: see pressure_part)
                s = pressure_part<T, KIND>(G, s, KIND == PAIR ? m : b, b, divb, divm, dive);
                S[0] -= GC(theta0) * dbx;
                S[1] -= GC(theta0) * dby;
            }
            S[f] = s;
        }
    }
}

template <typename T, int KIND, int SMAG>
__global__ void __launch_bounds__(NTHREADS, sizeof(T) == sizeof(float) ? 3 : 4)
plane3d(Geo G, const T* __restrict__ u, const T* __restrict__ v, const T* __restrict__ s0,
        const T* __restrict__ s1, T* __restrict__ P, Ctl* ctl, int check_done) {
    using SH = PlaneShape<T, KIND, SMAG>;
    constexpr int PY = SH::PY, SX = SH::SX, SP = SH::SP, XW = SH::XW, XN = SH::XN, YN = SH::YN, PPT = SH::PPT;
    if (KIND != ONE && check_done && ctl->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* st = reinterpret_cast<T*>(smem_raw);          // [NS][5][SP]: b fields, then m fields
    T* X = st + SH::NS * 5 * SP;                     // [5][PY][PX + 4]
    T* Y = X + 5 * XN;                               // [5][PY + 4][PX]
    const int x0 = blockIdx.x * PX, y0 = blockIdx.y * PY, gz = blockIdx.z;
    T ev[5] = {T(0), T(0), T(0), T(0), T(0)};
    if (KIND != ONE) {
#pragma unroll
        for (int f = 0; f < 5; ++f) ev[f] = eps_field<T>(ctl, f);
    }
    const size_t plane = (size_t)gz * G.ny * G.nx;
    // eddy values of the thread's points and of its arm point, in flight with the staging
    const int a = threadIdx.x;
    const bool yarm = a < 4 * PX, arm = a < 4 * (PX + PY);
    const int ar = yarm ? a / PX : (a - 4 * PX) & 3;
    const int ax = yarm ? a % PX : (ar < 2 ? ar - 2 : PX + ar - 2);
    const int ay = yarm ? (ar < 2 ? ar - 2 : PY + ar - 2) : (a - 4 * PX) >> 2;
    T kn[PPT + 1], kd[PPT + 1];
#pragma unroll
    for (int k = 0; k <= PPT; ++k) {
        kn[k] = kd[k] = T(0);
        if (SMAG && (k < PPT || arm)) {
            const int w = threadIdx.x + k * NTHREADS;
            const int px = k < PPT ? w % PX : ax, py = k < PPT ? w / PX : ay;
            const size_t o = plane + (size_t)wrap(y0 + py, G.ny) * G.nx + wrap(x0 + px, G.nx);
            kd[k] = s1[o];
            if (KIND == PAIR) kn[k] = s0[o];
        }
    }
    for (int idx = threadIdx.x; idx < SP; idx += NTHREADS) {
        const int ixl = idx % SX, iyl = idx / SX;
        const size_t o = plane + (size_t)wrap(y0 + iyl - HALO, G.ny) * G.nx + wrap(x0 + ixl - HALO, G.nx);
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            T m, b;
            load_mb<T, KIND>(u, v, ev[f], (size_t)f * G.npt + o, m, b);
            st[f * SP + idx] = b;
            if (KIND == PAIR) st[(5 + f) * SP + idx] = m;
        }
    }
    __syncthreads();
    T S[PPT][5];
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int w = threadIdx.x + k * NTHREADS, tx = w % PX, ty = w / PX;
        if (x0 + tx <= G.nx + 1 && y0 + ty <= G.ny + 1)      // else it feeds no output
            plane_point<T, KIND, SMAG, true, true>(G, st, (ty + HALO) * SX + tx + HALO, kn[k], kd[k],
                                                   X + ty * XW + tx + R, Y + (ty + R) * PX + tx, S[k]);
    }
    if (arm && x0 + ax <= G.nx + 1 && y0 + ay <= G.ny + 1) {
        T none[5];
        const int c = (ay + HALO) * SX + ax + HALO;
        if (yarm) plane_point<T, KIND, SMAG, false, true>(G, st, c, kn[PPT], kd[PPT], X, Y + (ay + R) * PX + ax, none);
        else plane_point<T, KIND, SMAG, true, false>(G, st, c, kn[PPT], kd[PPT], X + ay * XW + ax + R, Y, none);
    }
    __syncthreads();
    const T wx1 = GC(wx1), wx2 = GC(wx2), wy1 = GC(wy1), wy2 = GC(wy2);
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int w = threadIdx.x + k * NTHREADS, tx = w % PX, ty = w / PX;
        const int gx = x0 + tx, gy = y0 + ty;
        if (gx >= G.nx || gy >= G.ny) continue;
        const size_t off = plane + (size_t)gy * G.nx + gx;
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            const T* x = X + f * XN + ty * XW + tx + R;
            const T* y = Y + f * YN + (ty + R) * PX + tx;
            T s = wx1 * (x[1] - x[-1]);
            s += wx2 * (x[2] - x[-2]);
            s += wy1 * (y[PX] - y[-PX]);
            s += wy2 * (y[2 * PX] - y[-2 * PX]);
            s += S[k][f];
            if (KIND != PAIR && f == 3 && gz == 0 && G.heat != nullptr)
                s += T(G.heat[(size_t)gy * G.nx + gx] * G.heat_coef);
            P[(size_t)f * G.npt + off] = s;
        }
    }
}

// ============================================================================
// Column pass: the z terms, plus the plane pass's sum; writes the mode's
// output.  A CTA takes CW columns; a thread owns one field of one column (a
// warp has one field) and marches through zc planes with everything in
// registers: the last five values of its field and of its partner (p for w,
// w for the others), the last five fluxes Z_phi and the point-wise parts of the
// planes between flux and output.  No shared memory, no barrier, every load
// coalesced; the fields' warps share w and the eddy values through L1.  A
// plane's values enter at step l (plane z0 - 4 + l), the plane two below gets
// its flux, the plane four below its output.  The rings turn by an index fixed
// at compile time in five copies of the step, so nothing is moved.
//
// Bound: float64 the FP64 pipe (about 100 operations a point; the slab form
// that staged tiles in shared memory and rebuilt products at every tap took
// about 240), float32 HBM and load latency.  One thread for all five fields of
// a column needs 230-255 registers (float64 spills): one CTA per SM.
// Difference-form product at 256 x 256 x 64: 258 (slab) -> 107 us, with the
// operands loaded one step ahead into registers 209; float64 F at
// 256 x 256 x 128: 3.1 -> 1.9 ms.
// ============================================================================
constexpr int CW = 32;                               // columns per CTA
constexpr int COL_THREADS = 5 * CW;
constexpr int COL_STAGES = 4;                        // steps whose operands are in flight or in use

template <typename T, int KIND, int SMAG>
__global__ void __launch_bounds__(COL_THREADS, sizeof(T) == sizeof(float) ? 5 : 4)
column3d(Geo G, int mode, int zc, const T* __restrict__ u, const T* __restrict__ v, const T* __restrict__ Fu,
         const double* __restrict__ f, const T* __restrict__ s0, const T* __restrict__ s1, const T* __restrict__ P,
         T* __restrict__ out, T* __restrict__ out2, double* __restrict__ part, Ctl* ctl, int check_done) {
    constexpr int IW = 2, IT = 3, IP = 4;
    if (KIND != ONE && check_done && ctl->done) return;
    const size_t nxy_ = (size_t)G.ny * G.nx, np = (size_t)G.npt;
    const int q = threadIdx.x / CW, pq = q == IW ? IP : IW;             // field, partner field
    const size_t col = (size_t)blockIdx.x * CW + threadIdx.x % CW;
    const int z0 = blockIdx.y * zc, z1 = min(z0 + zc, G.nz);
    __shared__ T ring_s[COL_STAGES][KIND == ONE ? 5 : 8][COL_THREADS];
    double ar = 0.0, au = 0.0;
    if (col < nxy_) {
        const T w1 = GC(wz1), w2 = GC(wz2);
        T evq = T(0), evp = T(0), cf = T(0);         // eps scale, 1 / (eps scale)
        if (KIND != ONE) {
            evq = eps_field<T>(ctl, q);
            evp = eps_field<T>(ctl, pq);
            cf = inv_eps_field<T>(ctl, q);
        }
        const bool oddb = G.pb[q] < 0, oddt = G.pt[q] < 0, poddb = G.pb[pq] < 0, poddt = G.pt[pq] < 0;
        // offsets within a plane stack fit 32 bits (npt does): one wide multiply-add per access
        const int nxy = (int)nxy_;
        const size_t oq = q * np + col, op = pq * np + col;
        const T *uq = u + oq, *up = u + op, *vq = KIND != ONE ? v + oq : u, *vp = KIND != ONE ? v + op : u;
        const T *s0c = s0 + col, *s1c = s1 + col, *Pq = P + oq, *Fq = KIND == SHIFT ? Fu + oq : u;
        const double* fq = KIND == ONE && mode == MODE_RES ? f + oq : nullptr;
        T* outq = out + oq;
        T* out2q = out2 != nullptr ? out2 + oq : nullptr;
        T b[5], m[5] = {}, c[5], d[5] = {}, Z[5], S[5];        // rings: field (b, m), partner (c, d), flux, point-wise part
        const int steps = z1 - z0 + 8;
        // step l's operands, copied to this thread's own shared-memory slots
        // COL_STAGES - 1 steps ahead (no barrier: nobody else reads them)
        auto stage = [&](int l) {
            if (l < steps) {
                T(*st)[COL_THREADS] = ring_s[l % COL_STAGES];
                const int z = z0 - 4 + l;
                int side;
                const int o = mirror(z, G.nz, side) * nxy;
                cpa1(&st[0][threadIdx.x], uq + o);
                cpa1(&st[1][threadIdx.x], up + o);
                if (SMAG) cpa1(&st[2][threadIdx.x], s1c + max(eddy_row(z - 2, G.nz), 0) * nxy);   // plane z - 2
                if (l >= 8) {                        // operands of the output of plane z - 4
                    const int oo = (z - 4) * nxy;
                    cpa1(&st[3][threadIdx.x], Pq + oo);
                    if (KIND != ONE) cpa1(&st[4][threadIdx.x], vq + oo);
                    if (KIND == SHIFT) cpa1(&st[7][threadIdx.x], Fq + oo);
                    if constexpr (KIND == ONE && sizeof(T) == sizeof(double))
                        if (fq != nullptr) cpa1(&st[4][threadIdx.x], fq + oo);
                }
                if (KIND != ONE) {
                    cpa1(&st[5][threadIdx.x], vq + o);
                    cpa1(&st[6][threadIdx.x], vp + o);
                }
                if (KIND == PAIR && SMAG) cpa1(&st[7][threadIdx.x], s0c + max(eddy_row(z - 2, G.nz), 0) * nxy);
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        auto step = [&](auto ring, int l) {
            constexpr int r0 = decltype(ring)::value;                                                   // l mod 5
            constexpr int r1 = (r0 + 4) % 5, r2 = (r0 + 3) % 5, r3 = (r0 + 2) % 5, r4 = (r0 + 1) % 5;   // l-1 .. l-4
            const int z = z0 - 4 + l;
            stage(l + COL_STAGES - 1);
            asm volatile("cp.async.wait_group %0;\n" ::"n"(COL_STAGES - 1) : "memory");
            const T(*st)[COL_THREADS] = ring_s[l % COL_STAGES];
            auto arrived = [&](int k) { return st[k][threadIdx.x]; };
            if constexpr (KIND == PAIR) {
                b[r0] = evq * arrived(5);
                m[r0] = arrived(0) + T(0.5) * b[r0];
                c[r0] = evp * arrived(6);
                d[r0] = arrived(1) + T(0.5) * c[r0];
            } else {
                b[r0] = arrived(0);
                c[r0] = arrived(1);
                if (KIND == SHIFT) {
                    b[r0] += evq * arrived(5);
                    c[r0] += evp * arrived(6);
                }
            }
            if (z < 0 || z >= G.nz) {                // ghost plane: signs of the odd fields
                if (z < 0 ? oddb : oddt) {
                    b[r0] = flip(b[r0]);
                    if constexpr (KIND == PAIR) m[r0] = flip(m[r0]);
                }
                if (z < 0 ? poddb : poddt) {
                    c[r0] = flip(c[r0]);
                    if constexpr (KIND == PAIR) d[r0] = flip(d[r0]);
                }
            }
            const T kd = SMAG ? arrived(2) : T(0), ka = KIND == PAIR && SMAG ? arrived(7) : T(0);
            if (l >= 4) {                            // flux and point-wise part of plane z - 2
                const T bw = T(0.5) * (q == IW ? b[r2] : c[r2]);
                const T mw = KIND == PAIR ? T(0.5) * (q == IW ? m[r2] : d[r2]) : T(0);
                const T db = w1 * (b[r1] - b[r3]) + w2 * (b[r0] - b[r4]);
                const T dm = KIND == PAIR ? w1 * (m[r1] - m[r3]) + w2 * (m[r0] - m[r4]) : T(0);
                T s = T(0);
                if (q == IP) {
                    Z[r2] = flux_p<T, KIND>(mw, bw, m[r2], b[r2]);
                    const T dw = w1 * (c[r1] - c[r3]) + w2 * (c[r0] - c[r4]);
                    const T dwm = KIND == PAIR ? w1 * (d[r1] - d[r3]) + w2 * (d[r0] - d[r4]) : T(0);
                    s = pressure_part<T, KIND>(G, advect<T, KIND>(s, mw, bw, dm, db), KIND == PAIR ? m[r2] : b[r2], b[r2], dw, dwm,
                                               GC(ez) * dw);
                } else {
                    T km[2], dk[2];
                    coefs<T, KIND, SMAG>(G, ka, kd, true, km, dk);
                    Z[r2] = q == IT ? flux_of<T, KIND, SMAG>(km[1], dk[1], mw, bw, m[r2], b[r2], dm, db)
                                    : flux_of<T, KIND, SMAG>(km[0], dk[0], mw, bw, m[r2], b[r2], dm, db);
                    s = advect<T, KIND>(s, mw, bw, dm, db);
                    if (q == IW) s -= GC(theta0) * (w1 * (c[r1] - c[r3]) + w2 * (c[r0] - c[r4]));
                }
                S[r2] = s;
            }
            if (l < 8) return;
            const int o = (z - 4) * nxy;
            const T pv = arrived(3), xv = KIND != ONE ? arrived(4) : T(0);
            // output of plane z - 4: fluxes of planes l-2, l-3, l-5, l-6 (rings r2, r3, r0, r1)
            T Fv = w1 * (Z[r3] - Z[r0]);
            Fv += w2 * (Z[r2] - Z[r1]);
            Fv += S[r4];
            Fv += pv;
            if (KIND == PAIR) {
                outq[o] = GC(two_over_dt) * xv - Fv * cf;
            } else if (KIND == SHIFT) {              // plain forward difference against F(u)
                outq[o] = T(G.two_over_dt * (double)xv - ((double)Fv - (double)arrived(7)) * cf);
            } else if (mode == MODE_F) {
                outq[o] = Fv;
            } else {
                const double uo = (double)b[r4], Fd = (double)Fv;
                if (mode == MODE_RHS) {
                    outq[o] = T(G.two_over_dt * uo + Fd);
                    return;
                }
                double Rv;
                if (mode == MODE_RHSRES) {
                    // at u = u^n the residual 2u/dt - F(u) - f with f = 2u/dt + F(u) is -2 F(u)
                    outq[o] = T(G.two_over_dt * uo + Fd);
                    Rv = -2.0 * Fd;
                    out2q[o] = T(Rv);
                } else {
                    Rv = G.two_over_dt * uo - Fd - (sizeof(T) == sizeof(double) ? (double)arrived(4) : fq[o]);
                    outq[o] = T(Rv);
                    if (out2q != nullptr) out2q[o] = Fv;
                }
                ar = fma(Rv, Rv, ar);
                au = fma(uo, uo, au);
            }
        };
        for (int l = 0; l < COL_STAGES - 1; ++l) stage(l);
        for (int l = 0; l < steps; l += 5) {
            step(std::integral_constant<int, 0>(), l);
            if (l + 1 < steps) step(std::integral_constant<int, 1>(), l + 1);
            if (l + 2 < steps) step(std::integral_constant<int, 2>(), l + 2);
            if (l + 3 < steps) step(std::integral_constant<int, 3>(), l + 3);
            if (l + 4 < steps) step(std::integral_constant<int, 4>(), l + 4);
        }
    }
    if (KIND == ONE && (mode == MODE_RES || mode == MODE_RHSRES)) {
        const double i2 = G.inv_scale[q] * G.inv_scale[q];
        double acc[2] = {ar * i2, au * i2};
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

// ------------------------------------------------------------------ vectors
// The marching sweeps (field blocks, Helmholtz) give a thread W consecutive
// points along x: 16 bytes where nx allows it, one point otherwise.
template <typename T, int W> struct VecT;
template <> struct VecT<float, 4> { using type = float4; };
template <> struct VecT<double, 2> { using type = double2; };
template <> struct VecT<float, 2> { using type = float2; };
template <> struct VecT<float, 1> { using type = float; };
template <> struct VecT<double, 1> { using type = double; };

template <typename T, int W>
__device__ __forceinline__ void vload(const T* p, T (&v)[W]) {
    *reinterpret_cast<typename VecT<T, W>::type*>(v) = *reinterpret_cast<const typename VecT<T, W>::type*>(p);
}
template <typename T, int W>
__device__ __forceinline__ void vstore(T* p, const T (&v)[W]) {
    *reinterpret_cast<typename VecT<T, W>::type*>(p) = *reinterpret_cast<const typename VecT<T, W>::type*>(v);
}

template <typename T, int W> struct HelmTile;      // threads of a sweep's CTA along x, y
template <> struct HelmTile<float, 4> { static constexpr int NXT = 16, NYT = 16; };
template <> struct HelmTile<double, 2> { static constexpr int NXT = 32, NYT = 8; };
template <> struct HelmTile<float, 2> { static constexpr int NXT = 32, NYT = 8; };
template <typename T> struct HelmTile<T, 1> { static constexpr int NXT = 32, NYT = 8; };

template <typename T, int W>
__device__ __forceinline__ void cpa(T* dst, const T* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (W * sizeof(T) == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(W * (int)sizeof(T)) : "memory");
}

// ============================================================================
// Field-block Chebyshev sweep (same recurrence as the 2-D kernel, Section 2.5.2).
// One CTA = one field of a TX x TY column of zb planes: blockIdx.z = zblock * 5
// + field; p (field 4) is written by the last sweep.  A thread owns W
// consecutive points along x and marches in z with, in registers, the column's
// iterate at z-4 .. z+4, its eddy values at z .. z+2 and its vertical fluxes
// K D_z x at z-2 .. z+2 (each formed once, when its plane enters).  Per plane the
// column's own iterate and eddy values go to shared memory and only the rings
// around the tile (4 and 2 points) are fetched, by cp.async, one plane ahead
// into the other of two buffers: one barrier per plane.  The horizontal fluxes
// a point's D reads are formed by the point's own thread (8 for 4 points along
// x, 4 rows along y): about twice the arithmetic of sharing them, but no
// second exchange and no arm items.
//
// Bound: instruction issue and load latency (r and the eddy field read, z
// written: 44 B a point over the five fields with two sweeps).  Against the
// form with one point per thread, fluxes exchanged through shared memory and
// two barriers a plane: 175 -> 87 us per apply (two
// sweeps) at 256 x 256 x 64, float32.
// ============================================================================
template <typename T, int W, int SMAG, int FIRST, int LAST>
__global__ void __launch_bounds__(NTHREADS, 2)
cheb3d(Geo G, int k, int zb, const T* __restrict__ r, const T* __restrict__ zin, const T* __restrict__ din,
       T* __restrict__ zout, T* __restrict__ dout, const T* __restrict__ nu, double* part, Ctl* ctl,
       int check_done) {
    constexpr int NXT = HelmTile<T, W>::NXT, NYT = HelmTile<T, W>::NYT;
    constexpr int TX = NXT * W, TY = NYT, SX = TX + 2 * HALO, SY = TY + 2 * HALO;
    // eddy plane: the iterate's row layout (vectors stay aligned), a ring of 2 rows and of HALO columns
    constexpr int KY2 = TY + 2 * R;
    constexpr int NH = (2 * HALO * TX + 2 * HALO * TY) / W, HS = (NH + NTHREADS - 1) / NTHREADS;
    constexpr int KROWS = SMAG ? KY2 : 1;
    __shared__ __align__(16) T pl[2][SX * SY];
    __shared__ __align__(16) T kp[2][SX * KROWS];
    pdl_wait();
    const int done = check_done ? ctl->done : 0;
    const int fld = blockIdx.z % 5;
    const int z0 = (blockIdx.z / 5) * zb, nzb = min(zb, G.nz - z0);
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const T ith = cheb_coef<T>(ctl, fld, k, 0), a1 = cheb_coef<T>(ctl, fld, k, 1), a2 = cheb_coef<T>(ctl, fld, k, 2);
    const size_t nxy = (size_t)G.ny * G.nx;
    const T* fr = r + (size_t)fld * G.npt;
    const T* src = (FIRST ? r : zin) + (size_t)fld * G.npt;
    const T* fdin = FIRST ? nullptr : din + (size_t)fld * G.npt;
    T* fzo = zout + (size_t)fld * G.npt;
    T* fdo = LAST ? nullptr : dout + (size_t)fld * G.npt;
    const int tx = threadIdx.x % NXT, ty = threadIdx.x / NXT;
    const int gx = x0 + tx * W, gy = y0 + ty;
    const bool inside = gx < G.nx && gy < G.ny;
    const size_t own = (size_t)wrap(gy, G.ny) * G.nx + wrap(gx, G.nx);
    T acc[1] = {T(0)};
    if (done) return;
    if (fld == 4) {
        if (LAST && inside) {
            for (int z = z0; z < z0 + nzb; ++z) {
                const size_t o = (size_t)z * nxy + own;
                T v[W];
                vload<T, W>(fr + o, v);
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    v[i] *= ith;
                    acc[0] += v[i] * v[i];
                }
                vstore<T, W>(fzo + o, v);
            }
        }
    } else {
        int hdst[HS], hsrc[HS], kdst[HS];
#pragma unroll
        for (int q = 0; q < HS; ++q) {
            int h = threadIdx.x + q * NTHREADS;
            hdst[q] = kdst[q] = -1;
            hsrc[q] = 0;
            if (h < NH) {
                int ly, lx;                                  // staged row, column (relative to the tile origin)
                if (h < 2 * HALO * NXT) {
                    ly = h / NXT;
                    ly = ly < HALO ? ly - HALO : TY + ly - HALO;
                    lx = (h % NXT) * W;
                } else {
                    h -= 2 * HALO * NXT;
                    constexpr int PER = 2 * HALO / W;        // vectors of the two sides of a row
                    ly = h / PER;
                    const int c = h % PER;
                    lx = c < PER / 2 ? c * W - HALO : TX + (c - PER / 2) * W;
                }
                hdst[q] = (ly + HALO) * SX + lx + HALO;
                hsrc[q] = wrap(y0 + ly, G.ny) * G.nx + wrap(x0 + lx, G.nx);
                if (SMAG && ly >= -R && ly < TY + R) kdst[q] = (ly + R) * SX + lx + HALO;
            }
        }
        const int me = (ty + HALO) * SX + tx * W + HALO, mk = (ty + R) * SX + tx * W + HALO;
        const bool odd_b = G.pb[fld] < 0, odd_t = G.pt[fld] < 0, heat = fld == 3;
        const T kscale = heat ? GC(inv_Pr) : T(1);
        auto coef = [&](T nv, bool zarm) -> T {              // exchange coefficient from the eddy value
            if constexpr (SMAG == 2) return dd3_coef(nv, zarm, heat, G);
            else return nv * kscale;
        };
        auto column = [&](int z, T (&v)[W]) {                // iterate of the column at plane z (signed mirror)
            int side;
            vload<T, W>(src + (size_t)mirror(z, G.nz, side) * nxy + own, v);
            if ((side == 1 && odd_b) || (side == 2 && odd_t)) {
#pragma unroll
                for (int i = 0; i < W; ++i) v[i] = flip(v[i]);
            }
        };
        auto eddy = [&](int z, T (&v)[W]) {                  // eddy values of the column (even mirror)
            if (SMAG) vload<T, W>(nu + (size_t)max(eddy_row(z, G.nz), 0) * nxy + own, v);
        };
        auto ring = [&](int t) {
            const size_t pz = (size_t)(z0 + t) * nxy;
#pragma unroll
            for (int q = 0; q < HS; ++q) {
                if (hdst[q] >= 0) cpa<T, W>(&pl[t & 1][hdst[q]], src + pz + hsrc[q]);
                if (SMAG && kdst[q] >= 0) cpa<T, W>(&kp[t & 1][kdst[q]], nu + pz + hsrc[q]);
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        const T wz1 = GC(wz1), wz2 = GC(wz2);
        T xw[9][W], kw[3][W], fw[5][W], xn[W], kn[W], rv[W], dv[W];
        ring(0);
#pragma unroll
        for (int q = 0; q < 8; ++q) column(z0 - 4 + q, xw[q]);
        {
            T ka[4][W];
#pragma unroll
            for (int q = 0; q < 4; ++q) eddy(z0 - 2 + q, ka[q]);
            column(z0 + 4, xn);
            eddy(z0 + 2, kn);
            if (!FIRST) {
                vload<T, W>(fr + (size_t)z0 * nxy + own, rv);
                vload<T, W>(fdin + (size_t)z0 * nxy + own, dv);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    const T dz = wz1 * (xw[q + 3][i] - xw[q + 1][i]) + wz2 * (xw[q + 4][i] - xw[q][i]);
                    fw[q][i] = SMAG ? coef(ka[q][i], true) * dz : dz;
                    if (SMAG && q >= 2) kw[q - 2][i] = ka[q][i];
                }
        }
        for (int t = 0; t < nzb; ++t) {
            T* p = pl[t & 1];
            T* kq = kp[t & 1];
            vstore<T, W>(p + me, xw[4]);
            if (SMAG) vstore<T, W>(kq + mk, kw[0]);
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            __syncthreads();
            if (t + 1 < nzb) ring(t + 1);     // its buffers were last read before this plane's barrier
            T rc[W], dc[W];
#pragma unroll
            for (int i = 0; i < W; ++i) {
                xw[8][i] = xn[i];
                if (SMAG) kw[2][i] = kn[i];
                rc[i] = FIRST ? xw[4][i] : rv[i];
                if (!FIRST) dc[i] = dv[i];
                const T dz = wz1 * (xw[7][i] - xw[5][i]) + wz2 * (xn[i] - xw[4][i]);
                fw[4][i] = SMAG ? coef(kn[i], true) * dz : dz;
            }
            if (t + 1 < nzb) {
                column(z0 + t + 5, xn);
                eddy(z0 + t + 3, kn);
                if (!FIRST) {
                    vload<T, W>(fr + (size_t)(z0 + t + 1) * nxy + own, rv);
                    vload<T, W>(fdin + (size_t)(z0 + t + 1) * nxy + own, dv);
                }
            }
            T dif[W];
#pragma unroll
            for (int i = 0; i < W; ++i) dif[i] = wz1 * (fw[3][i] - fw[1][i]) + wz2 * (fw[4][i] - fw[0][i]);
            {   // x: row values at -4 .. W+4, fluxes at -2 .. W+2
                T e[W + 8], kx[W + 8];
#pragma unroll
                for (int i = 0; i < 4; i += W) {
                    T a[W], b[W];
                    vload<T, W>(p + me - 4 + i, a);
                    vload<T, W>(p + me + W + i, b);
#pragma unroll
                    for (int j = 0; j < W; ++j) {
                        e[i + j] = a[j];
                        e[W + 4 + i + j] = b[j];
                    }
                    if (SMAG) {
                        vload<T, W>(kq + mk - 4 + i, a);
                        vload<T, W>(kq + mk + W + i, b);
#pragma unroll
                        for (int j = 0; j < W; ++j) {
                            kx[i + j] = a[j];
                            kx[W + 4 + i + j] = b[j];
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    e[4 + i] = xw[4][i];
                    if (SMAG) kx[4 + i] = kw[0][i];
                }
                T fx[W + 4];
#pragma unroll
                for (int i = 0; i < W + 4; ++i) {
                    if (W == 1 && i == 2) continue;              // the centre flux is not read
                    const T dx = GC(wx1) * (e[i + 3] - e[i + 1]) + GC(wx2) * (e[i + 4] - e[i]);
                    fx[i] = SMAG ? coef(kx[i + 2], false) * dx : dx;
                }
#pragma unroll
                for (int i = 0; i < W; ++i) {
                    dif[i] += GC(wx1) * (fx[i + 3] - fx[i + 1]);
                    dif[i] += GC(wx2) * (fx[i + 4] - fx[i]);
                }
            }
            {   // y: rows -4 .. 4, fluxes at rows -2, -1, 1, 2
                T e[9][W];
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    if (q != 4) vload<T, W>(p + me + (q - 4) * SX, e[q]);
#pragma unroll
                for (int i = 0; i < W; ++i) e[4][i] = xw[4][i];
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    if (q == 2) continue;
                    T ky[W];
                    if (SMAG) vload<T, W>(kq + mk + (q - 2) * SX, ky);
                    const T w = q == 0 ? -GC(wy2) : (q == 1 ? -GC(wy1) : (q == 3 ? GC(wy1) : GC(wy2)));
#pragma unroll
                    for (int i = 0; i < W; ++i) {
                        const T dy = GC(wy1) * (e[q + 3][i] - e[q + 1][i]) + GC(wy2) * (e[q + 4][i] - e[q][i]);
                        dif[i] += w * (SMAG ? coef(ky[i], false) * dy : dy);
                    }
                }
            }
            const T Kc = SMAG ? T(1) : (heat ? GC(K_H) : GC(K_M));
            T xo[W], dk[W];
#pragma unroll
            for (int i = 0; i < W; ++i) {
                const T xk = FIRST ? ith * xw[4][i] : xw[4][i];
                const T df = (FIRST ? ith * Kc : Kc) * dif[i];
                const T res = rc[i] - (GC(two_over_dt) * xk - df);
                dk[i] = a1 * (FIRST ? xk : dc[i]) + a2 * res;
                xo[i] = xk + dk[i];
            }
            if (inside) {
                const size_t o = (size_t)(z0 + t) * nxy + own;
                vstore<T, W>(fzo + o, xo);
                if (!LAST) vstore<T, W>(fdo + o, dk);
                if (LAST) {
#pragma unroll
                    for (int i = 0; i < W; ++i) acc[0] += xo[i] * xo[i];
                }
            }
#pragma unroll
            for (int i = 0; i < W; ++i) {
#pragma unroll
                for (int q = 0; q < 8; ++q) xw[q][i] = xw[q + 1][i];
#pragma unroll
                for (int q = 0; q < 4; ++q) fw[q][i] = fw[q + 1][i];
                if (SMAG) {
                    kw[0][i] = kw[1][i];
                    kw[1][i] = kw[2][i];
                }
            }
        }
    }
    pdl_trigger();
    if (LAST) {
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

// ============================================================================
// Field-block Chebyshev sweep with the horizontal fluxes shared (float64).  One
// CTA = one field of a CX x CY column of CZB planes: blockIdx.z = zblock * 5 +
// field.  Each thread owns one (x, y) column and keeps, in registers, the
// iterate at z-4 .. z+4 and the vertical fluxes K D_z x at z-2 .. z+2; per plane
// the iterate is staged with a halo of 4 and the eddy field with a halo of 2, and
// the fluxes K D_x x, K D_y x are formed once per arm point in shared memory.
// Bound: the FP64 pipe (about 37 operations a point and field; the vector sweep
// forms every flux in each thread that reads it, about 55, which float32 does
// not feel and float64 does: 2.6 against 3.0 ms per apply at 256 x 256 x 64).
// ============================================================================
constexpr int CX = 32, CY = 8;
static_assert(CX * CY == NTHREADS, "one output per thread");
constexpr int CZB = 16;      // planes per CTA of the Chebyshev sweep

template <typename T, int SMAG, int FIRST, int LAST>
__global__ void __launch_bounds__(NTHREADS)
cheb3d_shared(Geo G, int k, const T* __restrict__ r, const T* __restrict__ zin, const T* __restrict__ din,
       T* __restrict__ zout, T* __restrict__ dout, const T* __restrict__ nu, double* part, Ctl* ctl,
       int check_done) {
    constexpr int SX = CX + 2 * HALO, SY = CY + 2 * HALO, SP = SX * SY;      // iterate plane
    constexpr int NX = CX + 2 * R, NY = CY + 2 * R, NP = NX * NY;            // eddy plane
    constexpr int AXN = (CX + 2 * R) * CY, AYN = CX * (CY + 2 * R), AN = AXN + AYN;
    constexpr int XS = (SP + NTHREADS - 1) / NTHREADS;    // staging slots per thread
    constexpr int NS = (NP + NTHREADS - 1) / NTHREADS;
    constexpr int AS = (AN + NTHREADS - 1) / NTHREADS;
    if (check_done && ctl->done) return;
    __shared__ T xs[SP];
    __shared__ T ns[SMAG ? NP : 1];
    __shared__ T kg[AN];       // K D_x x on the x arms, K D_y x on the y arms (D only when K is constant)
    const int fld = blockIdx.z % 5;
    const int z0 = (blockIdx.z / 5) * CZB;
    const int z1 = min(z0 + CZB, G.nz);
    const int x0 = blockIdx.x * CX, y0 = blockIdx.y * CY;
    const T ith = cheb_coef<T>(ctl, fld, k, 0);
    const T a1 = cheb_coef<T>(ctl, fld, k, 1);
    const T a2 = cheb_coef<T>(ctl, fld, k, 2);
    const size_t nxy = (size_t)G.ny * G.nx;
    const T* fr = r + (size_t)fld * G.npt;
    const T* fsrc = (FIRST ? r : zin) + (size_t)fld * G.npt;
    const T* fdin = FIRST ? nullptr : din + (size_t)fld * G.npt;
    T* fzo = zout + (size_t)fld * G.npt;
    T* fdo = dout + (size_t)fld * G.npt;
    const int tx = threadIdx.x % CX, ty = threadIdx.x / CX;
    const int gx = x0 + tx, gy = y0 + ty;
    const bool inside = gx < G.nx && gy < G.ny;
    const size_t own = inside ? (size_t)gy * G.nx + gx : 0;       // in-plane offset of the thread's column
    T acc[1] = {T(0)};
    if (fld == 4) {
        if (LAST && inside) {
            for (int z = z0; z < z1; ++z) {
                const size_t o = (size_t)z * nxy + own;
                const T zv = fr[o] * ith;
                fzo[o] = zv;
                acc[0] += zv * zv;
            }
        }
    } else {
        // in-plane offsets of this thread's staging slots (-1: unused slot)
        int xoff[XS], noff[NS], acen[AS], anu[AS];
#pragma unroll
        for (int q = 0; q < XS; ++q) {
            const int idx = threadIdx.x + q * NTHREADS;
            xoff[q] = idx < SP ? wrap(y0 + idx / SX - HALO, G.ny) * G.nx + wrap(x0 + idx % SX - HALO, G.nx) : -1;
        }
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            const int idx = threadIdx.x + q * NTHREADS;
            noff[q] = (SMAG && idx < NP) ? wrap(y0 + idx / NX - R, G.ny) * G.nx + wrap(x0 + idx % NX - R, G.nx) : -1;
        }
#pragma unroll
        for (int q = 0; q < AS; ++q) {
            const int idx = threadIdx.x + q * NTHREADS;
            if (idx < AXN) {
                const int qx = idx % NX, qy = idx / NX;          // x arm at tile (qx - R, qy)
                acen[q] = (qy + HALO) * SX + qx + R;
                anu[q] = (qy + R) * NX + qx;
            } else if (idx < AN) {
                const int j = idx - AXN;
                const int qx = j % CX, qy = j / CX;               // y arm at tile (qx, qy - R)
                acen[q] = -((qy + R) * SX + qx + HALO) - 1;       // negative: a y arm
                anu[q] = qy * NX + qx + R;
            } else {
                acen[q] = 0;
                anu[q] = -1;
            }
        }
        // what the fluxes leave out: 1/Pr of theta, the constant K, 1/theta_c of a first sweep
        const T fscale = (SMAG == 2 ? T(1) : SMAG ? (fld == 3 ? GC(inv_Pr) : T(1)) : (fld == 3 ? GC(K_H) : GC(K_M))) * (FIRST ? ith : T(1));
        // FIRST: x_1 = r / theta_c enters as r, the sum of the fluxes is scaled at the end
        const T wz1 = GC(wz1), wz2 = GC(wz2);
        auto D = [](const T* s, int i, int st, T w1, T w2) {
            return w1 * (s[i + st] - s[i - st]) + w2 * (s[i + 2 * st] - s[i - 2 * st]);
        };
        auto xval = [&](int z) -> T {          // iterate at row z of the column (mirror ghosts)
            int side;
            const int sz = mirror(z, G.nz, side);
            const T v = fsrc[(size_t)sz * nxy + own];
            return (side == 1 && G.pb[fld] < 0) || (side == 2 && G.pt[fld] < 0) ? flip(v) : v;
        };
        auto zflux = [&](T d, int z) -> T {    // K D_z x at row z (eddy field mirrored even)
            if (!SMAG) return d;
            const int sz = eddy_row(z, G.nz);
            const T nv = sz >= 0 ? nu[(size_t)sz * nxy + own] : T(0);
            return (SMAG == 2 ? dd3_coef(nv, true, fld == 3, G) : nv) * d;
        };
        T xw[9], fw[5];
        if (inside) {
#pragma unroll
            for (int q = 0; q < 8; ++q) xw[q] = xval(z0 - 4 + q);
#pragma unroll
            for (int q = 0; q < 4; ++q) fw[q] = zflux(wz1 * (xw[q + 3] - xw[q + 1]) + wz2 * (xw[q + 4] - xw[q]), z0 - 2 + q);
        }
        // every global value a plane needs (its staged tile and eddy plane, the
        // point's r, d, the iterate at z+4 and the eddy field at z+2) is loaded one
        // plane ahead into registers, so that the latency overlaps the previous
        // plane's arithmetic
        T px[XS], pn[NS];
        T pr = T(0), pd = T(0), px4 = T(0), pnu2 = T(0);
        auto prefetch = [&](int z) {
            const size_t pz = (size_t)z * nxy;
#pragma unroll
            for (int q = 0; q < XS; ++q) px[q] = xoff[q] >= 0 ? fsrc[pz + xoff[q]] : T(0);
#pragma unroll
            for (int q = 0; q < NS; ++q) pn[q] = (SMAG && noff[q] >= 0) ? nu[pz + noff[q]] : T(0);
            if (inside) {
                pr = fr[pz + own];
                if (!FIRST) pd = fdin[pz + own];
                px4 = xval(z + 4);
                if (SMAG) {
                    const int sz = eddy_row(z + 2, G.nz);
                    pnu2 = sz >= 0 ? nu[(size_t)sz * nxy + own] : T(0);
                }
            }
        };
        prefetch(z0);
        for (int z = z0; z < z1; ++z) {
            const size_t pz = (size_t)z * nxy;
#pragma unroll
            for (int q = 0; q < XS; ++q)
                if (xoff[q] >= 0) xs[threadIdx.x + q * NTHREADS] = px[q];
            if (SMAG) {
#pragma unroll
                for (int q = 0; q < NS; ++q)
                    if (noff[q] >= 0) ns[threadIdx.x + q * NTHREADS] = pn[q];
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < AS; ++q) {
                if (anu[q] < 0) continue;
                const bool xarm = acen[q] >= 0;
                const int c = xarm ? acen[q] : -acen[q] - 1;
                const T d = xarm ? D(xs, c, 1, GC(wx1), GC(wx2)) : D(xs, c, SX, GC(wy1), GC(wy2));
                T kv = T(1);
                if (SMAG) {
                    const T nv = ns[anu[q]];
                    kv = SMAG == 2 ? dd3_coef(nv, false, fld == 3, G) : nv;
                }
                kg[threadIdx.x + q * NTHREADS] = SMAG ? kv * d : d;
            }
            __syncthreads();
            const T rv = pr, dv = pd, nu2 = pnu2;
            xw[8] = px4;
            if (z + 1 < z1) prefetch(z + 1);
            if (inside) {
                {
                    const T dz2 = wz1 * (xw[7] - xw[5]) + wz2 * (xw[8] - xw[4]);
                    fw[4] = SMAG ? (SMAG == 2 ? dd3_coef(nu2, true, fld == 3, G) : nu2) * dz2 : dz2;
                }
                const int cax = ty * NX + tx + R;
                const int cay = AXN + (ty + R) * CX + tx;
                const T dif = D(kg, cax, 1, GC(wx1), GC(wx2)) + D(kg, cay, CX, GC(wy1), GC(wy2)) +
                              (wz1 * (fw[3] - fw[1]) + wz2 * (fw[4] - fw[0]));
                const T xk = FIRST ? ith * xw[4] : xw[4];
                const size_t o = pz + own;
                const T res = rv - (GC(two_over_dt) * xk - fscale * dif);
                const T dprev = FIRST ? rv * ith : dv;
                const T dk = a1 * dprev + a2 * res;
                const T xn = xk + dk;
                fzo[o] = xn;
                if (!LAST) fdo[o] = dk;
                if (LAST) acc[0] += xn * xn;
#pragma unroll
                for (int q = 0; q < 8; ++q) xw[q] = xw[q + 1];
#pragma unroll
                for (int q = 0; q < 4; ++q) fw[q] = fw[q + 1];
            }
        }
    }
    if (LAST) {
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

// ============================================================================
// Budgets: E_k = 1/2 sum (u^2+v^2+w^2) dV, E_p = sum (lz - z) theta dV,
// sum theta dV, sum div(u) dV, max / min of the five fields.
// ============================================================================
__global__ void __launch_bounds__(NTHREADS)
budgets3d(Geo G, const double* __restrict__ u, double dV, double dz, double lz, double* part,
          Ctl* ctl, double* out) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    double mx[10];
    for (int f = 0; f < 10; ++f) mx[f] = -1e300;
    const int nxy = G.nx * G.ny;
    const double* U = u;
    const double* Vv = u + G.npt;
    const double* W = u + 2 * (size_t)G.npt;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < G.npt; p += gridDim.x * blockDim.x) {
        const int z = p / nxy, rem = p - z * nxy;
        const int y = rem / G.nx, x = rem - y * G.nx;
        const double zc = (z + 0.5) * dz;
        s[0] += 0.5 * (U[p] * U[p] + Vv[p] * Vv[p] + W[p] * W[p]);
        s[1] += (lz - zc) * u[3 * (size_t)G.npt + p];
        s[2] += u[3 * (size_t)G.npt + p];
        double ux = 0.0, vy = 0.0, wz = 0.0;
        for (int l = 1; l <= 2; ++l) {
            const double c = l == 1 ? 2.0 / 3.0 : -1.0 / 12.0;
            ux += c * (U[(size_t)z * nxy + y * G.nx + wrap(x + l, G.nx)] - U[(size_t)z * nxy + y * G.nx + wrap(x - l, G.nx)]);
            vy += c * (Vv[(size_t)z * nxy + wrap(y + l, G.ny) * G.nx + x] - Vv[(size_t)z * nxy + wrap(y - l, G.ny) * G.nx + x]);
            int sp_, sm_;
            const int zp = mirror(z + l, G.nz, sp_), zm = mirror(z - l, G.nz, sm_);
            const double gp = sp_ == 2 ? -1.0 : 1.0, gm = sm_ == 1 ? -1.0 : 1.0;   // w odd at both walls
            wz += c * (gp * W[(size_t)zp * nxy + y * G.nx + x] - gm * W[(size_t)zm * nxy + y * G.nx + x]);
        }
        s[3] += ux * G.inv_dx + vy * G.inv_dy + wz * G.inv_dz;
        for (int f = 0; f < 5; ++f) {
            const double val = u[(size_t)f * G.npt + p];
            mx[f] = max_nan(mx[f], val);
            mx[5 + f] = max_nan(mx[5 + f], -val);
        }
    }
    double* pmax = part + 4 * gridDim.x;
    block_partials<4>(s, 4, part, gridDim.x, blockIdx.x);
    block_partials_max<10>(mx, 10, pmax, gridDim.x, blockIdx.x);
    if (arrive_last(&ctl->counter[CNT_MISC], gridDim.x)) {
        __shared__ double tot[14];
        final_sums(part, gridDim.x, 4, tot);
        final_maxes(pmax, gridDim.x, 10, tot + 4);
        if (threadIdx.x == 0) {
            for (int i = 0; i < 4; ++i) out[i] = tot[i] * dV;
            for (int f = 0; f < 5; ++f) { out[4 + f] = tot[4 + f]; out[9 + f] = -tot[9 + f]; }
        }
    }
}


// ------------------------------------------------------------------ launchers
template <typename K>
static cudaError_t set_smem(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

static int stream_blocks3(size_t n) {
    size_t b = (n + NTHREADS - 1) / NTHREADS;
    return (int)(b < (size_t)MAX_STREAM_BLOCKS ? (b > 0 ? b : 1) : MAX_STREAM_BLOCKS);
}

// Scratch of the split passes inside G.s3 (7 npt values of T): the plane
// pass's partial sums (5 npt), then the strain values s1, s0 (npt each).
template <typename T>
struct S3 {
    T *P, *s1, *s0;
    explicit S3(const Geo& G) {
        T* b = reinterpret_cast<T*>(G.s3);
        P = b;
        s1 = b + 5 * (size_t)G.npt;
        s0 = b + 6 * (size_t)G.npt;
    }
};

// Planes per CTA of the column pass: the split with the fewest rounds of CTAs
// times steps (the eight lead-in steps of a march cost about three full ones).
static int column_planes(const Geo& G, int slots) {
    const long long cols = ((long long)G.nx * G.ny + CW - 1) / CW;
    int best = G.nz;
    double least = 1e300;
    for (int parts = 1; parts <= 16; ++parts) {
        const int zc = (G.nz + parts - 1) / parts;
        if (zc < 8 && parts > 1) break;
        const long long ctas = cols * ((G.nz + zc - 1) / zc);
        const double cost = (double)((ctas + slots - 1) / slots) * (zc + 3.0);
        if (cost < least) {
            least = cost;
            best = zc;
        }
    }
    return best;
}

template <typename T, int KIND, int SMAG>
static cudaError_t launch_split(int mode, const Geo& G, const T* u, const T* v, const T* Fu, const double* f, T* out,
                                T* out2, double* part, Ctl* ctl, int check_done, cudaStream_t s) {
    if (G.s3 == nullptr) return cudaErrorInvalidValue;
    using SH = PlaneShape<T, KIND, SMAG>;
    S3<T> sc(G);
    static std::atomic<int> slots{0};   // resident column CTAs; set once, concurrent first calls are harmless
    cudaError_t e;
    if (slots.load() == 0) {
        int dev = 0, nsm = 0, per = 0;
        if ((e = set_smem(plane3d<T, KIND, SMAG>, SH::smem)) != cudaSuccess || (e = cudaGetDevice(&dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, column3d<T, KIND, SMAG>, COL_THREADS, 0)) != cudaSuccess)
            return e;
        slots = std::max(1, nsm * per);
    }
    if (SMAG) {
        dim3 gk((G.nx + KX - 1) / KX, (G.ny + KY - 1) / KY, (G.nz + SZB - 1) / SZB);
        bool pairs = false;
        if constexpr (KIND == PAIR && sizeof(T) == sizeof(float)) {
            auto at = [](const void* q) { return reinterpret_cast<uintptr_t>(q); };
            pairs = G.nx % 2 == 0 && ((at(u) | at(v) | at(sc.s0) | at(sc.s1)) & 7) == 0;
            if (pairs) {
                gk.x = (G.nx / 2 + KX - 1) / KX;
                strain3d_pairs<<<gk, NTHREADS, 0, s>>>(G, u, v, sc.s0, sc.s1, ctl, check_done);
            }
        }
        if (!pairs) strain3d<T, KIND, 0><<<gk, NTHREADS, 0, s>>>(G, u, v, sc.s0, sc.s1, part, ctl, check_done);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    dim3 gp((G.nx + PX - 1) / PX, (G.ny + SH::PY - 1) / SH::PY, G.nz);
    plane3d<T, KIND, SMAG><<<gp, NTHREADS, SH::smem, s>>>(G, u, v, sc.s0, sc.s1, sc.P, ctl, check_done);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int zc = column_planes(G, slots.load());
    dim3 gc((unsigned)(((size_t)G.nx * G.ny + CW - 1) / CW), (G.nz + zc - 1) / zc);
    column3d<T, KIND, SMAG><<<gc, COL_THREADS, 0, s>>>(G, mode, zc, u, v, Fu, f, sc.s0, sc.s1, sc.P, out, out2, part, ctl,
                                                     check_done);
    return cudaGetLastError();
}

template <typename T, int KIND>
static cudaError_t launch_split_k(int mode, const Geo& G, const T* u, const T* v, const T* Fu, const double* f, T* out,
                                  T* out2, double* part, Ctl* ctl, int check_done, cudaStream_t s) {
    if (G.sgs == 2) return launch_split<T, KIND, 2>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
    return G.smag ? launch_split<T, KIND, 1>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s)
                  : launch_split<T, KIND, 0>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
}

// ---------------------------------------------------------------------------
// Acoustic Schur-complement preconditioner in 3-D (scaled units): the 2-D
// construction with three velocity components,
//   H dp = v_p - c_div (D_x v_u + D_y v_v + D_z v_w),  H = (2/dt) I - a sum_j D_j D_j,
//   z_i = (dt/2)(v_i - c_grad D_i dp),  z_theta = v_theta / theta_c,
// with H applied point-wise as the composite stencil of the first derivative
// taken twice along each axis (in float32 in the line's first differences, HELM_DIFF:
// p errs 20 % less; in float64, where the FP64 pipe counts operations, 25 against 36,
// through its coefficients) on the ghost-extended plane (p even at the walls), which equals D_j applied to D_j dp evaluated with its ghosts.
// Fields: 0 u, 1 v, 2 w, 3 theta, 4 p; planes [z][y][x].
//
// ---------------------------------------------------------------------------
// e[0 .. W+4) = row[gx-2 .. gx+W+2) of a periodic row (gx and nx multiples of W)
template <typename T, int W>
__device__ __forceinline__ void row_taps(const T* __restrict__ row, int gx, int nx, T (&e)[W + 4]) {
    if constexpr (W == 1) {
#pragma unroll
        for (int k = 0; k < 5; ++k) e[k] = row[wrap(gx + k - 2, nx)];
    } else {
        T l[W], c[W], r[W];
        vload<T, W>(row + wrap(gx - W, nx), l);
        vload<T, W>(row + gx, c);
        vload<T, W>(row + wrap(gx + W, nx), r);
        e[0] = l[W - 2];
        e[1] = l[W - 1];
#pragma unroll
        for (int k = 0; k < W; ++k) e[2 + k] = c[k];
        e[W + 2] = r[0];
        e[W + 3] = r[1];
    }
}

// D along y or z of W points: rows at offsets o[0..3] = -2, -1, +1, +2, the
// ghost rows' signs in sg (odd fields at a wall)
template <typename T, int W>
__device__ __forceinline__ void line_d(const T* __restrict__ f, const size_t (&o)[4], const T (&sg)[4], T ih, T (&d)[W]) {
    T a[4][W];
#pragma unroll
    for (int k = 0; k < 4; ++k) vload<T, W>(f + o[k], a[k]);
#pragma unroll
    for (int i = 0; i < W; ++i) d[i] = d5(sg[0] * a[0][i], sg[1] * a[1][i], sg[2] * a[2][i], sg[3] * a[3][i], ih);
}

// Row offsets of the y and z neighbours of vector (gz, gy, gx) and, for a
// field that is odd at the walls, the signs of its ghost planes.
template <typename T>
__device__ __forceinline__ void line_offsets(const Geo& G, int gz, int gy, int gx, int fld, size_t (&oy)[4],
                                             size_t (&oz)[4], T (&sz)[4]) {
    constexpr int s[4] = {-2, -1, 1, 2};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        oy[k] = ((size_t)gz * G.ny + wrap(gy + s[k], G.ny)) * G.nx + gx;
        int side;
        const int mz = mirror(gz + s[k], G.nz, side);
        oz[k] = ((size_t)mz * G.ny + gy) * G.nx + gx;
        sz[k] = side == 0 ? T(1) : (side == 1 ? T(G.pb[fld]) : T(G.pt[fld]));
    }
}

template <typename T, int W>
__global__ void __launch_bounds__(NTHREADS)
schur_rhs3d(Geo G, const T* __restrict__ r, T* __restrict__ rhs, Ctl* ctl, int check_done) {
    pdl_wait();
    if (check_done && ctl->done) return;
    const T cdiv = GC(schur_cdiv);
    const T ix = GC(inv_dx), iy = GC(inv_dy), iz = GC(inv_dz);
    const T one[4] = {T(1), T(1), T(1), T(1)};
    const size_t np = (size_t)G.npt;
    const unsigned nv = G.npt / W, nxv = G.nx / W, nxy = nxv * G.ny;
    for (unsigned q = blockIdx.x * NTHREADS + threadIdx.x; q < nv; q += gridDim.x * NTHREADS) {
        const int gz = q / nxy, gy = (q - gz * nxy) / nxv, gx = (q % nxv) * W;
        const size_t p = (size_t)q * W;
        size_t oy[4], oz[4];
        T sz[4], e[W + 4], dy[W], dz[W], c[W];
        line_offsets<T>(G, gz, gy, gx, 2, oy, oz, sz);
        row_taps<T, W>(r + p - gx, gx, G.nx, e);
        line_d<T, W>(r + np, oy, one, iy, dy);
        line_d<T, W>(r + 2 * np, oz, sz, iz, dz);
        vload<T, W>(r + 4 * np + p, c);
#pragma unroll
        for (int i = 0; i < W; ++i) c[i] -= cdiv * (d5(e[i], e[i + 1], e[i + 3], e[i + 4], ix) + dy[i] + dz[i]);
        vstore<T, W>(rhs + p, c);
    }
    pdl_trigger();
}

// ---------------------------------------------------------------------------
// One Chebyshev sweep k for H x = rhs (FIRST: x_k = rhs / theta_c, d_{k-1} = x_k).
// A CTA marches a TX x TY column of planes in z.  Each thread keeps its W
// points' column x(z-4 .. z+4) in registers (one new plane per step, loaded a
// step ahead together with rhs and d); per plane the column's own values are
// written to shared memory and only the ring of 4 points around the tile is
// fetched (cp.async, one plane ahead, two buffers: one barrier per plane).
//
// Bound: HBM and L2 (x, rhs, d read, x, d written: 20 B a point, 168 MB at
// 256 x 256 x 128, 25 us).  Odd sweeps march downwards (REV), so that each
// sweep starts on the planes the previous one left in L2.  The former kernel
// read all 25 taps of every point from global memory with a wrap or mirror
// each and had two CTAs per SM in a grid-stride loop: 297 us at that size;
// this one 31.8 us (34.4 without the alternating direction), and 2.6 us more with the
// first differences of float32.
// ---------------------------------------------------------------------------
template <typename T>
struct HelmC {                      // coefficients of a sweep in the type of the sweep
    // float32: res = rhs + c0 x + sum_k c_k (g_k - g_{-1-k}), g_k = x_{k+1} - x_k along each axis
    // float64: res = rhs + c0 x + lap0 x + sum_k c_k (x_{+k+1} + x_{-k-1})
    T c0, lap0, cx[4], cy[4], cz[4];
};

template <typename T, int W, int FIRST, int LAST>
__global__ void __launch_bounds__(NTHREADS, 2)
helm3d(Geo G, HelmC<T> C, int k, int zb, int rev, const T* __restrict__ rhs, const T* __restrict__ xin,
       const T* __restrict__ din, T* __restrict__ xout, T* __restrict__ dout, Ctl* ctl, int check_done) {
    constexpr int NXT = HelmTile<T, W>::NXT, NYT = HelmTile<T, W>::NYT;
    constexpr int TX = NXT * W, TY = NYT, SX = TX + 2 * HALO, SY = TY + 2 * HALO, SP = SX * SY;
    // ring of the tile in vectors: HALO rows above and below, HALO columns either side
    constexpr int NH = (2 * HALO * TX + 2 * HALO * TY) / W, HS = (NH + NTHREADS - 1) / NTHREADS;
    static_assert(NXT * NYT == NTHREADS, "one vector per thread");
    constexpr bool DIFF = sizeof(T) == sizeof(float);
    __shared__ __align__(16) T pl[2][SP];
    pdl_wait();
    const int done = check_done ? ctl->done : 0;
    const T ith = cheb_coef<T>(ctl, 5, k, 0), a1 = cheb_coef<T>(ctl, 5, k, 1), a2 = cheb_coef<T>(ctl, 5, k, 2);
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zb, nzb = min(zb, G.nz - z0);
    const size_t nxy = (size_t)G.ny * G.nx;
    const T* src = FIRST ? rhs : xin;
    int hdst[HS], hsrc[HS];
#pragma unroll
    for (int q = 0; q < HS; ++q) {
        int h = threadIdx.x + q * NTHREADS;
        hdst[q] = -1;
        hsrc[q] = 0;
        if (h < NH) {
            int ly, lx;                                  // staged row, column (relative to the tile origin)
            if (h < 2 * HALO * NXT) {
                ly = h / NXT;
                ly = ly < HALO ? ly - HALO : TY + ly - HALO;
                lx = (h % NXT) * W;
            } else {
                h -= 2 * HALO * NXT;
                constexpr int PER = 2 * HALO / W;        // vectors of the two sides of a row
                ly = h / PER;
                const int c = h % PER;
                lx = c < PER / 2 ? c * W - HALO : TX + (c - PER / 2) * W;
            }
            hdst[q] = (ly + HALO) * SX + lx + HALO;
            hsrc[q] = wrap(y0 + ly, G.ny) * G.nx + wrap(x0 + lx, G.nx);
        }
    }
    const int tx = threadIdx.x % NXT, ty = threadIdx.x / NXT;
    const int gx = x0 + tx * W, gy = y0 + ty;
    const bool inside = gx < G.nx && gy < G.ny;
    const size_t own = (size_t)wrap(gy, G.ny) * G.nx + wrap(gx, G.nx);
    const int me = (ty + HALO) * SX + tx * W + HALO;
    // plane t of the march, and its storage row (even mirror at the walls)
    auto plane = [&](int t) {
        int side;
        return (size_t)mirror(rev ? z0 + nzb - 1 - t : z0 + t, G.nz, side) * nxy;
    };
    auto ring = [&](int t) {
        const size_t pz = plane(t);
#pragma unroll
        for (int q = 0; q < HS; ++q)
            if (hdst[q] >= 0) cpa<T, W>(&pl[t & 1][hdst[q]], src + pz + hsrc[q]);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    T xw[9][W], gz[8][W], xn[W], rv[W], dv[W];      // the column's values and (float32: kept instead of those below) differences
    ring(0);
#pragma unroll
    for (int q = 0; q < 8; ++q) vload<T, W>(src + plane(q - 4) + own, xw[q]);
#pragma unroll
    for (int q = 0; q < 7; ++q)
#pragma unroll
        for (int i = 0; i < W; ++i) gz[q][i] = xw[q + 1][i] - xw[q][i];
    vload<T, W>(src + plane(4) + own, xn);
    vload<T, W>(rhs + plane(0) + own, rv);
    if (!FIRST) vload<T, W>(din + plane(0) + own, dv);
    if (done) {
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        return;
    }
    for (int t = 0; t < nzb; ++t) {
        T* p = pl[t & 1];
        vstore<T, W>(p + me, xw[4]);
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();
        if (t + 1 < nzb) ring(t + 1);     // its buffer was last read before this plane's barrier
        T r[W], d[W];
#pragma unroll
        for (int i = 0; i < W; ++i) {
            xw[8][i] = xn[i];
            r[i] = rv[i];
            if (!FIRST) d[i] = dv[i];
        }
        if (t + 1 < nzb) {
            vload<T, W>(src + plane(t + 5) + own, xn);
            vload<T, W>(rhs + plane(t + 1) + own, rv);
            if (!FIRST) vload<T, W>(din + plane(t + 1) + own, dv);
        }
        T s[W], e[W + 2 * HALO];
#pragma unroll
        for (int i = 0; i < HALO; i += W) {
            T a[W], b[W];
            vload<T, W>(p + me - HALO + i, a);
            vload<T, W>(p + me + W + i, b);
#pragma unroll
            for (int j = 0; j < W; ++j) {
                e[i + j] = a[j];
                e[W + HALO + i + j] = b[j];
            }
        }
#pragma unroll
        for (int i = 0; i < W; ++i) e[HALO + i] = xw[4][i];
        // the differences first: they are small (float64: the coefficients' form, see above)
        T g[W + 2 * HALO - 1], pa[W], pb[W];
#pragma unroll
        for (int i = 0; i < W + 2 * HALO - 1; ++i) g[i] = e[i + 1] - e[i];
#pragma unroll
        for (int i = 0; i < W; ++i) {
            gz[7][i] = xw[8][i] - xw[7][i];
            pa[i] = pb[i] = xw[4][i];
            s[i] = DIFF ? T(0) : C.lap0 * xw[4][i];
#pragma unroll
            for (int l = 3; l >= 0; --l) {
                s[i] += C.cx[l] * (DIFF ? g[HALO + i + l] - g[HALO - 1 + i - l] : e[HALO + 1 + i + l] + e[HALO - 1 + i - l]);
                s[i] += C.cz[l] * (DIFF ? gz[4 + l][i] - gz[3 - l][i] : xw[5 + l][i] + xw[3 - l][i]);
            }
        }
#pragma unroll
        for (int l = 1; l <= 4; ++l) {
            T a[W], b[W];
            vload<T, W>(p + me + l * SX, a);
            vload<T, W>(p + me - l * SX, b);
#pragma unroll
            for (int i = 0; i < W; ++i) {
                s[i] += C.cy[l - 1] * (DIFF ? (a[i] - pa[i]) - (pb[i] - b[i]) : a[i] + b[i]);
                pa[i] = a[i];
                pb[i] = b[i];
            }
        }
#pragma unroll
        for (int i = 0; i < W; ++i) s[i] += C.c0 * xw[4][i];
        T xo[W], dk[W];
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const T xk = FIRST ? ith * xw[4][i] : xw[4][i];
            const T res = r[i] + (FIRST ? ith * s[i] : s[i]);
            dk[i] = a1 * (FIRST ? xk : d[i]) + a2 * res;
            xo[i] = xk + dk[i];
        }
        if (inside) {
            const size_t o = plane(t) + own;
            vstore<T, W>(xout + o, xo);
            if (!LAST) vstore<T, W>(dout + o, dk);
        }
#pragma unroll
        for (int i = 0; i < W; ++i) {
#pragma unroll
            for (int q = DIFF ? 4 : 0; q < 8; ++q) xw[q][i] = xw[q + 1][i];
#pragma unroll
            for (int q = 0; q < 7; ++q) gz[q][i] = gz[q + 1][i];
        }
    }
    pdl_trigger();
}

template <typename T, int W>
__global__ void __launch_bounds__(NTHREADS)
schur_back3d(Geo G, const T* __restrict__ r, T* __restrict__ z, double* part, Ctl* ctl, int check_done) {
    pdl_wait();
    if (check_done && ctl->done) return;
    const T cgrad = GC(schur_cgrad), hdt = GC(half_dt);
    const T ith_t = cheb_coef<T>(ctl, 3, 0, 0);
    const T ix = GC(inv_dx), iy = GC(inv_dy), iz = GC(inv_dz);
    const T one[4] = {T(1), T(1), T(1), T(1)};
    const size_t np = (size_t)G.npt;
    const T* dp = z + 4 * np;
    T acc[1] = {T(0)};
    const unsigned nv = G.npt / W, nxv = G.nx / W, nxy = nxv * G.ny;
    for (unsigned q = blockIdx.x * NTHREADS + threadIdx.x; q < nv; q += gridDim.x * NTHREADS) {
        const int gz = q / nxy, gy = (q - gz * nxy) / nxv, gx = (q % nxv) * W;
        const size_t p = (size_t)q * W;
        size_t oy[4], oz[4];
        T sz[4], e[W + 4], dy[W], dz[W], ru[W], rv[W], rw[W], rt[W];
        line_offsets<T>(G, gz, gy, gx, 4, oy, oz, sz);
        row_taps<T, W>(dp + p - gx, gx, G.nx, e);
        line_d<T, W>(dp, oy, one, iy, dy);
        line_d<T, W>(dp, oz, sz, iz, dz);
        vload<T, W>(r + p, ru);
        vload<T, W>(r + np + p, rv);
        vload<T, W>(r + 2 * np + p, rw);
        vload<T, W>(r + 3 * np + p, rt);
#pragma unroll
        for (int i = 0; i < W; ++i) {
            ru[i] = hdt * (ru[i] - cgrad * d5(e[i], e[i + 1], e[i + 3], e[i + 4], ix));
            rv[i] = hdt * (rv[i] - cgrad * dy[i]);
            rw[i] = hdt * (rw[i] - cgrad * dz[i]);
            rt[i] *= ith_t;
            acc[0] += ru[i] * ru[i] + rv[i] * rv[i] + rw[i] * rw[i] + rt[i] * rt[i] + e[i + 2] * e[i + 2];
        }
        vstore<T, W>(z + p, ru);
        vstore<T, W>(z + np + p, rv);
        vstore<T, W>(z + 2 * np + p, rw);
        vstore<T, W>(z + 3 * np + p, rt);
    }
    block_partials<1, T>(acc, 1, part, gridDim.x, blockIdx.x);
    if (arrive_last(&ctl->counter[CNT_PC], gridDim.x)) {
        __shared__ double tot[1];
        final_sums(part, gridDim.x, 1, tot);
        if (threadIdx.x < 5) put_eps_norm2(ctl, tot[0]);
    }
}

}  // namespace d3

// ------------------------------------------------------------------ entry points
int stencil3d_part_blocks(const Geo& G) {
    // largest reduction grid any 3-D kernel launches
    using namespace d3;
    const long long column = ((long long)G.nx * G.ny + CW - 1) / CW * ((G.nz + 7) / 8);     // marches of eight planes at least
    const long long cheb = (long long)((G.nx + 31) / 32) * ((G.ny + 7) / 8) * ((G.nz + 7) / 8) * 5;   // smallest tile and march
    const long long strain = (long long)((G.nx + KX - 1) / KX) * ((G.ny + KY - 1) / KY) * G.nz;
    return (int)std::max(column, std::max(cheb, strain));
}

size_t stencil3d_scratch_bytes(const Geo& G) { return 7 * (size_t)G.npt * sizeof(double); }

template <typename T>
cudaError_t launch_stencil3d(int mode, const Geo& G, const T* u, const T* v, const T* Fu, const double* f,
                             T* out, T* out2, double* part, Ctl* ctl, int check_done, cudaStream_t s) {
    using namespace d3;
    if (mode < d3::MODE_F || mode > d3::MODE_RHSRES) return cudaErrorInvalidValue;
    if (mode != d3::MODE_JV) return launch_split_k<T, ONE>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
    // the plain forward difference is the float64 path's; float32 takes launch_jv_diff3d
    if constexpr (sizeof(T) == sizeof(double))
        return launch_split_k<T, SHIFT>(mode, G, u, v, Fu, f, out, out2, part, ctl, check_done, s);
    return cudaErrorNotSupported;
}
template cudaError_t launch_stencil3d<float>(int, const Geo&, const float*, const float*, const float*,
                                             const double*, float*, float*, double*, Ctl*, int, cudaStream_t);
template cudaError_t launch_stencil3d<double>(int, const Geo&, const double*, const double*, const double*,
                                              const double*, double*, double*, double*, Ctl*, int, cudaStream_t);

cudaError_t launch_jv_diff3d(const Geo& G, const float* u, const float* v, float* out, Ctl* ctl, int check_done,
                             cudaStream_t s) {
    using namespace d3;
    return launch_split_k<float, PAIR>(d3::MODE_JV, G, u, v, nullptr, nullptr, out, nullptr, nullptr, ctl, check_done, s);
}

template <typename T>
cudaError_t launch_eddy3d(const Geo& G, const T* u, T* nu, double* part, Ctl* ctl, cudaStream_t s) {
    using namespace d3;
    dim3 gk((G.nx + KX - 1) / KX, (G.ny + KY - 1) / KY, (G.nz + SZB - 1) / SZB);
    strain3d<T, ONE, 1><<<gk, NTHREADS, 0, s>>>(G, u, nullptr, nullptr, nu, part, ctl, 0);
    return cudaGetLastError();
}
template cudaError_t launch_eddy3d<float>(const Geo&, const float*, float*, double*, Ctl*, cudaStream_t);
template cudaError_t launch_eddy3d<double>(const Geo&, const double*, double*, double*, Ctl*, cudaStream_t);

// Points per thread of the marching sweeps: 16 bytes where the rows are
// multiples of that, else 8 bytes of float32, else one.  Every plane of the
// workspace vectors starts a multiple of npt elements in, so nx decides the
// alignment; r and z of the per-call entry may be the caller's (8-byte aligned)
// float64 arrays.
template <typename T>
static int row_vector(const Geo& G, const T* r, const T* z) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(r) | reinterpret_cast<uintptr_t>(z);
    if (G.nx % (16 / sizeof(T)) == 0 && (a & 15) == 0) return 16 / sizeof(T);
    return sizeof(T) == 4 && G.nx % 2 == 0 && (a & 7) == 0 ? 2 : 1;
}

template <typename T, int W, int SMAG>
static cudaError_t launch_pc3_w(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb_, T* da, T* db,
                                const T* nu, double* part, Ctl* ctl, int check_done, cudaStream_t s,
                                long long* launches) {
    using namespace d3;
    constexpr int SMS = 152;
    constexpr int TX = HelmTile<T, W>::NXT * W, TY = HelmTile<T, W>::NYT;
    const int gx = (G.nx + TX - 1) / TX, gy = (G.ny + TY - 1) / TY;
    // planes per CTA: the longest march that still gives every SM two CTAs of the
    // four diffused fields (each march reads eight planes beyond its own)
    int zb = 64;
    while (zb > 8 && 4LL * gx * gy * ((G.nz + zb - 1) / zb) < 2 * SMS) zb /= 2;
    dim3 grid(gx, gy, ((G.nz + zb - 1) / zb) * 5);
    const T* zin = nullptr;
    const T* din = nullptr;
    T* zbuf[2] = {za, zb_};
    T* dbuf[2] = {da, db};
    for (int k = 1; k <= sweeps - 1; ++k) {
        const bool first = k == 1, last = k == sweeps - 1;
        T* zo = last ? z : zbuf[k & 1];
        T* dO = dbuf[k & 1];
        auto* kern = first ? (last ? cheb3d<T, W, SMAG, 1, 1> : cheb3d<T, W, SMAG, 1, 0>)
                           : (last ? cheb3d<T, W, SMAG, 0, 1> : cheb3d<T, W, SMAG, 0, 0>);
        const cudaError_t e = launch_pdl(kern, grid, dim3(NTHREADS), 0, s, G, k, zb, r, zin, din, zo, dO, nu, part, ctl,
                                         check_done);
        if (launches) ++*launches;
        if (e != cudaSuccess) return e;
        zin = zo;
        din = dO;
    }
    return cudaSuccess;
}

// float64: the sweep with shared fluxes.
template <int SMAG>
static cudaError_t launch_pc3_shared(const Geo& G, int sweeps, const double* r, double* z, double* za, double* zb,
                                     double* da, double* db, const double* nu, double* part, Ctl* ctl, int check_done,
                                     cudaStream_t s, long long* launches) {
    using namespace d3;
    using T = double;
    dim3 grid((G.nx + CX - 1) / CX, (G.ny + CY - 1) / CY, ((G.nz + CZB - 1) / CZB) * 5);
    const T* zin = nullptr;
    const T* din = nullptr;
    T* zbuf[2] = {za, zb};
    T* dbuf[2] = {da, db};
    for (int k = 1; k <= sweeps - 1; ++k) {
        const bool first = k == 1, last = k == sweeps - 1;
        T* zo = last ? z : zbuf[k & 1];
        T* dO = dbuf[k & 1];
        auto* kern = first ? (last ? cheb3d_shared<T, SMAG, 1, 1> : cheb3d_shared<T, SMAG, 1, 0>)
                           : (last ? cheb3d_shared<T, SMAG, 0, 1> : cheb3d_shared<T, SMAG, 0, 0>);
        kern<<<grid, NTHREADS, 0, s>>>(G, k, r, zin, din, zo, dO, nu, part, ctl, check_done);
        if (launches) ++*launches;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        zin = zo;
        din = dO;
    }
    return cudaSuccess;
}

template <typename T, int SMAG>
static cudaError_t launch_pc3(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                              const T* nu, double* part, Ctl* ctl, int check_done, cudaStream_t s,
                              long long* launches) {
    if constexpr (sizeof(T) == sizeof(double)) {
        return launch_pc3_shared<SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
    } else {
        switch (row_vector<T>(G, r, z)) {
            case 4: return launch_pc3_w<T, 4, SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
            case 2: return launch_pc3_w<T, 2, SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
            default: return launch_pc3_w<T, 1, SMAG>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
        }
    }
}

// Acoustic Schur complement (3-D): rhs in da, iterates in xa / xb, directions
// in db and db + npt, the last sweep into the p plane of z, back-substitution.
template <typename T, int W>
static cudaError_t launch_schur3d_w(const Geo& G, int sweeps, const T* r, T* z, T* xa, T* xb, T* da, T* db,
                                    double* part, Ctl* ctl, int check_done, cudaStream_t s, long long* launches) {
    using namespace d3;
    constexpr int SMS = 152;
    const size_t np = (size_t)G.npt;
    // eight CTAs per SM of the two point-wise kernels (a thread holds a dozen vector loads)
    const int nb = (int)std::min<size_t>((np / W + NTHREADS - 1) / NTHREADS, 8 * SMS);
    T* rhs = da;
    cudaError_t e = launch_pdl(schur_rhs3d<T, W>, dim3(nb), dim3(NTHREADS), 0, s, G, r, rhs, ctl, check_done);
    if (e != cudaSuccess) return e;
    if (launches) ++*launches;
    HelmC<T> C;
    const double ax = G.helm_a * G.inv_dx * G.inv_dx, ay = G.helm_a * G.inv_dy * G.inv_dy,
                 az = G.helm_a * G.inv_dz * G.inv_dz;
    constexpr double lap[5] = {-65.0 / 72.0, 1.0 / 9.0, 4.0 / 9.0, -1.0 / 9.0, 1.0 / 144.0};
    C.c0 = T(-G.two_over_dt);
    C.lap0 = T(lap[0] * (ax + ay + az));
    for (int l = 0; l < 4; ++l) {
        const double c = sizeof(T) == sizeof(float) ? HELM_DIFF[l] : lap[l + 1];
        C.cx[l] = T(c * ax);
        C.cy[l] = T(c * ay);
        C.cz[l] = T(c * az);
    }
    constexpr int TX = HelmTile<T, W>::NXT * W, TY = HelmTile<T, W>::NYT;
    const int gx = (G.nx + TX - 1) / TX, gy = (G.ny + TY - 1) / TY;
    // planes per CTA: the longest march that still gives three CTAs to two SMs
    // (each march reads eight planes beyond its own), eight at least; per sweep at
    // 256 x 256 x 128 with 8 / 16 / 32 / 64 planes: 36.7 / 34.5 / 31.8 / 45.8 us
    int zb = 64;
    while (zb > 8 && (long long)gx * gy * ((G.nz + zb - 1) / zb) < 3 * SMS / 2) zb /= 2;
    const dim3 grid(gx, gy, (G.nz + zb - 1) / zb);
    T* xbuf[2] = {xa, xb};
    T* dbuf[2] = {db, db + np};
    const T* xin = nullptr;
    const T* din = nullptr;
    for (int k = 1; k <= sweeps - 1; ++k) {
        const bool first = k == 1, last = k == sweeps - 1;
        T* xo = last ? z + 4 * np : xbuf[k & 1];
        T* dO = dbuf[k & 1];
        auto* kern = first ? (last ? helm3d<T, W, 1, 1> : helm3d<T, W, 1, 0>)
                           : (last ? helm3d<T, W, 0, 1> : helm3d<T, W, 0, 0>);
        e = launch_pdl(kern, grid, dim3(NTHREADS), 0, s, G, C, k, zb, k & 1, (const T*)rhs, xin, din, xo, dO, ctl,
                       check_done);
        if (e != cudaSuccess) return e;
        if (launches) ++*launches;
        xin = xo;
        din = dO;
    }
    e = launch_pdl(schur_back3d<T, W>, dim3(nb), dim3(NTHREADS), 0, s, G, r, z, part, ctl, check_done);
    if (launches) ++*launches;
    return e;
}

template <typename T>
static cudaError_t launch_schur3d(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                                  double* part, Ctl* ctl, int check_done, cudaStream_t s, long long* launches) {
    const int w = row_vector<T>(G, r, z);
    if (w == 16 / sizeof(T))
        return launch_schur3d_w<T, 16 / sizeof(T)>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches);
    if constexpr (sizeof(T) == sizeof(float))
        if (w == 2) return launch_schur3d_w<T, 2>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches);
    return launch_schur3d_w<T, 1>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches);
}

template <typename T>
cudaError_t launch_precond3d(const Geo& G, int sweeps, const T* r, T* z, T* za, T* zb, T* da, T* db,
                             const T* nu, double* part, Ctl* ctl, int check_done, cudaStream_t s,
                             long long* launches) {
    if (G.pc_schur) return launch_schur3d<T>(G, sweeps, r, z, za, zb, da, db, part, ctl, check_done, s, launches);
    if (G.sgs == 2) return launch_pc3<T, 2>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
    return G.smag ? launch_pc3<T, 1>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches)
                  : launch_pc3<T, 0>(G, sweeps, r, z, za, zb, da, db, nu, part, ctl, check_done, s, launches);
}
template cudaError_t launch_precond3d<float>(const Geo&, int, const float*, float*, float*, float*, float*,
                                             float*, const float*, double*, Ctl*, int, cudaStream_t, long long*);
template cudaError_t launch_precond3d<double>(const Geo&, int, const double*, double*, double*, double*,
                                              double*, double*, const double*, double*, Ctl*, int, cudaStream_t,
                                              long long*);

cudaError_t launch_budgets3d(const Geo& G, const double* u, double dV, double dz, double lz, double* part,
                             Ctl* ctl, double* out, cudaStream_t s) {
    d3::budgets3d<<<d3::stream_blocks3(G.npt), NTHREADS, 0, s>>>(G, u, dV, dz, lz, part, ctl, out);
    return cudaGetLastError();
}

}  // namespace jfnk
