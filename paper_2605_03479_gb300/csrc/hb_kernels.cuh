// Kernels of one HB-UGKS pseudo-time iteration (Sec 2.2 - 2.4) and of the state/field conversions.
//
// One iteration, for every active case of a batch (each kernel covers all cases through a per-case block
// offset table):
//   K1 face_moments : per (face, level): velocity sums of the limited, upwinded interface reconstruction
//                     (kinetic average, heat-flux moments, tangential slopes, free-transport flux moments);
//                     per (cell, level): raw moments of h^k for the heat flux q^k
//   K2 face_params  : per (face, level): interface Maxwellian, tau, dG_f (Eq. dt_face), C1..C5 (Eq. C_coeffs),
//                     slopes a^L, a^R, a_t and A (compatibility), diffuse-wall density (Eq. rho_wall), the
//                     macro flux (Eq. macro_flux) and the parameters the micro update needs
//   K3 macro_update : per (cell, level): W^{k+1} (Eq. fv_W with the spectral source), the collision coefficients
//                     of Eq. fv_h, the equilibrium tables; per cell the next local step (Eqs. dt_hb, nu_conv) and
//                     the level-0 residual partials
//   K4 micro_update : per (cell, 32 velocities): interface micro fluxes (Eq. micro_flux), spectral source
//                     across levels and the semi-implicit collision update (Eq. fv_h)
//   K5 finish       : per case: residual (Eq. benchmark_residuals), convergence / divergence status
#pragma once
#include "hb_common.cuh"

namespace hb {

// ------------------------------------------------------------------------------ geometry helpers

struct FaceGeo {
    int axis;            // 0: normal along x, 1: normal along y
    int iL, jL, iR, jR;  // low-side and high-side cells
    bool hasL, hasR;
    int wall;            // wall id when one side is missing
};

template <typename T>
__device__ __forceinline__ FaceGeo face_geo(const CaseDev<T>& cd, int f)
{
    FaceGeo g;
    if (f < cd.nfx) {
        int j = f / (cd.nx + 1), i = f - j * (cd.nx + 1);
        g.axis = 0;
        g.iL = i - 1; g.jL = j; g.iR = i; g.jR = j;
        g.hasL = i > 0; g.hasR = i < cd.nx;
        g.wall = (i == 0) ? 3 : 1;
    } else {
        int ff = f - cd.nfx;
        int j = ff / cd.nx, i = ff - j * cd.nx;
        g.axis = 1;
        g.iL = i; g.jL = j - 1; g.iR = i; g.jR = j;
        g.hasL = j > 0; g.hasR = j < cd.ny;
        g.wall = (j == 0) ? 0 : 2;
    }
    return g;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// heat flux from the 13 raw moments (h: 1,u,v,uu,uv,vv,uuu,uuv,uvv,vvv; b: 1,u,v) about (U, V):
// q = 1/2 sum w c (|c|^2 h + b)  (Eq. heatflux, reduced)
__device__ __forceinline__ void heat_flux_raw(const double* A, double U, double V, double& qx, double& qy)
{
    double cx3 = A[6] - 3.0 * U * A[3] + 3.0 * U * U * A[1] - U * U * U * A[0];
    double cxcy2 = A[8] - 2.0 * V * A[4] + V * V * A[1] - U * A[5] + 2.0 * U * V * A[2] - U * V * V * A[0];
    double cy3 = A[9] - 3.0 * V * A[5] + 3.0 * V * V * A[2] - V * V * V * A[0];
    double cycx2 = A[7] - 2.0 * U * A[4] + U * U * A[2] - V * A[3] + 2.0 * U * V * A[1] - V * U * U * A[0];
    qx = 0.5 * (cx3 + cxcy2 + A[11] - U * A[10]);
    qy = 0.5 * (cy3 + cycx2 + A[12] - V * A[10]);
}

// ------------------------------------------------------------------------------ K2 face parameters

// A CTA takes K2_ITEMS (face, level) items with one lane each in every one of its four warps, which divide the work:
//   A  interface state from the velocity sums (each warp for itself), then warp 0 the heat flux and Shakhov factor,
//      1 and 2 the slopes a^L and a^R, 3 the slope a_t;
//   B  all warps: the expm1 table of the interface Maxwellian (lanes over the nodes, one item after another) and its
//      27 sums per axis (lanes over the items, a warp per power);
//   C  warp 0 the compatibility condition (A), 1 the Shakhov moments, the relaxation time and the weights C1..C5, 2 and 3
//      the moments of the left and right slopes;
//   D  warp 0 the macro flux and the wall density, 1 and 2 the micro-flux parameters of the two upwind sides, 3 the rest.
// On small meshes the time is the chain of one thread, in large ones FP64 instructions and latency at few warps.
// Against one thread per item doing all of it (219 registers, nine FP64 instructions per division, polynomials in (u, v)
// whose axis was known at run time only): 57 -> 27 us (8x8, N_T 3), 0.210 -> 0.136 ms (64x64, 48x48, N_T 7),
// 5.49 -> 3.80 ms (48 uneven cavities), 1.12 -> 0.68 ms (128x128, 64x64, N_T 11); FP64 0.190 -> 0.077 ms (32x32, 24x24)
// and 2.97 -> 1.98 ms (twelve 64x64, 32x32).  32 items fill a warp; 4 warps balance the parts of A and C.
constexpr int K2_ITEMS = 32, K2_WARPS = 4, K2_NODES = 32;

// All polynomials are kept in the face's own velocity components, n along its normal and t along the other axis, in
// the order 1, n, t, n^2, nt, t^2, n^3, n^2 t, n t^2, t^3, so that a product by u_n is a shift of the 1-D sums by one
// power and every pattern of zero coefficients is known when compiling.

// place of coefficient k (0..9 a cubic, 10..12 a linear form) after exchanging the two components
__device__ __forceinline__ constexpr int nt_order(int k)
{
    constexpr int o[13] = {0, 2, 1, 5, 4, 3, 9, 8, 7, 6, 10, 12, 11};
    return o[k];
}

// P_h(a) = a0 + a1 u + a2 v + a3/2 (u^2 + v^2 + 1/(2 lam)) of a slope and P_b(a) = P_h(a) + a3/(2 lam): constant term,
// the addition for b, then the coefficients of n, t and n^2 (= that of t^2)
template <typename T>
__device__ __forceinline__ void slope_poly(const double w[4], double U, double V, double lam, double i2l, int ax,
                                           T (*o)[K2_ITEMS], int lane)
{
    double a[4];
    micro_slope(w, U, V, lam, i2l, a);
    o[0][lane] = T(a[0] + 0.5 * a[3] * i2l);
    o[1][lane] = T(a[3] * i2l);
    o[2][lane] = T(ax == 0 ? a[1] : a[2]);
    o[3][lane] = T(ax == 0 ? a[2] : a[1]);
    o[4][lane] = T(0.5 * a[3]);
}

// cubic Q = u_n P_h(a_side) + u_t P_h(a_t); dn, dt: the additions to its coefficients of n and t for b
template <typename T>
__device__ __forceinline__ void side_poly(const T (*ps)[K2_ITEMS], const T (*pt)[K2_ITEMS], int lane, T (&c)[10], T& dn, T& dt)
{
    c[0] = T(0);
    c[1] = ps[0][lane];
    c[2] = pt[0][lane];
    c[3] = ps[2][lane];
    c[4] = ps[3][lane] + pt[2][lane];
    c[5] = pt[3][lane];
    c[6] = c[8] = ps[4][lane];
    c[7] = c[9] = pt[4][lane];
    dn = ps[1][lane];
    dt = pt[1][lane];
}

// moments sum w psi [Q H ; R B] of the cubic c (CUB false: without nt and the cubic terms) times u_n^S, R = c + d0 +
// dn n + dt t, with the 1-D sums x along the normal and y along t of the selected grid part, H = pref e^{..}, B = H i2l:
// (sum Q H, sum u_n Q H, sum u_t Q H, 1/2 sum (|u|^2 Q H + R B)).  The inner sums over powers of n serve every moment.
template <int S, bool CUB, typename P>
__device__ __forceinline__ void mom4(const P (&c)[10], P d0, P dn, P dt, const P (&x)[9], const P (&y)[9], P pref, P i2l,
                                     P (&out)[4])
{
    P m[3][3];                                               // [power added to n][power added to t]
#pragma unroll
    for (int z = 0; z < 3; ++z) {
        const P *v = x + S + z;
        P t[4];
        t[0] = c[0] * v[0] + c[1] * v[1] + c[3] * v[2];
        t[1] = c[2] * v[0];
        t[2] = c[5] * v[0];
        t[3] = P(0);
        if (CUB) {
            t[0] += c[6] * v[3];
            t[1] += c[4] * v[1] + c[7] * v[2];
            t[2] += c[8] * v[1];
            t[3] = c[9] * v[0];
        }
#pragma unroll
        for (int k = 0; k + z < 3; ++k) {
            m[z][k] = t[0] * y[k] + t[1] * y[k + 1] + t[2] * y[k + 2];
            if (CUB) m[z][k] += t[3] * y[k + 3];
        }
    }
    const P ob = m[0][0] + (d0 * x[S] + dn * x[S + 1]) * y[0] + dt * x[S] * y[1];
    out[0] = pref * m[0][0];
    out[1] = pref * m[1][0];
    out[2] = pref * m[0][1];
    out[3] = P(0.5) * pref * (m[2][0] + m[0][2] + i2l * ob);
}

template <typename T>
__global__ void __launch_bounds__(K2_ITEMS * K2_WARPS) k2_face_params(Batch<T> B)
{
    __shared__ CaseDev<T> cd;
    int lb;
    copy_case(B.find(blockIdx.x, lb), cd);
    // uniform over the CTA: neither word changes while this kernel runs
    if (!cd.st->active || *(volatile int*)cd.err) return;
    __shared__ T pL[5][K2_ITEMS], pR[5][K2_ITEMS], pt[5][K2_ITEMS], pA[5][K2_ITEMS], shk_[13][K2_ITEMS], Cw[5][K2_ITEMS];
    __shared__ T tco[5][K2_ITEMS];                           // exponent coefficients of the table
    __shared__ T S[2][3][9][K2_ITEMS];                       // table sums per axis, node class (> 0, < 0, 0) and power
    __shared__ T se[K2_NODES][K2_ITEMS + 1];
    __shared__ T F1s[4][K2_ITEMS], F2L[4][K2_ITEMS], F2R[4][K2_ITEMS];
    __shared__ double dF1[4][K2_ITEMS], sdG[K2_ITEMS], st[10][K2_ITEMS];
    const int nt = cd.nt, nu = cd.nu, nv = cd.nv, nuv = nu + nv, nitems = cd.nf * nt;
    const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
    const int base = lb * K2_ITEMS;
    const bool valid = base + lane < nitems;
    const int item = valid ? base + lane : nitems - 1;       // lanes past the end repeat the last item and store nothing
    const int f = item / nt, n = item - f * nt;
    const FaceGeo g = face_geo(cd, f);
    const int ax = g.axis;
    const double* W = cd.W[cd.st->parity];
    const bool wall = !(g.hasL && g.hasR);
    const double nin = wall ? (g.hasL ? -1.0 : 1.0) : 0.0;
    const int inc_row = nin > 0 ? 2 : 1;                     // incident: u_n nin < 0
    const int refset = !wall ? 0 : ax == 0 ? (nin > 0 ? 2 : 1) : (nin > 0 ? 4 : 3);
    const int wsl = wall_slot(cd, n);
    const double* wc = wall ? cd.wconst + ((size_t)g.wall * cd.nslot + wsl) * WCN : nullptr;
    const int cL = g.jL * cd.nx + g.iL, cR = g.jR * cd.nx + g.iR;
    // Velocity sums of the upwinded reconstruction from the half-face sums of the face's cells: at an interior face the
    // low-side cell's u_n > 0 class plus the high-side cell's u_n < 0 class; at a wall the interior cell's class moving
    // into the wall, with the tangential-slope sums (13..17) over both classes.
    const int sp = ax == 0 ? 0 : 2;                          // half-face slot of the u_n > 0 class, sp + 1: u_n < 0
    const double* hL = g.hasL ? cd.hmom + ((size_t)cL * nt + n) * 4 * NM + sp * NM : nullptr;
    const double* hR = g.hasR ? cd.hmom + ((size_t)cR * nt + n) * 4 * NM + (sp + 1) * NM : nullptr;
    const double* ha = g.hasL ? hL : hR;
    const double* hb = wall ? (g.hasL ? hL + NM : hR - NM) : hR;   // at a wall: the other class
    auto msum = [&](int k) { return ha[k] + (!wall || (k >= 13 && k < 18) ? hb[k] : 0.0); };

    // ---- A: interface Maxwellian from the kinetic average; diffuse wall: its mixed with the free-transport estimate
    // of the re-emitted distribution (Eq. rho_wall)
    auto amix = [&](int k, double rhow0) {
        const double a = msum(k) + cd.refmom[refset * 13 + k];
        return wall ? fma(rhow0, wc[k], a) : a;
    };
    if (role == 0) {
        double rhow0 = 0.0;
        if (wall) rhow0 = -nin * (msum(ax == 0 ? 1 : 2) + cd.refmom[refset * 13 + (ax == 0 ? 1 : 2)]) * rcp64(wc[13]);
        const double w[4] = {amix(0, rhow0), amix(1, rhow0), amix(2, rhow0),
                             0.5 * (amix(3, rhow0) + amix(5, rhow0) + amix(10, rhow0))};
        double r, a, b, l;
        prim(w, r, a, b, l);
#pragma unroll
        for (int k = 0; k < 4; ++k) st[k][lane] = w[k];
        st[4][lane] = a;
        st[5][lane] = b;
        st[6][lane] = l;
        st[7][lane] = rcp64(r);
        st[8][lane] = 0.5 * rcp64(l);
        st[9][lane] = rhow0;
    }
    __syncthreads();
    const double rho0 = st[0][lane], U0 = st[4][lane], V0 = st[5][lane], lamf = st[6][lane], ir = st[7][lane],
                 i2ld = st[8][lane], il0 = rcp64(cd.lam0);
    if (role == 0) {
        double Am[13], q0x, q0y, sh[13];
#pragma unroll
        for (int k = 0; k < 13; ++k) Am[k] = amix(k, st[9][lane]);
        heat_flux_raw(Am, U0, V0, q0x, q0y);
        // Shakhov factor s (c.q)(2 lam |c|^2 - 4) and the b-part addition 2 s (c.q)
        shakhov_poly((1.0 - cd.pr) * 0.8 * lamf * lamf * ir, q0x, q0y, U0, V0, lamf, sh);
#pragma unroll
        for (int k = 0; k < 13; ++k) shk_[ax == 0 ? k : nt_order(k)][lane] = T(sh[k]);
    } else if (role < 3) {
        // equilibrium slopes a^L, a^R (normal); a wall face has the interior side's in both
        const bool low = role == 1 ? g.hasL : !g.hasR;
        const double* Wc = W + ((size_t)n * cd.nc + (low ? cL : cR)) * 4;
        const double d = ax == 0 ? cd.hx[low ? g.iL : g.iR] : cd.hy[low ? g.jL : g.jR];
        const double s = (low ? ir : -ir) * rcp64(d);
        double w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = (st[k][lane] - Wc[k]) * s;
        slope_poly<T>(w, U0, V0, lamf, i2ld, ax, role == 1 ? pL : pR, lane);
    } else {
        const double w[4] = {msum(13) * ir, msum(14) * ir, msum(15) * ir, 0.5 * (msum(16) + msum(17)) * ir};
        slope_poly<T>(w, U0, V0, lamf, i2ld, ax, pt, lane);
        tco[0][lane] = T(cd.lam0 - lamf);
        tco[1][lane] = T(2.0 * lamf * U0);
        tco[2][lane] = T(lamf * U0 * U0);
        tco[3][lane] = T(2.0 * lamf * V0);
        tco[4][lane] = T(lamf * V0 * V0);
    }
    __syncthreads();

    // ---- B: separable table of the interface Maxwellian and its 1-D sums.  The nodes are taken in the order of their
    // class (positive, negative, zero), so that a node adds to one sum only.
    for (int axis = 0; axis < 2; ++axis) {
        const int nn = axis == 0 ? nu : nv, e0 = cd.ncls[axis][0], e1 = cd.ncls[axis][1];
        const T* __restrict__ xn = axis == 0 ? cd.su1 : cd.sv1;
        const T* __restrict__ wq = axis == 0 ? cd.wxr : cd.wyr;
        const int* __restrict__ ord = axis == 0 ? cd.ou1 : cd.ov1;
        T* const tab = cd.ftab + (axis == 0 ? 0 : nu);
        T acc[3][3];                                         // powers role, role + 4, role + 8; node classes
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) acc[a][b] = T(0);
        for (int k0 = 0; k0 < nn; k0 += K2_NODES) {
            const int kn = min(K2_NODES, nn - k0);
            if (lane < kn) {
                const T x = __ldg(xn + k0 + lane);
                const int o = __ldg(ord + k0 + lane);
#pragma unroll 4
                for (int i = role; i < K2_ITEMS; i += K2_WARPS) {
                    const T e = t_expm1<T>(tco[0][i] * x * x + tco[1 + 2 * axis][i] * x - tco[2 + 2 * axis][i]);
                    se[lane][i] = e;
                    if (base + i < nitems) tab[(size_t)(base + i) * nuv + o] = e;
                }
            }
            __syncthreads();
            const int b0 = min(max(e0 - k0, 0), kn), b1 = min(max(e1 - k0, 0), kn);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const int q = role + K2_WARPS * a;
                if (q >= 9) break;
                const T* __restrict__ wk = wq + (size_t)q * nn + k0;
#pragma unroll 4
                for (int k = 0; k < b0; ++k) acc[a][0] += __ldg(wk + k) * se[k][lane];
#pragma unroll 4
                for (int k = b0; k < b1; ++k) acc[a][1] += __ldg(wk + k) * se[k][lane];
                for (int k = b1; k < kn; ++k) acc[a][2] += __ldg(wk + k) * se[k][lane];
            }
            __syncthreads();
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int q = role + K2_WARPS * a;
            if (q >= 9) break;
#pragma unroll
            for (int b = 0; b < 3; ++b) S[axis][b][q][lane] = acc[a][b];
        }
    }
    __syncthreads();

    // ---- C: velocity moments of the Maxwellian's polynomials
    const T pref = T(rho0 * lamf * M_1_PI), i2l = T(i2ld);
    // full 1-D sums of the interface Maxwellian over node subset r (0 all, 1 positive, 2 negative, 3 zero); dif: the
    // table part alone
    auto row = [&](int axis, int r, T (&o)[9]) {
        const T* ref = (axis == 0 ? cd.xr0t : cd.yr0t) + r * 9;
#pragma unroll
        for (int q = 0; q < 9; ++q)
            o[q] = ref[q] + (r == 0 ? S[axis][0][q][lane] + S[axis][1][q][lane] + S[axis][2][q][lane]
                                    : S[axis][r - 1][q][lane]);
    };
    auto rows = [&](int r, T (&x)[9], T (&y)[9]) { row(ax, r, x); row(1 - ax, 0, y); };   // subset r along the normal
    // moments back from (n, t) to (u, v) order
    auto put = [&](T (*o)[K2_ITEMS], const T (&m)[4]) {
        o[0][lane] = m[0];
        o[1][lane] = ax == 0 ? m[1] : m[2];
        o[2][lane] = ax == 0 ? m[2] : m[1];
        o[3][lane] = m[3];
    };
    const int half = wall ? inc_row : 0;                     // velocities carried by the integral solution
    T x[9], y[9];
    if (role == 0) {
        // compatibility: moments of (A.psi) g0 = - moments of (u_n a_n + u_t a_t) g0
        T c[10], d[10], dn, dt, en, M[4], tmp[4];
        side_poly(pL, pt, lane, c, dn, dt);
        rows(wall ? 0 : 1, x, y);
        mom4<0, true>(c, T(0), dn, dt, x, y, pref, i2l, M);
        if (!wall) {
            side_poly(pR, pt, lane, d, en, dt);
            rows(2, x, y);
            mom4<0, true>(d, T(0), en, dt, x, y, pref, i2l, tmp);
#pragma unroll
            for (int k = 0; k < 4; ++k) M[k] += tmp[k];
            if (cd.zeros) {
                // nodes with u_n = 0 take the average of both sides
#pragma unroll
                for (int k = 0; k < 10; ++k) c[k] = T(0.5) * (c[k] + d[k]);
                rows(3, x, y);
                mom4<0, true>(c, T(0), T(0.5) * (dn + en), dt, x, y, pref, i2l, tmp);
#pragma unroll
                for (int k = 0; k < 4; ++k) M[k] += tmp[k];
            }
        }
        const double w[4] = {-(double)M[0] * ir, -(double)(ax == 0 ? M[1] : M[2]) * ir, -(double)(ax == 0 ? M[2] : M[1]) * ir,
                             -(double)M[3] * ir};
        slope_poly<T>(w, U0, V0, lamf, i2ld, ax, pA, lane);
    } else if (role == 1) {
        // C1 term: moments of u_n s (c.q)(2 lam |c|^2 - 4)
        T c[10], o[4];
#pragma unroll
        for (int k = 0; k < 10; ++k) c[k] = shk_[k][lane];
        rows(half, x, y);
        mom4<1, true>(c, shk_[10][lane], shk_[11][lane], shk_[12][lane], x, y, pref, i2l, o);
        put(F1s, o);
        // face step (Eq. dt_face) and time-integration weights (Eq. C_coeffs), here beside warp 0's longer part
        double dGf;
        if (!g.hasL) dGf = cd.dG[cR];
        else if (!g.hasR) dGf = cd.dG[cL];
        else if (cd.face_step == 1) dGf = 2.0 * cd.dG[cL] * cd.dG[cR] * rcp64(cd.dG[cL] + cd.dG[cR]);
        else dGf = fmin(cd.dG[cL], cd.dG[cR]);
        sdG[lane] = dGf;
        T Ct[5];
        ugks_coeffs<T>(T(dGf), T(relax_time(cd.mu0, cd.w_vss, cd.lam0, il0, ir, lamf, i2ld)), Ct);
#pragma unroll
        for (int k = 0; k < 5; ++k) Cw[k][lane] = Ct[k];
    } else {
        // C2 term: u_n (u_n P(a_bar) + u_t P(a_t)), a_bar = a^L for u_n > 0 (warp 2), a^R for u_n < 0 (warp 3; at a wall
        // the incident velocities' one side is warp 2's)
        T o[4] = {T(0), T(0), T(0), T(0)};
        if (role == 2 || !wall) {
            T c[10], dn, dt;
            side_poly(role == 2 ? pL : pR, pt, lane, c, dn, dt);
            rows(wall ? inc_row : role - 1, x, y);
            mom4<1, true>(c, T(0), dn, dt, x, y, pref, i2l, o);
        }
        put(role == 2 ? F2L : F2R, o);
        if (role == 3) {
            // C1 term, Maxwellian part: moments of u_n psi (H0 - H_ref, B0 - B_ref), in FP64 from the reference sums
            const double rr = rho0 * lamf * il0, di2l = i2ld - 0.5 * il0, fac = cd.lam0 * M_1_PI;
            const int rx = ax == 0 ? half : 0, ry = ax == 0 ? 0 : half;
            const double* X0 = cd.xr0 + rx * 9;
            const double* Y0 = cd.yr0 + ry * 9;
            auto dif = [&](int axis, int r, int q) -> double {
                return r == 0 ? (double)(S[axis][0][q][lane] + S[axis][1][q][lane] + S[axis][2][q][lane])
                              : (double)S[axis][r - 1][q][lane];
            };
            // (lam0/pi) [(r - 1) X0 Y0 + r (dX Y0 + X0 dY + dX dY)] and (lam0/pi) X0 Y0
            auto Sd = [&](int p, int q) {
                const double x0 = X0[p], y0 = Y0[q], dx = dif(0, rx, p), dy = dif(1, ry, q);
                return fac * ((rr - 1.0) * x0 * y0 + rr * (dx * y0 + x0 * dy + dx * dy));
            };
            double o4[4];
            if (ax == 0) {
                const double s10 = Sd(1, 0);
                o4[0] = s10; o4[1] = Sd(2, 0); o4[2] = Sd(1, 1);
                o4[3] = 0.5 * (Sd(3, 0) + Sd(1, 2)) + 0.5 * (i2ld * s10 + di2l * fac * X0[1] * Y0[0]);
            } else {
                const double s01 = Sd(0, 1);
                o4[0] = s01; o4[1] = Sd(1, 1); o4[2] = Sd(0, 2);
                o4[3] = 0.5 * (Sd(2, 1) + Sd(0, 3)) + 0.5 * (i2ld * s01 + di2l * fac * X0[0] * Y0[1]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) dF1[k][lane] = o4[k];
        }
    }
    __syncthreads();

    // ---- D: macro flux deviation (Eq. macro_flux minus the flux of H_ref, which cancels in every cell balance) and the
    // parameters of the micro flux (delta form, divided by dG_f; level-major: a tile's faces of one level are rows)
    if (!valid) return;
    T* pp = cd.fpar + ((size_t)n * cd.nf + f) * NP;
    const double dGf = sdG[lane], idG = rcp64(dGf);
    const double rr = rho0 * lamf * il0;
    if (role == 0) {
        // C3 term: u_n P(A)
        const T c[10] = {pA[0][lane], pA[2][lane], pA[3][lane], pA[4][lane], T(0), pA[4][lane], T(0), T(0), T(0), T(0)};
        T o[4];
        rows(half, x, y);
        mom4<1, false>(c, pA[1][lane], T(0), T(0), x, y, pref, i2l, o);
        const T F3[4] = {o[0], ax == 0 ? o[1] : o[2], ax == 0 ? o[2] : o[1], o[3]};
        // C4 term: u_n psi (h_0 - H_ref) (reconstruction; incident velocities only at a wall); C5 term
        double F4[4], F5[4], I[4], F[4];
        if (ax == 0) { F4[0] = msum(1); F4[1] = msum(3); F4[2] = msum(4); F4[3] = 0.5 * (msum(6) + msum(8) + msum(11)); }
        else { F4[0] = msum(2); F4[1] = msum(4); F4[2] = msum(5); F4[3] = 0.5 * (msum(7) + msum(9) + msum(12)); }
        F5[0] = msum(18); F5[1] = msum(19); F5[2] = msum(20); F5[3] = 0.5 * (msum(21) + msum(22));
        double C[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) C[k] = (double)Cw[k][lane];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            I[k] = C[0] * (dF1[k][lane] + (double)F1s[k][lane]) + C[1] * (double)(F2L[k][lane] + F2R[k][lane]) +
                   C[2] * (double)F3[k] + C[3] * F4[k] + C[4] * F5[k];
        double rhow = 0.0;
        if (!wall) {
#pragma unroll
            for (int k = 0; k < 4; ++k) F[k] = I[k] * idG;
        } else {
            // impermeability (Eq. rho_wall) with the time-integrated incident mass flux; reflected part rho_w H_w
            const double* oc = cd.oconst + g.wall * 8;       // [0..3] incident flux of H_ref, [4..7] reflected
            rhow = -nin * (oc[0] + I[0] * idG) * rcp64(wc[13]);
#pragma unroll
            for (int k = 0; k < 4; ++k) F[k] = I[k] * idG + rhow * wc[14 + k] - oc[4 + k];
        }
        double* fo = cd.fflux + (size_t)item * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) fo[k] = F[k];
        if (wall) {
            const double* ws = cd.wall + ((size_t)g.wall * cd.nslot + wsl) * 3;
            const double lamw = cd.lam0 * rcp64(ws[2]), iw = 0.5 * rcp64(lamw);
            const double rw = rhow * lamw * il0;
            pp[F_WRM1] = T(rw - 1.0);
            pp[F_WR] = T(rw);
            pp[F_WI2L] = T(iw);
            pp[F_WDI2L] = T(iw - 0.5 * il0);
        } else {
            pp[F_WRM1] = pp[F_WR] = pp[F_WI2L] = pp[F_WDI2L] = T(0);
        }
    } else if (role < 3) {
        // for the upwind side: the cubic Q = C1' s(c.q)(2 lam |c|^2 - 4) + C2' (u_n P_h(a_side) + u_t P_h(a_t)) +
        // C3' P_h(A) and the linear b-part difference C1' 2 s (c.q) + C2' (u_n a_side,3 + u_t a_t,3)/(2 lam) +
        // C3' A_3/(2 lam)
        T c[10], dn, dt;
        side_poly(role == 1 ? pL : pR, pt, lane, c, dn, dt);
        const T C1p = T((double)Cw[0][lane] * idG), C2p = T((double)Cw[1][lane] * idG), C3p = T((double)Cw[2][lane] * idG);
        const T pa[10] = {pA[0][lane], pA[2][lane], pA[3][lane], pA[4][lane], T(0), pA[4][lane], T(0), T(0), T(0), T(0)};
        T* q = pp + (role == 1 ? F_QL : F_QR);
#pragma unroll
        for (int k = 0; k < 10; ++k) q[ax == 0 ? k : nt_order(k)] = C1p * shk_[k][lane] + C2p * c[k] + C3p * pa[k];
        T* l = pp + (role == 1 ? F_LBL : F_LBR);
        l[0] = C1p * shk_[10][lane] + C3p * pA[1][lane];
        l[ax == 0 ? 1 : 2] = C1p * shk_[11][lane] + C2p * dn;
        l[ax == 0 ? 2 : 1] = C1p * shk_[12][lane] + C2p * dt;
    } else {
        pp[F_RM1] = T(rr - 1.0);
        pp[F_R] = T(rr);
        pp[F_I2L] = T(i2ld);
        pp[F_DI2L] = T(i2ld - 0.5 * il0);
        pp[F_C1] = T((double)Cw[0][lane] * idG);
        pp[F_C4] = T((double)Cw[3][lane] * idG);
        pp[F_C5] = T((double)Cw[4][lane] * idG);
        pp[F_C1D] = T((double)Cw[0][lane] * idG * (i2ld - 0.5 * il0));
    }
}

// ------------------------------------------------------------------------------ local pseudo-time step

// nu_conv of one (cell, level) with the cell's 1/dx, 1/dy (Eq. nu_conv); k_steps and k3_macro form the same bits, so
// a state that is set from a checkpoint continues exactly
template <typename T>
__device__ __forceinline__ double nu_conv(const CaseDev<T>& cd, double U, double V, double lam, double rdx, double rdy)
{
    const double cs = sqrt(0.5 * cd.gam * rcp64(lam));
    return fma(fmax(fabs(cd.umax), fabs(U)) + cs, rdx, (fmax(fabs(cd.vmax), fabs(V)) + cs) * rdy);
}

// Eqs. dt_hb, nu_conv: dG_i = CFL / (max_n nu_conv,i,n + omega N_H)
template <typename T>
__device__ __forceinline__ double local_step(const CaseDev<T>& cd, double numax)
{
    return cd.dt_fixed > 0.0 ? cd.dt_fixed : cd.cfl / fma(cd.omega, (double)cd.nh, numax);
}

template <typename T>
__global__ void k_steps(Batch<T> B)
{
    int lb;
    const CaseDev<T>& cd = B.find(blockIdx.x, lb);
    int c = lb * blockDim.x + threadIdx.x;
    if (c >= cd.nc) return;
    const double rdx = rcp64(2.0 * cd.hx[c % cd.nx]), rdy = rcp64(2.0 * cd.hy[c / cd.nx]);
    double numax = 0.0;
    for (int n = 0; n < cd.nt; ++n) {
        double rho, U, V, lam;
        prim(cd.W[cd.st->parity] + ((size_t)n * cd.nc + c) * 4, rho, U, V, lam);
        numax = fmax(numax, nu_conv(cd, U, V, lam, rdx, rdy));
    }
    cd.dG[c] = local_step(cd, numax);
}

// ------------------------------------------------------------------------------ K3 macro update

// A CTA takes K3_CELLS cells on all their levels, in two halves of its warps: threads 0.. form W^k's primitive
// variables, heat flux and relaxation time of one (cell, level) each, threads half.. the new W and those of W^{k+1};
// they exchange what the other side needs through shared memory and each writes its equilibrium's parameters.  All
// warps then write the expm1 tables of the CTA's equilibria.  Bound by FP64 instructions, and on small meshes by
// the length of one thread's chain of them: the previous layout (a thread per cell running over its levels, then a
// kernel of 128 cell-levels per CTA for the tables) left most of the chip idle.  Measured before -> now, both parts:
// 115 -> 18 us (8x8 cells, N_T 3), 262 -> 51 us (64x64, N_T 7), 482 -> 215 us (128x128, N_T 11), 754 -> 45 us (32x32,
// N_T 11, spectral source at the new iterate), 236 -> 35 us (32x32, N_T 3, FP64 tables).  8 cells per CTA give a
// 32x32 mesh 128 CTAs and still fill three quarters of the lanes at N_T = 3.
constexpr int K3_MAXTHREADS = 2 * ((MAXNT * K3_CELLS + 31) / 32) * 32;
// warps of one half for nt levels, and threads of the launch for the largest nt of its cases (at least four warps,
// one per scheduler, for the tables)
__host__ __device__ constexpr int k3_half(int nt) { return (nt * K3_CELLS + 31) / 32 * 32; }
__host__ __device__ constexpr int k3_threads(int nt) { return 2 * k3_half(nt) < 128 ? 128 : 2 * k3_half(nt); }

template <typename T>
__global__ void __launch_bounds__(K3_MAXTHREADS) k3_macro(Batch<T> B)
{
    __shared__ CaseDev<T> cd;
    int lb;
    copy_case(B.find(blockIdx.x, lb), cd);
    // uniform over the CTA: neither word changes while this kernel runs
    if (!cd.st->active || *(volatile int*)cd.err) return;
    __shared__ T coef[K3_CELLS * MAXNT * 2][5];            // exponent coefficients of the tables, row (cell, level, e)
    __shared__ double sq[MAXNT * K3_CELLS][2], stau[MAXNT * K3_CELLS], snu[MAXNT * K3_CELLS];
    __shared__ double srhs[MAXNT * K3_CELLS][4], sinv[MAXNT * K3_CELLS];
    __shared__ double sM[MAXNT][MAXNT][K3_CELLS];
    const int nt = cd.nt, nc = cd.nc, half = k3_half(nt);
    const int role = (int)threadIdx.x / half;              // 0: W^k, 1: W^{k+1}, 2: helps with the tables only
    const int r = (int)threadIdx.x - role * half;
    const int n = r / K3_CELLS, ci = r % K3_CELLS, c = lb * K3_CELLS + ci;
    const bool work = role < 2 && n < nt && c < nc;
    const int p = cd.st->parity;
    const bool implicit = cd.spectral_implicit != 0;
    const double* W = cd.W[p];
    double* Wn = cd.W[p ^ 1];
    const double il0 = rcp64(cd.lam0);
    const int i = work ? c % cd.nx : 0, j = work ? c / cd.nx : 0;
    const double dx = 2.0 * cd.hx[i], dy = 2.0 * cd.hy[j], idx_ = rcp64(dx), idy = rcp64(dy);
    const double dG = work ? cd.dG[c] : 0.0;
    double rho = 1.0, U = 0.0, V = 0.0, lam = 1.0, tau = 1.0, qx = 0.0, qy = 0.0;
    double Wc[4], wn[4];                                   // this thread's W^k, W^{k+1}
    if (work) {
#pragma unroll
        for (int k = 0; k < 4; ++k) Wc[k] = W[((size_t)n * nc + c) * 4 + k];
        if (role == 0) {
            double A[13];
            const double* cm = cd.cmom + ((size_t)c * nt + n) * NCM;
#pragma unroll
            for (int k = 0; k < 13; ++k) A[k] = cm[k] + cd.refmom[k];
            prim(Wc, rho, U, V, lam);
            heat_flux_raw(A, U, V, qx, qy);
            tau = relax_time(cd.mu0, cd.w_vss, cd.lam0, il0, rcp64(rho), lam, 0.5 * rcp64(lam));
            sq[r][0] = qx;
            sq[r][1] = qy;
        } else {
            const int fL = j * (cd.nx + 1) + i, fB = cd.nfx + j * cd.nx + i;
            const double* FL = cd.fflux + ((size_t)fL * nt + n) * 4;
            const double* FR = FL + (size_t)nt * 4;
            const double* FB = cd.fflux + ((size_t)fB * nt + n) * 4;
            const double* FT = FB + (size_t)cd.nx * nt * 4;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double div = (FR[k] - FL[k]) * idx_ + (FT[k] - FB[k]) * idy;
                if (implicit) {
                    srhs[r][k] = Wc[k] - dG * div;
                } else {
                    double ew = 0.0;
                    for (int d = 1; d <= cd.nh; ++d) {
                        int nm = n - d; nm += nm < 0 ? nt : 0;
                        int np = n + d; np -= np >= nt ? nt : 0;
                        ew += cd.e[d] * (W[((size_t)nm * nc + c) * 4 + k] - W[((size_t)np * nc + c) * 4 + k]);
                    }
                    wn[k] = Wc[k] - dG * (div + cd.omega * ew);
                }
            }
            if (implicit) {
                // entry d = n of the inverse of the circulant I + a E, a = dG omega, whose eigenvalues are 1 + i a k:
                // (1/N_T) [1 + 2 sum_k (cos(2 pi k d / N_T) + a k sin(2 pi k d / N_T)) / (1 + a^2 k^2)]
                const double a = dG * cd.omega;
                double s = 0.0;
                for (int k = 1, m = n; k <= cd.nh; ++k, m += n) {
                    if (m >= nt) m -= nt;
                    const double ak = a * k;
                    s += (cd.ct[m] + ak * cd.snt[m]) * rcp64(1.0 + ak * ak);
                }
                sinv[r] = (1.0 + 2.0 * s) / nt;
            }
        }
    }
    if (implicit) {
        // spectral source at the new iterate: (I + dG omega E) W^{k+1} = W^k - dG div F for every variable
        __syncthreads();
        if (work && role == 1) {
#pragma unroll
            for (int k = 0; k < 4; ++k) wn[k] = 0.0;
            for (int m = 0; m < nt; ++m) {
                int d = n - m; d += d < 0 ? nt : 0;
                const double g = sinv[d * K3_CELLS + ci];
#pragma unroll
                for (int k = 0; k < 4; ++k) wn[k] += g * srhs[m * K3_CELLS + ci][k];
            }
        }
    }
    if (work && role == 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k) Wn[((size_t)n * nc + c) * 4 + k] = wn[k];
        prim(wn, rho, U, V, lam);
        tau = relax_time(cd.mu0, cd.w_vss, cd.lam0, il0, rcp64(rho), lam, 0.5 * rcp64(lam));
        stau[r] = tau;
        snu[r] = nu_conv(cd, U, V, lam, idx_, idy);        // for the next local step
    }
    if (role == 1 && r < 32) {
        // level-0 residual partials of the CTA's cells (lanes 0..7 of the half's first warp)
        double r2[4] = {0, 0, 0, 0};
        if (work && n == 0)
#pragma unroll
            for (int k = 0; k < 4; ++k) { const double d = wn[k] - Wc[k]; r2[k] = d * d; }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int o = K3_CELLS / 2; o > 0; o >>= 1) r2[k] += __shfl_xor_sync(0xffffffffu, r2[k], o);
        }
        if (r == 0)
#pragma unroll
            for (int k = 0; k < 4; ++k) cd.rpart[(size_t)lb * 4 + k] = r2[k];
    }
    __syncthreads();
    if (work) {
        T* cp = cd.cpar + ((size_t)n * nc + c) * NCP;
        const int row = (ci * nt + n) * 2 + role;
        coef[row][0] = T(cd.lam0 - lam);
        coef[row][1] = T(2.0 * lam * U);
        coef[row][2] = T(lam * U * U);
        coef[row][3] = T(2.0 * lam * V);
        coef[row][4] = T(lam * V * V);
        if (role == 0) {
            // collision coefficients of Eq. fv_h.  Explicit: the update divided by D; implicit: its right-hand side,
            // which the micro update then multiplies by minv across levels
            eq_cell(rho, U, V, lam, il0, cd.pr, qx, qy, cp + C_EQ0);
            const double h0 = 0.5 * dG * rcp64(tau), h1 = 0.5 * dG * rcp64(stau[r]);
            const double is = implicit ? 1.0 : rcp64(1.0 + h1);
            // kself, -kE, kp1, kp0, -kdx, -kdy, each stored twice (broadcast pairs for the (h, b) update)
            const double kk[6] = {(1.0 - h0) * is, implicit ? 0.0 : -dG * cd.omega * is, h1 * is, h0 * is,
                                  -dG * idx_ * is, -dG * idy * is};
#pragma unroll
            for (int q = 0; q < 6; ++q) cp[C_K + 2 * q] = cp[C_K + 2 * q + 1] = T(kk[q]);
        } else {
            // h+ of W^{k+1} takes the heat flux q^k
            eq_cell(rho, U, V, lam, il0, cd.pr, sq[r][0], sq[r][1], cp + C_EQ1);
            if (n == 0) {
                double numax = 0.0;
                for (int m = 0; m < nt; ++m) numax = fmax(numax, snu[m * K3_CELLS + ci]);
                cd.dG[c] = local_step(cd, numax);
            }
        }
    }
    if (implicit) {
        // inverse of diag(D_n) + dG omega E, D = 1 + dG/(2 tau^{k+1}), for the micro update of each cell (every
        // velocity): Gauss-Jordan in place, a thread per row and cell and the two halves on alternate columns.  No
        // pivoting is needed: E is skew-symmetric and D > 0, so the symmetric part is positive definite, and so is
        // that of every Schur complement the elimination meets.
        double D = 0.0;
        if (work) {
            D = 1.0 + 0.5 * dG * rcp64(stau[r]);
            for (int m = role; m < nt; m += 2) {
                int d = n - m; d += d < 0 ? nt : 0;        // E_{n, n-d} = e_d for d <= N_H, -e_{N_T - d} beyond
                const double e = d == 0 ? 0.0 : d <= cd.nh ? cd.e[d] : -cd.e[nt - d];
                sM[n][m][ci] = d == 0 ? D : dG * cd.omega * e;
            }
        }
        __syncthreads();
        for (int k = 0; k < nt; ++k) {
            double pv = 0.0, f = 0.0;
            if (work) {
                pv = rcp64(sM[k][k][ci]);
                f = sM[n][k][ci] * pv;
                if (n != k)
                    for (int m = role; m < nt; m += 2)
                        if (m != k) sM[n][m][ci] -= f * sM[k][m][ci];
            }
            __syncthreads();
            if (work) {
                if (n == k) {
                    for (int m = role; m < nt; m += 2) sM[k][m][ci] = m == k ? pv : sM[k][m][ci] * pv;
                } else if ((k & 1) == role) {
                    sM[n][k][ci] = -f;
                }
            }
            __syncthreads();
        }
        if (work) {
            T* mo = cd.minv + (size_t)c * nt * nt + n * nt;
            for (int m = role; m < nt; m += 2) mo[m] = T(sM[n][m][ci]);
        }
    }
    __syncthreads();
    // tables of expm1(lam0 x^2 - lam (x - U)^2) over the 1-D velocity nodes, so that for a Maxwellian of density rho:
    // H - H_ref = H_ref [(r - 1) + r (ex + ey + ex ey)], r = rho lam / lam0.  The entries of W^k and W^{k+1} lie side by
    // side (one load gives both); the CTA's rows are consecutive in memory.
    const int nuv = cd.nu + cd.nv, rows = min(K3_CELLS, nc - lb * K3_CELLS) * nt;
    P2<T>* dst = reinterpret_cast<P2<T>*>(cd.ctab) + (size_t)lb * K3_CELLS * nt * nuv;
    int row = (int)threadIdx.x / nuv, k = (int)threadIdx.x - row * nuv;
    for (int q = threadIdx.x; row < rows; q += blockDim.x) {
        const T* e = coef[2 * row];
        const T* e1 = coef[2 * row + 1];
        const bool isu = k < cd.nu;
        const T x = isu ? cd.tu1[k] : cd.tv1[k - cd.nu];
        dst[q] = pk(t_expm1<T>(e[0] * x * x + (isu ? e[1] : e[3]) * x - (isu ? e[2] : e[4])),
                    t_expm1<T>(e1[0] * x * x + (isu ? e1[1] : e1[3]) * x - (isu ? e1[2] : e1[4])));
        k += blockDim.x;
        while (k >= nuv) { k -= nuv; ++row; }
    }
}

// ------------------------------------------------------------------------------ K5 residual / status

constexpr int K5_THREADS = 128;

// residual, history and status of one case from nb partials; ends the iteration (swaps the state buffers)
template <typename T>
__device__ __forceinline__ void finish_case(const CaseDev<T>& cd, int nb)
{
    // every load is issued before the first is needed: the kernel is one CTA per case and waits for little else
    // (8.1 -> 6.1 us, 8x8 cells)
    CaseStatus* const st = cd.st;
    const double* __restrict__ rp = cd.rpart;
    double* const hist = cd.rhist;
    const double inv = rcp64((double)cd.nc);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int active = st->active, parity = st->parity, failed = *(volatile int*)cd.err;
    const long long iters = st->iters, iters_call = st->iters_call;
    const double tol = *cd.tol;
    // thread t sums variable t & 3 of every 32nd partial; then a fixed tree over lanes and warps
    __shared__ double part[K5_THREADS / 32][4];
    double s = 0.0;
    for (int b = threadIdx.x >> 2; b < nb; b += K5_THREADS / 4) s += rp[(size_t)b * 4 + (lane & 3)];
    if (!active || failed) return;                       // a failed wait leaves the iteration unfinished
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane < 4) part[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        // lanes 0..3: one variable each
        const int k = lane & 3;
        const double R = sqrt((part[0][k] + part[1][k] + part[2][k] + part[3][k]) * inv);
        const bool bad = __any_sync(0xffffffffu, !(R <= 1e10));   // also catches NaN
        if (lane < 4) {
            st->last[k] = R;
            hist[(iters % RING) * 4 + k] = R;
        }
        if (lane == 0) {
            st->iters = iters + 1;
            st->iters_call = iters_call + 1;
            st->parity = parity ^ 1;
            if (bad) st->diverged = 1;
            if (bad || (tol > 0.0 && iters + 1 >= 10 && R <= tol)) st->active = 0;
        }
    }
}

// LOOP: the last CTA also ends the pass of the device-side loop: one iteration fewer left; the loop goes on while
// iterations are left, some case is still iterating (not converged, not diverged) and no device wait has failed.  Every
// pass decrements the count, so the loop ends after at most the requested number of iterations.
struct LoopTest {
    cudaGraphConditionalHandle handle;
    int* left;                          // [0] iterations left, [1] CTAs of this pass that are done
    const CaseStatus* st;
    const int* err;
};

template <typename T, bool LOOP>
__global__ void __launch_bounds__(K5_THREADS) k5_finish(const CaseDev<T>* cases, int ncases, const int* k3off, LoopTest loop)
{
    finish_case(cases[blockIdx.x], k3off[blockIdx.x + 1] - k3off[blockIdx.x]);
    if constexpr (LOOP) {
        __syncthreads();
        if (threadIdx.x != 0) return;
        if (ncases > 1) {
            __threadfence();
            if (atomicAdd(loop.left + 1, 1) != ncases - 1) return;
            __threadfence();
            loop.left[1] = 0;
        }
        const int r = loop.left[0] - 1;
        loop.left[0] = r;
        int any = 0;
        for (int k = 0; k < ncases; ++k) any |= *(volatile const int*)&loop.st[k].active;
        cudaGraphSetConditional(loop.handle, (r > 0 && any && *(volatile const int*)loop.err == 0) ? 1u : 0u);
    }
}

// ------------------------------------------------------------------------------ conversions and fields

// sign class in which a node is stored first (classes in order 0..3: u > 0 first, then v > 0 first)
template <typename T>
__device__ __forceinline__ int first_class(const CaseDev<T>& cd, int can)
{
    const double u = cd.u1[can % cd.nu], v = cd.v1[can / cd.nu];
    return (u < 0 ? 1 : 0) | (v < 0 ? 2 : 0);
}

// H_ref of every stored velocity, formed once per case: an FP64 exponential costs a scheduler some 1000 cycles per warp,
// and the conversions below took one per value (set, 20 iterations, harmonics and get of a 32x32, 32x32, N_T 7 state:
// 22.1 -> 20.6 ms)
template <typename T>
__global__ void k_reference(CaseDev<T> cd)
{
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= cd.nvb * VB) return;
    cd.vref[a] = cd.vcan[a] >= 0 ? (cd.lam0 / M_PI) * exp(-cd.lam0 * (cd.vu[a] * cd.vu[a] + cd.vv[a] * cd.vv[a])) : 0.0;
}

// canonical FP64 level array (stage[c][a], a < nvel) -> delta-form internal layout of one level
template <typename T>
__global__ void k_set_level(CaseDev<T> cd, int n, int which, const double* stage)
{
    size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t tot = (size_t)cd.nc * cd.nvb * VB;
    if (k >= tot) return;
    int lane = k & 31;
    size_t r = k >> 5;
    int c = r % cd.nc, vb = r / cd.nc;
    int a = vb * VB + lane;
    double val = 0.0;
    const int can = cd.vcan[a];
    if (can >= 0) {
        const double href = cd.vref[a];
        double rv = which == 0 ? href : href * 0.5 / cd.lam0;
        val = stage[(size_t)c * cd.nvel + can] - rv;
    }
    T* dst = reinterpret_cast<T*>(cd.f[cd.st->parity]);
    dst[2 * sidx(cd.nc, cd.nt, vb, c, n, lane) + which] = T(val);
}

template <typename T>
__global__ void k_get_level(CaseDev<T> cd, int n, int which, double* stage)
{
    size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    size_t tot = (size_t)cd.nc * cd.nvb * VB;
    if (k >= tot) return;
    int lane = k & 31;
    size_t r = k >> 5;
    int c = r % cd.nc, vb = r / cd.nc;
    int a = vb * VB + lane;
    const int can = cd.vcan[a];
    // a node stored in several sign classes holds the same value in each; the first copy is read
    if (can < 0 || cd.vcls[vb] != first_class(cd, can)) return;
    const double href = cd.vref[a];
    double rv = which == 0 ? href : href * 0.5 / cd.lam0;
    const T* src = reinterpret_cast<const T*>(cd.f[cd.st->parity]);
    stage[(size_t)c * cd.nvel + can] = (double)src[2 * sidx(cd.nc, cd.nt, vb, c, n, lane) + which] + rv;
}

// Uniform reduced Maxwellian (rho, U, V, T) on every level, delta form; W = its continuous moments.  CTAs (x, vb): each
// thread forms the two values of its velocity once and writes them to INIT_ROWS (level, cell) rows (one pair of
// exponentials per stored value took 116 ms for the 128x128, 64x64, N_T 11 state, against a write of 5.9 GB).
constexpr int INIT_ROWS = 256;

template <typename T>
__global__ void __launch_bounds__(256) k_init_uniform(CaseDev<T> cd, double rho, double U, double V, double Tt)
{
    const int p = cd.st->parity, rows = cd.nc * cd.nt;
    const int lane = threadIdx.x & 31, first = blockIdx.x * INIT_ROWS;
    if (blockIdx.y == 0) {
        for (int k = first + threadIdx.x; k < min(first + INIT_ROWS, rows); k += blockDim.x) {
            double* W = cd.W[p] + (size_t)k * 4;
            W[0] = rho; W[1] = rho * U; W[2] = rho * V; W[3] = 0.5 * rho * (U * U + V * V) + 0.75 * rho * Tt;
        }
    }
    for (int vb = blockIdx.y; vb < cd.nvb; vb += gridDim.y) {
        const int a = vb * VB + lane;
        double dhv = 0.0, dbv = 0.0;
        if (cd.vcan[a] >= 0) {
            double uu = cd.vu[a], vv = cd.vv[a];
            double lam = cd.lam0 / Tt;
            double H = rho * (lam / M_PI) * exp(-lam * ((uu - U) * (uu - U) + (vv - V) * (vv - V)));
            double href = (cd.lam0 / M_PI) * exp(-cd.lam0 * (uu * uu + vv * vv));
            dhv = H - href;
            dbv = H * 0.5 / lam - href * 0.5 / cd.lam0;
        }
        const P2<T> x = pk(T(dhv), T(dbv));
        P2<T>* o = cd.f[p] + (size_t)vb * rows * VB + lane;
        for (int k = first + (int)(threadIdx.x >> 5); k < min(first + INIT_ROWS, rows); k += blockDim.x >> 5)
            o[(size_t)k * VB] = x;
    }
}

// fields of one level from the moments of h, b: out[f * nc + c], f = rho, U, V, T, tau_xy, qx, qy, p
template <typename T>
__global__ void k_fields(CaseDev<T> cd, int n, double* out)
{
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (c >= cd.nc) return;
    const int p = cd.st->parity;
    double A[13];
#pragma unroll
    for (int k = 0; k < 13; ++k) A[k] = 0.0;
    for (int vb = 0; vb < cd.nvb; ++vb) {
        int a = vb * VB + lane;
        double w = cd.vw[a], u = cd.vu[a], v = cd.vv[a];
        const P2<T> fv = cd.f[p][sidx(cd.nc, cd.nt, vb, c, n, lane)];
        double wd = w * (double)fv.x, we = w * (double)fv.y;
        A[0] += wd; A[1] += wd * u; A[2] += wd * v; A[3] += wd * u * u; A[4] += wd * u * v; A[5] += wd * v * v;
        A[6] += wd * u * u * u; A[7] += wd * u * u * v; A[8] += wd * u * v * v; A[9] += wd * v * v * v;
        A[10] += we; A[11] += we * u; A[12] += we * v;
    }
#pragma unroll
    for (int k = 0; k < 13; ++k) A[k] = warp_sum(A[k]) + cd.refmom[k];
    if (lane == 0) {
        double Wm[4] = {A[0], A[1], A[2], 0.5 * (A[3] + A[5] + A[10])};
        double rho, U, V, lam, qx, qy;
        prim(Wm, rho, U, V, lam);
        heat_flux_raw(A, U, V, qx, qy);
        double txy = A[4] - V * A[1] - U * A[2] + U * V * A[0];
        const int nc = cd.nc;
        out[0 * nc + c] = rho;
        out[1 * nc + c] = U;
        out[2 * nc + c] = V;
        out[3 * nc + c] = cd.lam0 / lam;
        out[4 * nc + c] = txy;
        out[5 * nc + c] = qx;
        out[6 * nc + c] = qy;
        out[7 * nc + c] = rho / (2.0 * lam);
    }
}

// Eq. dft_general on fields of all levels (lv[n][8][nc]) -> re/im of harmonic k
__global__ void k_dft(const double* lv, int nt, int nc, int k, double* re, double* im)
{
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 8 * nc) return;
    double sr = 0.0, si = 0.0;
    for (int n = 0; n < nt; ++n) {
        double th = 2.0 * M_PI * (double)k * (double)n / (double)nt;
        double val = lv[(size_t)n * 8 * nc + idx];
        sr += val * cos(th);
        si -= val * sin(th);
    }
    re[idx] = sr / nt;
    im[idx] = si / nt;
}

}  // namespace hb
