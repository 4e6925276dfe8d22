// Micro update of one HB-UGKS iteration (K4): interface micro fluxes (Eq. micro_flux), spectral source and the
// semi-implicit collision update (Eq. fv_h) of every cell, level and velocity.
//
// A group of warps, one per level, takes a strip of TX columns, a segment of rows and VPL blocks of 32 velocities of
// one sign class; a CTA holds one or several groups, which share nothing (registers are given to a CTA for four warps
// at a time, so CTAs of three or five warps would waste a quarter or more of them).  A group's warps march along the rows in the direction of v and, within a row, along the
// columns in the direction of u: a cell's upwind fluxes are then the ones the same lane has just computed (the
// x-flux of the cell before, the y-flux of the row before), so no flux and no slope passes through shared memory and
// no CTA barrier separates levels.  Columns and rows are counted from the upwind side ("mirrored": column p is
// i = p or nx - 1 - p); in these coordinates both velocity components are positive, a slope along an axis changes sign
// with it, and u s_x, u (F_downwind - F_upwind) keep theirs, so one code serves the four sign classes.  Only the
// strip's upwind column and the segment's upwind row are computed twice (one flux each).
//
// Bound by instruction issue in single precision: 232 warp instructions per 32 updates, some 130 of them floating
// point, where the previous kernel (a tile of cells per CTA, fluxes through shared memory, one barrier per level) needed
// 422.  The shared-memory loads serve two velocities per lane, the expm1 factors are loaded ahead of their use (their L2
// latency was 46 % of the stalls), and the x direction is a template parameter so that all offsets within a row are
// constants.  Strips of two columns with 128 registers hold more warps per SM and win up to 7 levels (0.83 against
// 1.02 ms, 64x64, 48x48, N_T 7), strips of four with 168 recompute less and win above (8.2 ms, 128x128, 64x64, N_T 11).
// Bound by the FP64 pipe in FP64.  Previous kernel
// -> this one: 16.25 -> 8.23 ms (128x128, 64x64, N_T 11), 1.50 -> 0.83 ms (64x64, 48x48, N_T 7), 44.5 -> 25.9 ms (48
// uneven cavities), 0.60 -> 0.32 ms (90x90, 28x28, N_T 3), 0.56 -> 0.68 ms where a class is one block (160x160, 10x10, N_T
// 7: the second half of every pair repeats it); FP64 with kept slopes 58.1 -> 35.1 ms (twelve 64x64, 32x32, N_T 3) and
// 25.8 -> 16.2 ms (64x64, 48x48, N_T 7).
#pragma once
#include "hb_cells.cuh"

namespace hb {

// the VPL velocities of a lane side by side: a scalar, or a pair handled by packed instructions
template <typename T, int VPL> struct LanesOf { using type = T; };
template <> struct LanesOf<float, 2> { using type = float2; };

template <typename L> struct Lane1;
template <> struct Lane1<float> {
    static __device__ __forceinline__ float all(float x) { return x; }
    static __device__ __forceinline__ float at(float x, int) { return x; }
    static __device__ __forceinline__ float of(const float* x) { return x[0]; }
};
template <> struct Lane1<double> {
    static __device__ __forceinline__ double all(double x) { return x; }
    static __device__ __forceinline__ double at(double x, int) { return x; }
    static __device__ __forceinline__ double of(const double* x) { return x[0]; }
};
template <> struct Lane1<float2> {
    static __device__ __forceinline__ float2 all(float x) { return make_float2(x, x); }
    static __device__ __forceinline__ float at(float2 x, int k) { return k ? x.y : x.x; }
    static __device__ __forceinline__ float2 of(const float* x) { return make_float2(x[0], x[1]); }
};

// Maxwellian part of the micro flux divided by dG_f and u_n (delta form): C1' dH + H Q for h and i2l (C1' dH + H Qb) +
// C1' (i2l - i2l0) H_ref for b (Qb = Q + lin), from the face's parameters fp (shared memory; cubic at qo, linear term at
// lo: the upwind side's), the expm1 factors (ex, ey) of the interface Maxwellian and H_ref (hr) at the lane's velocities;
// c4, c5: C4', C5'.  H/H_ref is multiplied by H_ref before anything else: far out on a wide velocity grid in hot gas it
// nears the largest float, which its product with Q would pass.
template <typename T, typename L>
__device__ __forceinline__ void flux_core(const T* fp, int qo, int lo, L ex, L ey, L u, L v, L hr, L& mh, L& mb, T& c4, T& c5)
{
    using A = Lane1<L>;
    T sc[8], c[12], l[4];          // sc: r - 1, r, 1/(2 lam), 1/(2 lam) - 1/(2 lam0), C1', C4', C5', C1' times slot 3
    load_par(fp + F_RM1, sc);
    load_par(fp + qo, c);
    load_par(fp + lo, l);
    c4 = sc[5];
    c5 = sc[6];
    const L G = pfma(A::all(sc[1]), pfma(ex, ey, padd(ex, ey)), A::all(sc[0]));
    const L dH = pmul(hr, G), H = pfma(hr, G, hr), cH = pmul(A::all(sc[4]), dH);
    // Horner form of the bivariate cubic with monomials 1, u, v, u^2, uv, v^2, u^3, u^2 v, u v^2, v^3
    const L y0 = pfma(v, pfma(v, pfma(v, A::all(c[9]), A::all(c[5])), A::all(c[2])), A::all(c[0]));
    const L y1 = pfma(v, pfma(v, A::all(c[8]), A::all(c[4])), A::all(c[1]));
    const L y2 = pfma(u, A::all(c[6]), pfma(v, A::all(c[7]), A::all(c[3])));
    const L Q = pfma(u, pfma(u, y2, y1), y0);
    const L Qb = pfma(v, A::all(l[2]), pfma(u, A::all(l[1]), padd(Q, A::all(l[0]))));
    mh = pfma(H, Q, cH);
    mb = pfma(A::all(sc[2]), pfma(H, Qb, cH), pmul(hr, A::all(sc[7])));
}

// Equilibrium (H+ - H_ref, B+ - B_ref) of one cell-parameter slot q at the lane's velocities: dH and i2l dH +
// (i2l - i2l0) H_ref of the Maxwellian (cell table factors ex, ey; hr = H_ref), and with the Shakhov model dH + H sk,
// sk = L Q, for h and the same with sk + 2 L for b (L, Q the linear and quadratic factors of s (c.q)(2 lam |c|^2 - 4);
// r2 = u^2 + v^2)
template <bool SHAKHOV, typename T, typename L>
__device__ __forceinline__ void eq_core(const T* qp, L ex, L ey, L u, L v, L r2, L hr, L& mh, L& mb)
{
    using A = Lane1<L>;
    T q[12];
    load_par(qp, q);
    const L dH = pmul(hr, pfma(A::all(q[E_R]), pfma(ex, ey, padd(ex, ey)), A::all(q[E_RM1])));
    const L i2l = A::all(q[E_I2L]), dB = pmul(hr, A::all(q[E_DI2L]));
    if constexpr (!SHAKHOV) {
        mh = dH;
        mb = pfma(i2l, dH, dB);
        return;
    }
    const L Lf = pfma(A::all(q[E_L + 2]), v, pfma(A::all(q[E_L + 1]), u, A::all(q[E_L])));
    const L Qs = pfma(A::all(q[E_Q + 3]), r2,
                      pfma(A::all(q[E_Q + 2]), v, pfma(A::all(q[E_Q + 1]), u, A::all(q[E_Q]))));
    const L sk = pmul(Lf, Qs), sb = pfma(A::all(T(2)), Lf, sk), H = padd(hr, dH);
    mh = pfma(H, sk, dH);
    mb = pfma(i2l, pfma(H, sb, dH), dB);
}

constexpr int K4_MAXROWS = 32;   // rows per segment

// Shared memory of one group of k4_march for nt levels (bytes): three rows of the strip with its halo on every level
// (two columns upwind, one downwind), two rows of parameters (x-faces, y-faces downwind, cells) on every level, and
// with the spectral source at the new iterate one row of right-hand sides.
template <typename T, int TX, int VPL>
struct K4Layout {
    using V = P2<T>;
    static constexpr int NCOL = TX + 3;
    static constexpr uint32_t COL = VB * sizeof(V), BLK = NCOL * COL, ROW = VPL * BLK;
    static constexpr uint32_t PX = (TX + 1) * NP * sizeof(T), PY = TX * NP * sizeof(T), PC = TX * NCP * sizeof(T);
    static constexpr uint32_t PAR = PX + PY + PC;
    // spacings: widths and inverse distances of the strip's columns, then of the segment's rows
    static constexpr int GX = TX + 2, GH = TX + 1, GY = K4_MAXROWS + 3;
    static constexpr size_t GEO = ((GX + GH + 2 * GY) * sizeof(T) + 15) / 16 * 16;
    static constexpr size_t bytes(int nt, bool imp)
    {
        return (size_t)nt * (3 * ROW + 2 * PAR + (imp ? (uint32_t)(VPL * TX) * COL : 0u)) + GEO;
    }
};

// Threads the instances are compiled for, and so their registers: 128 for up to 15 warps (every level count with strips
// of two columns, up to 7 levels with strips of four), 168 for strips of four columns on up to 11 levels, one CTA per SM.
constexpr int K4_T2 = MAXNT * 32, K4_T4L = 11 * 32;
constexpr int K4_NT4 = 7, K4_NT4L = 11;

// spectral source of NC consecutive cells of a row on level n: sum_d e_d (f_{n-d} - f_{n+d}) for (h, b) (Eq. D_explicit in paired
// form); row: the first cell on level 0, level stride ls, column step CS and block step BLK in bytes
template <int NH, int CS, int BLK, typename T, typename V, int NC, int VPL>
__device__ __forceinline__ void spectral_cells(const char* row, uint32_t ls, int n, int nt, const T* et, V (&e)[NC][VPL])
{
#pragma unroll
    for (int t = 0; t < NC; ++t)
#pragma unroll
        for (int h = 0; h < VPL; ++h) e[t][h] = bc(T(0));
#pragma unroll
    for (int d = 1; d <= NH; ++d) {
        int nm = n - d; nm += nm < 0 ? nt : 0;
        int np = n + d; np -= np >= nt ? nt : 0;
        const char* pm = row + (uint32_t)nm * ls;
        const char* pp = row + (uint32_t)np * ls;
        const V ed = bc(et[d]);
#pragma unroll
        for (int t = 0; t < NC; ++t)
#pragma unroll
            for (int h = 0; h < VPL; ++h)
                e[t][h] = pfma(ed, psub(*reinterpret_cast<const V*>(pm + t * CS + h * BLK),
                                        *reinterpret_cast<const V*>(pp + t * CS + h * BLK)), e[t][h]);
    }
}

// One bulk copy of the per-row batches, formed once per warp: in batch b (lo <= b <= hi) it reads src + (b - 1) stride
// and lands at dst, plus the slot of the row it belongs to.
struct alignas(16) K4Copy {
    const char* src;
    long long stride;
    uint32_t dst, bytes;
    int lo, hi;
};
static_assert(sizeof(K4Copy) == 32);

template <class P, int TX, int VPL, bool IMP, int MAXT>
__global__ void __launch_bounds__(MAXT) k4_march(const __grid_constant__ P B, int rows, int groups)
{
    using T = typename P::value_type;
    using Y = K4Layout<T, TX, VPL>;
    using V = P2<T>;
    using L = typename LanesOf<T, VPL>::type;
    using A = Lane1<L>;
    // strips of four columns are always full (the last one overlaps its neighbour and writes the same bits there);
    // those of two may be partial
    constexpr bool FULL = TX == 4;
    constexpr int NCOPY = VPL + 3;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t full_[MAXNT][2], done_[MAXNT], meet_[IMP ? MAXNT : 1];   // per group
    __shared__ int abort_flag;                               // set by the first warp whose wait runs out
    __shared__ K4Copy copies[MAXNT][NCOPY];                  // per warp
    int lb;
    const CaseDev<T>& cd = B.find(blockIdx.x, lb);
    if (!cd.st->active) return;
    // another CTA may set the error word while this one starts: decide for the whole CTA at once
    if (__syncthreads_or(*(volatile int*)cd.err != 0)) return;
    const bool expire = *(volatile const int*)cd.expire != 0;
    const int nx = cd.nx, ny = cd.ny, nt = cd.nt, nc = cd.nc, nfx = cd.nfx, nuv = cd.nu + cd.nv;
    const int lane = threadIdx.x & 31;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
    constexpr bool ALONE = MAXT == K4_T4L;                   // one group per CTA
    const int gi = ALONE ? 0 : warp / nt, n = ALONE ? warp : warp - gi * nt;   // the warp's group and level
    const int tid = (int)threadIdx.x - gi * nt * 32, nthreads = nt * 32;   // in the group
    uint64_t* const full = full_[gi];
    uint64_t* const done = &done_[gi];
    uint64_t* const meet = &meet_[IMP ? gi : 0];             // (implicit source)
    // CTA order: velocity group fastest (the CTAs of one strip share its parameters in L2), then strips, segments
    int ng = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) ng += (cd.cls_end[c] - (c ? cd.cls_end[c - 1] : 0) + VPL - 1) / VPL;
    const int work = ALONE ? lb : lb * groups + gi, tile = work / ng;
    int g = work - tile * ng, cls = 0, vb = 0, vend = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int first = c ? cd.cls_end[c - 1] : 0, cnt = (cd.cls_end[c] - first + VPL - 1) / VPL;
        if (g >= 0 && g < cnt) { cls = c; vb = first + g * VPL; vend = cd.cls_end[c]; }
        g -= cnt;
    }
    const bool xneg = (cls & 1) != 0, yneg = (cls & 2) != 0;
    const int nstrip = (nx + TX - 1) / TX;
    const int p0 = FULL ? min((tile % nstrip) * TX, nx - TX) : (tile % nstrip) * TX;
    const int q0 = (tile / nstrip) * rows, nr = min(rows, ny - q0);
    const bool idle = !ALONE && q0 >= ny;                    // past the case's last group
    char* const srow = reinterpret_cast<char*>(smem_raw) + (ALONE ? 0 : (size_t)gi * Y::bytes(nt, IMP));
    char* const spar = srow + (size_t)3 * nt * Y::ROW;
    V* const srhs = reinterpret_cast<V*>(spar + (size_t)2 * nt * Y::PAR);   // right-hand sides (implicit source)
    __shared__ T geo[ALONE ? Y::GEO / sizeof(T) : 1];        // (a fixed address saves the lone group's registers)
    T* const gxw = ALONE ? geo : reinterpret_cast<T*>(srow + Y::bytes(nt, IMP) - Y::GEO);
    T *const gxh = gxw + Y::GX, *const gyw = gxh + Y::GH, *const gyh = gyw + Y::GY;
    const uint32_t slot_b = (uint32_t)nt * Y::ROW, pslot_b = (uint32_t)nt * Y::PAR;
    if (threadIdx.x == 0) abort_flag = 0;
    if (tid == 0) {
        mbar_init(&full[0], nt);
        mbar_init(&full[1], nt);
        mbar_init(done, nt);
        if (IMP) mbar_init(meet, nt);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // spacings in mirrored order: gxw[k] twice the inverse distance of columns p0 - 2 + k and p0 - 1 + k, gxh[k] half
    // the width of column p0 - 1 + k; gyw[r], gyh[r] of stream rows r (row q = q0 - 2 + r) and r, r + 1
    for (int k = tid; k < TX + 2; k += nthreads) {
        const int p = p0 - 2 + k, i = xneg ? nx - 2 - p : p;
        gxw[k] = (i >= 0 && i < nx - 1) ? T(2) * T(cd.rdx[i]) : T(0);
        const int ph = p + 1, ih = xneg ? nx - 1 - ph : ph;
        if (k < TX + 1) gxh[k] = (ih >= 0 && ih < nx) ? T(cd.hx[ih]) : T(0);
    }
    for (int r = tid; r < nr + 3; r += nthreads) {
        const int q = q0 - 2 + r, j = yneg ? ny - 2 - q : q, jh = yneg ? ny - 1 - q : q;
        gyw[r] = (j >= 0 && j < ny - 1) ? T(2) * T(cd.rdy[j]) : T(0);
        gyh[r] = (jh >= 0 && jh < ny) ? T(cd.hy[jh]) : T(0);
    }
    const int par = cd.st->parity;
    const size_t bstride = (size_t)nt * nc * VB;             // pairs between consecutive velocity blocks
    const bool two = VPL == 2 && vb + 1 < vend;              // a class's last block may go alone (computed twice)
    // The warp's copies.  Batch b >= 1 holds stream row b + 1 of every block and the parameters of stream row b
    // (y-faces downwind of it; x-faces and cells of the rows that are computed, b = 2..nr + 1) on the warp's level and
    // completes, with the other warps' parts, on full[b & 1]; batch 0 holds rows 0 and 1.  Shared memory keeps columns,
    // faces and cells in natural order from lowc, lowf, lowo on (which may lie outside the domain: clipped copies).
    const int lowc = xneg ? nx - 1 - (p0 + TX) : p0 - 2, c0 = max(lowc, 0), c1 = min(lowc + Y::NCOL, nx);
    const int lowf = xneg ? nx - (p0 + TX) : p0, f0_ = max(lowf, 0), f1_ = min(lowf + TX + 1, nx + 1);
    const int lowo = lowf, o0 = max(lowo, 0), o1 = min(lowo + TX, nx);
    const uint32_t rb = (uint32_t)(c1 - c0) * Y::COL, xb = (uint32_t)(f1_ - f0_) * (uint32_t)(NP * sizeof(T)),
                   yb = (uint32_t)(o1 - o0) * (uint32_t)(NP * sizeof(T)),
                   cb = (uint32_t)(o1 - o0) * (uint32_t)(NCP * sizeof(T));
    const long long ysgn = yneg ? -1 : 1;                    // (row strides in bytes may pass 31 bits)
    if (lane < NCOPY) {
        const int q = q0 - 1, j = yneg ? ny - 1 - q : q, fj = yneg ? ny - 1 - q : q + 1;   // stream row 1
        K4Copy c;
        if (lane < VPL) {
            c.src = reinterpret_cast<const char*>(cd.f[par] + (size_t)(vb + (two ? lane : 0)) * bstride +
                                                  (size_t)n * nc * VB + ((long long)(j + ysgn) * nx + c0) * VB);
            c.stride = ysgn * nx * (long long)Y::COL;
            c.dst = smem_u32(srow) + n * Y::ROW + lane * Y::BLK + (uint32_t)(c0 - lowc) * Y::COL;
            c.bytes = rb;
            c.lo = 1;
            c.hi = ny - q0;
        } else {
            const uint32_t base = smem_u32(spar) + n * Y::PAR;
            if (lane == VPL) {
                c.src = reinterpret_cast<const char*>(cd.fpar + ((long long)n * cd.nf + (long long)j * (nx + 1) + f0_) * NP);
                c.stride = ysgn * (nx + 1) * (long long)(NP * sizeof(T));
                c.dst = base + (uint32_t)((f0_ - lowf) * NP * sizeof(T));
                c.bytes = xb;
            } else if (lane == VPL + 1) {
                c.src = reinterpret_cast<const char*>(cd.fpar + ((long long)n * cd.nf + nfx + (long long)fj * nx + o0) * NP);
                c.stride = ysgn * nx * (long long)(NP * sizeof(T));
                c.dst = base + Y::PX + (uint32_t)((o0 - lowo) * NP * sizeof(T));
                c.bytes = yb;
            } else {
                c.src = reinterpret_cast<const char*>(cd.cpar + ((long long)n * nc + (long long)j * nx + o0) * NCP);
                c.stride = ysgn * nx * (long long)(NCP * sizeof(T));
                c.dst = base + Y::PX + Y::PY + (uint32_t)((o0 - lowo) * NCP * sizeof(T));
                c.bytes = cb;
            }
            c.lo = lane == VPL + 1 ? 1 : 2;
            c.hi = nr + 1;
        }
        copies[warp][lane] = c;
    }
    __syncthreads();
    if (idle) return;

    // this warp's part of batch b >= 1, its row into row slot `slot`
    auto issue = [&](int b, uint32_t slot) {
        uint64_t* bar = &full[b & 1];
        if (lane == 0) mbar_arrive_expect(bar, (b <= ny - q0 ? VPL * rb : 0u) + yb + (b >= 2 ? xb + cb : 0u));
        __syncwarp();
        if (lane < NCOPY) {
            const K4Copy c = copies[warp][lane];
            if (b >= c.lo && b <= c.hi)
                bulk_g2s_at(c.dst + (lane < VPL ? slot * slot_b : (uint32_t)(b & 1) * pslot_b),
                            c.src + (b - 1) * c.stride, c.bytes, bar);
        }
    };
    if (lane == 0) {
        // batch 0: rows 0 and 1, where they exist
        const uint32_t have = (q0 >= 2 ? 1u : 0u) + (q0 >= 1 ? 1u : 0u);
        if (have) mbar_arrive_expect(&full[0], have * VPL * rb);
        else mbar_arrive(&full[0]);
    }
    __syncwarp();
    if (lane < 2 * VPL) {
        const int row = lane / VPL;
        const K4Copy c = copies[warp][lane % VPL];
        if (q0 + row >= 2)
            bulk_g2s_at(c.dst + (uint32_t)row * slot_b, c.src + (row - 2) * c.stride, c.bytes, &full[0]);
    }
    issue(1, 2);
    int issued = 1;

    // the lane's velocities
    T u[VPL], v[VPL];
    T um[VPL], vm[VPL];                                      // |u|, |v|
    T hr[VPL], rr2[VPL];
    uint32_t iu[VPL], iv[VPL];                               // byte offsets of the lane's entries in a table row
#pragma unroll
    for (int h = 0; h < VPL; ++h) {
        const int av = (vb + (two ? h : 0)) * VB + lane;
        u[h] = __ldg(cd.tu + av);
        v[h] = __ldg(cd.tv + av);
        um[h] = xneg ? -u[h] : u[h];
        vm[h] = yneg ? -v[h] : v[h];
        hr[h] = __ldg(cd.thref + av);
        rr2[h] = pfma(u[h], u[h], pmul(v[h], v[h]));
        iu[h] = (uint32_t)__ldg(cd.viu + av) * (uint32_t)sizeof(T);
        iv[h] = (uint32_t)(cd.nu + __ldg(cd.viv + av)) * (uint32_t)sizeof(T);
    }
    const L uL = A::of(u), vL = A::of(v), r2L = A::of(rr2), hL = A::of(hr);
    const bool shakhov = cd.shakhov != 0;
    const bool implicit = IMP && cd.spectral_implicit != 0;
    const int nh = implicit ? 0 : cd.nh;
    int* err = cd.err;
    const int qx_ = xneg ? F_QR : F_QL, lx_ = xneg ? F_LBR : F_LBL;
    const int qy_ = yneg ? F_QR : F_QL, ly_ = yneg ? F_LBR : F_LBL;
    // expm1 factors of the lane's velocities from a table row; of both equilibria from a cell's row (W^k, W^{k+1})
    auto pair_at = [&](const char* tb, const uint32_t (&ix)[VPL]) {
        T x[VPL];
#pragma unroll
        for (int h = 0; h < VPL; ++h) x[h] = __ldg(reinterpret_cast<const T*>(tb + ix[h]));
        return A::of(x);
    };
    auto pairs_at = [&](const char* tb, const uint32_t (&ix)[VPL], L& a0, L& a1) {
        T x[VPL], y[VPL];
#pragma unroll
        for (int h = 0; h < VPL; ++h) {
            const V z = __ldg(reinterpret_cast<const V*>(tb + 2 * ix[h]));
            x[h] = z.x;
            y[h] = z.y;
        }
        a0 = A::of(x);
        a1 = A::of(y);
    };
    // flux pairs (divided by dG_f and the speed) of a diffuse wall's re-emitted distribution rho_w H_w
    auto wall_flux = [&](const char* fp, int wall, V (&F)[VPL]) {
        const T* wp = reinterpret_cast<const T*>(fp) + F_WRM1;
        const char* tb = reinterpret_cast<const char*>(cd.wtab + (size_t)(wall * cd.nslot + wall_slot(cd, n)) * nuv);
#pragma unroll
        for (int h = 0; h < VPL; ++h) {
            const T ex = __ldg(reinterpret_cast<const T*>(tb + iu[h])), ey = __ldg(reinterpret_cast<const T*>(tb + iv[h]));
            const T dHw = pmul(hr[h], pfma(wp[1], pfma(ex, ey, padd(ex, ey)), wp[0]));
            F[h] = pk(dHw, pfma(dHw, wp[2], pmul(hr[h], wp[3])));
        }
    };
    // flux pairs through a face (divided by dG_f and the speed): d0 the reconstruction, gr = u s_x + v s_y
    auto face_flux = [&](const char* fp, int qo, int lo, L ex, L ey, const V (&d0)[VPL], const V (&gr)[VPL], V (&F)[VPL]) {
        L mh, mb;
        T c4, c5;
        flux_core<T, L>(reinterpret_cast<const T*>(fp), qo, lo, ex, ey, uL, vL, hL, mh, mb, c4, c5);
#pragma unroll
        for (int h = 0; h < VPL; ++h)
            F[h] = pfma(bc(c4), d0[h], pfma(bc(c5), gr[h], pk(A::at(mh, h), A::at(mb, h))));
    };
    // a wait ran out: this warp waits (bounded) for the batches from b on that it has issued and not seen complete, so
    // that none still lands in shared memory after the CTA exits
    auto give_up = [&](int b) {
        for (int k = b; k <= issued; ++k) mbar_drain(&full[k & 1], (uint32_t)((k >> 1) & 1));
    };
    // The group's warps meet twice per row with the implicit source, so the phases are 0 and 1 in turn.  Bounded like every
    // wait: a warp that has given up elsewhere never arrives here.
    auto group_meet = [&](uint32_t phase) {
        __syncwarp();
        if (lane == 0) mbar_arrive(meet);
        return mbar_wait(meet, phase, err, &abort_flag);
    };
    if (!mbar_wait(&full[0], 0, err, &abort_flag)) { give_up(0); return; }
    if (expire) {
        // the test hook reports the first wait as expired after it has completed
        if (threadIdx.x == 0) atomicExch(err, 1);
        give_up(1);
        return;
    }

    // XN: u < 0.  With the direction along x fixed, columns, faces and cells lie at constant offsets from each other.
    auto march = [&](auto xn_tag) {
        constexpr bool XN = decltype(xn_tag)::value;
        constexpr int SG = XN ? -1 : 1, CS = SG * (int)Y::COL, FS = SG * (int)(NP * sizeof(T)), ES = SG * (int)(NCP * sizeof(T));
        constexpr int COL0 = XN ? (Y::NCOL - 1) * (int)Y::COL : 0;           // column 0 (p0 - 2) of a row
        constexpr int FX0 = XN ? TX * (int)(NP * sizeof(T)) : 0;             // x-face upwind of the strip
        constexpr int FY0 = (int)Y::PX + (XN ? (TX - 1) * (int)(NP * sizeof(T)) : 0);
        constexpr int CE0 = (int)(Y::PX + Y::PY) + (XN ? (TX - 1) * (int)(NCP * sizeof(T)) : 0);
        const int i0 = XN ? nx - 1 - p0 : p0, fi0 = XN ? nx - p0 : p0;
        // Bytes between the table rows of consecutive faces.  The lone-group instance, short of registers, keeps them in 32
        // bits (its launch rule sees to it that eight of them fit).
        using Off = std::conditional_t<ALONE, int, long long>;
        const Off tstep = (Off)SG * nt * nuv * (int)sizeof(T);
        auto ahead = [tstep](const char* tb, int k) { return tb + k * tstep; };
        char* const rown = srow + n * Y::ROW + lane * sizeof(V) + COL0;      // row slot 0, this level and lane
        auto at = [](const char* row, int c, int h) -> V {                   // mirrored column c (2 is p0) of block h
            return *reinterpret_cast<const V*>(row + c * CS + h * (int)Y::BLK);
        };
        V dyp[TX + 1][VPL];                                  // y difference towards the row before, columns -1..TX-1
        V Fy[TX][VPL];                                       // y-flux through the upwind face of the current row
#pragma unroll
        for (int k = 0; k < TX; ++k)
#pragma unroll
            for (int h = 0; h < VPL; ++h) Fy[k][h] = bc(T(0));
        // FP64: the slopes the face sums have kept, in mirrored direction (elsewhere they are formed here again)
        const bool kept = sizeof(T) == 8 && cd.sl != nullptr;
        auto kept_slopes = [&](int jr, int t, V& sx, V& sy) {                // of column p0 + t of row jr
            const V* o = cd.sl + (((size_t)vb * nt + n) * nc + (size_t)(jr * nx + i0 + t * SG)) * 2 * VB + lane;
            const V a = __ldg(o), b = __ldg(o + VB);
            sx = XN ? pk(-a.x, -a.y) : a;
            sy = yneg ? pk(-b.x, -b.y) : b;
        };
        // differences between the rows in slots a and b (row r and r + 1) along y, of every column
        auto row_diff = [&](const char* ra, const char* rb2, int r) {
#pragma unroll
            for (int k = 0; k <= TX; ++k)
#pragma unroll
                for (int h = 0; h < VPL; ++h) dyp[k][h] = pmul(psub(at(rb2, k + 1, h), at(ra, k + 1, h)), bc(gyw[r]));
        };
        // The table entries of a face or cell come from L2 and are loaded one cell ahead: xe, xv of the next x-face, ye,
        // yv of the next y-face, and with registers to spare (one CTA per SM) ce, cv (and those of W^{k+1}) of the next
        // cell, in the order they are used.
        constexpr bool EARLY = ALONE;
        L xe, xv, ye, yv, ce0, cv0, ce1, cv1;
        auto load_x = [&](const char* tb) { xe = pair_at(tb, iu); xv = pair_at(tb, iv); };
        auto load_y = [&](const char* tb) { ye = pair_at(tb, iu); yv = pair_at(tb, iv); };
        auto load_c = [&](const char* tb) { pairs_at(tb, iu, ce0, ce1); pairs_at(tb, iv, cv0, cv1); };
        // table rows of row q: the x-face upwind of the strip, the y-face downwind of column 0, the cell of column 0
        auto row_tables = [&](int q, const char*& tx, const char*& ty, const char*& tc) {
            const int j = yneg ? ny - 1 - q : q, fj = yneg ? j : j + 1;
            tx = reinterpret_cast<const char*>(cd.ftab + ((size_t)(j * (nx + 1) + fi0) * nt + n) * nuv);
            ty = reinterpret_cast<const char*>(cd.ftab + ((size_t)(nfx + fj * nx + i0) * nt + n) * nuv);
            tc = reinterpret_cast<const char*>(cd.ctab + ((size_t)(j * nx + i0) * nt + n) * 2 * nuv);
        };
        const char *tx0, *ty0, *tc0;
        row_tables(q0, tx0, ty0, tc0);
        load_x(p0 > 0 ? tx0 : ahead(tx0, 1));
        load_y(ty0);
        if (EARLY) load_c(tc0);
        row_diff(rown, rown + slot_b, 0);                    // (unused where the segment starts at a wall)
        __syncwarp();
        if (lane == 0) mbar_arrive(done);

        uint32_t slot = 0;
        for (int r = 1; r <= nr + 1; ++r) {
            slot = slot == 2 ? 0 : slot + 1;
            const uint32_t nslot = slot == 2 ? 0 : slot + 1;
            const char* rc = rown + slot * slot_b;           // row r
            const char* rn = rown + nslot * slot_b;          // row r + 1
            const int q = q0 - 2 + r, j = yneg ? ny - 1 - q : q;
            const char* pr = spar + (r & 1) * pslot_b + n * Y::PAR;
            if (!mbar_wait(&full[r & 1], (uint32_t)((r >> 1) & 1), err, &abort_flag)) { give_up(r); return; }
            // the next batch: once every warp has left row r - 1, whose slots it refills
            auto refill = [&]() -> bool {
                if (r > nr) return true;
                if (!mbar_wait(done, (uint32_t)((r - 1) & 1), err, &abort_flag)) return false;
                issue(r + 1, nslot == 2 ? 0 : nslot + 1);
                issued = r + 1;
                return true;
            };
            const bool lastrow = q == ny - 1;
            const T wy = gyw[r];
            // limited slope along y of column c with value f0; the difference to the next row becomes dp
            auto yslope = [&](int c, int h, V f0, V& dp) -> V {
                V dn = pmul(psub(at(rn, c, h), f0), bc(wy));
                if (lastrow) dn = dp;
                const V s = vleer2(dp, dn);
                dp = dn;
                return s;
            };
            if (r == 1) {
                // ---- y-fluxes through the upwind faces of the segment's first row: of the row before, or of the wall
                if (q0 == 0) {
                    for (int t = 0; t < TX; ++t)
                        if (FULL || p0 + t < nx) {
                            V F[VPL];
                            wall_flux(pr + FY0 + t * FS, yneg ? 2 : 0, F);
#pragma unroll
                            for (int z = 0; z < TX; ++z)
#pragma unroll
                                for (int h = 0; h < VPL; ++h)
                                    if (z == t) Fy[z][h] = F[h];
                        }
                    if (!refill()) { give_up(r + 1); return; }
                    // no row before the first: its one-sided difference is the one to the next row (row 3, batch 2)
                    if (!mbar_wait(&full[0], 1u, err, &abort_flag)) { give_up(2); return; }
                    if (ny > 1) {
                        row_diff(rown + 2 * slot_b, rown, 2);
                    } else {
#pragma unroll
                        for (int k = 0; k <= TX; ++k)
#pragma unroll
                            for (int h = 0; h < VPL; ++h) dyp[k][h] = bc(T(0));
                    }
                } else {
                    V dxp[VPL], fc[VPL];
#pragma unroll
                    for (int h = 0; h < VPL; ++h) {
                        fc[h] = at(rc, 2, h);
                        // the column upwind exists unless the strip starts at a wall
                        dxp[h] = p0 > 0 ? pmul(psub(fc[h], at(rc, 1, h)), bc(gxw[1]))
                                        : nx > 1 ? pmul(psub(at(rc, 3, h), fc[h]), bc(gxw[2])) : bc(T(0));
                        dyp[0][h] = pmul(psub(at(rn, 1, h), at(rc, 1, h)), bc(wy));   // used where column -1 exists
                    }
                    if (!refill()) { give_up(r + 1); return; }
                    const char* th =
                        reinterpret_cast<const char*>(cd.ftab + ((size_t)(nfx + (yneg ? j : j + 1) * nx + i0) * nt + n) * nuv);
#pragma unroll
                    for (int t = 0; t < TX; ++t) {
                        if (!FULL && p0 + t >= nx) break;
                        V d0[VPL], gr[VPL];
#pragma unroll
                        for (int h = 0; h < VPL; ++h) {
                            const V fe = at(rc, t + 3, h);
                            V sx, sy;
                            if (kept) {
                                kept_slopes(j, t, sx, sy);
                            } else {
                                V dxn = pmul(psub(fe, fc[h]), bc(gxw[t + 2]));
                                if ((!FULL || t == TX - 1) && p0 + t == nx - 1) dxn = dxp[h];
                                sx = vleer2(dxp[h], dxn);
                                sy = yslope(t + 2, h, fc[h], dyp[t + 1][h]);
                                dxp[h] = dxn;
                            }
                            d0[h] = pfma(sy, bc(gyh[r]), fc[h]);
                            gr[h] = pfma(bc(um[h]), sx, pmul(bc(vm[h]), sy));
                            fc[h] = fe;
                        }
                        face_flux(pr + FY0 + t * FS, qy_, ly_, pair_at(ahead(th, t), iu), pair_at(ahead(th, t), iv), d0,
                                  gr, Fy[t]);
                    }
                }
            } else {
                V dxp[VPL], fc[VPL], Fx[VPL], e[2][VPL];
#pragma unroll
                for (int h = 0; h < VPL; ++h) fc[h] = at(rc, 2, h);
                if (p0 > 0) {
                    // ---- x-flux through the strip's upwind face, from the column before
                    V d0[VPL], gr[VPL];
#pragma unroll
                    for (int h = 0; h < VPL; ++h) {
                        const V fw = at(rc, 1, h);
                        V sx, sy;
                        if (kept) {
                            kept_slopes(j, -1, sx, sy);
                        } else {
                            dxp[h] = pmul(psub(fc[h], fw), bc(gxw[1]));
                            V dxm = pmul(psub(fw, at(rc, 0, h)), bc(gxw[0]));
                            if (p0 == 1) dxm = dxp[h];       // (an overlapping strip next to the wall)
                            sx = vleer2(dxm, dxp[h]);
                            sy = yslope(1, h, fw, dyp[0][h]);
                        }
                        d0[h] = pfma(sx, bc(gxh[0]), fw);
                        gr[h] = pfma(bc(um[h]), sx, pmul(bc(vm[h]), sy));
                    }
                    face_flux(pr + FX0, qx_, lx_, xe, xv, d0, gr, Fx);
                    load_x(ahead(tx0, 1));
                } else {
                    wall_flux(pr + FX0, XN ? 1 : 3, Fx);
#pragma unroll
                    for (int h = 0; h < VPL; ++h)
                        dxp[h] = nx > 1 ? pmul(psub(at(rc, 3, h), fc[h]), bc(gxw[2])) : bc(T(0));
                }
                if (!refill()) { give_up(r + 1); return; }
                V* const on = cd.f[par ^ 1] + (size_t)vb * bstride + (size_t)n * nc * VB + (size_t)(j * nx + i0) * VB + lane;
#pragma unroll
                for (int t = 0; t < TX; ++t) {
                    if (!FULL && p0 + t >= nx) break;
                    if (t % 2 == 0) {
                        const char* own = srow + slot * slot_b + lane * sizeof(V) + COL0 + (2 + t) * CS;
                        constexpr int BL = (int)Y::BLK;
                        switch (nh) {
                            case 0: spectral_cells<0, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            case 1: spectral_cells<1, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            case 2: spectral_cells<2, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            case 3: spectral_cells<3, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            case 4: spectral_cells<4, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            case 5: spectral_cells<5, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            case 6: spectral_cells<6, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                            default: spectral_cells<7, CS, BL, T, V, 2, VPL>(own, Y::ROW, n, nt, cd.et, e); break;
                        }
                    }
                    // ---- reconstruction and fluxes through the cell's downwind faces
                    V f0[VPL], dx0[VPL], dy0[VPL], gr[VPL], Fn[VPL], dX[VPL], dY[VPL];
#pragma unroll
                    for (int h = 0; h < VPL; ++h) {
                        f0[h] = fc[h];
                        fc[h] = at(rc, t + 3, h);
                        V sx, sy;
                        if (kept) {
                            kept_slopes(j, t, sx, sy);
                        } else {
                            V dxn = pmul(psub(fc[h], f0[h]), bc(gxw[t + 2]));
                            if ((!FULL || t == TX - 1) && p0 + t == nx - 1) dxn = dxp[h];
                            sx = vleer2(dxp[h], dxn);
                            sy = yslope(t + 2, h, f0[h], dyp[t + 1][h]);
                            dxp[h] = dxn;
                        }
                        dx0[h] = pfma(sx, bc(gxh[t + 1]), f0[h]);
                        dy0[h] = pfma(sy, bc(gyh[r]), f0[h]);
                        gr[h] = pfma(bc(um[h]), sx, pmul(bc(vm[h]), sy));
                    }
                    const bool more = t + 1 < TX && (FULL || p0 + t + 1 < nx);   // another cell in this row
                    const char* tcell = ahead(tc0, 2 * t);
                    if (!more) {
                        // the tables of the next row from here on (after the segment's last row: its own, unused)
                        row_tables(min(q + 1, q0 + nr - 1), tx0, ty0, tc0);
                    }
                    face_flux(pr + FX0 + (t + 1) * FS, qx_, lx_, xe, xv, dx0, gr, Fn);
                    load_x(more ? ahead(tx0, t + 2) : p0 > 0 ? tx0 : ahead(tx0, 1));
#pragma unroll
                    for (int h = 0; h < VPL; ++h) { dX[h] = psub(Fn[h], Fx[h]); Fx[h] = Fn[h]; }
                    face_flux(pr + FY0 + t * FS, qy_, ly_, ye, yv, dy0, gr, Fn);
                    load_y(more ? ahead(ty0, t + 1) : ty0);
#pragma unroll
                    for (int h = 0; h < VPL; ++h) { dY[h] = psub(Fn[h], Fy[t][h]); Fy[t][h] = Fn[h]; }
                    // ---- Eq. fv_h (delta form) with the equilibria of W^{k+1} (slot 1) and W^k (slot 0)
                    const T* cp = reinterpret_cast<const T*>(pr + CE0 + t * ES);
                    if (!EARLY) load_c(tcell);
                    const L ex0 = ce0, ey0 = cv0, ex1 = ce1, ey1 = cv1;
                    if (EARLY) load_c(more ? ahead(tc0, 2 * (t + 1)) : tc0);
                    L h1, b1, h0, b0;
                    if (shakhov) {
                        eq_core<true, T, L>(cp + C_EQ1, ex1, ey1, uL, vL, r2L, hL, h1, b1);
                        eq_core<true, T, L>(cp + C_EQ0, ex0, ey0, uL, vL, r2L, hL, h0, b0);
                    } else {
                        eq_core<false, T, L>(cp + C_EQ1, ex1, ey1, uL, vL, r2L, hL, h1, b1);
                        eq_core<false, T, L>(cp + C_EQ0, ex0, ey0, uL, vL, r2L, hL, h0, b0);
                    }
                    T kp[12];                                // kself, -kE, kp1, kp0, -kdx, -kdy, each twice
                    load_par(cp + C_K, kp);
#pragma unroll
                    for (int h = 0; h < VPL; ++h) {
                        V x = pmul(pk(kp[0], kp[1]), f0[h]);
                        x = pfma(bc(kp[8] * um[h]), dX[h], x);
                        x = pfma(bc(kp[10] * vm[h]), dY[h], x);
                        x = pfma(pk(kp[2], kp[3]), e[t & 1][h], x);
                        x = pfma(pk(kp[4], kp[5]), pk(A::at(h1, h), A::at(b1, h)), x);
                        x = pfma(pk(kp[6], kp[7]), pk(A::at(h0, h), A::at(b0, h)), x);
                        if (implicit) srhs[(size_t)((n * TX + t) * VPL + h) * VB + lane] = x;
                        else if (h == 0 || two) on[h * bstride + t * SG * VB] = x;
                    }
                }
                if (implicit) {
                    // spectral source at the new iterate: f^{k+1} = minv (right-hand sides over the levels), per cell
                    if (!group_meet(0)) { give_up(r + 1); return; }
#pragma unroll
                    for (int t = 0; t < TX; ++t) {
                        if (!FULL && p0 + t >= nx) break;
                        const T* Mi = cd.minv + ((size_t)(j * nx + i0 + t * SG) * nt + n) * nt;
                        V acc[VPL];
#pragma unroll
                        for (int h = 0; h < VPL; ++h) acc[h] = bc(T(0));
                        for (int m = 0; m < nt; ++m) {
                            const V w = bc(__ldg(Mi + m));
#pragma unroll
                            for (int h = 0; h < VPL; ++h)
                                acc[h] = pfma(w, srhs[(size_t)((m * TX + t) * VPL + h) * VB + lane], acc[h]);
                        }
#pragma unroll
                        for (int h = 0; h < VPL; ++h)
                            if (h == 0 || two) on[h * bstride + t * SG * VB] = acc[h];
                    }
                    if (!group_meet(1)) { give_up(r + 1); return; }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(done);
        }
    };
    if (xneg) march(std::true_type{});
    else march(std::false_type{});
}

}  // namespace hb
