// Per-velocity kernels of one HB-UGKS iteration on sign-pure velocity blocks.
//
// The discrete velocities are stored in blocks of 32 (one warp lane each) in which u and v each keep one sign
// (a zero node is stored once in each of the adjacent sign classes with its weight split between the copies).
// The upwind side of every x-face is then the same for all lanes of a block, and so is that of every y-face,
// so each cell reconstructs once per velocity block and the result serves the one x-face and the one y-face
// lying downwind of it (Sec 2.2, upwind interface reconstruction):
//   k1_cells : per (cell, level): velocity sums of the reconstruction of h^k at the cell's downwind faces,
//              kept per sign class (half-face sums), and the raw moments of h^k;
//   k4_march : per (cell, level, velocity): interface micro fluxes, spectral source and update (hb_micro.cuh).
// A CTA of k1_cells owns a tile of cells and one level and runs over all velocity blocks; a CTA of k4_march
// owns a strip of cells and one or two velocity blocks of one sign class on all levels.  Both stage
// their cells with a halo in shared memory with bulk copies (TMA) completing on an mbarrier.  The distributions
// h and b of a velocity are stored side by side and carried as one pair (hb_common.cuh): one 8-byte access
// and, in single precision, one packed FP32x2 instruction for both wherever they see the same arithmetic
// (differences, limited slopes, reconstruction, the flux combination, velocity sums with a common weight,
// spectral source and update).
#pragma once
#include "hb_common.cuh"

namespace hb {

// van Leer limiter of a pair: 2 s1 s2 / (s1 + s2) where s1 s2 > 0, else 0.  Single precision: the limited slope
// needs no correctly rounded division (approximate reciprocal, 2 ulp); double precision: rcp64_normal
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// (All products that feed a sum are written as fused ones here and in hb_micro.cuh, so that every instance of a kernel,
// whether it finds its case in a table or as a parameter, rounds alike.)
// The arguments are twice the one-sided slopes, so that the limited slope 2 s1 s2 / (s1 + s2) is their product over
// their sum.
__device__ __forceinline__ float2 vleer2(float2 s1, float2 s2)
{
    const float2 p = pmul(s1, s2);
    const float2 den = padd(s1, s2);
    const float2 q = pmul(p, make_float2(rcp_approx(den.x), rcp_approx(den.y)));
    return make_float2(p.x > 0.f ? q.x : 0.f, p.y > 0.f ? q.y : 0.f);
}
// x > 0 by integer arithmetic, off the FP64 pipe (false for NaN)
__device__ __forceinline__ bool pos64(double x)
{
    return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7ff0000000000000ull;
}
__device__ __forceinline__ double2 vleer2(double2 s1, double2 s2)
{
    const double px = s1.x * s2.x, py = s1.y * s2.y;
    // where the product is positive the sum lies above 2^-537, a normal number
    const double qx = px * rcp64_normal(__dadd_rn(s1.x, s2.x)), qy = py * rcp64_normal(__dadd_rn(s1.y, s2.y));
    return make_double2(pos64(px) ? qx : 0.0, pos64(py) ? qy : 0.0);
}

// Limited slope of (h, b) of a cell from its two neighbours along one axis, wm = 2/(x_i - x_{i-1}),
// wp = 2/(x_{i+1} - x_i) (non-uniform spacing); a missing neighbour (wall) makes the available one-sided
// difference the slope, a single cell along the axis has none
template <typename V, typename T>
__device__ __forceinline__ V slope2(V fm, V f0, V fp, T wm, T wp, bool has_m, bool has_p, bool several)
{
    V s1 = pmul(psub(f0, fm), bc(wm)), s2 = pmul(psub(fp, f0), bc(wp));
    if (!has_m) s1 = s2;
    if (!has_p) s2 = s1;
    return several ? vleer2(s1, s2) : bc(T(0));
}
// both neighbours present
template <typename V, typename T>
__device__ __forceinline__ V slope2i(V fm, V f0, V fp, T wm, T wp)
{
    return vleer2(pmul(psub(f0, fm), bc(wm)), pmul(psub(fp, f0), bc(wp)));
}

__device__ __forceinline__ void mbar_setup(uint64_t* bars, int n)
{
    if (threadIdx.x == 0) {
        for (int k = 0; k < n; ++k) mbar_init(bars + k, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
}

// Sum over the 32 lanes of each of v[0..N-1] (N <= 32), recursive halving: after the step with distance d the
// lanes with bit d set hold the upper half of the remaining values.  Returns, on lane l, the total of v[l]
// (0 for l >= N).  v is destroyed.
template <int N, typename T>
__device__ __forceinline__ T lane_totals(T (&v)[N], int lane)
{
    T x[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) x[k] = k < N ? v[k] : T(0);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const bool hi = (lane & d) != 0;
#pragma unroll
        for (int k = 0; k < d; ++k) {
            const T send = hi ? x[k] : x[k + d];
            const T keep = hi ? x[k + d] : x[k];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, send, d);
        }
    }
    return x[0];
}

// N parameters (a multiple of 4) from shared memory by 16-byte loads
template <int N>
__device__ __forceinline__ void load_par(const float* p, float (&o)[N])
{
#pragma unroll
    for (int k = 0; k < N; k += 4) {
        const float4 x = *reinterpret_cast<const float4*>(p + k);
        o[k] = x.x; o[k + 1] = x.y; o[k + 2] = x.z; o[k + 3] = x.w;
    }
}
template <int N>
__device__ __forceinline__ void load_par(const double* p, double (&o)[N])
{
#pragma unroll
    for (int k = 0; k < N; k += 2) {
        const double2 x = *reinterpret_cast<const double2*>(p + k);
        o[k] = x.x; o[k + 1] = x.y;
    }
}

// ------------------------------------------------------------------------------ K1: half-face sums

// Velocity sums of one cell's reconstruction at its downwind faces.  Slots of the 23 sums (as for an
// interface with normal n and tangent t, u_n = u.n):
//   0..9   w d0 (1, u, v, u^2, uv, v^2, u^3, u^2 v, u v^2, v^3),  d0 the reconstructed h deviation at the face
//   10..12 w e0 (1, u, v),                                         e0 the same for b
//   13..16 w s_t (1, u, v, |u|^2), 17 w s_t^b                      tangential slopes of h and b
//   18..21 w u_n (u_n s_n + u_t s_t) (1, u, v, |u|^2), 22 the same for b
// A wall face takes 0..12 and 18..22 from the velocities moving into the wall only and 13..17 from all.
// Half-face slots per (cell, level): 0 x-face of the u > 0 class (the right face), 1 u < 0 (left face),
// 2 v > 0 (top face), 3 v < 0 (bottom face).
// Every one of these sums is linear in f0, the slope s_x and the slope s_y of the cell (d0 = f0 +- h_x s_x at the
// x-face, f0 +- h_y s_y at the y-face; u_n s_n + u_t s_t = u s_x + v s_y at both), with factors that are the same for
// the whole sign class.  So a lane keeps moments of f0, s_x and s_y only and the face sums are formed from them when
// the class changes: 47 sums per velocity instead of 59 and no reconstruction (the b sums need the weights 1, u, v of
// f0; 1, u, v, u^2, uv of s_x; 1, u, v, uv, v^2 of s_y).
// With SEP the case's velocity grid has no zero node and each sign class has 1, 2, 4, 8, 16 or 32 u-nodes, so a
// lane sees the same u in every block of a class (blocks hold whole rows of the class, u fastest): every sum
// w u^a v^b d factors into w_u u^a (the lane's) times sum over the lane's velocities of w_v v^b d, and the lane
// keeps only those v-moments (20 sums: of f0 v^0..3 for h and v^0..1 for b, of s_x the same, of s_y v^0..4 and
// v^0..2), multiplying by w_u u^a when the class changes.
// Bound by FP64 instructions in FP64 (62 per velocity with SEP, the limiter's reciprocals included); in FP32 by waiting
// for the staged blocks (three times the tile's own cells pass from L2) at 56 % issue.  Against 59 sums with the
// reconstruction formed per velocity, divisions in the limiter and weights formed per lane from two loads: 36.98 ->
// 22.2 ms (twelve 64x64 cavities, 32x32 velocities, N_T 3, FP64, SEP), 18.22 -> 11.3 ms (64x64, 48x48, N_T 7, FP64),
// 4.83 -> 3.34 ms (128x128, 64x64, N_T 11, FP32, SEP), 0.543 -> 0.457 ms (64x64, 48x48, FP32).  Tiles of 4x2 cells:
// 4x4 4.11 ms, 6x4 3.96, 8x3 4.14 on the 128x128 case, whose larger CTAs wait for their slowest warp.
// Weights of a velocity block in global and shared memory, T [K1_WT]: SEP four per lane (w_v v^0..3), then w_v v^4 per
// lane; general four, four and four per lane (w times 1, u, v, uu; uv, vv, uuu, uuv; uvv, vvv, uu|u|^2, vv|u|^2), then
// w uv|u|^2 per lane.  Products formed in FP64 when the case is uploaded.
template <bool SEP> constexpr int K1_WT = SEP ? 160 : 416;

template <class P, int TX, int TY, int G, int S, bool SEP, int CTAS>
__global__ void __launch_bounds__(TX * TY * 32, CTAS) k1_cells(const __grid_constant__ P B)
{
    using T = typename P::value_type;
    using V = P2<T>;
    constexpr int PX = TX + 2, PY = TY + 2, NR = PX * PY, NWC = TX * TY;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint64_t bars[S], empty[S];
    __shared__ T sacc[NWC][4][NM];
    __shared__ int abort_flag;                               // set by the first warp whose wait runs out
    int lb;
    const CaseDev<T>& cd = B.find(blockIdx.x, lb);
    if (!cd.st->active) return;
    // another CTA may set the error word while this one starts: decide for the whole CTA at once
    if (__syncthreads_or(*(volatile int*)cd.err != 0)) return;
    const int ntx = (cd.nx + TX - 1) / TX, nty = (cd.ny + TY - 1) / TY;
    const int tx = lb % ntx, ty = (lb / ntx) % nty, n = lb / (ntx * nty);
    const int i0 = tx * TX, j0 = ty * TY;
    const int nt = cd.nt, nc = cd.nc, nx = cd.nx, ny = cd.ny, nvb = cd.nvb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ti = warp % TX, tj = warp / TX, i = i0 + ti, j = j0 + tj;
    const bool valid = i < nx && j < ny;
    for (int k = lane; k < 4 * NM; k += 32) sacc[warp][k / NM][k % NM] = T(0);
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int k = 0; k < S; ++k) mbar_init(empty + k, NWC);   // one arrival per warp: slot read
    }
    mbar_setup(bars, S);
    // staged rectangle: columns i0-1 .. i0+TX, rows j0-1 .. j0+TY; S slots of [G][NR][32] (h, b) pairs
    constexpr size_t blk = (size_t)NR * VB;
    constexpr int WT = K1_WT<SEP>;
    constexpr size_t SLOT = G * (blk * sizeof(V) + WT * sizeof(T));   // bytes: G blocks, then their weights
    const int p = cd.st->parity;
    const V* gf = cd.f[p];
    const int c0 = max(i0 - 1, 0), c1 = min(i0 + TX + 1, nx);
    const uint32_t row_b = (uint32_t)((c1 - c0) * VB * sizeof(V));
    uint32_t rbytes = 0;
    for (int r = 0; r < PY; ++r) {
        const int jj = j0 - 1 + r;
        if (jj >= 0 && jj < ny) rbytes += row_b;
    }
    // chunks of up to G blocks of one sign class (the classes occupy consecutive blocks)
    int nchunk = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) nchunk += (cd.cls_end[c] - (c ? cd.cls_end[c - 1] : 0) + G - 1) / G;
    int* err = cd.err;
    int pvb = 0, pcls = 0;                                   // next block to copy and its class (warp 0)
    auto issue = [&](int k) {
        while (pvb >= cd.cls_end[pcls]) ++pcls;
        const int gk = min(G, cd.cls_end[pcls] - pvb);
        unsigned char* dst = smem_raw + (size_t)(k % S) * SLOT;
        const uint32_t wb = (uint32_t)(gk * WT * (int)sizeof(T));
        if (lane == 0) mbar_arrive_expect(&bars[k % S], (uint32_t)gk * rbytes + wb);
        __syncwarp();
        for (int q = lane; q <= gk * PY; q += 32) {
            if (q == gk * PY) {
                bulk_g2s(dst + G * blk * sizeof(V), cd.wrow + (size_t)pvb * WT, wb, &bars[k % S]);
                break;
            }
            const int r = q % PY, g = q / PY;
            const int jj = j0 - 1 + r;
            if (jj < 0 || jj >= ny) continue;
            const size_t src = ((size_t)(pvb + g) * nt + n) * nc * VB + ((size_t)jj * nx + c0) * VB;
            bulk_g2s(dst + ((size_t)g * blk + (size_t)(r * PX + c0 - (i0 - 1)) * VB) * sizeof(V), gf + src, row_b,
                     &bars[k % S]);
        }
        __syncwarp();
        pvb += gk;
    };
    if (warp == 0)
        for (int k = 0; k < S - 1 && k < nchunk; ++k) issue(k);
    int issued = min(S - 1, nchunk);                         // chunks warp 0 has issued (kept on warp 0)
    // a wait ran out: warp 0, which issued the copies, waits (bounded) for every chunk from k on that it has not
    // seen complete, so that none still lands in shared memory after the CTA exits; the other warps just leave
    auto give_up = [&](int k) {
        if (warp == 0)
            for (int q = k; q < issued; ++q) mbar_drain(&bars[q % S], (uint32_t)((q / S) & 1));
    };

    // the warp's cell: neighbours, spacings, half widths (uniform over the warp)
    const bool hm = i > 0, hp = i < nx - 1, vm = j > 0, vp = j < ny - 1, sx = nx > 1, sy = ny > 1;
    const T wxm = valid && hm ? T(2) * T(cd.rdx[i - 1]) : T(0), wxp = valid && hp ? T(2) * T(cd.rdx[i]) : T(0);
    const T wym = valid && vm ? T(2) * T(cd.rdy[j - 1]) : T(0), wyp = valid && vp ? T(2) * T(cd.rdy[j]) : T(0);
    const T hxh = valid ? T(cd.hx[i]) : T(0), hyh = valid ? T(cd.hy[j]) : T(0);
    const bool inner = hm && hp && vm && vp;                 // every neighbour present: no wall branches
    const int kc = (tj + 1) * PX + ti + 1;
    // A sum of h and the sum of b with the same weight are kept as one pair (one packed FMA), the others of h alone:
    //   SEP      f: pairs v^0 v^1, h v^2 v^3;  x: the same;  y: pairs v^0 v^1 v^2, h v^3 v^4
    //   general  f: pairs 1 u v, h uu uv vv uuu uuv uvv vvv;  x: pairs 1 u v uu uv, h vv uuu uuv uvv vvv uu|u|^2 uv|u|^2;
    //            y: pairs 1 u v uv vv, h uu uuu uuv uvv vvv vv|u|^2 uv|u|^2;  and in wall cells the part of f0 +- h s
    //            of nodes parallel to the wall, which the wall face leaves out: zx pairs 1 v, h vv vvv; zy pairs 1 u,
    //            h uu uuu
    constexpr int NFP = SEP ? 2 : 3, NFS = SEP ? 2 : 7, NXP = SEP ? 2 : 5, NXS = SEP ? 2 : 7, NYP = SEP ? 3 : 5,
                  NYS = SEP ? 2 : 7, NZ = SEP ? 0 : 1;
    V fp_[NFP], xp[NXP], yp[NYP], zxp[2 * NZ + 1], zyp[2 * NZ + 1];
    T fs_[NFS], xs[NXS], ys[NYS], zxs[2 * NZ + 1], zys[2 * NZ + 1], ac[NCM];
    auto zero_sums = [&]() {
#pragma unroll
        for (int q = 0; q < NFP; ++q) fp_[q] = bc(T(0));
#pragma unroll
        for (int q = 0; q < NFS; ++q) fs_[q] = T(0);
#pragma unroll
        for (int q = 0; q < NXP; ++q) xp[q] = bc(T(0));
#pragma unroll
        for (int q = 0; q < NXS; ++q) xs[q] = T(0);
#pragma unroll
        for (int q = 0; q < NYP; ++q) yp[q] = bc(T(0));
#pragma unroll
        for (int q = 0; q < NYS; ++q) ys[q] = T(0);
#pragma unroll
        for (int q = 0; q < 2 * NZ; ++q) { zxp[q] = bc(T(0)); zyp[q] = bc(T(0)); zxs[q] = T(0); zys[q] = T(0); }
    };
    zero_sums();
#pragma unroll
    for (int q = 0; q < NCM; ++q) ac[q] = T(0);
    int cur = 0;                                             // current sign class
    T ul = T(0), wul = T(0);                                 // SEP: the lane's u and w_u in the current class
    // the 23 face sums of one face from its v-moments (SEP): D, DB of d0 and e0, S, SB tangential slopes, N, NB normal
    auto unfold = [&](const T (&D)[4], const T (&DB)[2], const T (&S_)[3], T SB, const T (&N)[3], T NB, T (&o)[NM]) {
        const T w1 = wul, w2 = w1 * ul, w3 = w2 * ul, w4 = w3 * ul;     // w_u u^a
        o[0] = w1 * D[0]; o[1] = w2 * D[0]; o[2] = w1 * D[1]; o[3] = w3 * D[0]; o[4] = w2 * D[1];
        o[5] = w1 * D[2]; o[6] = w4 * D[0]; o[7] = w3 * D[1]; o[8] = w2 * D[2]; o[9] = w1 * D[3];
        o[10] = w1 * DB[0]; o[11] = w2 * DB[0]; o[12] = w1 * DB[1];
        o[13] = w1 * S_[0]; o[14] = w2 * S_[0]; o[15] = w1 * S_[1]; o[16] = pfma(w3, S_[0], w1 * S_[2]);
        o[17] = w1 * SB;
        o[18] = w1 * N[0]; o[19] = w2 * N[0]; o[20] = w1 * N[1]; o[21] = pfma(w3, N[0], w1 * N[2]);
        o[22] = w1 * NB;
    };
    // add the sums of the current sign class to its two half-face slots and to the cell's moments
    auto flush = [&]() {
        const T sx_ = (cur & 1) ? -hxh : hxh, sy_ = (cur & 2) ? -hyh : hyh;
        T ox[NM], oy[NM];
        if constexpr (SEP) {
            const T F[4] = {fp_[0].x, fp_[1].x, fs_[0], fs_[1]}, FB[2] = {fp_[0].y, fp_[1].y};
            const T X[4] = {xp[0].x, xp[1].x, xs[0], xs[1]}, XB[2] = {xp[0].y, xp[1].y};
            const T Y[5] = {yp[0].x, yp[1].x, yp[2].x, ys[0], ys[1]}, YB[3] = {yp[0].y, yp[1].y, yp[2].y};
            T D[4], DB[2], S_[3], N[3];
#pragma unroll
            for (int q = 0; q < 4; ++q) D[q] = pfma(sx_, X[q], F[q]);
#pragma unroll
            for (int q = 0; q < 2; ++q) DB[q] = pfma(sx_, XB[q], FB[q]);
#pragma unroll
            for (int q = 0; q < 3; ++q) { S_[q] = Y[q]; N[q] = ul * pfma(ul, X[q], Y[q + 1]); }
            unfold(D, DB, S_, YB[0], N, ul * pfma(ul, XB[0], YB[1]), ox);
#pragma unroll
            for (int q = 0; q < 4; ++q) D[q] = pfma(sy_, Y[q], F[q]);
#pragma unroll
            for (int q = 0; q < 2; ++q) DB[q] = pfma(sy_, YB[q], FB[q]);
#pragma unroll
            for (int q = 0; q < 3; ++q) { S_[q] = X[q]; N[q] = pfma(ul, X[q + 1], Y[q + 2]); }
            unfold(D, DB, S_, XB[0], N, pfma(ul, XB[1], YB[2]), oy);
            const T w1 = wul, w2 = w1 * ul, w3 = w2 * ul, w4 = w3 * ul;
            ac[0] = pfma(w1, F[0], ac[0]); ac[1] = pfma(w2, F[0], ac[1]); ac[2] = pfma(w1, F[1], ac[2]); ac[3] = pfma(w3, F[0], ac[3]);
            ac[4] = pfma(w2, F[1], ac[4]); ac[5] = pfma(w1, F[2], ac[5]); ac[6] = pfma(w4, F[0], ac[6]); ac[7] = pfma(w3, F[1], ac[7]);
            ac[8] = pfma(w2, F[2], ac[8]); ac[9] = pfma(w1, F[3], ac[9]);
            ac[10] = pfma(w1, FB[0], ac[10]); ac[11] = pfma(w2, FB[0], ac[11]); ac[12] = pfma(w1, FB[1], ac[12]);
        } else {
            // monomials 1, u, v, uu, uv, vv, uuu, uuv, uvv, vvv
            const T F[10] = {fp_[0].x, fp_[1].x, fp_[2].x, fs_[0], fs_[1], fs_[2], fs_[3], fs_[4], fs_[5], fs_[6]};
            const T X[10] = {xp[0].x, xp[1].x, xp[2].x, xp[3].x, xp[4].x, xs[0], xs[1], xs[2], xs[3], xs[4]};
            const T Y[10] = {yp[0].x, yp[1].x, yp[2].x, ys[0], yp[3].x, yp[4].x, ys[1], ys[2], ys[3], ys[4]};
#pragma unroll
            for (int q = 0; q < 10; ++q) {
                ox[q] = pfma(sx_, X[q], F[q]);
                oy[q] = pfma(sy_, Y[q], F[q]);
                ac[q] += F[q];
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                ox[10 + q] = pfma(sx_, xp[q].y, fp_[q].y);
                oy[10 + q] = pfma(sy_, yp[q].y, fp_[q].y);
                ac[10 + q] += fp_[q].y;
                ox[13 + q] = Y[q];
                oy[13 + q] = X[q];
            }
            ox[16] = Y[3] + Y[5]; ox[17] = yp[0].y;
            oy[16] = X[3] + X[5]; oy[17] = xp[0].y;
            ox[18] = X[3] + Y[4]; ox[19] = X[6] + Y[7]; ox[20] = X[7] + Y[8]; ox[21] = xs[5] + ys[6];
            ox[22] = xp[3].y + yp[3].y;
            oy[18] = X[4] + Y[5]; oy[19] = X[7] + Y[8]; oy[20] = X[8] + Y[9]; oy[21] = xs[6] + ys[5];
            oy[22] = xp[4].y + yp[4].y;
            ox[0] -= zxp[0].x; ox[2] -= zxp[1].x; ox[5] -= zxs[0]; ox[9] -= zxs[1]; ox[10] -= zxp[0].y; ox[12] -= zxp[1].y;
            oy[0] -= zyp[0].x; oy[1] -= zyp[1].x; oy[3] -= zys[0]; oy[6] -= zys[1]; oy[10] -= zyp[0].y; oy[11] -= zyp[1].y;
        }
        const T tx_ = lane_totals<NM>(ox, lane), ty_ = lane_totals<NM>(oy, lane);
        if (lane < NM) {
            sacc[warp][(cur & 1) ? 1 : 0][lane] += tx_;
            sacc[warp][(cur & 2) ? 3 : 2][lane] += ty_;
        }
        zero_sums();
    };

    // Ring of S slots: chunk k lands in slot k % S (mbarrier bars); each warp arrives on empty once it has
    // read the slot, and warp 0 refills a slot only after every warp has released it, so warps run up to
    // S - 1 chunks apart instead of meeting at a CTA barrier per chunk.
    [[maybe_unused]] V* const slo =
        cd.sl ? cd.sl + ((size_t)n * nc + (valid ? j * nx + i : 0)) * 2 * VB + lane : nullptr;
    [[maybe_unused]] const size_t slstride = (size_t)nt * nc * 2 * VB;
    int k = 0, slot = 0, vb = 0;                             // chunk, its slot, its first block
    uint32_t ph = 0;                                         // phase of the slot's barrier
    for (cur = 0; cur < 4; ++cur) {
        const int vend = cd.cls_end[cur];
        if (vb >= vend) continue;
        if (SEP) {
            ul = __ldg(cd.tu + vb * VB + lane);
            wul = __ldg(cd.twu + vb * VB + lane);
        }
        for (; vb < vend; vb += G, ++k) {
            if (warp == 0 && k + S - 1 < nchunk) {
                const int kk = k + S - 1;
                if (kk >= S && !mbar_wait(&empty[kk % S], (uint32_t)((kk / S - 1) & 1), err, &abort_flag)) {
                    give_up(k);
                    return;
                }
                issue(kk);
                issued = kk + 1;
            }
            if (!mbar_wait(&bars[slot], ph, err, &abort_flag)) {
                give_up(k);
                return;
            }
            const unsigned char* cb = smem_raw + (size_t)slot * SLOT;
            const int gk = min(G, vend - vb);
            // one block of the chunk; INNER: every neighbour of the warp's cell exists (no wall branches)
            auto block = [&](auto inner_tag, int g, const V* pc, const T* wp) {
                constexpr bool INNER = decltype(inner_tag)::value;
                const V f0 = pc[0];
                V sxv, syv;
                if constexpr (INNER) {
                    sxv = slope2i(pc[-VB], f0, pc[VB], wxm, wxp);
                    syv = slope2i(pc[-PX * VB], f0, pc[PX * VB], wym, wyp);
                } else {
                    sxv = slope2(pc[-VB], f0, pc[VB], wxm, wxp, hm, hp, sx);
                    syv = slope2(pc[-PX * VB], f0, pc[PX * VB], wym, wyp, vm, vp, sy);
                }
                if constexpr (sizeof(T) == 8) {
                    // kept for the micro update, which would spend a quarter of its FP64 instructions on them again
                    if (slo) {
                        V* o = slo + (size_t)(vb + g) * slstride;
                        o[0] = sxv;
                        o[VB] = syv;
                    }
                }
                T a[4];
                load_par(wp + lane * 4, a);
                if constexpr (SEP) {
                    const T c4 = wp[4 * VB + lane];
                    const V bw = bc(a[0]), bc1 = bc(a[1]);
                    fp_[0] = pfma(f0, bw, fp_[0]); fp_[1] = pfma(f0, bc1, fp_[1]);
                    xp[0] = pfma(sxv, bw, xp[0]); xp[1] = pfma(sxv, bc1, xp[1]);
                    yp[0] = pfma(syv, bw, yp[0]); yp[1] = pfma(syv, bc1, yp[1]); yp[2] = pfma(syv, bc(a[2]), yp[2]);
                    fs_[0] = pfma(f0.x, a[2], fs_[0]); fs_[1] = pfma(f0.x, a[3], fs_[1]);
                    xs[0] = pfma(sxv.x, a[2], xs[0]); xs[1] = pfma(sxv.x, a[3], xs[1]);
                    ys[0] = pfma(syv.x, a[3], ys[0]); ys[1] = pfma(syv.x, c4, ys[1]);
                } else {
                    T d[4], e[4];                            // a: 1 u v uu, d: uv vv uuu uuv, e: uvv vvv uu|u|^2 vv|u|^2
                    load_par(wp + 4 * VB + lane * 4, d);
                    load_par(wp + 8 * VB + lane * 4, e);
                    const T wr = wp[12 * VB + lane];
                    const V bw = bc(a[0]), bu = bc(a[1]), bv = bc(a[2]), buv = bc(d[0]);
                    fp_[0] = pfma(f0, bw, fp_[0]); fp_[1] = pfma(f0, bu, fp_[1]); fp_[2] = pfma(f0, bv, fp_[2]);
                    xp[0] = pfma(sxv, bw, xp[0]); xp[1] = pfma(sxv, bu, xp[1]); xp[2] = pfma(sxv, bv, xp[2]);
                    xp[3] = pfma(sxv, bc(a[3]), xp[3]); xp[4] = pfma(sxv, buv, xp[4]);
                    yp[0] = pfma(syv, bw, yp[0]); yp[1] = pfma(syv, bu, yp[1]); yp[2] = pfma(syv, bv, yp[2]);
                    yp[3] = pfma(syv, buv, yp[3]); yp[4] = pfma(syv, bc(d[1]), yp[4]);
                    fs_[0] = pfma(f0.x, a[3], fs_[0]); fs_[1] = pfma(f0.x, d[0], fs_[1]); fs_[2] = pfma(f0.x, d[1], fs_[2]); fs_[3] = pfma(f0.x, d[2], fs_[3]);
                    fs_[4] = pfma(f0.x, d[3], fs_[4]); fs_[5] = pfma(f0.x, e[0], fs_[5]); fs_[6] = pfma(f0.x, e[1], fs_[6]);
                    xs[0] = pfma(sxv.x, d[1], xs[0]); xs[1] = pfma(sxv.x, d[2], xs[1]); xs[2] = pfma(sxv.x, d[3], xs[2]); xs[3] = pfma(sxv.x, e[0], xs[3]);
                    xs[4] = pfma(sxv.x, e[1], xs[4]); xs[5] = pfma(sxv.x, e[2], xs[5]); xs[6] = pfma(sxv.x, wr, xs[6]);
                    ys[0] = pfma(syv.x, a[3], ys[0]); ys[1] = pfma(syv.x, d[2], ys[1]); ys[2] = pfma(syv.x, d[3], ys[2]); ys[3] = pfma(syv.x, e[0], ys[3]);
                    ys[4] = pfma(syv.x, e[1], ys[4]); ys[5] = pfma(syv.x, e[3], ys[5]); ys[6] = pfma(syv.x, wr, ys[6]);
                    if constexpr (!INNER) {
                        // a velocity parallel to a wall (u w = 0; not u^2 w, which a small u brings below the smallest
                        // 32-bit value) carries nothing into it
                        const bool xn = (cur & 1) != 0, yn = (cur & 2) != 0;
                        if ((xn ? !hm : !hp) && a[1] == T(0)) {
                            const V z = pfma(sxv, bc(xn ? -hxh : hxh), f0);
                            zxp[0] = pfma(z, bw, zxp[0]); zxp[1] = pfma(z, bv, zxp[1]);
                            zxs[0] = pfma(z.x, d[1], zxs[0]); zxs[1] = pfma(z.x, e[1], zxs[1]);
                        }
                        if ((yn ? !vm : !vp) && a[2] == T(0)) {
                            const V z = pfma(syv, bc(yn ? -hyh : hyh), f0);
                            zyp[0] = pfma(z, bw, zyp[0]); zyp[1] = pfma(z, bu, zyp[1]);
                            zys[0] = pfma(z.x, a[3], zys[0]); zys[1] = pfma(z.x, d[2], zys[1]);
                        }
                    }
                }
            };
            auto run_blocks = [&](auto inner_tag) {
                const V* pc = reinterpret_cast<const V*>(cb) + (size_t)kc * VB + lane;
                const T* wp = reinterpret_cast<const T*>(cb + G * blk * sizeof(V));
                if (gk == G) {
#pragma unroll
                    for (int g = 0; g < G; ++g) block(inner_tag, g, pc + g * blk, wp + g * WT);
                } else {
                    for (int g = 0; g < gk; ++g) block(inner_tag, g, pc + g * blk, wp + g * WT);
                }
            };
            if (valid) {
                if (inner) run_blocks(std::true_type{});
                else run_blocks(std::false_type{});
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[slot]);
            if (++slot == S) { slot = 0; ph ^= 1; }
        }
        vb = vend;
        if (valid) flush();
    }
    if (!valid) return;
    const T cm = lane_totals<NCM>(ac, lane);
    __syncwarp();
    const int c = j * nx + i;
    if (lane < NCM) cd.cmom[((size_t)c * nt + n) * NCM + lane] = (double)cm;
    double* hmo = cd.hmom + ((size_t)c * nt + n) * 4 * NM;
    for (int k = lane; k < 4 * NM; k += 32) hmo[k] = (double)sacc[warp][k / NM][k % NM];
}

template <typename T, int TX, int TY, int G, int S, bool SEP>
constexpr size_t k1_cells_smem()
{
    return (size_t)S * G * ((TX + 2) * (TY + 2) * VB * sizeof(P2<T>) + K1_WT<SEP> * sizeof(T));
}

}  // namespace hb
