// Matrix-free operators on the grid:
//  - B x (Eq. Bdec): the regular 27-point compact stencil of Eqs. A27/As_qs
//    rebuilt on the fly from the 1D metrics, sum-factorised as
//      A x = sum_r Lz[r] (sum_q Ly[q] XR + Ry[q] XL) + Rz[r] (sum_q Ly[q] XL),
//      XR = sum_p Rx[p] x,  XL = sum_p Lx[p] x,
//    with the y-pass results of three planes kept in registers while a thread
//    (FP64, most FP32 grids) or a shared-memory ring's consumer (large FP32
//    grids whose width fills its tiles) marches in z; the rows of irregular
//    points, with their modified-stencil corrections, in a kernel beside it;
//    solid rows are zero.
//  - the right-hand side of Eq. Bu=q and helpers of the solves.
#include <algorithm>

#include "cfp_internal.cuh"
#include "cfp_tc.cuh"

namespace cfp {

template <>
Grid<double> grid_view<double>(cfp_ctx* c) {
    Grid<double> g;
    int64_t off = 0;
    for (int d = 0; d < 3; ++d) {
        const int n = c->n[d];
        double* b = c->dcoef64 + off;
        g.ax[d] = Axis<double>{b, b + n, b + 2 * n, b + 3 * n, b + 4 * n, b + 5 * n, b + 6 * n, b + 7 * n};
        off += 8 * (int64_t)n;
    }
    g.nx = c->n[0];
    g.ny = c->n[1];
    g.nz = c->n[2];
    return g;
}

template <>
Grid<float> grid_view<float>(cfp_ctx* c) {
    Grid<float> g;
    int64_t off = 0;
    for (int d = 0; d < 3; ++d) {
        const int n = c->n[d];
        float* b = c->dcoef32 + off;
        g.ax[d] = Axis<float>{b, b + n, b + 2 * n, b + 3 * n, b + 4 * n, b + 5 * n, b + 6 * n, b + 7 * n};
        off += 8 * (int64_t)n;
    }
    g.nx = c->n[0];
    g.ny = c->n[1];
    g.nz = c->n[2];
    return g;
}

template <>
Side<double> side_view<double>(cfp_ctx* c) {
    return Side<double>{c->slot, c->corr_ptr, c->corr_off, c->corr_val, c->krow};
}

template <>
Side<float> side_view<float>(cfp_ctx* c) {
    return Side<float>{c->slot, c->corr_ptr, c->corr_off, c->corr_val32, c->krow32};
}

namespace {

__device__ __forceinline__ void block_reduce2(double& a, double& b) {
    __shared__ double sa[32], sb[32];
    const int tid = threadIdx.x + blockDim.x * threadIdx.y;
    const int lane = tid & 31, wid = tid >> 5;
    for (int o = 16; o; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
        sa[wid] = a;
        sb[wid] = b;
    }
    __syncthreads();
    const int nw = (blockDim.x * blockDim.y) >> 5;
    if (wid == 0) {
        a = lane < nw ? sa[lane] : 0.0;
        b = lane < nw ? sb[lane] : 0.0;
        for (int o = 16; o; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
    }
}

// Fused multiply-add in either precision: the apply's sums are written as
// explicit chains so that every kernel and tile shape rounds each row the same
// way.
__device__ __forceinline__ float fmat(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmat(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mult(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mult(double a, double b) { return __dmul_rn(a, b); }

// Packed FP32 pairs: one fma.rn.f32x2 instruction does the (IEEE,
// round-to-nearest) arithmetic of both halves (two rows of a streaming thread,
// two columns of a ring consumer), with the results of two scalar fmaf calls.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 f2b(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// DotAcc<float> on both halves at once: a running sum and its lost
// low-order part per half, the latter kept negated (cn = -c), so that no
// step needs a negation: v = x y - c = fma(x, y, cn); t = s + v; the new
// c = (t - s) - v, that is cn = (s - t) + v, with s - t formed exactly as
// fma(t, -1, s).  Round-to-nearest is symmetric, so every value is the
// negation of the plain form's, bit for bit.
struct DotAcc2 {
    float2 s = {0.f, 0.f}, cn = {0.f, 0.f};
    __device__ __forceinline__ void add(float2 x, float2 y) {
        const float2 v = fma2(x, y, cn);
        const float2 t = add2(s, v);
        cn = add2(fma2(t, make_float2(-1.f, -1.f), s), v);
        s = t;
    }
    __device__ __forceinline__ double total() const {
        return ((double)s.x + (double)cn.x) + ((double)s.y + (double)cn.y);
    }
};

// Regular part of B x at the unknowns in FP32 (the streaming kernel; the ring
// below takes large grids that fill its tiles).  A warp is 32 columns x TY
// consecutive rows (a lane each) and marches the planes k0 .. k1 - 1 of its z
// chunk (kc planes, at most kMaxPlanes); a CTA is four warps, one above the
// other in y.
// Per plane a thread loads the values x(i-1..i+1, j) of the rows j0-1 .. j0+TY
// (the x and y neighbours come from L1/L2; the loads of the next plane are
// issued once the x pass has used this one's), forms the x-pass XR = Rx x,
// XL = Lx x of those rows (each shared by up to three output rows), the y-pass
// P = Ly XR + Ry XL, Q = Ly XL of its rows, and keeps P, Q of three planes in
// registers for the z-pass
//   out(k) = Lz (P(k-1), P(k), P(k+1)) + Rz (Q(k-1), Q(k), Q(k+1)).
// Rows t and t + TY / 2 are the halves of packed instructions.  The kernel is
// bound by the latency of the loads (long scoreboard 6.3 cycles per issue, 20 %
// of the L1 and DRAM rates at 321 x 257 x 289), so each lane also asks L2 for 32
// bytes of the rows kAhead planes on: 513^3 460 -> 390 us.  With the dot: 385^3
// 224 -> 181 us, 129^3 16.6 -> 12.4, 33^3 9.7 -> 6.2 against one column of 2
// rows x 64 planes per thread, scalar, in CTAs of 128 columns.  No barriers in
// the march; the z coefficients of the chunk are staged in shared memory once,
// each twice.  Solid rows are zero; the rows of
// irregular points are left to k_apply_irr, which runs beside this kernel on
// a second stream.  (Gathering the corrections inside this kernel, at each plane or
// from a per-warp list after the march, measured 1.57x slower at 513^3: the
// dependent side-list loads stall the streaming march, and the CTAs near the
// bodies become the tail.)
// DOT = 0: y only; 1: partial (d0, y); 2: partials (d0, y) and (y, y).
constexpr int kMaxPlanes = 64;
constexpr int kA32Warps = 4;
constexpr int kAhead = 3;  // planes; 5: 0 to 3 % slower

// the pairs (row p, row p + NP), p = 0 .. NP + 1, of the 2 NP + 2 rows a thread
// holds, from the NP + 1 distinct ones: d[0 .. NP - 1] those, d[NP] the last two rows
template <int NP>
__device__ __forceinline__ void row_pairs(const float2 (&d)[NP + 1], float2 (&w)[NP + 2]) {
#pragma unroll
    for (int p = 0; p < NP; ++p) w[p] = d[p];
    w[NP] = f2(d[0].y, d[NP].x);
    w[NP + 1] = f2(NP == 1 ? d[1].x : d[NP - 1].y, d[NP].y);
}

template <int DOT, int TY>
__global__ void __launch_bounds__(32 * kA32Warps, TY == 4 ? 4 : 6)
    k_apply32(Grid<float> G, const uint8_t* __restrict__ type, const float* __restrict__ x, float* __restrict__ y,
              const float* __restrict__ d0, double* __restrict__ partial, int kc) {
    constexpr int NP = TY / 2;
    constexpr int R = TY + 2;  // rows loaded per plane
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int i = 1 + blockIdx.x * 32 + threadIdx.x;
    const int j0 = 1 + (blockIdx.y * kA32Warps + threadIdx.y) * TY;
    const int k0 = 1 + blockIdx.z * kc;
    const int k1 = min(k0 + kc, nz - 1);
    // z coefficients of the chunk's output planes k0 .. k1 - 1: a, c, ar, br, cr twice each, two unused
    __shared__ float4 zc[3 * kMaxPlanes];
    for (int q = threadIdx.x + 32 * threadIdx.y; q < k1 - k0; q += 32 * kA32Warps) {
        const int k = k0 + q;
        const float a = G.ax[2].a[k], c = G.ax[2].c[k], ar = G.ax[2].ar[k], br = G.ax[2].br[k], cr = G.ax[2].cr[k];
        zc[3 * q] = make_float4(a, a, c, c);
        zc[3 * q + 1] = make_float4(ar, ar, br, br);
        zc[3 * q + 2] = make_float4(cr, cr, 0.f, 0.f);
    }
    __syncthreads();
    DotAcc2 dacc0, dacc1;
    if (j0 <= ny - 2) {
        const bool iin = i <= nx - 2;
        const int ic = iin ? i : 1;  // clamped: every load stays inside the grid
        // node offsets fit in 32 bits: contexts hold fewer than 2^31 nodes
        const unsigned sy = (unsigned)nx, sz = (unsigned)nx * (unsigned)ny;
        const float2 ax = f2b(G.ax[0].a[ic]), cx = f2b(G.ax[0].c[ic]);
        const float2 arx = f2b(G.ax[0].ar[ic]), brx = f2b(G.ax[0].br[ic]), crx = f2b(G.ax[0].cr[ic]);
        float2 ay[NP], cy[NP], ary[NP], bry[NP], cry[NP];
        bool ok[TY];
        unsigned l[TY];  // the output nodes of the step's plane
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const int ja = min(j0 + q, ny - 2), jb = min(j0 + q + NP, ny - 2);
            ay[q] = f2(G.ax[1].a[ja], G.ax[1].a[jb]);
            cy[q] = f2(G.ax[1].c[ja], G.ax[1].c[jb]);
            ary[q] = f2(G.ax[1].ar[ja], G.ax[1].ar[jb]);
            bry[q] = f2(G.ax[1].br[ja], G.ax[1].br[jb]);
            cry[q] = f2(G.ax[1].cr[ja], G.ax[1].cr[jb]);
        }
#pragma unroll
        for (int t = 0; t < TY; ++t) {
            ok[t] = iin && j0 + t <= ny - 2;
            l[t] = (unsigned)(k0 - 2) * sz + (unsigned)min(j0 + t, ny - 2) * sy + (unsigned)ic;
        }
        unsigned roff[R];
#pragma unroll
        for (int r = 0; r < R; ++r) roff[r] = (unsigned)min(j0 - 1 + r, ny - 1) * sy;
        const float* p = x + ((unsigned)(k0 - 1) * sz + (unsigned)ic);
        float n[3 * R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float* q = p + roff[r];
            n[3 * r] = q[-1];
            n[3 * r + 1] = q[0];
            n[3 * r + 2] = q[1];
        }
        // what this lane fetches into L2 ahead of the warp's loads: 32 bytes of one of its rows of x
        // (lanes 8 t .. 8 t + 3), d0 (8 t + 4 .. 8 t + 7) or, second, of type (lane t)
        const int pt = threadIdx.x >> 3, pc = (int)blockIdx.x * 32 + 1 + 8 * (int)(threadIdx.x & 3);
        const bool pd = threadIdx.x & 4;
        const bool pin = pt < TY && (DOT || !pd) && j0 + pt <= ny - 2 && pc <= nx - 2;
        const float* pf = (DOT && pd ? d0 : x) + ((unsigned)(k0 - 1 + kAhead) * sz +
                                                  (unsigned)min(j0 + pt, ny - 2) * sy + (unsigned)pc);
        const bool tin = threadIdx.x < TY && j0 + (int)threadIdx.x <= ny - 2;
        const uint8_t* tf = type + ((unsigned)(k0 - 1 + kAhead) * sz +
                                    (unsigned)min(j0 + (int)threadIdx.x, ny - 2) * sy + blockIdx.x * 32 + 1);
        float2 Pm[NP], P0[NP], Pp[NP], Qm[NP], Q0[NP], Qp[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) Pm[q] = P0[q] = Pp[q] = Qm[q] = Q0[q] = Qp[q] = f2b(0.f);
#pragma unroll 1
        for (int kk = k0 - 1; kk <= k1; ++kk) {
            // the output plane is kk - 1, from step k0 + 1 on
            uint8_t ty[TY];
            float d[TY];
            if (kk > k0) {
#pragma unroll
                for (int t = 0; t < TY; ++t) {
                    ty[t] = type[l[t]];
                    d[t] = DOT ? d0[l[t]] : 0.f;
                }
            }
            float2 XR[NP + 2], XL[NP + 2];
            {
                float2 xr[NP + 1], xl[NP + 1];
#pragma unroll
                for (int q = 0; q <= NP; ++q) {
                    const int ra = q < NP ? q : 2 * NP, rb = q < NP ? q + NP : 2 * NP + 1;
                    const float2 m = f2(n[3 * ra], n[3 * rb]), o = f2(n[3 * ra + 1], n[3 * rb + 1]),
                                 u = f2(n[3 * ra + 2], n[3 * rb + 2]);
                    xr[q] = fma2(crx, u, fma2(brx, o, mul2(arx, m)));
                    xl[q] = fma2(cx, u, fma2(ax, m, o));
                }
                row_pairs<NP>(xr, XR);
                row_pairs<NP>(xl, XL);
            }
            if (kk + kAhead <= k1) {
                if (pin) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf));
                if (tin) asm volatile("prefetch.global.L2 [%0];" ::"l"(tf));
                pf += sz;
                tf += sz;
            }
            if (kk < k1) {  // the next plane's loads, ahead of the y and z passes
                p += sz;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float* q = p + roff[r];
                    n[3 * r] = q[-1];
                    n[3 * r + 1] = q[0];
                    n[3 * r + 2] = q[1];
                }
            }
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                Pm[q] = P0[q];
                P0[q] = Pp[q];
                Qm[q] = Q0[q];
                Q0[q] = Qp[q];
                Pp[q] = fma2(cry[q], XL[q + 2],
                             fma2(bry[q], XL[q + 1],
                                  fma2(ary[q], XL[q], fma2(cy[q], XR[q + 2], fma2(ay[q], XR[q], XR[q + 1])))));
                Qp[q] = fma2(cy[q], XL[q + 2], fma2(ay[q], XL[q], XL[q + 1]));
            }
            if (kk > k0) {
                const float4 z0 = zc[3 * (kk - 1 - k0)], z1 = zc[3 * (kk - 1 - k0) + 1], z2 = zc[3 * (kk - 1 - k0) + 2];
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    float2 v = add2(fma2(f2(z0.z, z0.w), Pp[q], fma2(f2(z0.x, z0.y), Pm[q], P0[q])),
                                    fma2(f2(z2.x, z2.y), Qp[q], fma2(f2(z1.z, z1.w), Q0[q], mul2(f2(z1.x, z1.y), Qm[q]))));
                    const int ta = q, tb = q + NP;
                    // solid rows are zero; irregular rows belong to k_apply_irr
                    v = f2(ok[ta] && ty[ta] == CFP_REGULAR ? v.x : 0.f, ok[tb] && ty[tb] == CFP_REGULAR ? v.y : 0.f);
                    if (ok[ta] && ty[ta] != CFP_IRREGULAR) y[l[ta]] = v.x;
                    if (ok[tb] && ty[tb] != CFP_IRREGULAR) y[l[tb]] = v.y;
                    if (DOT >= 1) dacc0.add(f2(ok[ta] ? d[ta] : 0.f, ok[tb] ? d[tb] : 0.f), v);
                    if (DOT == 2) dacc1.add(v, v);
                }
            }
#pragma unroll
            for (int t = 0; t < TY; ++t) l[t] += sz;
        }
    }
    if (DOT) {
        double acc0 = dacc0.total(), acc1 = dacc1.total();
        block_reduce2(acc0, acc1);
        if (threadIdx.x == 0 && threadIdx.y == 0) {
            const int64_t b = blockIdx.x + (int64_t)gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
            partial[2 * b] = acc0;
            partial[2 * b + 1] = acc1;
        }
    }
}

// The FP64 apply.  GB300 issues about two FP64 instructions per SM and clock,
// so the kernel is bound by their number (20.5 per node with four rows to a
// thread: 5 per loaded row, 7 and 6 per output in y and z), not by memory.
// (Folding the x operator's centre weight into the y weights would save one
// per loaded row, and one chain for the z pass one per output, but both round
// worse: 1.4 to 2.3 times the error on smooth fields of stretched grids for
// the first.)
// A warp is 32 columns x TY rows and marches its own z chunk of kc planes:
// no lane beyond the row's last 32-column tile, and small grids still spread
// over the SMs (apply64_shape; a CTA is four warps, one above the other in y).
// Before: 128-column CTAs of 4 x 64 columns x planes at every
// size.  With the irregular rows and the dot: 33^3 98 -> 8 us, 97 x 65 x 82
// 194 -> 36 us, 129^3 199 -> 110 us; 513^3 is as before (5.0 ms).
// DOT, solid and irregular rows as in k_apply32.
constexpr int kA64Warps = 4;

template <int DOT, int TY>
__global__ void __launch_bounds__(32 * kA64Warps, TY == 4 ? 3 : 4)
    k_apply64(Grid<double> G, const uint8_t* __restrict__ type, const double* __restrict__ x, double* __restrict__ y,
              const double* __restrict__ d0, double* __restrict__ partial, int kc) {
    constexpr int R = TY + 2;  // rows loaded per plane
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int i = 1 + blockIdx.x * 32 + threadIdx.x;
    const int j0 = 1 + (blockIdx.y * kA64Warps + threadIdx.y) * TY;
    const int k0 = 1 + blockIdx.z * kc;
    const int k1 = min(k0 + kc, nz - 1);
    double acc0 = 0.0, acc1 = 0.0;
    if (j0 <= ny - 2) {
        const bool iin = i <= nx - 2;
        const int ic = iin ? i : 1;  // clamped: every load stays inside the grid
        const unsigned sy = (unsigned)nx, sz = (unsigned)nx * (unsigned)ny;
        const double ax = G.ax[0].a[ic], cx = G.ax[0].c[ic];
        const double arx = G.ax[0].ar[ic], brx = G.ax[0].br[ic], crx = G.ax[0].cr[ic];
        double ay[TY], cy[TY], ary[TY], bry[TY], cry[TY];
        bool jin[TY];
        unsigned lout0[TY];
#pragma unroll
        for (int t = 0; t < TY; ++t) {
            jin[t] = j0 + t <= ny - 2;
            const int jc = jin[t] ? j0 + t : j0;
            ay[t] = G.ax[1].a[jc];
            cy[t] = G.ax[1].c[jc];
            ary[t] = G.ax[1].ar[jc];
            bry[t] = G.ax[1].br[jc];
            cry[t] = G.ax[1].cr[jc];
            lout0[t] = (unsigned)k0 * sz + (unsigned)jc * sy + (unsigned)ic;
        }
        unsigned roff[R];
#pragma unroll
        for (int r = 0; r < R; ++r) roff[r] = (unsigned)min(j0 - 1 + r, ny - 1) * sy;
        const double* p = x + ((unsigned)(k0 - 1) * sz + (unsigned)ic);
        double n[3 * R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double* q = p + roff[r];
            n[3 * r] = q[-1];
            n[3 * r + 1] = q[0];
            n[3 * r + 2] = q[1];
        }
        double Pm[TY], P0[TY], Pp[TY], Qm[TY], Q0[TY], Qp[TY];
#pragma unroll
        for (int t = 0; t < TY; ++t) Pm[t] = P0[t] = Pp[t] = Qm[t] = Q0[t] = Qp[t] = 0.0;
#pragma unroll 1
        for (int kk = k0 - 1; kk <= k1; ++kk) {
            double XR[R], XL[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                XR[r] = fmat(crx, n[3 * r + 2], fmat(brx, n[3 * r + 1], mult(arx, n[3 * r])));
                XL[r] = fmat(cx, n[3 * r + 2], fmat(ax, n[3 * r], n[3 * r + 1]));
            }
            if (kk < k1) {  // the next plane's loads, ahead of the y and z passes
                p += sz;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const double* q = p + roff[r];
                    n[3 * r] = q[-1];
                    n[3 * r + 1] = q[0];
                    n[3 * r + 2] = q[1];
                }
            }
#pragma unroll
            for (int t = 0; t < TY; ++t) {
                Pm[t] = P0[t];
                P0[t] = Pp[t];
                Qm[t] = Q0[t];
                Q0[t] = Qp[t];
                Pp[t] = fmat(cry[t], XL[t + 2],
                             fmat(bry[t], XL[t + 1],
                                  fmat(ary[t], XL[t], fmat(cy[t], XR[t + 2], fmat(ay[t], XR[t], XR[t + 1])))));
                Qp[t] = fmat(cy[t], XL[t + 2], fmat(ay[t], XL[t], XL[t + 1]));
            }
            if (kk >= k0 + 1) {
                const int k = kk - 1;
                const double az = G.ax[2].a[k], cz = G.ax[2].c[k];
                const double arz = G.ax[2].ar[k], brz = G.ax[2].br[k], crz = G.ax[2].cr[k];
#pragma unroll
                for (int t = 0; t < TY; ++t) {
                    const unsigned l = lout0[t] + (unsigned)(k - k0) * sz;
                    const uint8_t tl = type[l];
                    const double v = fmat(cz, Pp[t], fmat(az, Pm[t], P0[t])) +
                                     fmat(crz, Qp[t], fmat(brz, Q0[t], mult(arz, Qm[t])));
                    // solid rows are zero; irregular rows belong to k_apply_irr
                    if (!iin || !jin[t]) continue;
                    const bool reg = tl == CFP_REGULAR;
                    if (tl != CFP_IRREGULAR) y[l] = reg ? v : 0.0;
                    if (DOT >= 1 && reg) acc0 = fmat(d0[l], v, acc0);
                    if (DOT == 2 && reg) acc1 = fmat(v, v, acc1);
                }
            }
        }
    }
    if (DOT) {
        block_reduce2(acc0, acc1);
        if (threadIdx.x == 0 && threadIdx.y == 0) {
            const int64_t b = blockIdx.x + (int64_t)gridDim.x * (blockIdx.y + (int64_t)gridDim.y * blockIdx.z);
            partial[2 * b] = acc0;
            partial[2 * b + 1] = acc1;
        }
    }
}

// The FP32 apply fed by a ring of bulk copies (the TMA engine) through shared
// memory.  The streaming kernel above keeps one plane of loads in flight per
// thread, too few bytes per SM to cover the HBM latency.  Here a producer
// warp copies each plane of a tile several planes ahead of the consumers
// into one of kRingStages stages: the x rows of the tile and of its two
// neighbours with their halo columns, and for the output planes the dot operand
// and the type bytes of its rows.  A tile is TX columns x 1024 / TX rows x KC
// planes, TX = 512 or, on grids up to 258 wide, 256 (ring_tx).  When it
// spans the whole row width (n_x <= TX + 2), its rows are contiguous in the
// natural layout and each array's rows of a plane are one bulk copy; wider
// grids copy row by row.  Rows start at any 4-byte offset (n_x is odd in the
// benchmark grids), so each copy starts at the 16-byte boundary at or below
// its first element and the consumers add that offset.  A copy never passes
// the array's last 16-byte boundary; the elements after it (at the end of
// the array only) are stored into the stage by the producer lane itself.
// Tiles go to a persistent grid, rows fastest within a z chunk; 256 consumer
// threads in groups of TX / 2 own two columns TX / 2 apart of two rows each and march the
// planes with the same sum-factorised arithmetic and fused multiply-add
// chains as k_apply32, so both give the same bits.  Solid rows are zero;
// irregular rows are left to k_apply_irr.
// A wait that runs out (1 s) records a code in *wait_err (31: producer, stage
// free; 32: producer, final drain; 33: consumer, stage filled).  A producer
// whose wait ran out issues no further copy and waits (bounded) for the
// copies it issued; a consumer whose wait ran out stops waiting (every index
// stays in bounds whatever a stage holds), so the launch still ends.
constexpr int kRingCons = 256;  // consumer threads: two columns and two rows each
constexpr int kRingThreads = kRingCons + 32;
constexpr int kRingStages = 6;
// a tile of TX columns
template <int TX>
struct RingTile {
    static constexpr int rows = 4 * kRingCons / TX;
    static constexpr int span_nx = TX + 2;   // widest grid copied as whole-plane spans
    static constexpr int xrow = TX + 8;      // floats per x row (row-by-row copies): TX + 2 + alignment
    static constexpr int drow = TX + 4;      // floats per dot-operand row: TX + alignment
    static constexpr int trow = TX + 16;     // bytes per type row: TX + alignment
    // the regions hold either copy pattern
    static constexpr int xbytes = (std::max((rows + 2) * xrow, (rows + 2) * span_nx + 8) * 4 + 127) / 128 * 128;
    static constexpr int dbytes = (std::max(rows * drow, rows * span_nx + 8) * 4 + 15) / 16 * 16;
    static constexpr int tbytes = std::max(rows * trow, rows * span_nx + 32);
    static constexpr int doff = xbytes, toff = doff + dbytes;
    static constexpr int stage = (toff + tbytes + 127) / 128 * 128;
    static constexpr int smem = kRingStages * stage + 2 * kRingStages * 8;  // + barriers
    static_assert(doff % 16 == 0 && toff % 16 == 0 && xrow % 4 == 0 && drow % 4 == 0 && trow % 16 == 0,
                  "bulk copies want 16-byte destinations");
    static_assert(2 * rows + rows + 2 <= 32, "a producer lane per row copy");
};

// Elements e .. e + want - 1 of an array of n elements of esize bytes into
// the stage at dst, which receives the array from e0 = the 16-byte boundary
// at or below e onward.  The bulk copy stops at the array's last 16-byte
// boundary (and at the end of what is wanted, rounded up); the producer lane
// stores the remaining elements itself.  Returns the bytes the bulk copy
// delivers (0: none to issue) and its source in *src_out.
__device__ __forceinline__ unsigned ring_copy(unsigned char* dst, const unsigned char* base, int64_t e, int want,
                                              int esize, int64_t n, const unsigned char** src_out) {
    const int per16 = 16 / esize;
    const int64_t e0 = e & ~(int64_t)(per16 - 1);
    const int64_t end = e + want;                   // one past the last wanted element
    const int64_t nal = n & ~(int64_t)(per16 - 1);  // the array's last 16-byte boundary, in elements
    int64_t stop = (end + per16 - 1) & ~(int64_t)(per16 - 1);
    if (stop > nal) stop = nal;
    bool tail = false;
    for (int64_t q = max(stop, e0); q < min(end, n); ++q) {  // the tail after the last boundary
        for (int b = 0; b < esize; ++b) dst[(q - e0) * esize + b] = base[q * esize + b];
        tail = true;
    }
    // order these generic stores before later bulk (async-proxy) writes into
    // the stage; only the rare copies with a tail pay for the fence
    if (tail) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    *src_out = base + e0 * esize;
    return stop > e0 ? (unsigned)((stop - e0) * esize) : 0u;
}

template <int DOT, bool SPAN, int TX>
__global__ void __launch_bounds__(kRingThreads, 2)
    k_apply_ring(Grid<float> G, const uint8_t* __restrict__ type, const float* __restrict__ x, float* __restrict__ y,
                 const float* __restrict__ d0, double* __restrict__ partial, int ntx, int nty, int ntz, int kc,
                 int* __restrict__ wait_err) {
    using namespace tc;
    using Tile = RingTile<TX>;
    constexpr int kRingRows = Tile::rows, HX = TX / 2;  // the halves of a thread are HX columns apart
    // indexed from the __shared__ array itself, so that every stage access
    // is a shared-memory load with a 32-bit address
    extern __shared__ __align__(16) unsigned char ring_smem[];
    const float* sf = reinterpret_cast<const float*>(ring_smem);
    uint64_t* full = reinterpret_cast<uint64_t*>(ring_smem + kRingStages * Tile::stage);  // filled: 32 producer lanes
    uint64_t* empty = full + kRingStages;  // released by the consumer warps
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int q = 0; q < kRingStages; ++q) {
            mbar_init(&full[q], 32);
            mbar_init(&empty[q], kRingCons / 32);
        }
        mbar_fence_init();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const unsigned sy = (unsigned)nx, sz = (unsigned)nx * (unsigned)ny;
    const int64_t N = (int64_t)sz * nz;
    const int ntiles = ntx * nty * ntz;
    DotAcc2 dacc0, dacc1;
    if (warp == kRingCons / 32) {
        // producer warp.  SPAN (one tile column): lane 0 copies
        // x, lane 1 the dot operand, lane 2 the type bytes, each as one span
        // of whole rows.  Otherwise a lane per row copies the x rows, then the
        // dot rows, then the type rows.  Every lane arrives on the stage's barrier
        // once per plane with the bytes its copy will deliver.
        constexpr int nxl = SPAN ? 1 : kRingRows + 2, per = SPAN ? 1 : kRingRows;
        const bool xl = lane < nxl, dl = !xl && lane < nxl + per, tl = !xl && !dl && lane < nxl + 2 * per;
        const int r = xl ? lane : dl ? lane - nxl : lane - nxl - per;  // row of a row copy
        const unsigned char* arr = xl ? (const unsigned char*)x : dl ? (const unsigned char*)d0 : type;
        const int esize = tl ? 1 : 4;
        const int dst_off = xl ? r * Tile::xrow * 4 : dl ? Tile::doff + r * Tile::drow * 4 : Tile::toff + r * Tile::trow;
        unsigned g = 0;  // planes issued; plane g uses stage g % kRingStages
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
            const int tyi = tile % nty, rest = tile / nty, tx = rest % ntx, tz = rest / ntx;
            const int i0 = 1 + tx * TX, j0 = 1 + tyi * kRingRows, k0 = 1 + tz * kc;
            const int k1 = min(k0 + kc, nz - 1);
            int64_t rowe;  // the copy's first element within a plane
            int w;         // elements wanted
            if (SPAN) {
                rowe = (int64_t)(xl ? j0 - 1 : j0) * sy;
                w = (xl ? min(kRingRows + 2, ny - (j0 - 1)) : min(kRingRows, ny - j0)) * nx;  // the rows that exist
            } else {
                rowe = xl ? (int64_t)min(j0 - 1 + r, ny - 1) * sy + (i0 - 1) : (int64_t)min(j0 + r, ny - 2) * sy + i0;
                w = xl ? TX + 2 : TX;
            }
            for (int k = k0 - 1; k <= k1; ++k, ++g) {
                const int st = g % kRingStages;
                if (g >= kRingStages) {  // refill only a stage every consumer warp released
                    bool okw = true;
                    if (lane == 0) okw = mbar_wait(&empty[st], ((g / kRingStages) - 1) & 1);
                    if (!__shfl_sync(0xffffffffu, okw, 0)) {
                        ok = false;
                        if (lane == 0) atomicExch(wait_err, 31);
                        break;
                    }
                }
                const bool outp = k >= k0 && k < k1;  // an output plane
                const bool act = xl || (outp && (tl || (dl && DOT)));
                unsigned bytes = 0;
                const unsigned char* src = nullptr;
                unsigned char* dst = ring_smem + st * Tile::stage + dst_off;
                if (act) bytes = ring_copy(dst, arr, (int64_t)k * sz + rowe, w, esize, N, &src);
                mbar_arrive_expect_tx(&full[st], bytes);
                if (bytes) bulk_load(dst, src, bytes, &full[st]);
            }
        }
        // every copy issued has landed before the CTA may end (after a
        // timeout too): only the last kRingStages planes can be in flight
        if (lane == 0)
            for (unsigned q = g > (unsigned)kRingStages ? g - kRingStages : 0; q < g; ++q)
                if (!mbar_wait(&full[q % kRingStages], (q / kRingStages) & 1)) atomicExch(wait_err, 32);
        __syncwarp();
    } else {
        // consumer: columns i0 + lx (low half) and i0 + HX + lx (high half)
        // of the rows j0 + jg, j0 + jg + 1
        const int lx = threadIdx.x % HX, jg = threadIdx.x / HX * 2;
        int st = 0;       // stage of the next plane
        unsigned ph = 0;  // and its phase
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            const int tyi = tile % nty, rest = tile / nty, tx = rest % ntx, tz = rest / ntx;
            const int i0 = 1 + tx * TX, j0 = 1 + tyi * kRingRows, k0 = 1 + tz * kc;
            const int k1 = min(k0 + kc, nz - 1);
            const int c = i0 + lx;  // the low half's column; the high half's is c + HX
            const int jr = j0 + jg;  // the thread's first row
            const bool in0 = c <= nx - 2 && jr <= ny - 2, in1 = c + HX <= nx - 2;
            const int c0i = min(c, nx - 2), c1i = min(c + HX, nx - 2);
            const float2 AX = f2(G.ax[0].a[c0i], G.ax[0].a[c1i]), CX = f2(G.ax[0].c[c0i], G.ax[0].c[c1i]);
            const float2 ARX = f2(G.ax[0].ar[c0i], G.ax[0].ar[c1i]), BRX = f2(G.ax[0].br[c0i], G.ax[0].br[c1i]);
            const float2 CRX = f2(G.ax[0].cr[c0i], G.ax[0].cr[c1i]);
            float2 AY[2], CY[2], ARY[2], BRY[2], CRY[2];
            const bool jin1 = jr + 1 <= ny - 2;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int jc = min(jr + t, ny - 2);
                AY[t] = f2b(G.ax[1].a[jc]);
                CY[t] = f2b(G.ax[1].c[jc]);
                ARY[t] = f2b(G.ax[1].ar[jc]);
                BRY[t] = f2b(G.ax[1].br[jc]);
                CRY[t] = f2b(G.ax[1].cr[jc]);
            }
            // stage positions: element (row q, column col) of a plane at
            // xb[q] + ((kp + xa[q]) & 3) + col, kp = the plane's first element
            // (SPAN: rows n_x apart, one offset for all); likewise for the
            // output rows.  kx, ko carry kp of the plane being read and of the
            // one being written, kept below 16 (only their low bits count).
            const int xrow = SPAN ? nx : Tile::xrow, drow = SPAN ? nx : Tile::drow, trow = SPAN ? nx : Tile::trow;
            const int xcol = (SPAN ? c : c - (i0 - 1)) + jg * xrow, ocol = SPAN ? c : c - i0;
            const int tcol = ocol + jg * trow, dcol = ocol + jg * drow;
            unsigned xa[4], oa[2];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                xa[q] = SPAN ? ((unsigned)(j0 - 1) * sy) & 3u
                             : ((unsigned)min(jr - 1 + q, ny - 1) * sy + (unsigned)(i0 - 1)) & 3u;
#pragma unroll
            for (int t = 0; t < 2; ++t)
                oa[t] = ((SPAN ? (unsigned)j0 : (unsigned)min(jr + t, ny - 2)) * sy + (SPAN ? 0u : (unsigned)i0)) & 15u;
            unsigned kx = ((unsigned)(k0 - 1) * sz) & 15u, ko = 0;
            float2 Pm[2], P0[2], Pp[2], Qm[2], Q0[2], Qp[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) Pm[t] = P0[t] = Pp[t] = Qm[t] = Q0[t] = Qp[t] = f2b(0.f);
            // z coefficients of the plane the next step outputs, loaded a step ahead
            const float* zp = G.ax[2].a + k0;  // a, c, ar, br, cr follow at n_z
            float zn[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
            float* yr = y + ((unsigned)k0 * sz + (unsigned)jr * sy + (unsigned)c);
            int sprev = 0;  // stage of the plane before
            for (int kk = k0 - 1; kk <= k1; ++kk) {
                const float2 AZ = f2b(zn[0]), CZ = f2b(zn[1]), ARZ = f2b(zn[2]), BRZ = f2b(zn[3]), CRZ = f2b(zn[4]);
                if (kk >= k0 && kk < k1) {
#pragma unroll
                    for (int q = 0; q < 5; ++q) zn[q] = zp[q * nz];
                    ++zp;
                }
                if (ok && !mbar_wait(&full[st], ph)) {
                    ok = false;
                    atomicExch(wait_err, 33);
                }
                const float* xs = sf + st * (Tile::stage / 4) + xcol + (SPAN ? (int)((kx + xa[0]) & 3u) : 0);
                float2 XR[4], XL[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float* row = xs + q * xrow + (SPAN ? 0 : (int)((kx + xa[q]) & 3u));
                    const float2 xm = f2(row[-1], row[HX - 1]), x0 = f2(row[0], row[HX]),
                                 xp = f2(row[1], row[HX + 1]);
                    XR[q] = fma2(CRX, xp, fma2(BRX, x0, mul2(ARX, xm)));
                    XL[q] = fma2(CX, xp, fma2(AX, xm, x0));
                }
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    Pm[t] = P0[t];
                    P0[t] = Pp[t];
                    Qm[t] = Q0[t];
                    Q0[t] = Qp[t];
                    Pp[t] = fma2(CRY[t], XL[t + 2],
                                 fma2(BRY[t], XL[t + 1],
                                      fma2(ARY[t], XL[t], fma2(CY[t], XR[t + 2], fma2(AY[t], XR[t], XR[t + 1])))));
                    Qp[t] = fma2(CY[t], XL[t + 2], fma2(AY[t], XL[t], XL[t + 1]));
                }
                if (kk >= k0) {  // plane kk - 1 (stage sprev): output (from kk = k0 + 1 on), then released
                    if (kk >= k0 + 1) {
                        if (in0) {
                            const unsigned char* ts =
                                ring_smem + sprev * Tile::stage + Tile::toff + tcol + (SPAN ? (int)((ko + oa[0]) & 15u) : 0);
                            const float* ds =
                                sf + sprev * (Tile::stage / 4) + Tile::doff / 4 + dcol + (SPAN ? (int)((ko + oa[0]) & 3u) : 0);
#pragma unroll
                            for (int t = 0; t < 2; ++t) {
                                if (t && !jin1) continue;
                                float2 v = add2(fma2(CZ, Pp[t], fma2(AZ, Pm[t], P0[t])),
                                                fma2(CRZ, Qp[t], fma2(BRZ, Q0[t], mul2(ARZ, Qm[t]))));
                                const unsigned char* tr = ts + t * trow + (SPAN ? 0 : (int)((ko + oa[t]) & 15u));
                                // solid rows are zero; irregular rows belong to k_apply_irr
                                const uint8_t t0 = tr[0], t1 = in1 ? tr[HX] : (uint8_t)CFP_SOLID;
                                if (t0 != CFP_REGULAR) v.x = 0.f;
                                if (t1 != CFP_REGULAR) v.y = 0.f;
                                float* yt = yr + t * nx;
                                if (t0 != CFP_IRREGULAR) yt[0] = v.x;
                                if (in1 && t1 != CFP_IRREGULAR) yt[HX] = v.y;
                                if (DOT >= 1) {
                                    const float* dr = ds + t * drow + (SPAN ? 0 : (int)((ko + oa[t]) & 3u));
                                    dacc0.add(f2(dr[0], in1 ? dr[HX] : 0.f), v);
                                }
                                if (DOT == 2) dacc1.add(v, v);
                            }
                        }
                        yr += sz;
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[sprev]);
                }
                ko = kx;
                kx = (kx + sz) & 15u;
                sprev = st;
                if (++st == kRingStages) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[sprev]);  // the tile's last plane
        }
    }
    if (DOT) {
        double acc0 = dacc0.total(), acc1 = dacc1.total();
        block_reduce2(acc0, acc1);
        if (threadIdx.x == 0) {
            partial[2 * blockIdx.x] = acc0;
            partial[2 * blockIdx.x + 1] = acc1;
        }
    }
}

// ---- the right-hand side of Eq. Bu=q: k_rhs_box gathers the Dirichlet
// values of the box, k_rhs_source writes Q-bar f at every interior node,
// k_rhs_shell subtracts the box values times their matrix entries from the
// rows next to the box, and k_rhs_irr finishes the irregular rows.  Each node
// of f is read once and each of rhs written once, plus the shell and the
// irregular points; as separate full-grid passes (lift, B times the lift, Q,
// difference) it took 685 us at 321 x 257 x 289, now 345.

// f(l) at every box node l: the two z faces, the y faces without their z
// edges, the x faces without theirs
template <class F>
__device__ __forceinline__ void for_box(int nx, int ny, int nz, F f) {
    const int64_t sz = (int64_t)nx * ny;
    const int64_t nA = 2 * sz, nB = 2 * (int64_t)(nz - 2) * nx, nC = 2 * (int64_t)(nz - 2) * (ny - 2);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nA + nB + nC;
         q += (int64_t)gridDim.x * blockDim.x) {
        if (q < nA) {
            f(q < sz ? q : (int64_t)(nz - 1) * sz + (q - sz));
        } else if (q < nA + nB) {
            const int64_t t = (q - nA) >> 1;
            f((1 + t / nx) * sz + ((q - nA) & 1 ? (int64_t)(ny - 1) * nx : 0) + t % nx);
        } else {
            const int64_t t = (q - nA - nB) >> 1;
            f((1 + t / (ny - 2)) * sz + (1 + t % (ny - 2)) * nx + ((q - nA - nB) & 1 ? nx - 1 : 0));
        }
    }
}

// gb = g at the box nodes and rhs = 0 there; the other entries of gb are never read
__global__ void k_rhs_box(const double* __restrict__ g, double* __restrict__ gb, double* __restrict__ rhs, int nx, int ny,
                          int nz) {
    for_box(nx, ny, nz, [=](int64_t l) {
        gb[l] = g[l];
        rhs[l] = 0.0;
    });
}

// y = 0 at the box nodes: what an apply does not write itself
template <class T>
__global__ void k_zero_box(T* __restrict__ y, int nx, int ny, int nz) {
    for_box(nx, ny, nz, [=](int64_t l) { y[l] = T(0); });
}

// The source term of Eq. q with the weights of solid points set to zero
// (Q-bar): the tensor product Q = Lx Ly Lz applied to f with its solid
// entries replaced by zero (SOLID: there may be some), sum-factorised and
// marched in z like k_apply64, whose launch shape it shares: 7 FP64
// instructions per node with four rows per thread, which is what bounds it
// (265 us at 321 x 257 x 289).  Interior solid nodes get 0.
template <int TY, bool SOLID>
__global__ void __launch_bounds__(32 * kA64Warps)
    k_rhs_source(Grid<double> G, const uint8_t* __restrict__ type, const double* __restrict__ f,
                 double* __restrict__ rhs, int kc) {
    constexpr int R = TY + 2;
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int i = 1 + blockIdx.x * 32 + threadIdx.x;
    const int j0 = 1 + (blockIdx.y * kA64Warps + threadIdx.y) * TY;
    const int k0 = 1 + blockIdx.z * kc;
    const int k1 = min(k0 + kc, nz - 1);
    if (j0 > ny - 2) return;
    const bool iin = i <= nx - 2;
    const int ic = iin ? i : 1;  // clamped: every load stays inside the grid
    const unsigned sy = (unsigned)nx, sz = (unsigned)nx * (unsigned)ny;
    const double ax = G.ax[0].a[ic], cx = G.ax[0].c[ic];
    double ay[TY], cy[TY];
    bool jin[TY];
#pragma unroll
    for (int t = 0; t < TY; ++t) {
        jin[t] = j0 + t <= ny - 2;
        const int jc = jin[t] ? j0 + t : j0;
        ay[t] = G.ax[1].a[jc];
        cy[t] = G.ax[1].c[jc];
    }
    unsigned roff[R];
#pragma unroll
    for (int r = 0; r < R; ++r) roff[r] = (unsigned)min(j0 - 1 + r, ny - 1) * sy + (unsigned)ic;
    double n[3 * R];
    uint8_t own[R], prev[R] = {};  // type of (i, row) in the plane just loaded, and in the one before
    auto load = [&](int k) {
        const unsigned pz = (unsigned)k * sz;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const unsigned q = pz + roff[r];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const uint8_t t = SOLID ? type[q + d - 1] : (uint8_t)CFP_REGULAR;
                n[3 * r + d] = SOLID && t == CFP_SOLID ? 0.0 : f[q + d - 1];
                if (d == 1) own[r] = t;
            }
        }
    };
    load(k0 - 1);
    double Qm[TY], Q0[TY], Qp[TY];
#pragma unroll
    for (int t = 0; t < TY; ++t) Qm[t] = Q0[t] = Qp[t] = 0.0;
#pragma unroll 1
    for (int kk = k0 - 1; kk <= k1; ++kk) {
        double XL[R];
        uint8_t tout[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            XL[r] = fmat(cx, n[3 * r + 2], fmat(ax, n[3 * r], n[3 * r + 1]));
            tout[r] = prev[r];
            prev[r] = own[r];
        }
        if (kk < k1) load(kk + 1);  // ahead of the y and z passes
#pragma unroll
        for (int t = 0; t < TY; ++t) {
            Qm[t] = Q0[t];
            Q0[t] = Qp[t];
            Qp[t] = fmat(cy[t], XL[t + 2], fmat(ay[t], XL[t], XL[t + 1]));
        }
        if (kk >= k0 + 1 && iin) {
            const int k = kk - 1;
            const double az = G.ax[2].a[k], cz = G.ax[2].c[k];
#pragma unroll
            for (int t = 0; t < TY; ++t)
                if (jin[t])
                    rhs[(unsigned)k * sz + (unsigned)(j0 + t) * sy + (unsigned)i] =
                        SOLID && tout[t + 1] == CFP_SOLID ? 0.0 : fmat(cz, Qp[t], fmat(az, Qm[t], Q0[t]));
        }
    }
}

// One axis' operators at a node: L = (a, 1, c), R = (ar, br, cr)
struct Ops3 {
    double L[3], R[3];
    __device__ __forceinline__ Ops3(const Axis<double>& A, int i) : L{A.a[i], 1.0, A.c[i]}, R{A.ar[i], A.br[i], A.cr[i]} {}
};

// The row of B at a node of exactly one face shell, applied to the box values
// of that face: nine nodes, a tensor product of the face's two axes (u, v)
// times entry s of the normal axis (w): Lw[s] (Lv Ru + Rv Lu) + Rw[s] Lv Lu.
__device__ __forceinline__ double face_lift(const Ops3& U, const Ops3& V, const Ops3& W, int s, const double* p,
                                            int64_t su, int64_t sv) {
    double P = 0.0, Q = 0.0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double* x = p + (q - 1) * sv;
        const double xr = U.R[0] * x[-su] + U.R[1] * x[0] + U.R[2] * x[su];
        const double xl = U.L[0] * x[-su] + x[0] + U.L[2] * x[su];
        P += V.L[q] * xr + V.R[q] * xl;
        Q += V.L[q] * xl;
    }
    return W.L[s] * P + W.R[s] * Q;
}

// rhs -= B gb on the shell of interior nodes next to the box, the only rows
// that reach it (solid rows stay zero; irregular rows get their corrections
// from k_rhs_irr).  The inner nodes of each face (face_lift) and the nodes
// next to two or three faces (27 weights, the box nodes among them read) are
// separate ranges of q, so that a warp takes one path: 24 to 30 FP64
// instructions per node instead of 135.  An axis with fewer than three
// interior nodes has no inner ones: every shell node then takes the second.
__global__ void k_rhs_shell(Grid<double> G, const uint8_t* __restrict__ type, const double* __restrict__ gb,
                            double* __restrict__ rhs) {
    const int nx = G.nx, ny = G.ny, nz = G.nz;
    const int64_t ax = nx - 2, ay = ny - 2, az = nz - 2;  // interior nodes per axis
    const bool thin = ax < 3 || ay < 3 || az < 3;
    const int64_t bx = ax - 2, by = ay - 2, bz = az - 2;
    const int64_t nA = thin ? 0 : 2 * bx * by, nB = thin ? 0 : 2 * bx * bz, nC = thin ? 0 : 2 * by * bz;
    // edges: 4 lines along z (corners included), 4 along y, 4 along x; thin: the whole interior
    const int64_t nE = thin ? ax * ay * az : 4 * az + 4 * by + 4 * bx;
    const int64_t sy = nx, sz = (int64_t)nx * ny;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nA + nB + nC + nE;
         q += (int64_t)gridDim.x * blockDim.x) {
        int i, j, k, face = -1;
        if (q < nA) {
            const int64_t t = q % (bx * by);
            i = 2 + (int)(t % bx), j = 2 + (int)(t / bx), k = q < bx * by ? 1 : nz - 2, face = 2;
        } else if (q < nA + nB) {
            const int64_t u = q - nA, t = u % (bx * bz);
            i = 2 + (int)(t % bx), k = 2 + (int)(t / bx), j = u < bx * bz ? 1 : ny - 2, face = 1;
        } else if (q < nA + nB + nC) {
            const int64_t u = q - nA - nB, t = u % (by * bz);
            j = 2 + (int)(t % by), k = 2 + (int)(t / by), i = u < by * bz ? 1 : nx - 2, face = 0;
        } else {
            const int64_t u = q - nA - nB - nC;
            if (thin) {
                i = 1 + (int)(u % ax), j = 1 + (int)((u / ax) % ay), k = 1 + (int)(u / (ax * ay));
                if (i > 1 && i < nx - 2 && j > 1 && j < ny - 2 && k > 1 && k < nz - 2) continue;
            } else if (u < 4 * az) {
                i = u & 1 ? nx - 2 : 1, j = u & 2 ? ny - 2 : 1, k = 1 + (int)(u >> 2);
            } else if (u < 4 * az + 4 * by) {
                const int64_t t = u - 4 * az;
                i = t & 1 ? nx - 2 : 1, k = t & 2 ? nz - 2 : 1, j = 2 + (int)(t >> 2);
            } else {
                const int64_t t = u - 4 * az - 4 * by;
                j = t & 1 ? ny - 2 : 1, k = t & 2 ? nz - 2 : 1, i = 2 + (int)(t >> 2);
            }
        }
        const int64_t l = (int64_t)k * sz + (int64_t)j * sy + i;
        if (type[l] == CFP_SOLID) continue;
        const Ops3 X(G.ax[0], i), Y(G.ax[1], j), Z(G.ax[2], k);
        double v = 0.0;
        if (face == 2) {
            const int s = k == 1 ? 0 : 2;
            v = face_lift(X, Y, Z, s, gb + l + (s - 1) * sz, 1, sy);
        } else if (face == 1) {
            const int s = j == 1 ? 0 : 2;
            v = face_lift(X, Z, Y, s, gb + l + (s - 1) * sy, 1, sz);
        } else if (face == 0) {
            const int s = i == 1 ? 0 : 2;
            v = face_lift(Y, Z, X, s, gb + l + (s - 1), sy, sz);
        } else {
            for (int c = 0; c < 3; ++c)
                for (int b = 0; b < 3; ++b)
                    for (int a = 0; a < 3; ++a) {
                        const int ii = i + a - 1, jj = j + b - 1, kk = k + c - 1;
                        if (ii > 0 && jj > 0 && kk > 0 && ii < nx - 1 && jj < ny - 1 && kk < nz - 1) continue;
                        const double w = X.R[a] * Y.L[b] * Z.L[c] + X.L[a] * Y.R[b] * Z.L[c] + X.L[a] * Y.L[b] * Z.R[c];
                        v += w * gb[l + (a - 1) + (b - 1) * sy + (c - 1) * sz];
                    }
        }
        rhs[l] -= v;
    }
}

// The irregular rows' share: the corrections of the modified lines (the C
// part of Eq. Bdec) times the box values they reach, and the IBI term of Eqs.
// bc / qb_case2; one thread per irregular point.  A correction lies at most
// six nodes away (a line of the 3 x 3 x 3 block, then at most five grid nodes
// along it), so only points that near to the box look for box nodes.
__global__ void __launch_bounds__(128)
    k_rhs_irr(Side<double> S, const uint8_t* __restrict__ type, const int32_t* __restrict__ irr_lin, int64_t n_irr,
              const int32_t* __restrict__ bib_ptr, const int32_t* __restrict__ bib_idx,
              const double* __restrict__ bib_val, const double* __restrict__ gb, const double* __restrict__ g_ibi,
              double* __restrict__ rhs, int nx, int ny, int nz) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_irr;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int l = irr_lin[s];
        const int k = l / (nx * ny), rem = l - k * nx * ny, j = rem / nx, i = rem - j * nx;
        double v = rhs[l];
        if (min(min(min(i, nx - 1 - i), min(j, ny - 1 - j)), min(k, nz - 1 - k)) <= 6) {
            double cor = 0.0;
            for (int e = S.corr_ptr[s]; e < S.corr_ptr[s + 1]; ++e) {
                const int m = l + S.corr_off[e];
                if (type[m] == CFP_BOUNDARY) cor += S.corr_val[e] * gb[m];
            }
            v -= cor;
        }
        for (int e = bib_ptr[s]; e < bib_ptr[s + 1]; ++e) v -= bib_val[e] * g_ibi[bib_idx[e]];
        rhs[l] = v;
    }
}

// The rows of the irregular points, whole (Eq. Bdec): the regular 27-point
// part with the arithmetic of the factorised kernels -- the same fused
// multiply-add chains on the same 27 values, so that part has the same bits
// as there -- plus the side-list corrections of the row's modified lines
// (Eqs. A27_mod, cor, cor_case2).  One thread per irregular point.  The
// regular rows' kernels leave these rows alone, so this kernel runs beside
// them on a second stream; its dot terms go to its own partials.
constexpr int kIrrGroup = 8;
template <class T, int DOT>
__global__ void __launch_bounds__(128)
    k_apply_irr(Grid<T> G, Side<T> S, const int32_t* __restrict__ irr_lin, int64_t n_irr, const T* __restrict__ x,
                T* __restrict__ y, const T* __restrict__ d0, double* __restrict__ partial) {
    const int nx = G.nx, ny = G.ny;
    const int64_t sy = nx, sz = (int64_t)nx * ny;
    double acc0 = 0.0, acc1 = 0.0;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_irr;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = irr_lin[s];
        // the corrections, summed in entry order: the offsets and weights of the
        // next eight are fetched while this eight's values are on their way
        const int e0 = S.corr_ptr[s], e1 = S.corr_ptr[s + 1];
        int off[kIrrGroup];
        T w[kIrrGroup];
        auto fetch = [&](int e) {
#pragma unroll
            for (int q = 0; q < kIrrGroup; ++q) {
                const bool in = e + q < e1;
                off[q] = in ? S.corr_off[e + q] : 0;
                w[q] = in ? S.corr_val[e + q] : T(0);
            }
        };
        fetch(e0);
        const unsigned lu = (unsigned)l, k = lu / (unsigned)sz, rem = lu - k * (unsigned)sz, j = rem / (unsigned)nx,
                       i = rem - j * (unsigned)nx;
        const T ax = G.ax[0].a[i], cx = G.ax[0].c[i], arx = G.ax[0].ar[i], brx = G.ax[0].br[i], crx = G.ax[0].cr[i];
        const T ay = G.ax[1].a[j], cy = G.ax[1].c[j], ary = G.ax[1].ar[j], bry = G.ax[1].br[j], cry = G.ax[1].cr[j];
        const T az = G.ax[2].a[k], cz = G.ax[2].c[k], arz = G.ax[2].ar[k], brz = G.ax[2].br[k], crz = G.ax[2].cr[k];
        T P[3], Q[3];
#pragma unroll
        for (int dz = 0; dz < 3; ++dz) {
            T XR[3], XL[3];
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const T* q = x + l + (dz - 1) * sz + (dy - 1) * sy;
                XR[dy] = fmat(crx, q[1], fmat(brx, q[0], mult(arx, q[-1])));
                XL[dy] = fmat(cx, q[1], fmat(ax, q[-1], q[0]));
            }
            P[dz] = fmat(cry, XL[2], fmat(bry, XL[1], fmat(ary, XL[0], fmat(cy, XR[2], fmat(ay, XR[0], XR[1])))));
            Q[dz] = fmat(cy, XL[2], fmat(ay, XL[0], XL[1]));
        }
        T v = fmat(cz, P[2], fmat(az, P[0], P[1])) + fmat(crz, Q[2], fmat(brz, Q[1], mult(arz, Q[0])));
        T cor = T(0);
        for (int e = e0; e < e1; e += kIrrGroup) {
            T xv[kIrrGroup], wv[kIrrGroup];
#pragma unroll
            for (int q = 0; q < kIrrGroup; ++q) {
                xv[q] = x[l + off[q]];
                wv[q] = w[q];
            }
            fetch(e + kIrrGroup);
#pragma unroll
            for (int q = 0; q < kIrrGroup; ++q)
                if (e + q < e1) cor = fmat(wv[q], xv[q], cor);
        }
        v = v + cor;
        y[l] = v;
        if (DOT >= 1) acc0 += (double)d0[l] * (double)v;
        if (DOT == 2) acc1 += (double)v * (double)v;
    }
    if (DOT) {
        block_reduce2(acc0, acc1);
        if (threadIdx.x == 0) {
            partial[2 * blockIdx.x] = acc0;
            partial[2 * blockIdx.x + 1] = acc1;
        }
    }
}

template <class T>
__global__ void k_mask_copy(const uint8_t* __restrict__ type, const T* __restrict__ in, T* __restrict__ out,
                            int64_t N) {
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < N; l += (int64_t)gridDim.x * blockDim.x) {
        const uint8_t t = type[l];
        out[l] = (t == CFP_REGULAR || t == CFP_IRREGULAR) ? in[l] : T(0);
    }
}

__global__ void k_boundary_lift(const uint8_t* __restrict__ type, const double* __restrict__ g,
                                double* __restrict__ gb, int64_t N) {
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < N; l += (int64_t)gridDim.x * blockDim.x)
        gb[l] = type[l] == CFP_BOUNDARY ? g[l] : 0.0;
}

__global__ void k_finish_solution(const uint8_t* __restrict__ type, const double* __restrict__ x,
                                  const double* __restrict__ g, double* __restrict__ u, int64_t N) {
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < N; l += (int64_t)gridDim.x * blockDim.x) {
        const uint8_t t = type[l];
        u[l] = t == CFP_BOUNDARY ? g[l] : (t == CFP_SOLID ? 0.0 : x[l]);
    }
}

// Eq. app_xxx (compact, b = 1) and Eq. 2ndorder_coef at interior nodes;
// layout per axis: a, c, ar, br, cr, ka, kb, kc (n each), zero at the ends.
__global__ void k_metrics(const double* __restrict__ x, int n, double* __restrict__ out, float* __restrict__ out32) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (i > 0 && i < n - 1) {
            const double f = x[i + 1] - x[i];
            const double b = x[i] - x[i - 1];
            const double D = f * f * f + 4.0 * f * f * b + 4.0 * f * b * b + b * b * b;
            v[0] = f * (b * b + b * f - f * f) / D;
            v[1] = b * (f * f + b * f - b * b) / D;
            v[2] = 12.0 * f / D;
            v[3] = -12.0 / (f * f + 3.0 * f * b + b * b);
            v[4] = 12.0 * b / D;
            v[5] = 2.0 / (b * (f + b));
            v[6] = -2.0 / (b * f);
            v[7] = 2.0 / (f * (f + b));
        }
        for (int q = 0; q < 8; ++q) {
            out[(int64_t)q * n + i] = v[q];
            out32[(int64_t)q * n + i] = (float)v[q];
        }
    }
}

unsigned flat_grid(int64_t n) {
    const int64_t b = (n + 255) / 256;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

}  // namespace


namespace {

// the ring's tile width: 256 only where a tile spans the row (copied row by row,
// 256-column tiles of 513^3 took 443 us, 512-column ones 354)
int ring_tx(const cfp_ctx* c) { return c->n[0] <= RingTile<256>::span_nx ? 256 : 512; }
// planes per z chunk by grid size: some 1024 tiles, of 64 to 128 planes (513^3:
// 128 336 us, 64 354); beside the irregular rows' kernel, whose CTAs delay some
// of the ring's, few rounds of tiles lose least (bodies, 257^3: 64 67 us, 24 87;
// 513^3: 64 412, 128 422)
int ring_planes_by_size(const cfp_ctx* c, bool irregular) {
    const int tx = ring_tx(c), rows = 4 * kRingCons / tx;
    const int64_t col = (int64_t)((c->n[0] - 2 + tx - 1) / tx) * ((c->n[1] - 2 + rows - 1) / rows);
    return irregular ? 64 : (int)std::max<int64_t>(64, std::min<int64_t>(128, col * (c->n[2] - 2) / 1024));
}
int ring_planes(const cfp_ctx* c) {
    return c->apply_kc[1] ? std::max(32, c->apply_kc[1]) : ring_planes_by_size(c, c->n_irr > 0);
}
// the apply's kernel of precision q (0 FP64, 1 FP32) by grid size: in FP64 the
// streaming kernel, in FP32 the ring from 2^23 nodes on where its tiles' columns
// are at least 85 % filled (257^3 55 us against the streaming kernel's 68, 225^3
// 45 : 55, 449 x 385 x 321 174 : 180, 513^3 337 : 406; but 257 x 129 x 65 18 : 12,
// 385^3 205 : 181) and else the streaming kernel
int kind_by_size(const cfp_ctx* c, int q) {
    if (q == 1 && c->ring_grid > 0) {
        const int cols = c->n[0] - 2, tx = ring_tx(c), tiles = (cols + tx - 1) / tx;
        const int64_t nodes = (int64_t)cols * (c->n[1] - 2) * (c->n[2] - 2);
        if (nodes >= (int64_t)1 << 23 && cols * 100 >= 85 * tiles * tx) return CFP_APPLY_RING;
    }
    return CFP_APPLY_STREAM;
}
int apply_kind(const cfp_ctx* c, int q) { return c->apply_kind[q] ? c->apply_kind[q] : kind_by_size(c, q); }

// k_apply64's rows per thread and planes per z chunk
struct Shape {
    int ty, kc;
    dim3 grid(const cfp_ctx* c) const {
        const int rows = ty * kA64Warps;
        return dim3((unsigned)((c->n[0] - 2 + 31) / 32), (unsigned)((c->n[1] - 2 + rows - 1) / rows),
                    (unsigned)((c->n[2] - 2 + kc - 1) / kc));
    }
    int64_t ctas(const cfp_ctx* c) const {
        const dim3 g = grid(c);
        return (int64_t)g.x * g.y * g.z;
    }
};

// The launch shape of k_apply64 (where the tuner set none) and k_rhs_source by
// grid size: the one with the smallest estimate.  A warp issues w = (kc + 2)
// (row (ty + 2) + yout ty) + zout kc ty FP64 instructions (row per loaded row,
// yout and zout per output row in y and z: 5, 7, 6 in the apply; its two halo
// planes do the x and y passes only), a CTA 4 w; the estimate is the busiest of
// 152 SMs, the latency of a plane's loads (about 130 slots per plane), which
// counts where few CTAs share an SM, and, past four CTAs per SM, half of a last
// one that runs alone.  Large grids take 4 rows and 64 planes, 129^3 and 257^3
// 4 x 16 (109 and 712 us; 4 x 64 250 and 895), 97 x 65 x 82 2 x 8; 33^3 takes
// 128 CTAs of 1 x 2, where 4 x 64 would leave the work to 8 SMs.  (CTAs of one
// warp share a scheduler: 33^3 14.5 us with them, 10.4 with four warps in the
// same shape.)
Shape shape64(const cfp_ctx* c, double row, double yout, double zout) {
    Shape best{4, 64};
    double est_best = 1e300;
    for (int t : {4, 2, 1})
        for (int q : {64, 32, 16, 8, 4, 2}) {
            const Shape sh{t, q};
            const double cta = kA64Warps * ((q + 2) * (row * (t + 2) + yout * t) + zout * q * t);
            const double per = (double)((sh.ctas(c) + 151) / 152);
            const double est = per * cta + 130.0 * (q + 2) + (per > 4 ? 0.5 * cta : 0.0);
            if (est < est_best * 0.99) {
                est_best = est;
                best = sh;
            }
        }
    return best;
}
Shape apply64_by_size(const cfp_ctx* c) { return shape64(c, 5.0, 7.0, 6.0); }
Shape apply64_shape(const cfp_ctx* c) {
    if (c->apply_ty[0] && c->apply_kc[0]) return Shape{c->apply_ty[0], c->apply_kc[0]};
    return apply64_by_size(c);
}

// The FP32 streaming kernel is bound by the latency of a plane's loads, so its
// time goes with the rounds of resident CTAs (four with 4 rows, six with 2 per
// SM) times the planes each marches, about 1 us per plane with 4 rows, and some
// 6 for a round's start (257^3: 4 x 64 68 us, 4 x 8 78; 129^3: 4 x 8 12.4, 4 x
// 16 14.5; 321 x 257 x 289: 4 x 32 91, 4 x 64 106).  Without a dot product 2
// rows take 0.65 of it (513^3 361 us against 390), with one more (448 against
// 406).
Shape apply32_by_size(const cfp_ctx* c, bool dot) {
    Shape best{4, 64};
    double est_best = 1e300;
    for (int t : {4, 2})
        for (int q : {64, 32, 16, 8, 4, 2}) {
            if (t == 2 && dot) continue;
            const Shape sh{t, q};
            const int64_t per = 152 * (t == 4 ? 4 : 6);
            const double est = (double)((sh.ctas(c) + per - 1) / per) * (q + 8) * (t == 4 ? 1.0 : 0.65);
            if (est < est_best) {
                est_best = est;
                best = sh;
            }
        }
    return best;
}

Shape apply32_shape(const cfp_ctx* c, bool dot) {
    // (a ring's planes, where the streaming kernel takes its place, may be more
    // than it stages coefficients for)
    if (c->apply_ty[1] && c->apply_kc[1]) return Shape{c->apply_ty[1], std::min(c->apply_kc[1], kMaxPlanes)};
    return apply32_by_size(c, dot);
}

}  // namespace

// the kernel and tile shape the apply of precision q runs with (FP32: with a
// dot product, as in a solve)
void apply_shape(const cfp_ctx* c, int q, int* kernel, int* rows, int* planes) {
    *kernel = apply_kind(c, q);
    if (*kernel == CFP_APPLY_RING) {
        *rows = 2;
        *planes = ring_planes(c);
        return;
    }
    const Shape sh = q == 0 ? apply64_shape(c) : apply32_shape(c, true);
    *rows = sh.ty;
    *planes = sh.kc;
}

// Whether a shape is one that apply_shape reports for contexts of this grid
// size that no tuner touched, with or without irregular points, before and
// after their ring is set up.  *own: it is what this context would run with.
bool shape_by_size(const cfp_ctx* c, int q, int kernel, int rows, int planes, bool* own) {
    *own = false;
    if (kernel == CFP_APPLY_RING) {
        if (q == 0 || rows != 2) return false;
        *own = kind_by_size(c, q) == CFP_APPLY_RING && planes == ring_planes_by_size(c, c->n_irr > 0);
        return planes == ring_planes_by_size(c, false) || planes == ring_planes_by_size(c, true);
    }
    const Shape sh = q == 0 ? apply64_by_size(c) : apply32_by_size(c, true);
    const bool same = kernel == CFP_APPLY_STREAM && rows == sh.ty && planes == sh.kc;
    *own = same && kind_by_size(c, q) == CFP_APPLY_STREAM;
    return same;
}

namespace {

// the ring's launch: tile width, planes per z chunk, tiles per axis
struct RingShape {
    int tx, kc, ntx, nty, ntz;
    int tiles() const { return ntx * nty * ntz; }
};
RingShape ring_shape(const cfp_ctx* c) {
    RingShape r{ring_tx(c), ring_planes(c), 0, 0, 0};
    const int rows = 4 * kRingCons / r.tx;
    r.ntx = (c->n[0] - 2 + r.tx - 1) / r.tx;
    r.nty = (c->n[1] - 2 + rows - 1) / rows;
    r.ntz = (c->n[2] - 2 + r.kc - 1) / r.kc;
    return r;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

void launch_metrics(cfp_ctx* c) {
    int64_t off = 0;
    for (int d = 0; d < 3; ++d) {
        const int n = c->n[d];
        k_metrics<<<(n + 255) / 256, 256, 0, c->stream>>>(c->dX[d], n, c->dcoef64 + off, c->dcoef32 + off);
        off += 8 * (int64_t)n;
    }
    c->launches += 3;
}

// CTAs of k_apply_irr (128 threads, one irregular point each per pass; at
// most 152 x 8)
int irr_blocks(const cfp_ctx* c) {
    if (c->n_irr <= 0) return 0;
    return (int)std::min<int64_t>((c->n_irr + 127) / 128, 152 * 8);
}

// the most CTAs any apply tile shape launches, with the irregular rows' kernel's
// (dot-product partials per launch); the ring's persistent grid never has
// more CTAs than the streaming kernel with 2 rows x 16 planes
int apply_blocks(cfp_ctx* c) {
    int64_t m = 0;
    for (int ty : {2, 4})
        for (int kc : {16, 32, 64}) m = std::max(m, Shape{ty, kc}.ctas(c));
    m = std::max(m, std::max(apply64_shape(c).ctas(c), apply32_shape(c, true).ctas(c)));
    if (c->ring_grid > 0) m = std::max<int64_t>(m, std::min(ring_shape(c).tiles(), c->ring_grid));
    return (int)m + irr_blocks(c);
}

// the FP64 regular rows' kernel
template <int DOT>
void apply64_launch(cfp_ctx* c, const Shape& sh, const double* x, double* y, const double* d0, double* partial,
                    cudaStream_t s) {
    const dim3 g = sh.grid(c), b(32, kA64Warps);
    if (sh.ty == 4) k_apply64<DOT, 4><<<g, b, 0, s>>>(grid_view<double>(c), c->type, x, y, d0, partial, sh.kc);
    else if (sh.ty == 2) k_apply64<DOT, 2><<<g, b, 0, s>>>(grid_view<double>(c), c->type, x, y, d0, partial, sh.kc);
    else k_apply64<DOT, 1><<<g, b, 0, s>>>(grid_view<double>(c), c->type, x, y, d0, partial, sh.kc);
}

// the FP32 ring
template <int DOT, int TX>
void ring_launch_tx(cfp_ctx* c, const RingShape& r, int ctas, const float* x, float* y, const float* d0,
                    double* partial, cudaStream_t s) {
    auto k = k_apply_ring<DOT, true, TX>;
    if constexpr (TX == 512)
        if (c->n[0] > RingTile<TX>::span_nx) k = k_apply_ring<DOT, false, TX>;
    k<<<ctas, kRingThreads, RingTile<TX>::smem, s>>>(grid_view<float>(c), c->type, x, y, d0, partial, r.ntx, r.nty,
                                                     r.ntz, r.kc, c->dwait);
}
template <int DOT>
void ring_launch(cfp_ctx* c, const RingShape& r, int ctas, const float* x, float* y, const float* d0, double* partial,
                 cudaStream_t s) {
    if (r.tx == 512) ring_launch_tx<DOT, 512>(c, r, ctas, x, y, d0, partial, s);
    else ring_launch_tx<DOT, 256>(c, r, ctas, x, y, d0, partial, s);
}

// B x: the regular rows' kernel on s and, forked onto the context's second
// stream and joined back before anything later on s, the irregular rows'
// kernel; dot partials: the main kernel's CTAs, then k_apply_irr's.
template <class T, int DOT>
void apply_launch(cfp_ctx* c, const T* x, T* y, const T* d0, double* partial, cudaStream_t s, int* nb) {
    int nmain = 0;
    bool ring = false;
    Shape sh{0, 0};
    RingShape rs{0, 0, 0, 0, 0};
    if constexpr (sizeof(T) == 8) {
        sh = apply64_shape(c);
        nmain = (int)sh.ctas(c);
    } else {
        ring = apply_kind(c, 1) == CFP_APPLY_RING && c->ring_grid > 0 && aligned16(x) && (!DOT || aligned16(d0));
        if (ring) {
            rs = ring_shape(c);
            nmain = std::min(rs.tiles(), c->ring_grid);
        } else {
            sh = apply32_shape(c, DOT > 0);
            nmain = (int)sh.ctas(c);
        }
    }
    const int nirr = irr_blocks(c);
    if (nirr) {
        cudaEventRecord(c->ev_fork, s);
        cudaStreamWaitEvent(c->aux, c->ev_fork, 0);
        k_apply_irr<T, DOT><<<nirr, 128, 0, c->aux>>>(grid_view<T>(c), side_view<T>(c), c->irr_lin, c->n_irr, x, y,
                                                      d0, partial ? partial + 2 * (int64_t)nmain : nullptr);
    }
    if constexpr (sizeof(T) == 8) {
        apply64_launch<DOT>(c, sh, x, y, d0, partial, s);
    } else if (ring) {
        ring_launch<DOT>(c, rs, nmain, x, y, d0, partial, s);
    } else if (sh.ty == 4) {
        k_apply32<DOT, 4><<<sh.grid(c), dim3(32, kA64Warps), 0, s>>>(grid_view<float>(c), c->type, x, y, d0, partial, sh.kc);
    } else {
        k_apply32<DOT, 2><<<sh.grid(c), dim3(32, kA64Warps), 0, s>>>(grid_view<float>(c), c->type, x, y, d0, partial, sh.kc);
    }
    if (nirr) {
        cudaEventRecord(c->ev_join, c->aux);
        cudaStreamWaitEvent(s, c->ev_join, 0);
    }
    c->launches += nirr ? 1 : 0;
    if (nb) *nb = nmain + nirr;
}

namespace {
template <int DOT, bool SPAN, int TX>
bool ring_attr(int* per) {
    const auto k = k_apply_ring<DOT, SPAN, TX>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, RingTile<TX>::smem) != cudaSuccess) return false;
    int p = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, k, kRingThreads, RingTile<TX>::smem) != cudaSuccess) return false;
    *per = std::min(*per, p);
    return true;
}
template <bool SPAN, int TX>
bool ring_attrs(int* per) {
    return ring_attr<0, SPAN, TX>(per) && ring_attr<1, SPAN, TX>(per) && ring_attr<2, SPAN, TX>(per);
}
}  // namespace

// The ring's launch attributes and persistent grid (CTAs resident on every
// SM at once), once per context before any capture.
bool setup_apply_ring(cfp_ctx* c) {
    if (c->ring_grid) return c->ring_grid > 0;
    int per = 1 << 20, nsm = 0;
    const bool ok = ring_attrs<true, 512>(&per) && ring_attrs<false, 512>(&per) && ring_attrs<true, 256>(&per) &&
                    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device) == cudaSuccess;
    cudaGetLastError();
    c->ring_grid = ok && per >= 1 ? per * nsm : -1;
    return c->ring_grid > 0;
}

template <class T>
void launch_apply(cfp_ctx* c, const T* x, T* y, const T* d0, int dotmode, double* partial, cudaStream_t s,
                  int* nblocks_out) {
    if (dotmode == 0) apply_launch<T, 0>(c, x, y, d0, partial, s, nblocks_out);
    else if (dotmode == 1) apply_launch<T, 1>(c, x, y, d0, partial, s, nblocks_out);
    else apply_launch<T, 2>(c, x, y, d0, partial, s, nblocks_out);
    c->launches += 1;
}

template <class T>
void launch_zero_box(cfp_ctx* c, T* y, cudaStream_t s) {
    const int nx = c->n[0], ny = c->n[1], nz = c->n[2];
    const int64_t box = 2 * ((int64_t)nx * ny + (int64_t)nx * nz + (int64_t)ny * nz);
    k_zero_box<T><<<flat_grid(box), 256, 0, s>>>(y, nx, ny, nz);
    c->launches += 1;
}
template void launch_zero_box<double>(cfp_ctx*, double*, cudaStream_t);
template void launch_zero_box<float>(cfp_ctx*, float*, cudaStream_t);

// `sweeps` red-black sweeps from phi = 0 (sweeps = 0: masked copy).  The
// sweeps run on the fine level's red/black split arrays of the multigrid
// hierarchy (the first red half-sweep reads rho, the last black one writes
// phi at every interior node), which ensure_mg provides.
template <class T>
void launch_precond_rbgs(cfp_ctx* c, int sweeps, const T* rho, T* phi, cudaStream_t s) {
    if (sweeps <= 0) {
        c->launches += 1;
        k_mask_copy<T><<<flat_grid(c->N), 256, 0, s>>>(c->type, rho, phi, c->N);
        return;
    }
    launch_rbgs_split<T>(c, sweeps, rho, phi, s);
}

template <class T>
void launch_precond(cfp_ctx* c, int sweeps, const T* rho, T* phi, cudaStream_t s) {
    if (c->precond_kind == CFP_PRECOND_MG) launch_precond_mg<T>(c, rho, phi, s);
    else if (c->precond_kind == CFP_PRECOND_ILU && sweeps > 0) launch_precond_ilu<T>(c, sweeps, rho, phi, s);
    else launch_precond_rbgs<T>(c, sweeps, rho, phi, s);
}

template void launch_apply<double>(cfp_ctx*, const double*, double*, const double*, int, double*, cudaStream_t,
                                   int*);
template void launch_apply<float>(cfp_ctx*, const float*, float*, const float*, int, double*, cudaStream_t, int*);
template void launch_precond<double>(cfp_ctx*, int, const double*, double*, cudaStream_t);
template void launch_precond<float>(cfp_ctx*, int, const float*, float*, cudaStream_t);

// rhs (at every node) from f, g and g_ibi; gb: work field, overwritten at the
// box nodes; rhs overlaps neither f nor gb
void launch_rhs(cfp_ctx* c, const double* f, const double* g, const double* g_ibi, double* gb, double* rhs,
                cudaStream_t s) {
    const int nx = c->n[0], ny = c->n[1], nz = c->n[2];
    const Grid<double> G = grid_view<double>(c);
    const int64_t box = 2 * ((int64_t)nx * ny + (int64_t)nx * nz + (int64_t)ny * nz);
    k_rhs_box<<<flat_grid(box), 256, 0, s>>>(g, gb, rhs, nx, ny, nz);
    const Shape sh = shape64(c, 2.0, 2.0, 2.0);
    const dim3 gr = sh.grid(c), b(32, kA64Warps);
    // no solid points: no bodies, and the fluid outside them (the inside of no
    // body is no fluid at all)
    const bool solid = !c->bodies.empty() || c->fluid_inside;
#define CFP_SOURCE(TY)                                                                                     \
    (solid ? k_rhs_source<TY, true><<<gr, b, 0, s>>>(G, c->type, f, rhs, sh.kc)                            \
           : k_rhs_source<TY, false><<<gr, b, 0, s>>>(G, c->type, f, rhs, sh.kc))
    if (sh.ty == 4) CFP_SOURCE(4);
    else if (sh.ty == 2) CFP_SOURCE(2);
    else CFP_SOURCE(1);
#undef CFP_SOURCE
    const bool thin = nx < 5 || ny < 5 || nz < 5;
    k_rhs_shell<<<flat_grid(thin ? c->N : box), 256, 0, s>>>(G, c->type, gb, rhs);
    c->launches += 3;
    if (c->n_irr > 0) {
        k_rhs_irr<<<(unsigned)std::min<int64_t>((c->n_irr + 127) / 128, 152 * 16), 128, 0, s>>>(
            side_view<double>(c), c->type, c->irr_lin, c->n_irr, c->bib_ptr, c->bib_idx, c->bib_val, gb, g_ibi, rhs, nx,
            ny, nz);
        c->launches += 1;
    }
}

void launch_boundary_lift(cfp_ctx* c, const double* g, double* gb, cudaStream_t s) {
    c->launches += 1;
    k_boundary_lift<<<flat_grid(c->N), 256, 0, s>>>(c->type, g, gb, c->N);
}

void launch_finish_solution(cfp_ctx* c, const double* x, const double* g, double* u, cudaStream_t s) {
    c->launches += 1;
    k_finish_solution<<<flat_grid(c->N), 256, 0, s>>>(c->type, x, g, u, c->N);
}

void launch_mask_unknowns(cfp_ctx* c, const double* in, double* out, cudaStream_t s) {
    c->launches += 1;
    k_mask_copy<double><<<flat_grid(c->N), 256, 0, s>>>(c->type, in, out, c->N);
}

}  // namespace cfp
