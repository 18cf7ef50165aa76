// Kernels of the learned part (an extension of the method, not in the
// paper): a 3D convolutional U-Net on the solver's grid, BF16 activations
// and weights, FP32 accumulation in tensor memory (tcgen05).
//
// Layout.  A level of the network holds its activations on the level's grid
// padded by one node on every side (nxp = nx + 2, ...), channels last: channel
// c of padded voxel (i, j, k) at ((k nyp + j) nxp + i) C + c.  The padding
// nodes hold zeros, so a 3x3x3 convolution with zero padding reads, for the
// tap of offset (dx, dy, dz), the rows v + dx + nxp (dy + nyp dz) of the
// activation matrix: 128 consecutive output rows read 128 consecutive input
// rows.  Weights: [Cout][27][Cin], tap t for (dz, dy, dx) = (t/9 - 1,
// (t/3)%3 - 1, t%3 - 1):
//     out[v][co] = bias[co] + sum_t sum_ci W[co][t][ci] in[v + off(t)][ci].
//
// Forward convolution (k_conv_tc; k_conv_march for 16 -> 16 and 16 -> 32
// channels and some 32 -> 64 ones): the implicit GEMM D (128 voxels x Cout) =
// sum over taps of A_t (128 x Cin) B_t^T.  For each (dy, dz) pair one window
// of 130 rows (the 128 outputs and one row either side) serves the three taps
// dx = -1, 0, 1, whose A operands start 0, 16 and 32 bytes into it (K-major,
// no swizzle).  The weights of the three taps come with it, in the operand
// layout (k_wpack), as one bulk copy.  The input gradient is the same kernel
// on flipped, transposed weights.
// The operand layout scatters a row's 8-channel pieces over planes.  With 32
// channels or more in and out the windows come by TMA, a box per plane.  With
// fewer the MMAs of a window are over before the TMA engine has placed it 16
// bytes at a time (2340 pieces per tile bound the 16-channel layers to 5 % of
// the tensor pipe), and four producer warps copy the windows with 16-byte
// cp.async at the shared-memory write rate instead.
// Weight gradient (k_wgrad_tc): D_t (Cin x Cout) = sum over voxels of
// X(v + off_t)^T G(v), both operands MN-major, the voxel shift again a
// start-address offset, windows by cp.async.  The windows of 128 / Cin (dy,
// dz) pairs lie one after the other in a stage, so one MMA's 128 rows are that
// many pairs' channels (with 16 channels a single pair would leave seven of
// eight rows idle, and reading the operand is what an MMA of 16 columns
// costs).  Per-chunk partials are summed in a fixed order (deterministic).
#pragma once

#include <cuda_bf16.h>

#include "cfp_tc.cuh"

namespace cfp {
namespace nn {

struct Pad {
    int nx, ny, nz;     // the level's grid
    int nxp, nyp, nzp;  // padded
    int Np;             // padded voxels (< 2^31)
};

enum { F_RELU = 1, F_MASK = 2, F_OUT_F32 = 4, F_ACCUM = 8 };

constexpr int kWin = 130;             // rows of a window: 128 outputs + one either side
// bytes of one 8-channel plane of a window / of a 128-voxel gradient tile: an
// odd number of 16-byte rows, so that the pieces of a voxel row, written
// together, fall into different banks
constexpr int kPlane = 137 * 16;
constexpr int kGPlane = 129 * 16;
constexpr int kTmaPlane = 136 * 16;   // of a window copied by TMA (destinations on 128-byte boundaries)
constexpr int kConvThreads = 288;     // warps 0-3 epilogue, 4-7 producers, 8 MMA issuer
constexpr int kProd = 128;            // producer threads

// 16 bytes global -> shared, asynchronous; zeros where ok is false (src is then
// not read)
__device__ __forceinline__ void copy16(unsigned dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
// one arrival on bar when every copy this thread has issued so far has landed.
// The thread goes on to the next stage at once; the MMA thread, which waits on
// bar, orders the copies before the tensor core's reads (async_after).  (With
// the fence on the producer's side a stage took the whole latency of its
// copies: the fence waits for the later stages' copies too.)
__device__ __forceinline__ void copy_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void copy_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void async_after() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// producer thread p's share of rows row0 .. row0 + nrows - 1 of an (Np x C)
// activation, channels 8 c0 .. 8 c0 + 8 NPL - 1, into NPL planes of PLANE bytes;
// rows outside [0, Np) become zeros
template <int NPL, int PLANE>
__device__ __forceinline__ void copy_rows(unsigned dst, const uint16_t* __restrict__ a, int C, int c0, int row0,
                                          int nrows, int Np, int p) {
#pragma unroll 4
    for (int q = p; q < nrows * NPL; q += kProd) {
        const int r = q / NPL, c = q % NPL, row = row0 + r;  // NPL is a power of two
        const bool ok = row >= 0 && row < Np;
        copy16(dst + c * PLANE + r * 16, a + (size_t)(ok ? row : 0) * C + 8 * (c0 + c), ok);
    }
}

__host__ __device__ constexpr int pow2ceil(int v) {
    int p = 32;
    while (p < v) p <<= 1;
    return p;
}
__host__ __device__ constexpr int rup(int v, int m) { return (v + m - 1) / m * m; }

__device__ __forceinline__ float bf2f(uint16_t h) { return __uint_as_float((uint32_t)h << 16); }
__device__ __forceinline__ uint16_t f2bf(float f) {
    const __nv_bfloat16 b = __float2bfloat16_rn(f);
    return *reinterpret_cast<const uint16_t*>(&b);
}
__device__ __forceinline__ bool bf_pos(uint16_t h) { return !(h & 0x8000u) && (h & 0x7fffu); }

__device__ __forceinline__ bool interior(const Pad& P, int row) {
    const int i = row % P.nxp, r = row / P.nxp, j = r % P.nyp, k = r / P.nyp;
    return i >= 1 && i <= P.nxp - 2 && j >= 1 && j <= P.nyp - 2 && k >= 1 && k <= P.nzp - 2;
}

// ------------------------------------------------------ forward convolution
template <int CIN, int COUT>
struct ConvCfg {
    static constexpr int KB = CIN < 64 ? CIN : 64;  // input channels per stage
    static constexpr int NKB = CIN / KB;
    static constexpr int NCH = KB / 8;              // 8-channel planes per stage
    // The windows by TMA (one producer thread), or by cp.async (four warps) where
    // a stage has few channels in or out: the TMA engine takes about two cycles
    // per 16-byte piece whatever the MMAs that wait for it do, the threads'
    // copies cost issue slots and a fence.  By TMA and by cp.async, us: 32 -> 32
    // at 129^3 369 : 427 (k_conv_march), 64 -> 64 736 : 807, 64 -> 128 at 65^3
    // 132 : 146, 128 -> 128 at 129^3 1667 : 1789, at 17^3 19.9 : 21.2; but 32 ->
    // 16 at 65^3 55 : 52, 16 -> 32 42 : 30 (k_conv_march).
    static constexpr bool TMA = CIN >= 32 && COUT >= 32;
    using In = std::conditional_t<TMA, CUtensorMap, const uint16_t*>;
    static constexpr int PWARPS = TMA ? 1 : kProd / 32;
    static constexpr int THREADS = 32 * (5 + PWARPS);
    static constexpr int PLANE = TMA ? kTmaPlane : kPlane;
    static constexpr int A_BYTES = NCH * PLANE;
    static constexpr int W_TAP = NCH * COUT * 16;   // one tap's weights for the stage's channels
    static constexpr int W_BYTES = 3 * W_TAP;
    static constexpr unsigned TX = W_BYTES + (TMA ? NCH * kWin * 16 : 0);  // bytes counted on a stage's barrier
    static constexpr int STAGE = rup(A_BYTES + W_BYTES, 128);
    static constexpr int S0 = (196 * 1024) / STAGE;
    static constexpr int STAGES = S0 > 8 ? 8 : S0;
    static_assert(STAGES >= 2, "shared memory");
    static constexpr int SPT = 9 * NKB;             // stages per 128-voxel tile
    static constexpr int TCOLS = pow2ceil(2 * COUT);  // two accumulators
    static constexpr int SMEM = 128 + STAGES * STAGE + (2 * STAGES + 5) * 8 + 16;
    // CTAs per SM: shared memory, tensor-memory columns and registers permitting, up to three
    static constexpr int PER0 = (220 * 1024) / SMEM;
    static constexpr int PER1 = 512 / TCOLS < PER0 ? 512 / TCOLS : PER0;
    static constexpr int PER = PER1 < 1 ? 1 : PER1 > 3 ? 3 : PER1;
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT <= 128, "channel counts");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// Packed weights of a convolution for k_conv_tc: for stage (kb, g), g = 3
// (dz + 1) + (dy + 1), the taps dx = -1, 0, 1, each as NCH planes of COUT
// rows x 8 input channels (16 bytes): element (kb, g, dx, c, co, e) =
// W[co][3 g + dx + 1][kb KB + 8 c + e].  FLIP: the weights of the input
// gradient of a layer whose weights w are [CIN][27][COUT] (this kernel's
// COUT and CIN swapped): W'[co][t][ci] = w[ci][26 - t][co].
template <int CIN, int COUT, bool FLIP>
__global__ void k_wpack(const uint16_t* __restrict__ w, uint16_t* __restrict__ out) {
    using C = ConvCfg<CIN, COUT>;
    const int n = COUT * 27 * CIN;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        int r = e;
        const int el = r % 8;
        r /= 8;
        const int co = r % COUT;
        r /= COUT;
        const int c = r % C::NCH;
        r /= C::NCH;
        const int dx = r % 3;
        r /= 3;
        const int g = r % 9;
        const int kb = r / 9;
        const int t = 3 * g + dx;
        const int ci = kb * C::KB + 8 * c + el;
        out[e] = FLIP ? w[((int64_t)ci * 27 + (26 - t)) * COUT + co] : w[((int64_t)co * 27 + t) * CIN + ci];
    }
}

// The epilogue of channels c0 .. c0 + 15 of one row, accumulated in v: bias,
// RELU, MASK, ACCUM as below; a padding row (in false) gets zeros.
template <int COUT>
__device__ __forceinline__ void conv_row16(float (&v)[16], int c0, int row, bool in, const float* __restrict__ bias,
                                           const uint16_t* __restrict__ act, int flags,
                                           uint16_t* __restrict__ out_bf, float* __restrict__ out_f) {
    if (!in) {
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = 0.f;
    } else {
        uint16_t am[16], ac[16];
        if (flags & F_MASK) {
            const uint4* ap = reinterpret_cast<const uint4*>(act + (size_t)row * COUT + c0);
            *reinterpret_cast<uint4*>(am) = ap[0];
            *reinterpret_cast<uint4*>(am + 8) = ap[1];
        }
        if ((flags & F_ACCUM) && !(flags & F_OUT_F32)) {
            const uint4* op = reinterpret_cast<const uint4*>(out_bf + (size_t)row * COUT + c0);
            *reinterpret_cast<uint4*>(ac) = op[0];
            *reinterpret_cast<uint4*>(ac + 8) = op[1];
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            float x = v[q] + (bias ? __ldg(bias + c0 + q) : 0.f);
            if (flags & F_RELU) x = fmaxf(x, 0.f);
            if ((flags & F_MASK) && !bf_pos(am[q])) x = 0.f;
            if ((flags & F_ACCUM) && !(flags & F_OUT_F32)) x += bf2f(ac[q]);
            v[q] = x;
        }
    }
    if (flags & F_OUT_F32) {
        float4* op = reinterpret_cast<float4*>(out_f + (size_t)row * COUT + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float4 o = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            if (flags & F_ACCUM) {
                const float4 p = op[q];
                o.x += p.x;
                o.y += p.y;
                o.z += p.z;
                o.w += p.w;
            }
            op[q] = o;
        }
    } else {
        uint16_t h[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) h[q] = f2bf(v[q]);
        uint4* op = reinterpret_cast<uint4*>(out_bf + (size_t)row * COUT + c0);
        op[0] = *reinterpret_cast<uint4*>(h);
        op[1] = *reinterpret_cast<uint4*>(h + 8);
    }
}

// The epilogue of one warp's 32 rows (this lane's: row), accumulated at acc;
// rows that are not valid are left alone (their lanes still take part in the
// tensor-memory loads, which are the whole warp's).
template <int COUT>
__device__ __forceinline__ void conv_rows(unsigned acc, int row, bool valid, const Pad& P, const float* __restrict__ bias,
                                          const uint16_t* __restrict__ act, int flags, uint16_t* __restrict__ out_bf,
                                          float* __restrict__ out_f) {
    const bool in = valid && interior(P, row);
#pragma unroll 1
    for (int c16 = 0; c16 < COUT / 16; ++c16) {
        float v[16];
        tc::tmem_ld16(acc + 16 * c16, v);
        if (valid) conv_row16<COUT>(v, 16 * c16, row, in, bias, act, flags, out_bf, out_f);
    }
}

// out (Np x COUT) = epilogue(conv(in, W) + bias): RELU max(., 0); MASK times
// [act > 0]; ACCUM adds the values already in out (BF16); OUT_F32 FP32
// output.  Padding rows get 0.  Bounded waits: a wait that runs out records
// a code in *err and that role stops issuing; every issued copy and MMA is
// waited for (bounded) before the tensor memory is released.
template <int CIN, int COUT>
__global__ void __launch_bounds__(ConvCfg<CIN, COUT>::THREADS, ConvCfg<CIN, COUT>::PER)
    k_conv_tc(const __grid_constant__ typename ConvCfg<CIN, COUT>::In in, const uint16_t* __restrict__ wpk,
              const float* __restrict__ bias, const uint16_t* __restrict__ act, Pad P, int flags,
              uint16_t* __restrict__ out_bf, float* __restrict__ out_f, int* __restrict__ err) {
    using C = ConvCfg<CIN, COUT>;
    constexpr int S = C::STAGES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    uint64_t* full = (uint64_t*)(base + S * C::STAGE);
    uint64_t* empty = full + S;
    uint64_t* accf = empty + S;  // accumulator b filled
    uint64_t* acce = accf + 2;   // accumulator b read out by the four epilogue warps
    uint64_t* fin = acce + 2;    // every MMA of this CTA completed
    unsigned* tslot = (unsigned*)(fin + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int q = 0; q < S; ++q) {
            tc::mbar_init(&full[q], C::TMA ? 1 : 1 + kProd);  // the bytes counted; the copying threads
            tc::mbar_init(&empty[q], 1);
        }
        for (int q = 0; q < 2; ++q) {
            tc::mbar_init(&accf[q], 1);
            tc::mbar_init(&acce[q], 4);
        }
        tc::mbar_init(fin, 1);
        tc::mbar_fence_init();
    }
    if (warp == 0) tc::tmem_alloc<C::TCOLS>(tslot);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = *tslot;
    const int ntiles = (P.Np + 127) / 128;

    if (warp >= 4 && warp < 4 + C::PWARPS && (!C::TMA || lane == 0)) {  // producers
        const int p = threadIdx.x - 128;
        unsigned g = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
            for (int s = 0; s < C::SPT; ++s, ++g) {
                const int kb = s / 9, gi = s % 9, st = g % S;
                int free = 1;
                if (g >= S && lane == 0 && !tc::mbar_wait(&empty[st], ((g / S) - 1) & 1)) {
                    free = 0;
                    atomicExch(err, 11);
                }
                ok = C::TMA ? free : __shfl_sync(0xffffffffu, free, 0);
                if (!ok) break;
                unsigned char* buf = base + st * C::STAGE;
                const int row0 = tile * 128 + ((gi / 3 - 1) * P.nyp + (gi % 3 - 1)) * P.nxp - 1;
                if (p == 0) {
                    tc::mbar_arrive_expect_tx(&full[st], C::TX);
                    if constexpr (C::TMA)
#pragma unroll
                        for (int c = 0; c < C::NCH; ++c)
                            tc::tma_load_2d(buf + c * C::PLANE, &in, &full[st], (kb * C::NCH + c) * 8, row0);
                    tc::bulk_load(buf + C::A_BYTES, wpk + (size_t)(kb * 9 + gi) * (C::W_BYTES / 2), C::W_BYTES, &full[st]);
                }
                if constexpr (!C::TMA) {
                    copy_rows<C::NCH, C::PLANE>(tc::smem_u32(buf), in, CIN, kb * C::NCH, row0, kWin, P.Np, p);
                    copy_arrive(&full[st]);
                }
            }
        }
        if constexpr (!C::TMA) copy_wait_all();
        if (p == 0)  // every bulk copy issued has landed before the CTA may end
            for (unsigned q = g > (unsigned)S ? g - S : 0; q < g; ++q)
                if (!tc::mbar_wait(&full[q % S], (q / S) & 1)) atomicExch(err, 12);
    } else if (warp == 4 + C::PWARPS && lane == 0) {  // MMA issuer
        constexpr unsigned idesc = tc::idesc_bf16(128, COUT, 0, 0);
        unsigned g = 0, tl = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++tl) {
            const unsigned b = tl & 1;
            if (tl >= 2 && !tc::mbar_wait(&acce[b], ((tl / 2) - 1) & 1)) {
                ok = false;
                atomicExch(err, 13);
                break;
            }
            tc::fence_after();
            const unsigned d = tmem + b * COUT;
            for (int s = 0; s < C::SPT; ++s, ++g) {
                const int st = g % S;
                if (!tc::mbar_wait(&full[st], (g / S) & 1)) {
                    ok = false;
                    atomicExch(err, 14);
                    break;
                }
                if constexpr (!C::TMA) async_after();
                tc::fence_after();
                const unsigned ab = tc::smem_u32(base + st * C::STAGE), wb = ab + C::A_BYTES;
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int q = 0; q < C::NCH / 2; ++q) {
                        const uint64_t da = tc::sdesc(ab + dx * 16 + q * 2 * C::PLANE, C::PLANE, 128);
                        const uint64_t db = tc::sdesc(wb + dx * C::W_TAP + q * 2 * COUT * 16, COUT * 16, 128);
                        tc::mma_bf16(d, da, db, idesc, (s | dx | q) != 0);
                    }
                tc::mma_commit(&empty[st]);
            }
            if (!ok) break;
            tc::mma_commit(&accf[b]);
        }
        tc::mma_commit(fin);
        if (!tc::mbar_wait(fin, 0)) atomicExch(err, 15);
    } else if (warp < 4) {  // epilogue: warp w reads tensor-memory lanes 32w .. 32w + 31
        unsigned tl = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++tl) {
            const unsigned b = tl & 1;
            int ok = 1;
            if (lane == 0 && !tc::mbar_wait(&accf[b], (tl / 2) & 1)) {
                ok = 0;
                atomicExch(err, 16);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            tc::fence_after();
            const int row = tile * 128 + 32 * warp + lane;
            conv_rows<COUT>(tmem + ((unsigned)(32 * warp) << 16) + b * COUT, row, row < P.Np, P, bias, act, flags, out_bf,
                            out_f);
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&acce[b]);
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        tc::tmem_free<C::TCOLS>(tmem);
    }
}

// The same convolution for few input channels, marching planes: a tile is 128
// consecutive voxels of a plane and a CTA takes it through a chunk of planes,
// so that a plane's three windows (dy = -1, 0, 1) are copied once and serve the
// outputs of three planes, and the 27 taps' weights stay in shared memory.
// k_conv_tc copies nine windows and the weights per tile, and with 16 channels
// those copies' issue bounds it (129 x 97 x 65, 16 -> 16: 58 % of the issue
// slots, 7 % of the tensor pipe, 76 us).  Here it takes 58 us, bound by a
// plane's chain of copy, 27 small MMAs and epilogue: two CTAs per SM instead of
// three take a third longer.  The products are added in the same order: the
// same bits.
template <int CIN, int COUT>
struct MarchCfg {
    static constexpr int NCH = CIN / 8;
    static constexpr int STAGE = rup(NCH * kPlane, 128);  // a window
    static constexpr int W_TAP = NCH * COUT * 16;
    static constexpr int W_BYTES = 27 * W_TAP;
    static constexpr int FIXED = W_BYTES + 128 + (2 * 18 + 6) * 8 + 16;
    static constexpr int TCOLS = pow2ceil(2 * COUT);
    // nine windows serve an output; CTAs per SM while twelve fit
    static constexpr int PER = 3 * (FIXED + 12 * STAGE) <= 220 * 1024   ? 3
                               : 2 * (FIXED + 12 * STAGE) <= 220 * 1024 ? 2
                                                                        : 1;
    static constexpr int S0 = (220 * 1024 / PER - FIXED) / STAGE;
    static constexpr int STAGES = S0 > 18 ? 18 : S0;
    static constexpr int SMEM = FIXED + STAGES * STAGE;
    static constexpr bool fits = (CIN == 16 || (CIN == 32 && COUT == 64)) && STAGES >= 12;
};

struct March {
    int tiles;     // 128-voxel tiles of a plane
    int planes;    // of a chunk
    int chunks;
    int64_t cost;  // planes that the SM with the most works through, one after the other
};

// as k_conv_tc; one CTA per unit (tile, chunk), tile fastest
template <int CIN, int COUT>
__global__ void __launch_bounds__(kConvThreads, MarchCfg<CIN, COUT>::PER)
    k_conv_march(const uint16_t* __restrict__ in, const uint16_t* __restrict__ wpk, const float* __restrict__ bias,
                 const uint16_t* __restrict__ act, Pad P, March M, int flags, uint16_t* __restrict__ out_bf,
                 float* __restrict__ out_f, int* __restrict__ err) {
    using C = MarchCfg<CIN, COUT>;
    constexpr unsigned S = C::STAGES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    unsigned char* wsm = base + S * C::STAGE;
    uint64_t* full = (uint64_t*)(wsm + C::W_BYTES);
    uint64_t* empty = full + S;
    uint64_t* accf = empty + S;  // accumulator b filled
    uint64_t* acce = accf + 2;   // accumulator b read out by the four epilogue warps
    uint64_t* wful = acce + 2;   // the weights
    uint64_t* fin = wful + 1;    // every MMA of this CTA completed
    unsigned* tslot = (unsigned*)(fin + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (unsigned q = 0; q < S; ++q) {
            tc::mbar_init(&full[q], kProd);
            tc::mbar_init(&empty[q], 1);
        }
        for (int q = 0; q < 2; ++q) {
            tc::mbar_init(&accf[q], 1);
            tc::mbar_init(&acce[q], 4);
        }
        tc::mbar_init(wful, 1);
        tc::mbar_init(fin, 1);
        tc::mbar_fence_init();
    }
    if (warp == 0) tc::tmem_alloc<C::TCOLS>(tslot);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = *tslot;
    const int plane = P.nxp * P.nyp;
    const int v0 = (int)(blockIdx.x % M.tiles) * 128;
    const int k0 = (int)(blockIdx.x / M.tiles) * M.planes, k1 = min(k0 + M.planes, P.nzp);

    if (warp >= 4 && warp < 8) {  // producers: windows (plane k0 - 1, dy = -1), (k0 - 1, 0), ...
        const int p = threadIdx.x - 128;
        if (p == 0) {
            tc::mbar_arrive_expect_tx(wful, C::W_BYTES);
            tc::bulk_load(wsm, wpk, C::W_BYTES, wful);
        }
        const unsigned nw = 3 * (k1 - k0 + 2);
        for (unsigned g = 0; g < nw; ++g) {
            const unsigned st = g % S;
            int free = 1;
            if (g >= S && lane == 0 && !tc::mbar_wait(&empty[st], ((g / S) - 1) & 1)) {
                free = 0;
                atomicExch(err, 17);
            }
            if (!__shfl_sync(0xffffffffu, free, 0)) break;
            const int row0 = (k0 - 1 + (int)(g / 3)) * plane + v0 + ((int)(g % 3) - 1) * P.nxp - 1;
            copy_rows<C::NCH, kPlane>(tc::smem_u32(base + st * C::STAGE), in, CIN, 0, row0, kWin, P.Np, p);
            copy_arrive(&full[st]);
        }
        copy_wait_all();
        if (p == 0 && !tc::mbar_wait(wful, 0)) atomicExch(err, 12);  // landed before the CTA may end
    } else if (warp == 8 && lane == 0) {  // MMA issuer
        constexpr unsigned idesc = tc::idesc_bf16(128, COUT, 0, 0);
        bool ok = tc::mbar_wait(wful, 0);
        if (!ok) atomicExch(err, 18);
        const unsigned wb = tc::smem_u32(wsm);
        unsigned got = 0;  // windows waited for
        for (int k = k0; k < k1 && ok; ++k) {
            const unsigned tl = k - k0, b = tl & 1;
            if (tl >= 2 && !tc::mbar_wait(&acce[b], ((tl / 2) - 1) & 1)) {
                atomicExch(err, 13);
                break;
            }
            tc::fence_after();
            const unsigned d = tmem + b * COUT;
            for (unsigned s = 0; s < 9; ++s) {  // 3 (dz + 1) + (dy + 1)
                const unsigned g = 3 * tl + s, st = g % S;
                if (g == got) {
                    if (!tc::mbar_wait(&full[st], (g / S) & 1)) {
                        ok = false;
                        atomicExch(err, 14);
                        break;
                    }
                    async_after();
                    tc::fence_after();
                    ++got;
                }
                const unsigned ab = tc::smem_u32(base + st * C::STAGE);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int q = 0; q < C::NCH / 2; ++q) {
                        const uint64_t da = tc::sdesc(ab + dx * 16 + q * 2 * kPlane, kPlane, 128);
                        const uint64_t db = tc::sdesc(wb + (3 * s + dx) * C::W_TAP + q * 2 * COUT * 16, COUT * 16, 128);
                        tc::mma_bf16(d, da, db, idesc, (s | dx | q) != 0);
                    }
            }
            if (!ok) break;
            tc::mma_commit(&accf[b]);
            for (unsigned s = 0; s < 3; ++s) tc::mma_commit(&empty[(3 * tl + s) % S]);  // plane k - 1 has served
        }
        tc::mma_commit(fin);
        if (!tc::mbar_wait(fin, 0)) atomicExch(err, 15);
    } else if (warp < 4) {  // epilogue: warp w reads tensor-memory lanes 32w .. 32w + 31
        for (int k = k0; k < k1; ++k) {
            const unsigned tl = k - k0, b = tl & 1;
            int ok = 1;
            if (lane == 0 && !tc::mbar_wait(&accf[b], (tl / 2) & 1)) {
                ok = 0;
                atomicExch(err, 16);
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            tc::fence_after();
            const int v = v0 + 32 * warp + lane;
            conv_rows<COUT>(tmem + ((unsigned)(32 * warp) << 16) + b * COUT, k * plane + v, v < plane, P, bias, act, flags,
                            out_bf, out_f);
            tc::fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&acce[b]);
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        tc::tmem_free<C::TCOLS>(tmem);
    }
}

// ------------------------------------------------------- weight gradient
template <int CIN, int COUT>
struct WgCfg {
    static constexpr int NCA = CIN / 8;                    // planes of one X window
    static constexpr int NCB = COUT / 8;                   // planes of the gradient tile
    static constexpr int GP = 16 / NCA;                    // (dy, dz) pairs of a unit: 128 rows of an MMA
    static constexpr int NU = (9 + GP - 1) / GP;           // units of the nine pairs
    static constexpr int A_BYTES = 16 * kPlane;
    static constexpr int B_BYTES = NCB * kGPlane;
    static constexpr int STAGE = rup(A_BYTES + B_BYTES, 128);
    static constexpr int U0 = 512 / (3 * COUT);
    static constexpr int UMAX = U0 > NU ? NU : U0;         // units per CTA
    static constexpr int NSETS = (NU + UMAX - 1) / UMAX;
    static constexpr int TCOLS = pow2ceil(3 * UMAX * COUT);
    static constexpr int S0 = (200 * 1024) / STAGE;
    static constexpr int STAGES = S0 > 8 ? 8 : S0;
    static_assert(STAGES >= 2, "shared memory");
    static constexpr int SMEM0 = 128 + STAGES * STAGE + (2 * STAGES + 3) * 8 + 16;
    // at least half an SM's shared memory: one CTA per SM, as it may take all
    // 512 tensor-memory columns
    static constexpr int SMEM = SMEM0 > 116 * 1024 ? SMEM0 : 116 * 1024;
    static_assert(CIN % 16 == 0 && CIN <= 128, "channel counts");
    static_assert(SMEM <= 227 * 1024, "shared memory");
    static_assert(TCOLS <= 512, "tensor memory");
};

// Partial weight gradient of one voxel chunk and one set of units:
// part[chunk][t][ci][co] = sum over the chunk's 128-voxel tiles of
// X[v + off(t)][ci] G[v][co].  Grid: (NSETS, nchunks); chunk q owns tiles
// [q * tpc, min((q + 1) * tpc, ntiles)).  A stage holds one tile's windows of
// one unit and its gradient tile; the rows of an MMA past the ninth pair are
// whatever the stage holds there, and are not read back.
template <int CIN, int COUT>
__global__ void __launch_bounds__(kConvThreads, 1)
    k_wgrad_tc(const uint16_t* __restrict__ x, const uint16_t* __restrict__ gr, Pad P, int tpc,
               float* __restrict__ part, int* __restrict__ err) {
    using C = WgCfg<CIN, COUT>;
    constexpr int S = C::STAGES;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    uint64_t* full = (uint64_t*)(base + S * C::STAGE);
    uint64_t* empty = full + S;
    uint64_t* accf = empty + S;
    uint64_t* fin = accf + 1;
    unsigned* tslot = (unsigned*)(fin + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int set = blockIdx.x, chunk = blockIdx.y;
    const int u0 = set * C::UMAX, nu = min(C::NU - u0, C::UMAX);
    const int ntiles = (P.Np + 127) / 128;
    const int t0 = chunk * tpc, t1 = min(ntiles, t0 + tpc);
    if (threadIdx.x == 0) {
        for (int q = 0; q < S; ++q) {
            tc::mbar_init(&full[q], kProd);
            tc::mbar_init(&empty[q], 1);
        }
        tc::mbar_init(accf, 1);
        tc::mbar_init(fin, 1);
        tc::mbar_fence_init();
    }
    if (warp == 0) tc::tmem_alloc<C::TCOLS>(tslot);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = *tslot;
    const int nst = (t1 > t0 ? t1 - t0 : 0) * nu;

    if (warp >= 4 && warp < 8) {  // producers
        const int p = threadIdx.x - 128;
        unsigned g = 0;
        for (; (int)g < nst; ++g) {
            const int tile = t0 + (int)g / nu, u = u0 + (int)g % nu, st = g % S;
            int free = 1;
            if (g >= (unsigned)S && lane == 0 && !tc::mbar_wait(&empty[st], ((g / S) - 1) & 1)) {
                free = 0;
                atomicExch(err, 21);
            }
            if (!__shfl_sync(0xffffffffu, free, 0)) break;
            const unsigned buf = tc::smem_u32(base + st * C::STAGE);
#pragma unroll
            for (int q = 0; q < C::GP; ++q) {
                const int gi = u * C::GP + q;
                if (gi < 9)
                    copy_rows<C::NCA, kPlane>(buf + q * C::NCA * kPlane, x, CIN, 0,
                                              tile * 128 + ((gi / 3 - 1) * P.nyp + (gi % 3 - 1)) * P.nxp - 1, kWin, P.Np, p);
            }
            copy_rows<C::NCB, kGPlane>(buf + C::A_BYTES, gr, COUT, 0, tile * 128, 128, P.Np, p);
            copy_arrive(&full[st]);
        }
        copy_wait_all();
    } else if (warp == 8 && lane == 0) {  // MMA issuer
        constexpr unsigned idesc = tc::idesc_bf16(128, COUT, 1, 1);
        for (int g = 0; g < nst; ++g) {
            const int st = g % S, first = g < nu;  // the chunk's first tile: the accumulators start
            const int ul = g % nu;
            if (!tc::mbar_wait(&full[st], (g / S) & 1)) {
                atomicExch(err, 23);
                break;
            }
            async_after();
            tc::fence_after();
            const unsigned ab = tc::smem_u32(base + st * C::STAGE), bb = ab + C::A_BYTES;
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                const unsigned d = tmem + (unsigned)((ul * 3 + dx) * COUT);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint64_t da = tc::sdesc(ab + dx * 16 + q * 256, 128, kPlane);
                    const uint64_t db = tc::sdesc(bb + q * 256, 128, kGPlane);
                    tc::mma_bf16(d, da, db, idesc, !(first && q == 0));
                }
            }
            tc::mma_commit(&empty[st]);
        }
        tc::mma_commit(accf);
        tc::mma_commit(fin);
        if (!tc::mbar_wait(fin, 0)) atomicExch(err, 24);
    } else if (warp < 4) {  // epilogue: row 32 warp + lane is channel ci of pair `pair` of a unit
        int ok = 1;
        if (nst > 0) {
            if (lane == 0 && !tc::mbar_wait(accf, 0)) {
                ok = 0;
                atomicExch(err, 25);
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
        }
        if (ok) {
            tc::fence_after();
            const int row = 32 * warp + lane, pair = row / CIN, ci = row % CIN;
            for (int ul = 0; ul < nu; ++ul)
                for (int dx = 0; dx < 3; ++dx) {
                    const int gi = (u0 + ul) * C::GP + pair, t = 3 * gi + dx;
#pragma unroll 1
                    for (int c16 = 0; c16 < COUT / 16; ++c16) {
                        float v[16];
                        tc::tmem_ld16(tmem + ((unsigned)(32 * warp) << 16) + (unsigned)((ul * 3 + dx) * COUT + 16 * c16), v);
                        if (gi < 9) {
                            float4* op = reinterpret_cast<float4*>(
                                part + (((size_t)chunk * 27 + t) * CIN + ci) * COUT + 16 * c16);
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                op[q] = nst > 0 ? make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3])
                                                : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
                    }
                }
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        tc::tmem_free<C::TCOLS>(tmem);
    }
}

}  // namespace nn
}  // namespace cfp
