// Weight and bias gradients of the surrogate's periodic 3x3x3 convolutions on
// the 5th-generation tensor cores (tcgen05.mma, accumulators in TMEM):
//   dW[o][co][ci] = sum_v dz[v][co] x[v + off(o)][ci],  db[co] = sum_v dz[v][co].
//
// The contraction runs over voxels, so both operands are MN-major: with
// channels last a voxel's eight channels are one 16-byte row of a no-swizzle
// core matrix and eight voxels of a grid row one core matrix.  Per 16 voxels
// of a row (K = 16) one MMA takes
//   A (M = 128): dz of the planes q-1, q, q+1 (and a fourth, ignored),
//                channels of one plane after the other -- dz offsets +1, 0, -1
//                of x plane q;
//   B (N = 3 Cin): x plane q at the rows y-1, y, y+1, started one of three
//                voxels apart for dx = -1, 0, +1;
// and adds to the TMEM block of its dx, so three MMAs serve all 27 offsets.
// The rows y-1 .. y+1 of x and the planes of dz must follow each other at one
// stride (a descriptor has one per direction): x is stored [row][Cin / 8]
// [18 voxels][8], dz [row][plane slot][Cout / 8][16 voxels + 2][8].  A window
// of dz slots must not wrap, so the first two of seven slots are written twice
// (after the seventh again).  288-byte runs keep the copies' 16-byte writes
// off each other's banks.
//
// A CTA marches planes of 16 x 8 voxel columns, an equal run of (column,
// plane) steps for every SM, and keeps its sums in TMEM throughout (3 x 96
// columns); the slices are added up in CTA order by a second kernel, so the
// result is the same every run.  Roles, meeting at mbarriers: three
// threads issue MMAs (one per dx, each into its own TMEM block, so that one
// thread's waits and commits hide behind the others' MMAs), eight warps copy
// (cp.async, three steps in flight, proxy fence once landed), one warp adds
// up dz for the bias.  Every wait is bounded and reports ST_TIMEOUT, which the
// calls that hand out or use the gradients turn into RKL_ERR_TIMEOUT.
//
// 32 -> 32 channels: 128^3 121 us with the slices' sum (the warp-level
// mma.sync kernel before it: about 360), 96^3 64 us (about 180).  The MMAs alone
// (three of 128 x 96 x 16 per 16 voxels, a quarter of M idle) take 97 us of
// the 121, the copies alone 113; with one issuing thread it was 157 us, with
// a window of three steps 222 us (each step then waited for the one before).
#include <algorithm>
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "rkl_conv.h"
#include "rkl_pair.cuh"

namespace rkl {
namespace conv {
namespace {

using x2::cp16;
using x2::cp_commit;
using x2::cp_wait;
using x2::mbar_init;
using x2::mbar_try_wait;
using x2::smem_u32;

constexpr int BX = 16, BY = 8;                  // voxels of a step
constexpr int HXW = BX + 2, HYW = BY + 2;       // x plane with its halo
constexpr int RUN = HXW * 16;                   // bytes of one (row, 8 channels) run
constexpr int WIN = 5, LAG = 2;                 // steps the copies run ahead of the MMAs; of them, in flight
constexpr int NZS = WIN + 2, NPOS = NZS + 3;    // dz slots; and with the repeated two and one that a window may touch
constexpr int NXS = WIN + 1;                    // x slots
constexpr int NB = 8;                           // barriers per kind
constexpr int NMW = 3, NLW = 8, NLT = 32 * NLW; // MMA warps (one per dx), copy warps
constexpr int NTHR_W = 32 * (NMW + NLW + 1);    // and one for the bias
constexpr int TMEM_ALL = 512;

template <int CIN, int COUT>
struct WSmem {
    static constexpr int NCI = CIN / 8, NCO = COUT / 8;
    alignas(128) unsigned char X[NXS][HYW * NCI * RUN];
    // with 16 channels the last row's window reaches past its slots (ignored rows of M)
    alignas(128) unsigned char Z[BY * NPOS * NCO * RUN + (NCO == 2 ? 4 * NCO * RUN : 0)];
    unsigned long long full[NB], empty[NB], done;
    unsigned tmem;
};

__device__ __forceinline__ uint64_t sdesc_w(unsigned addr, unsigned lbo, unsigned sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// kind::f16: FP32 accumulator, BF16 A and B, both MN-major, M = 128
template <int N>
__device__ __forceinline__ unsigned idesc_w()
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((unsigned)(N >> 3) << 17) |
           ((unsigned)(128 >> 4) << 24);
}
__device__ __forceinline__ void mma_w(unsigned dtmem, uint64_t a, uint64_t b, unsigned id, unsigned accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(id), "r"(accumulate));
}
__device__ __forceinline__ void commit_w(unsigned bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}
__device__ __forceinline__ void arrive_w(unsigned bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void zero16(unsigned d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};\n" ::"r"(d), "r"(0u) : "memory");
}
__device__ __forceinline__ void tmem_ld16w(unsigned taddr, float* v)
{
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// Bounded wait; false if it gave up.
__device__ __forceinline__ bool wait_w(unsigned long long& bar, unsigned parity, int limit = 1 << 24)
{
    for (int it = 0; it < limit; ++it)
        if (mbar_try_wait(smem_u32(&bar), parity)) return true;
    return false;
}
__device__ __forceinline__ int wrapw(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// The CTA's run of (column, plane) units as segments of one column each.
// Per segment of planes [z0, z1) the steps q = z0 - 3 .. z1 follow: step q
// brings x plane q and dz plane q + 1; dz planes outside the segment are
// zero, the first two steps bring only those and issue no MMA.
struct Seg {
    int col, z0, z1;
};
__device__ __forceinline__ bool next_seg(int& u, int u1, int D, Seg& s)
{
    if (u >= u1) return false;
    s.col = u / D;
    s.z0 = u % D;
    s.z1 = min(D, s.z0 + (u1 - u));
    u += s.z1 - s.z0;
    return true;
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(NTHR_W, 1)
wgrad_tc_kernel(const __nv_bfloat16* __restrict__ dz, const __nv_bfloat16* __restrict__ x, float* __restrict__ part,
                float* __restrict__ partb, int D, int H, int W, int per, unsigned* status)
{
    using S = WSmem<CIN, COUT>;
    constexpr int NCI = S::NCI, NCO = S::NCO, N = 3 * CIN;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    S& sm = *reinterpret_cast<S*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ncolx = W / BX, units = ncolx * (H / BY) * D;
    const int ubeg = blockIdx.x * per, u1 = min(units, ubeg + per);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&sm.tmem)),
                     "r"(TMEM_ALL)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < NB; ++i) {
            mbar_init(smem_u32(&sm.full[i]), NLW);
            mbar_init(smem_u32(&sm.empty[i]), NMW + 1u);      // MMAs of the step, bias warp
        }
        mbar_init(smem_u32(&sm.done), NMW);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tbase = sm.tmem;
    const unsigned xbase = smem_u32(&sm.X[0][0]), zbase = smem_u32(&sm.Z[0]);
    // bounded waits; a thread whose wait gave up skips its later ones
    bool ok = true;
    auto wait = [&](unsigned long long& bar, unsigned parity) { ok = ok && wait_w(bar, parity); };

    Seg sg;
    int u = ubeg;
    unsigned t = 0;                              // steps so far
    if (warp < NMW) {
        if (lane == 0) {
            const int j = warp;
            const unsigned id = idesc_w<N>();
            unsigned acc = 0u;
            while (next_seg(u, u1, D, sg))
                for (int q = sg.z0 - 3; q <= sg.z1; ++q, ++t) {
                    wait(sm.full[t % NB], (t / NB) & 1u);
                    if (q >= sg.z0 - 1) {
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        // dz planes q - 1, q, q + 1 came with steps t - 2, t - 1, t
                        const unsigned wz = (t - 2) % NZS;
                        const uint64_t a0 = sdesc_w(zbase + wz * (NCO * RUN), 128, RUN);
                        const uint64_t b0 = sdesc_w(xbase + (t % NXS) * (unsigned)sizeof(sm.X[0]), 128, RUN);
#pragma unroll
                        for (int y = 0; y < BY; ++y)
                            mma_w(tbase + j * N, a0 + (uint64_t)((y * NPOS * NCO * RUN) >> 4),
                                  b0 + (uint64_t)((y * NCI * RUN + j * 16) >> 4), id, acc | (unsigned)(y > 0));
                        acc = 1u;
                    }
                    commit_w(smem_u32(&sm.empty[t % NB]));
                }
            commit_w(smem_u32(&sm.done));
        }
    } else if (warp < NMW + NLW) {
        const int lt = tid - 32 * NMW;
        constexpr int NZT = BX * BY * NCO / NLT, NXT = (HXW * HYW * NCI + NLT - 1) / NLT;
        static_assert(BX * BY * NCO % NLT == 0, "dz copies");
        unsigned zdst[NZT], xdst[NXT];
        int zoff[NZT], xoff[NXT];
#pragma unroll
        for (int i = 0; i < NZT; ++i) {
            const int k = lt + i * NLT, m = k / NCO, cc = k % NCO;
            zdst[i] = (unsigned)(((m / BX) * NPOS * NCO + cc) * RUN + (m % BX) * 16);
        }
#pragma unroll
        for (int i = 0; i < NXT; ++i) {
            const int k = lt + i * NLT, hv = k / NCI, cc = k % NCI;
            xdst[i] = (unsigned)(((hv / HXW) * NCI + cc) * RUN + (hv % HXW) * 16);
        }
        auto land = [&](unsigned s) {            // step s's copies of this thread have landed
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) arrive_w(smem_u32(&sm.full[s % NB]));
        };
        while (next_seg(u, u1, D, sg)) {
            const int x0 = (sg.col % ncolx) * BX, y0 = (sg.col / ncolx) * BY;
#pragma unroll
            for (int i = 0; i < NZT; ++i) {
                const int k = lt + i * NLT, m = k / NCO, cc = k % NCO;
                zoff[i] = ((y0 + m / BX) * W + x0 + m % BX) * COUT + cc * 8;
            }
#pragma unroll
            for (int i = 0; i < NXT; ++i) {
                const int k = lt + i * NLT, hv = k / NCI, cc = k % NCI;
                xoff[i] = k < HXW * HYW * NCI ? (wrapw(y0 + hv / HXW - 1, H) * W + wrapw(x0 + hv % HXW - 1, W)) * CIN + cc * 8
                                              : -1;
            }
            for (int q = sg.z0 - 3; q <= sg.z1; ++q, ++t) {
                // x slot t % 6 was last read by step t - 6, dz slot t % 7 by step t - 5
                if (t >= WIN) {
                    if (lane == 0) wait(sm.empty[(t - WIN) % NB], ((t - WIN) / NB) & 1u);
                    __syncwarp();
                }
                const unsigned zs = t % NZS, zb = zbase + zs * (NCO * RUN);
                if (q + 1 >= sg.z0 && q + 1 < sg.z1) {
                    const __nv_bfloat16* p = dz + (int64_t)(q + 1) * H * W * COUT;
#pragma unroll
                    for (int i = 0; i < NZT; ++i) {
                        cp16(zb + zdst[i], p + zoff[i]);
                        if (zs < 2) cp16(zb + NZS * NCO * RUN + zdst[i], p + zoff[i]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < NZT; ++i) {
                        zero16(zb + zdst[i]);
                        if (zs < 2) zero16(zb + NZS * NCO * RUN + zdst[i]);
                    }
                }
                if (q >= sg.z0 - 1) {
                    const __nv_bfloat16* p = x + (int64_t)wrapw(q, D) * H * W * CIN;
                    const unsigned xb = xbase + (t % NXS) * (unsigned)sizeof(sm.X[0]);
#pragma unroll
                    for (int i = 0; i < NXT; ++i)
                        if (xoff[i] >= 0) cp16(xb + xdst[i], p + xoff[i]);
                }
                cp_commit();
                if (t >= LAG) {
                    cp_wait<LAG>();
                    land(t - LAG);
                }
            }
        }
        cp_wait<0>();
        for (unsigned k = t >= LAG ? t - LAG : 0u; k < t; ++k) land(k);
    } else {
        // bias: a lane adds up 8 channels (chunk lane % 4) of every eighth voxel
        const int cc = lane & 3, v0 = lane >> 2;
        float s8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        while (next_seg(u, u1, D, sg))
            for (int q = sg.z0 - 3; q <= sg.z1; ++q, ++t) {
                wait(sm.full[t % NB], (t / NB) & 1u);
                if (COUT == 32 && q + 1 >= sg.z0 && q + 1 < sg.z1) {
                    const unsigned char* Z = sm.Z + ((t % NZS) * NCO + cc) * RUN + v0 * 16;
#pragma unroll
                    for (int k = 0; k < BX * BY / 8; ++k) {
                        const uint4 v = *reinterpret_cast<const uint4*>(Z + (k / 2) * (NPOS * NCO * RUN) + (k % 2) * 128);
                        const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            s8[2 * c] += __uint_as_float(w[c] << 16);
                            s8[2 * c + 1] += __uint_as_float(w[c] & 0xffff0000u);
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) arrive_w(smem_u32(&sm.empty[t % NB]));
            }
        if (COUT == 32) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) s8[c] += __shfl_xor_sync(0xffffffffu, s8[c], o);
                if (v0 == 0) partb[(int64_t)blockIdx.x * COUT + cc * 8 + c] = s8[c];
            }
        }
    }
    // drain: TMEM lane = row of M = (plane r, channel co), r = 0, 1, 2 for dz
    // offsets +1, 0, -1; warps 4 .. 7 reach the lane quarters 0 .. 3
    __syncwarp();
    if (warp >= 4 && warp < 8) {
        // also after a wait that gave up: TMEM is given back only once the MMAs have ended
        ok = wait_w(sm.done, 0u) && ok;
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const int m = (warp & 3) * 32 + lane, r = m / COUT, co = m % COUT;
        const unsigned tl = tbase + ((unsigned)((warp & 3) * 32) << 16);
        if ((warp & 3) * 32 < 3 * COUT) {        // whole warps
            float* dst = part + (int64_t)blockIdx.x * (27 * COUT * CIN) + (int64_t)(2 - r) * 9 * COUT * CIN + co * CIN;
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int c = 0; c < N; c += 16) {
                    float v[16];
                    tmem_ld16w(tl + j * N + c, v);
                    if (r < 3) {
                        float4* o = reinterpret_cast<float4*>(dst + ((c / CIN) * 3 + j) * COUT * CIN + c % CIN);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            o[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
                    }
                }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tbase), "r"(TMEM_ALL) : "memory");
    }
    if (!ok && status) atomicOr(status, ST_TIMEOUT);
}

// One wait of the kernel above, short, on a barrier that nothing arrives at.
__global__ void wait_selftest_kernel(unsigned* status)
{
    __shared__ unsigned long long bar;
    mbar_init(smem_u32(&bar), 1u);
    if (!wait_w(bar, 0u, 64)) atomicOr(status, ST_TIMEOUT);
}

// dW[i] = sum of the slices part[b][i] in a fixed order (eight strided runs,
// then their sums), and db likewise from the last block.
constexpr int kSumRuns = 8;
__global__ void __launch_bounds__(32 * kSumRuns)
sum_slices_kernel(const float* __restrict__ part, const float* __restrict__ partb, int nparts, int n, int nb,
                  bool with_bias, float* __restrict__ dW, float* __restrict__ db)
{
    const int l = threadIdx.x & 31, r = threadIdx.x >> 5;
    const bool bias = with_bias && blockIdx.x == gridDim.x - 1;
    const float* p = bias ? partb : part;
    const int len = bias ? nb : n, i = bias ? l : blockIdx.x * 32 + l;
    float s = 0.f;
    if (i < len) {
#pragma unroll 8
        for (int b = r; b < nparts; b += kSumRuns) s += p[(int64_t)b * len + i];
    }
    __shared__ float sh[kSumRuns][32];
    sh[r][l] = s;
    __syncthreads();
    if (r == 0 && i < len) {
        float a = 0.f;
#pragma unroll
        for (int k = 0; k < kSumRuns; ++k) a += sh[k][l];
        (bias ? db : dW)[i] = a;
    }
}

// Bias gradient of the head (16 channels).  Its dz is the adjoint of a
// divergence, so the channel sums cancel down to the rounding of their terms
// and the order of the additions decides the digits that are left: they keep
// one fixed order, over tiles of 4 x 8 x 16 voxels (block b takes tiles b, b +
// gridDim, ...), 32 voxel classes a tile, then the classes, then the blocks.
// The tiles stream through shared memory, three in flight, so that the fixed
// order costs no memory latency (reading them where they are added took 65
// us at 96^3).
constexpr int kHeadThreads = 512, kHeadStages = 4, kHeadTile = 4 * 8 * 16;
__global__ void __launch_bounds__(kHeadThreads)
head_bias_kernel(const __nv_bfloat16* __restrict__ dz, float* __restrict__ partb, int D, int H, int W)
{
    constexpr int TZ = 4, TY = 8, TX = 16, COUT = 16, NC = 32;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __nv_bfloat16* buf = reinterpret_cast<__nv_bfloat16*>(smem_raw);          // [kHeadStages][512][16]
    const int tid = threadIdx.x, ch = tid % COUT, k = tid / COUT;
    const int tilesx = W / TX, tilesy = H / TY, ntiles = tilesx * tilesy * (D / TZ);
    auto load = [&](int tile, int slot) {
        if (tile < ntiles) {
            const int x0 = tile % tilesx * TX, y0 = tile / tilesx % tilesy * TY, z0 = tile / (tilesx * tilesy) * TZ;
#pragma unroll
            for (int i = 0; i < 2; ++i) {                                     // 1024 chunks of 16 bytes
                const int q = tid + i * kHeadThreads, m = q >> 1;
                const int64_t gv = ((int64_t)(z0 + m / (TX * TY)) * H + y0 + m / TX % TY) * W + x0 + m % TX;
                cp16(smem_u32(buf + (slot * kHeadTile + m) * COUT + (q & 1) * 8), dz + gv * COUT + (q & 1) * 8);
            }
        }
        cp_commit();
    };
    const int step = gridDim.x;
    for (int i = 0; i < kHeadStages - 1; ++i) load(blockIdx.x + i * step, i);
    float s = 0.f;
    int slot = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += step) {
        cp_wait<kHeadStages - 2>();
        __syncthreads();
        load(tile + (kHeadStages - 1) * step, (slot + kHeadStages - 1) % kHeadStages);
        const __nv_bfloat16* b = buf + slot * kHeadTile * COUT;
#pragma unroll
        for (int m = 0; m < kHeadTile; m += NC) s += __bfloat162float(b[(m + k) * COUT + ch]);
        slot = (slot + 1) % kHeadStages;
    }
    cp_wait<0>();
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem_raw);
    red[tid] = s;
    __syncthreads();
    if (tid < COUT) {
        float t = 0.f;
        for (int q = 0; q < NC; ++q) t += red[q * COUT + tid];
        partb[(int64_t)blockIdx.x * COUT + tid] = t;
    }
}

// db[c] = sum of partb[b][c], b ascending
__global__ void head_bias_sum_kernel(const float* __restrict__ partb, int nparts, float* __restrict__ db)
{
    constexpr int COUT = 16;
    __shared__ float sh[256 * COUT];
    float t = 0.f;
    for (int b0 = 0; b0 < nparts; b0 += 256) {
        const int n = min(256, nparts - b0) * COUT;
        for (int i = threadIdx.x; i < n; i += blockDim.x) sh[i] = partb[(int64_t)b0 * COUT + i];
        __syncthreads();
        if (threadIdx.x < COUT) {
#pragma unroll 8
            for (int i = threadIdx.x; i < n; i += COUT) t += sh[i];
        }
        __syncthreads();
    }
    if (threadIdx.x < COUT) db[threadIdx.x] = t;
}

template <int CIN, int COUT>
cudaError_t wgrad_tc_t(const void* dz, const void* x, float* dW, float* db, float* part, int D, int H, int W,
                       unsigned* status, cudaStream_t st)
{
    // more than half an SM's shared memory: one CTA (and its TMEM) per SM
    const int smem = (int)std::max<size_t>(sizeof(WSmem<CIN, COUT>), 116 * 1024);
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(wgrad_tc_kernel<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const int64_t units = (int64_t)(W / BX) * (H / BY) * D;
    const int per = (int)std::max<int64_t>(4, (units + wgrad_max_ctas() - 1) / wgrad_max_ctas());
    const int grid = (int)((units + per - 1) / per);
    float* partb = part + (size_t)wgrad_max_ctas() * 27 * COUT * CIN;
    wgrad_tc_kernel<CIN, COUT><<<grid, NTHR_W, smem, st>>>(static_cast<const __nv_bfloat16*>(dz),
                                                          static_cast<const __nv_bfloat16*>(x), part, partb, D, H, W,
                                                          per, status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int n = 27 * COUT * CIN;
    // the last block adds up the bias slices
    sum_slices_kernel<<<n / 32 + (COUT == 32), 32 * kSumRuns, 0, st>>>(part, partb, grid, n, COUT, COUT == 32, dW, db);
    if ((e = cudaGetLastError()) != cudaSuccess || COUT == 32) return e;
    const int ntiles = (D / 4) * (H / BY) * (W / BX), nb = std::min(ntiles, wgrad_max_ctas());
    constexpr int hsm = kHeadStages * kHeadTile * 16 * 2;
    static bool hattr = false;
    if (!hattr) {
        if ((e = cudaFuncSetAttribute(head_bias_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, hsm)) != cudaSuccess)
            return e;
        hattr = true;
    }
    head_bias_kernel<<<nb, kHeadThreads, hsm, st>>>(static_cast<const __nv_bfloat16*>(dz), partb, D, H, W);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    head_bias_sum_kernel<<<1, 512, 0, st>>>(partb, nb, db);
    return cudaGetLastError();
}

}  // namespace

cudaError_t wait_selftest(unsigned* status, cudaStream_t st)
{
    wait_selftest_kernel<<<1, 1, 0, st>>>(status);
    return cudaGetLastError();
}

cudaError_t conv_wgrad_tc(int cin, int cout, const void* dz, const void* x, float* dW, float* db, float* part, int D,
                          int H, int W, unsigned* status, cudaStream_t st)
{
    if (H % BY || W % BX || D % 4) return cudaErrorInvalidValue;
    if ((int64_t)H * W * 32 > ((int64_t)1 << 31)) return cudaErrorInvalidValue;       // 31-bit in-plane offsets
    if (cin == 16 && cout == 32) return wgrad_tc_t<16, 32>(dz, x, dW, db, part, D, H, W, status, st);
    if (cin == 32 && cout == 32) return wgrad_tc_t<32, 32>(dz, x, dW, db, part, D, H, W, status, st);
    if (cin == 32 && cout == 16) return wgrad_tc_t<32, 16>(dz, x, dW, db, part, D, H, W, status, st);
    return cudaErrorInvalidValue;
}

}  // namespace conv
}  // namespace rkl
