// 3x3 periodic convolutions of the surrogate on the 5th-generation tensor
// cores, warp-specialised: 64 -> 64 (forward layers and input gradients), 16 ->
// 64 (the lift layer and the projection's input gradient) and 64 -> 16 (the
// projection, four channels of which are kept, in FP32).
//
// The output is cut into rows of 128 pixels (one MMA M); a CTA walks down
// 128-pixel strips, each a contiguous run of rows. Roles, handing over by
// mbarriers only (every wait bounded in time):
//   warp 0        tensor copies of the input rows (64 channels) into a ring of
//                 slots: 128 pixels, and 8 more on each side of which one is
//                 the periodic halo (8-pixel boxes start on the 1024-byte
//                 atoms of the 128-byte swizzle; narrow strips are filled by
//                 8-pixel boxes only);
//   warps 12-15   apply ReLU to a slot in place (where the layer wants it); with
//                 16 channels they copy the rows, 16 bytes at a time, six rows
//                 ahead;
//   warp 1        issues the MMAs, input-stationary: input row li feeds output
//                 rows li - 2, li - 1 and li through taps dy = +1, 0, -1, whose
//                 weights sit side by side in N, so one MMA (M = 128 pixels, N =
//                 3 COUT, K = 16) applies one (dx, 16-channel) step to three
//                 output rows. Output row t accumulates in block t % 8 of tensor
//                 memory (COUT columns); a step is cut in two where the blocks
//                 wrap around. The epilogue leaves a block zeroed, so every MMA
//                 accumulates. Each output sums its 9 CIN / 16 K-steps in the
//                 order (dy, dx, channel chunk);
//   warps 4-11    two epilogue groups of 4 warps take the output rows in turn:
//                 tensor memory -> registers (a thread is a pixel), bias, mask,
//                 residual, ReLU, BF16, into one of the group's two staging
//                 rows, from where one tensor store writes it. The residual row
//                 is brought into the same staging row by a tensor copy, one row
//                 of the group ahead. Masks are kept as one bit per channel: 8
//                 bytes per pixel instead of the 128 of the activation whose sign
//                 they are, written by the forward layer that computes it. The
//                 projection's four FP32 channels go straight to memory, 16 bytes
//                 a thread.
//
// What bounds it (1024 x 1024, one image): 268 MB per 64 -> 64 layer without and
// 402 MB with the residual, 40 and 59 us at the measured copy bandwidth, against 35 us
// of MMAs; without the residual copies the 12 layers of a forward pass take 133
// us less, without any epilogue 230 us less. A forward pass takes 1269 us where
// the layers with two block barriers per row and copies by the threads took
// 1889, a training step on 8 x 256 x 256 3310 instead of 4625. The lift and the
// projection, 168 MB each (25 us), take 47.6 and 42.5 us instead of 74.9 and 92.6 (the
// forward pass by then 1103 -> 992). The descriptors have to be warp-uniform: with
// one lane walking the rows each MMA cost its thread about 130 cycles (1428 us per
// forward pass).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "lbm_conv.h"
#include "lbm_conv64.cuh"
#include "lbm_launch.cuh"
#include "lbm_ptx.cuh"
#include "lbm_tc.cuh"

namespace lbm {
namespace {

constexpr int C6_BLK = 8;                  // accumulator blocks in tensor memory
constexpr int C6_THREADS = 512;

template <int CIN, int COUT>
struct TcCfg {
    static constexpr int KC = CIN / 16;                      // K steps of 16 channels
    static constexpr int SLOTS = CIN == 64 && COUT == 64 ? 4 : 8;  // input-row ring
    // Input rows. 64 channels: one 128-byte row per pixel, 128-byte swizzle. 16:
    // [2 groups of 8 channels][pixel][16 bytes], no swizzle (rows of 32 bytes are
    // a fourth of the line the copy engine moves at a time, so these are copied
    // by threads).
    static constexpr int GS = (C6_W + 3) * 16;               // bytes of a channel group
    static constexpr int SLOT = CIN == 64 ? C6_SLOT : (2 * GS + 127) / 128 * 128;
    // weights of one dx: rows n = block (dy = +1, 0, -1) * COUT + co, laid out as
    // the input
    static constexpr int WGS = 3 * COUT * 16;
    static constexpr int WROW = CIN == 64 ? 128 : 16;        // bytes from one n to the next
    static constexpr int WDX = CIN == 64 ? 3 * COUT * 128 : 2 * WGS;
    static constexpr int OFF_IN = 3 * WDX;
    static constexpr int OFF_OUT = OFF_IN + SLOTS * SLOT;    // staging rows of BF16 outputs
    static constexpr int BYTES = (COUT == 64 ? (OFF_OUT + 1023) / 1024 * 1024 + 4 * C6_ROW : OFF_OUT) + 1024;
    static constexpr int TMEM = C6_BLK * COUT;               // tensor-memory columns
    static_assert(BYTES <= 227 * 1024 && WDX % 1024 == 0 && (CIN == 16 || SLOT % 1024 == 0), "shared memory");
    static_assert(TMEM <= 512 && (TMEM & (TMEM - 1)) == 0, "tensor memory");
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

struct C6Maps {
    CUtensorMap in, in8, out, out8, res, res8;  // boxes of 128 and of 8 pixels
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(C6_THREADS, 1)
    k_conv_tc(const __grid_constant__ C6Maps tm, const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias, int N,
              int H, int W, int in_relu, int out_relu, int with_res, const uint2* mbits, uint2* __restrict__ obits,
              const float4* res32, float4* __restrict__ out32, int* __restrict__ status) {
    using Cf = TcCfg<CIN, COUT>;
    constexpr int C6_SLOTS = Cf::SLOTS, OFF_OUT = (Cf::OFF_OUT + 1023) / 1024 * 1024;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[C6_SLOTS], ready[C6_SLOTS], empty[C6_SLOTS], acc_full[C6_BLK], acc_empty[C6_BLK],
        side[2][2];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float s_bias[COUT];
    __shared__ int dead_flag;
    volatile int* dead = &dead_flag;
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid / 32, 0), lane = tid % 32;

    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"((uint32_t)Cf::TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < C6_SLOTS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&ready[s], 4);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < C6_BLK; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4);
        }
        for (int b = 0; b < 4; ++b) mbar_init(&side[b / 2][b % 2], 1);
        fence_mbar_init();
        dead_flag = 0;
    }
    if (tid < COUT) s_bias[tid] = bias ? __ldcg(bias + tid) : 0.f;
    // weights [9 taps (dy, dx)][co][ci] -> [3 dx][n][channels], 16-byte chunks swizzled by the row, or [3 dx][group of 8
    // channels][n][8 channels]
    constexpr int KG = CIN / 8;
    for (int e = tid; e < 9 * COUT * KG; e += C6_THREADS) {
        const int kg = e % KG, co = (e / KG) % COUT, tap = e / (KG * COUT);
        const int n = (2 - tap / 3) * COUT + co;
        const int at = CIN == 64 ? n * 128 + ((kg ^ (n & 7)) * 16) : kg * Cf::WGS + n * 16;
        *reinterpret_cast<uint4*>(smem + (tap % 3) * Cf::WDX + at) =
            __ldcg(reinterpret_cast<const uint4*>(w + ((size_t)tap * COUT + co) * CIN + kg * 8));
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    if (warp >= 4 && warp < 8) {  // every accumulator block starts zeroed
#pragma unroll 1
        for (int c = 0; c < Cf::TMEM; c += 32) tc_st_zero32(tmem + ((uint32_t)(32 * (warp % 4)) << 16) + (uint32_t)c);
        tc_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    after_previous_grid();  // (the weights and biases are older: see ConvArgs)

    const StripRuns R(N, H, W);
    const long long r_begin = R.rows * blockIdx.x / gridDim.x, r_end = R.rows * (blockIdx.x + 1) / gridDim.x;
    using Run = StripRun;
    auto run_at = [&](long long r) { return R.at(r, r_end); };

    if (warp == 0) {
        if (CIN == 64 && lane == 0) {
            unsigned q = 0;  // input rows issued
            bool ok = true;
            for (long long r = r_begin; r < r_end && ok;) {
                const Run u = run_at(r);
                r += u.L;
                const int xl = u.x0 == 0 ? W - 8 : u.x0 - 8, xr = u.x0 + u.nv == W ? 0 : u.x0 + u.nv;
                for (int li = 0; li < u.L + 2; ++li, ++q) {
                    const unsigned s = q % C6_SLOTS;
                    if (q >= C6_SLOTS && !role_wait(&empty[s], (q / C6_SLOTS - 1) & 1u, dead)) {
                        ok = false;
                        break;
                    }
                    const int row = u.n * H + R.wrap(u.y0 - 1 + li);
                    const uint32_t dst = sbase + Cf::OFF_IN + s * Cf::SLOT;
                    mbar_arrive_expect_tx(&full[s], (uint32_t)(u.nv + 16) * 128u);
                    tma_load_rows(dst, &tm.in8, xl, row, &full[s]);
                    if (u.nv == C6_W) {
                        tma_load_rows(dst + 1024, &tm.in, u.x0, row, &full[s]);
                    } else {
                        for (int x = 0; x < u.nv; x += 8) tma_load_rows(dst + 1024 + x * 128, &tm.in8, u.x0 + x, row, &full[s]);
                    }
                    tma_load_rows(dst + 1024 + u.nv * 128, &tm.in8, xr, row, &full[s]);
                }
            }
            // every copy issued lands before the shared memory is given up
            for (unsigned j = 0; j < C6_SLOTS && j < q; ++j) land(&full[(q - 1 - j) % C6_SLOTS], ((q - 1 - j) / C6_SLOTS) & 1u);
        }
    } else if (warp == 1) {
        // The whole warp walks the rows, so that descriptors and addresses are
        // warp-uniform; one elected lane issues.
        // D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 = 1), K-major, M >> 4 at bits 24-28; N >> 3 (bits 17-22)
        // per MMA
        const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(C6_W >> 4) << 24);
        const uint64_t b_desc = CIN == 64 ? sdesc_sw128(sbase) : sdesc(sbase, Cf::WGS, 128);
        const uint64_t a_desc = CIN == 64 ? sdesc_sw128(sbase + Cf::OFF_IN + 1024 - 128) : sdesc(sbase + Cf::OFF_IN, Cf::GS, 128);
        constexpr int ADX = CIN == 64 ? 128 : 16;  // one pixel further
        const uint32_t ahi = (uint32_t)(a_desc >> 32), bhi = (uint32_t)(b_desc >> 32);
        unsigned q = 0, t0 = 0;
        bool ok = true;
        for (long long r = r_begin; r < r_end && ok;) {
            const Run u = run_at(r);
            r += u.L;
            for (int li = 0; li < u.L + 2; ++li, ++q) {
                const unsigned s = q % C6_SLOTS;
                if (li < u.L) {  // the block that output row li starts in
                    const unsigned t = t0 + li;
                    if (t >= C6_BLK && !role_wait_warp(&acc_empty[t % C6_BLK], (t / C6_BLK - 1) & 1u, dead)) {
                        ok = false;
                        break;
                    }
                }
                if (!role_wait_warp(CIN == 16 || in_relu ? &ready[s] : &full[s], (q / C6_SLOTS) & 1u, dead)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                // output rows tlo .. thi, in one MMA per step, or two where the
                // accumulator blocks wrap around to block 0 at row wr
                const int tlo = li - 2 > 0 ? li - 2 : 0, thi = li < u.L - 1 ? li : u.L - 1;
                const int to_wrap = C6_BLK - (int)((t0 + tlo) % C6_BLK);  // rows up to the wrap
                const int wr = tlo + to_wrap <= thi ? tlo + to_wrap : thi + 1;
                const uint32_t d0 = tmem + ((t0 + tlo) % C6_BLK) * (uint32_t)COUT;
                const uint32_t b0 = (uint32_t)b_desc + (uint32_t)((tlo - li + 2) * COUT * Cf::WROW >> 4);
                const uint32_t b1 = (uint32_t)b_desc + (uint32_t)((wr - li + 2) * COUT * Cf::WROW >> 4);
                const uint32_t i0 = idesc0 | ((uint32_t)(wr - tlo) * (COUT / 8) << 17), i1 = idesc0 | ((uint32_t)(thi + 1 - wr) * (COUT / 8) << 17);
                const uint32_t a0 = (uint32_t)a_desc + ((s * Cf::SLOT) >> 4);
                const bool two = wr <= thi;
                if (elect_one()) {
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int kc = 0; kc < Cf::KC; ++kc)
                            tc_mma_acc(d0, a0 + ((dx * ADX + kc * 32) >> 4), ahi, b0 + ((dx * Cf::WDX + kc * 32) >> 4), bhi, i0);
                    if (two) {
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                            for (int kc = 0; kc < Cf::KC; ++kc)
                                tc_mma_acc(tmem, a0 + ((dx * ADX + kc * 32) >> 4), ahi, b1 + ((dx * Cf::WDX + kc * 32) >> 4), bhi,
                                           i1);
                    }
                    tc_commit(&empty[s]);
                    if (li >= 2) tc_commit(&acc_full[(t0 + li - 2) % C6_BLK]);
                }
                __syncwarp();
            }
            t0 += u.L;
        }
        // the MMAs issued are done with the slots before the block ends
        for (unsigned j = 0; j < C6_SLOTS && j < q; ++j) land(&empty[(q - 1 - j) % C6_SLOTS], ((q - 1 - j) / C6_SLOTS) & 1u);
    } else if (warp >= 12) {
        if constexpr (CIN == 16) {
            // the input rows, 16 bytes a copy, up to AHEAD rows in flight
            constexpr int AHEAD = 6;
            static_assert(AHEAD < C6_SLOTS, "a slot waited for has been handed over");
            const int rt = tid - 12 * 32;
            unsigned q = 0;  // rows issued
            bool ok = true;
            auto hand_over = [&](unsigned j) {  // row j has landed
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ready[j % C6_SLOTS]);
            };
            for (long long r = r_begin; r < r_end && ok;) {
                const Run u = run_at(r);
                r += u.L;
                for (int li = 0; li < u.L + 2; ++li) {
                    const unsigned s = q % C6_SLOTS;
                    if (q >= C6_SLOTS && !role_wait_warp(&empty[s], (q / C6_SLOTS - 1) & 1u, dead)) {
                        ok = false;
                        break;
                    }
                    const __nv_bfloat16* row = in + (size_t)(u.n * (long long)H + R.wrap(u.y0 - 1 + li)) * W * 16;
                    const uint32_t dst = sbase + Cf::OFF_IN + s * Cf::SLOT;
                    // pixels -1 .. nv of the strip, 2 vectors each
                    for (int e = rt; e < (u.nv + 2) * 2; e += 128) {
                        const int kg = e & 1, px = e >> 1;
                        int gx = u.x0 - 1 + px;
                        gx = gx < 0 ? gx + W : (gx >= W ? gx - W : gx);
                        cp_async16(dst + kg * Cf::GS + px * 16, row + (size_t)gx * 16 + kg * 8);
                    }
                    cp_async_commit();
                    ++q;
                    if (q > AHEAD) {
                        cp_async_wait<AHEAD>();
                        hand_over(q - 1 - AHEAD);
                    }
                }
            }
            cp_async_wait<0>();
            if (ok)
                for (unsigned j = q > AHEAD ? q - AHEAD : 0; j < q; ++j) hand_over(j);
        } else if (in_relu) {
            const int rt = tid - 12 * 32;
            unsigned q = 0;
            bool ok = true;
            for (long long r = r_begin; r < r_end && ok;) {
                const Run u = run_at(r);
                r += u.L;
                // pixels -1 .. nv of the strip, 8 vectors each
                const int nvec = (u.nv + 2) * 8;
                for (int li = 0; li < u.L + 2; ++li, ++q) {
                    const unsigned s = q % C6_SLOTS;
                    if (!role_wait_warp(&full[s], (q / C6_SLOTS) & 1u, dead)) {
                        ok = false;
                        break;
                    }
                    uint4* v = reinterpret_cast<uint4*>(smem + Cf::OFF_IN + s * Cf::SLOT + 1024 - 128);
#pragma unroll 4
                    for (int e = rt; e < nvec; e += 128) v[e] = relu8(v[e]);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ready[s]);
                }
            }
        }
    } else if (warp >= 4) {
        const int grp = (warp - 4) / 4;
        const int px = 32 * (warp % 4) + lane;  // pixel = tensor-memory lane
        const uint32_t t_lane = tmem + ((uint32_t)(32 * (warp % 4)) << 16);
        const bool leader = warp == 4 + 4 * grp && lane == 0;
        // the group's output rows, one after another through the CTA's runs
        struct Rows {
            long long r;  // where the next run starts
            Run u;
            int t;        // row of the run
            unsigned t0;  // output rows of the CTA before the run
            bool more;
        };
        auto settle = [&](Rows& c) {  // on to the next run while the row lies beyond this one
            while (c.more && c.t >= c.u.L) {
                c.t0 += c.u.L;
                if (c.r >= r_end) {
                    c.more = false;
                } else {
                    c.u = run_at(c.r);
                    c.r += c.u.L;
                    c.t = (int)((c.t0 ^ (unsigned)grp) & 1u);
                }
            }
        };
        Rows c;
        c.more = r_begin < r_end;
        if (c.more) {
            c.u = run_at(r_begin);
            c.r = r_begin + c.u.L;
            c.t = grp;
            c.t0 = 0;
            settle(c);
        }
        auto stage = [&](unsigned k) { return OFF_OUT + (2 * grp + (int)(k & 1u)) * C6_ROW; };
        // the residual of a row into its staging row (leader)
        auto bring = [&](const Rows& d, unsigned k) {
            const int row = d.u.n * H + d.u.y0 + d.t;
            uint64_t* bar = &side[grp][k & 1u];
            const uint32_t dst = sbase + stage(k);
            mbar_arrive_expect_tx(bar, (uint32_t)d.u.nv * 128u);
            if (d.u.nv == C6_W) {
                tma_load_rows(dst, &tm.res, d.u.x0, row, bar);
            } else {
                for (int x = 0; x < d.u.nv; x += 8) tma_load_rows(dst + x * 128, &tm.res8, d.u.x0 + x, row, bar);
            }
        };
        unsigned k = 0, brought = 0;  // rows of the group done; residuals asked for (leader)
        if (with_res && leader && c.more) {
            bring(c, 0);
            brought = 1;
        }
        while (c.more) {
            const unsigned tt = c.t0 + c.t;
            const size_t pix = ((size_t)c.u.n * H + c.u.y0 + c.t) * W + c.u.x0 + px;
            if constexpr (COUT == 16) {  // the first four channels in FP32, a pixel per thread
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
                if (res32 && px < c.u.nv) o = res32[pix];
                if (!role_wait_warp(&acc_full[tt % C6_BLK], (tt / C6_BLK) & 1u, dead)) break;
                tc_fence_after();
                float v[16];
                tc_ld16(t_lane + (tt % C6_BLK) * 16u, v);
                tc_st_zero16(t_lane + (tt % C6_BLK) * 16u);
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[tt % C6_BLK]);
                const float4 b = *reinterpret_cast<const float4*>(s_bias);
                o.x += v[0] + b.x;
                o.y += v[1] + b.y;
                o.z += v[2] + b.z;
                o.w += v[3] + b.w;
                if (px < c.u.nv) out32[pix] = o;
                c.t += 2;
                settle(c);
            } else {
                uint2 mw = make_uint2(0xffffffffu, 0xffffffffu);
                if (mbits && px < c.u.nv) mw = mbits[pix];
                // A warp whose wait runs out skips the row, but not the barrier that
                // ends it: the group leaves together.
                bool failed = true;
                do {
                    if (!role_wait_warp(&acc_full[tt % C6_BLK], (tt / C6_BLK) & 1u, dead)) break;
                    tc_fence_after();
                    float v[64];
                    tc_ld32(t_lane + (tt % C6_BLK) * 64u, v);
                    tc_ld32(t_lane + (tt % C6_BLK) * 64u + 32u, v + 32);
                    tc_wait_ld(v);
                    tc_st_zero32(t_lane + (tt % C6_BLK) * 64u);
                    tc_st_zero32(t_lane + (tt % C6_BLK) * 64u + 32u);
                    tc_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[tt % C6_BLK]);
                    if (with_res && !role_wait_warp(&side[grp][k & 1u], (k >> 1) & 1u, dead)) break;
                    unsigned char* orow = smem + stage(k) + px * 128;
                    uint32_t bits[2] = {0u, 0u};
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        float* x = v + 8 * q;
                        const int at = (q ^ (px & 7)) * 16;
#pragma unroll
                        for (int j = 0; j < 8; j += 4) {
                            const float4 b = *reinterpret_cast<const float4*>(s_bias + 8 * q + j);
                            x[j] += b.x;
                            x[j + 1] += b.y;
                            x[j + 2] += b.z;
                            x[j + 3] += b.w;
                        }
                        if (mbits) {
                            // bit j of a word: channel 2 j of its 32, bit 16 + j: channel 2 j + 1
                            const uint32_t m = q < 4 ? mw.x : mw.y;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                if (!(m & (1u << (4 * (q & 3) + j)))) x[2 * j] = 0.f;
                                if (!(m & (0x10000u << (4 * (q & 3) + j)))) x[2 * j + 1] = 0.f;
                            }
                        }
                        if (with_res) {
                            const uint4 m = *reinterpret_cast<const uint4*>(orow + at);
                            const __nv_bfloat16* mh = reinterpret_cast<const __nv_bfloat16*>(&m);
#pragma unroll
                            for (int j = 0; j < 8; ++j) x[j] += __bfloat162float(mh[j]);
                        }
                        uint4 o;
                        __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
                        for (int j = 0; j < 4; ++j) oh[j] = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
                        if (obits) {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                bits[q / 4] |= __hgt2_mask(oh[j], __floats2bfloat162_rn(0.f, 0.f)) & (0x10001u << (4 * (q & 3) + j));
                        }
                        if (out_relu) o = relu8(o);
                        *reinterpret_cast<uint4*>(orow + at) = o;
                    }
                    if (obits && px < c.u.nv) obits[pix] = make_uint2(bits[0], bits[1]);
                    failed = false;
                } while (false);
                Rows d = c;  // the row after this one
                d.t += 2;
                settle(d);
                if (leader && !failed) {
                    // the other staging row is free once the store before has been read
                    bulk_wait_read0();
                    if (with_res && d.more) {
                        bring(d, k + 1);
                        ++brought;
                    }
                }
                fence_proxy_async();
                if (group_any(grp, failed)) break;
                if (leader) {
                    const int row = c.u.n * H + c.u.y0 + c.t;
                    const uint32_t src = sbase + stage(k);
                    if (c.u.nv == C6_W) {
                        tma_store_rows(&tm.out, c.u.x0, row, src);
                    } else {
                        for (int x = 0; x < c.u.nv; x += 8) tma_store_rows(&tm.out8, c.u.x0 + x, row, src + x * 128);
                    }
                    bulk_commit();
                }
                c = d;
                ++k;
            }
        }
        if (leader) {
            // after a wait that ran out: the residuals still in flight
            for (unsigned j = k; j < brought; ++j) land(&side[grp][j & 1u], (j >> 1) & 1u);
            bulk_wait_all();
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && dead_flag) atomicOr(status, 1);
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)Cf::TMEM) : "memory");
    }
}

using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled get_encoder() {
    static EncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    });
    return fn;
}

}  // namespace

cudaError_t encode_rows64(const void* base, long long rows, int W, int px, CUtensorMap* m) {
    EncodeTiled enc = get_encoder();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {64, (cuuint64_t)W, (cuuint64_t)rows}, strides[2] = {128, (cuuint64_t)W * 128};
    const cuuint32_t box[3] = {64, (cuuint32_t)px, 1}, ones[3] = {1, 1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, ones,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess
               : cudaErrorInvalidValue;
}

namespace {

template <int CIN, int COUT>
cudaError_t conv_tc_t(const ConvArgs& a, cudaStream_t s, int sms, int* status) {
    using Cf = TcCfg<CIN, COUT>;
    const long long rows = (long long)a.N * a.H, tiles = rows * ((a.W + C6_W - 1) / C6_W);
    if (rows >= (1ll << 31)) return cudaErrorInvalidValue;
    C6Maps m{};
    const struct {
        const void* p;
        CUtensorMap *wide, *narrow;
    } t[3] = {{CIN == 64 ? a.in : nullptr, &m.in, &m.in8}, {a.out16, &m.out, &m.out8}, {a.res16, &m.res, &m.res8}};
    for (const auto& e : t) {
        if (!e.p) continue;
        cudaError_t rc = encode_rows64(e.p, rows, a.W, C6_W, e.wide);
        if (rc == cudaSuccess) rc = encode_rows64(e.p, rows, a.W, 8, e.narrow);
        if (rc != cudaSuccess) return rc;
    }
    const cudaError_t e = cudaFuncSetAttribute(k_conv_tc<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cf::BYTES);
    if (e != cudaSuccess) return e;
    const int grid = tiles < sms ? (int)tiles : sms;
    return launch_early(k_conv_tc<CIN, COUT>, grid, C6_THREADS, Cf::BYTES, s, m, a.in, a.w, a.bias, a.N, a.H, a.W, a.in_relu,
                        a.out_relu, (int)(a.res16 != nullptr), reinterpret_cast<const uint2*>(a.mbits),
                        reinterpret_cast<uint2*>(a.obits), reinterpret_cast<const float4*>(a.res32),
                        reinterpret_cast<float4*>(a.out32), status);
}

}  // namespace

cudaError_t launch_conv_tc(int cin, int cout, const ConvArgs& a, cudaStream_t s, int sms, int* status) {
    if (a.N < 1 || a.H < 1 || a.W < 16 || a.W % 16 != 0 || !status || sms < 1 || a.mask) return cudaErrorInvalidValue;
    if (cin == 64 && cout == 64 && a.out16) return conv_tc_t<64, 64>(a, s, sms, status);
    if (cin == 16 && cout == 64 && a.out16 && !a.in_relu) return conv_tc_t<16, 64>(a, s, sms, status);
    if (cin == 64 && cout == 16 && a.out32 && !a.out16 && !a.res16) return conv_tc_t<64, 16>(a, s, sms, status);
    return cudaErrorInvalidValue;
}

}  // namespace lbm
