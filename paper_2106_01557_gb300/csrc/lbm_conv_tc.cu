// 3x3 periodic convolution of the surrogate's lift and projection layers (16 ->
// 64, 64 -> 16 channels; lbm_conv64.cu has the 64 -> 64 layers) on the 5th-generation tensor
// cores: tcgen05.mma (kind::f16: BF16 operands in shared memory, FP32
// accumulators in tensor memory), completion tracked by tcgen05.commit on an
// mbarrier (every wait bounded in time).
//
// Work: the output is cut into rows of TC_TW = 128 pixels (one MMA M); the
// rows of all (image, 128-pixel strip) columns are dealt out to the CTAs in
// contiguous runs, so a CTA walks down a strip and loads each input row once,
// into a ring of TC_NSLOT halo'd input rows in shared memory filled by
// cp.async copies issued TC_NSLOT - 2 rows ahead of their use (ReLU, where
// the layer wants it, is applied in place by the thread that copied the
// vector).
//
// The MMAs are input-stationary: input row li of a run (image row y0 - 1 +
// li) feeds output rows t = li - 2, li - 1 and li of the run through taps
// dy = +1, 0 and -1; the weights of the three dy taps sit side by side in
// N, so one MMA (M = 128 pixels, N = 3 COUT, K = 16) applies one (dx,
// 16-channel) step of input row li to all three output rows at once.
// Output row t accumulates in block t % TC_NBLK of tensor memory (COUT
// columns each); where the blocks of the rows wrap around, or where a row
// starts its accumulator (its first step, accumulate flag off), the step is
// split into two or three MMAs over adjacent blocks. Per output row this
// reads the input operand 3 CIN / 16 times instead of 9 CIN / 16 and issues
// about 3 CIN / 16 + 1 MMAs instead of 9 CIN / 16; every output still sums
// its 9 CIN / 16 K-steps in the order (dy, dx, channel chunk).
//
// Roles: warps 0 .. TC_EPI_WARPS - 1 copy, apply ReLU and run the epilogue;
// the last warp only issues the MMAs (one elected lane), so the next input
// row's MMAs never wait for an epilogue. The epilogue of output row t runs
// once input row t + 2 is done, while the MMAs of input row t + 3 run: it
// reads the row out with tcgen05.ld (warp w reads lanes 32 (w % 4) .. + 31
// = pixels, a share of the columns), adds the bias and stages FP32 values in
// one of two shared tiles (16-byte chunks XOR-swizzled by pixel, no bank
// conflicts); in the next iteration the tile leaves in coalesced 16-byte
// stores, where the mask and the residual (loaded a row ahead) are applied,
// while the other tile takes the next row.
//
// Shared-memory operand layouts (K-major). With CIN = 64 both operands use
// the tensor core's 128-byte swizzle: one 128-byte row of 64 channels per
// pixel (A) or per N row (B), the 16-byte chunk c of a row stored at chunk
// c ^ (row address bits 7-9), 1024-byte atoms of 8 rows (SBO); the K step
// of 16 channels moves the descriptor start 32 bytes along the rows.
//   input row slot [TC_TW + 2 pixels][128 B] (1024-byte aligned): the window
//     of tap dx is the same operand started dx + 1 rows in.
//   weights [3 dx][3 blocks: dy = +1, 0, -1][COUT][128 B].
// With CIN = 16 (the lift layer), no swizzle; a core matrix is 8 rows of 16
// bytes:
//   input row slot [CIN/8 channel groups][TC_TW + 2 pixels, stride 16 B],
//     channel-group stride GS = (TC_TW + 3) * 16 B (LBO), SBO = 128; the
//     window of tap dx starts (1 + dx) * 16 B in.
//   weights [3 dx][CIN/8][3 blocks][COUT][8 channels]: LBO = 3 COUT * 16,
//     SBO = 128.
// The block of tap dy for output row t and input row li is t - li + 2, so
// adjacent output rows take adjacent blocks in N, as they take adjacent
// blocks of tensor memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_conv.h"
#include "lbm_launch.cuh"
#include "lbm_ptx.cuh"
#include "lbm_tc.cuh"

namespace lbm {
namespace {

constexpr int TC_TW = 128;          // pixels per output row segment (MMA M)
constexpr int TC_EPI_WARPS = 16;    // warps 0 .. TC_EPI_WARPS - 1: copies and epilogue
constexpr int TC_EPI_THREADS = 32 * TC_EPI_WARPS;
constexpr int TC_THREADS = TC_EPI_THREADS + 32;  // + one warp: MMA issue
constexpr int TC_NSLOT = 5;         // input-row ring: 1 row in use, 1 ready, the rest in flight
constexpr int TC_NBLK = 8;          // accumulator blocks in tensor memory (output rows in flight)

template <int CIN, int COUT>
struct TcCfg {
    static constexpr int KG = CIN / 8;                  // 8-channel groups
    static constexpr int PIX = TC_TW + 2;               // halo'd pixels per row
    static constexpr int GS = (TC_TW + 3) * 16;         // bytes between channel groups
    // input rows: with CIN = 64, one 128-byte row per pixel, 16-byte chunks
    // swizzled by the pixel's address (the tensor core's 128-byte swizzle);
    // otherwise no swizzle, channel groups GS bytes apart
    static constexpr bool ASW = CIN == 64;
    static constexpr int SLOT_BYTES = ASW ? (PIX * 128 + 1023) / 1024 * 1024 : KG * GS;
    // weights: with CIN = 64, one 128-byte row of channels per N row, 16-byte
    // chunks swizzled by the row (the tensor core's 128-byte swizzle);
    // otherwise no swizzle, channel groups WGS bytes apart
    static constexpr bool WSW = CIN == 64;
    static constexpr int WGS = 3 * COUT * 16;
    static constexpr int WDX = WSW ? 3 * COUT * 128 : KG * WGS;  // bytes per tap dx
    static constexpr int W_BYTES = 3 * WDX;
    static constexpr int TILE = TC_TW * COUT;            // FP32 values of one output row
    static constexpr int OUT_BYTES = 2 * TILE * 4;      // two staging tiles (rows t and t - 1)
    static constexpr int BYTES = W_BYTES + TC_NSLOT * SLOT_BYTES + OUT_BYTES + 1024;  // + alignment slack
    static constexpr int ROW_VECS = KG * PIX;           // 16-byte vectors per halo'd row
    static constexpr int VPT = (ROW_VECS + TC_EPI_THREADS - 1) / TC_EPI_THREADS;
    static constexpr int TMEM_COLS = TC_NBLK * COUT < 32 ? 32 : TC_NBLK * COUT;  // power of two
    // warps reading the accumulator (4 per lane quarter group, >= 8 columns each)
    static constexpr int TW_WARPS = TC_EPI_WARPS < COUT / 2 ? TC_EPI_WARPS : COUT / 2;
    static constexpr int EPI_COLS = COUT / (TW_WARPS / 4);  // accumulator columns per reading warp
    static constexpr int NC = EPI_COLS < 16 ? EPI_COLS : 16;        // columns per tcgen05.ld
    static constexpr int EPI_CH = EPI_COLS / NC;        // tcgen05.ld per thread and row
    static constexpr int CPP = COUT / 4;                // 16-byte FP32 chunks per pixel in the tile
    static constexpr int SWZ = (CPP < 8 ? CPP : 8) - 1; // chunk swizzle mask
    static constexpr int N16 = TC_TW * COUT / 8;        // 16-byte BF16 output chunks of a row
    static constexpr int O16 = (N16 + TC_EPI_THREADS - 1) / TC_EPI_THREADS;  // BF16 chunks per thread
    static_assert(CIN % 16 == 0 && COUT % 16 == 0 && 3 * COUT <= 256, "tcgen05 f16 shape");
    static_assert((TMEM_COLS & (TMEM_COLS - 1)) == 0 && TC_NBLK >= 4, "accumulator blocks");
    static_assert(WDX % 1024 == 0, "swizzle atoms of the weights start on 1024-byte boundaries");
    static_assert(TW_WARPS % 4 == 0 && COUT % (TW_WARPS / 4) == 0 && (NC == 8 || NC == 16), "tile split");
    static_assert(TMEM_COLS <= 512, "tensor memory");
    static_assert(BYTES <= 227 * 1024, "shared memory");
};

// barrier of the epilogue threads only (the issue warp does not wait)
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"r"(TC_EPI_THREADS) : "memory"); }

// bounded wait on an mbarrier phase; true when it completed in time
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
    const uint64_t t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity))
        if (globaltimer_ns() - t0 > WAIT_NS) return false;
    return true;
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int CIN, int COUT>
__global__ void __launch_bounds__(TC_THREADS, 1)
    k_conv_tc(const __nv_bfloat16* in, const __nv_bfloat16* w, const float* bias,
              int N, int H, int W, int in_relu, const __nv_bfloat16* mask,
              const __nv_bfloat16* res16, const float* res32,
              __nv_bfloat16* __restrict__ out16, float* __restrict__ out32, int* __restrict__ status) {
    using Cf = TcCfg<CIN, COUT>;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t tmem_base;
    __shared__ __align__(16) float s_bias[COUT];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char* s_w = smem;
    unsigned char* s_in = s_w + Cf::W_BYTES;
    unsigned char* s_out = s_in + TC_NSLOT * Cf::SLOT_BYTES;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const bool is_epi = tid < TC_EPI_THREADS;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"((uint32_t)Cf::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    for (int c = tid; c < COUT; c += TC_THREADS) s_bias[c] = bias ? __ldcg(bias + c) : 0.f;
    // weights [9 taps (dy, dx)][COUT][CIN] -> per dx, N rows n = block (dy = +1,
    // 0, -1) * COUT + co: [3 dx][n][64 channels, chunk kg at kg ^ (n % 8)]
    // (CIN = 64) or [3 dx][CIN/8][n][8 channels]
    for (int e = tid; e < 9 * COUT * Cf::KG; e += TC_THREADS) {
        const int kg = e % Cf::KG, co = (e / Cf::KG) % COUT, tap = e / (Cf::KG * COUT);
        const int dyi = tap / 3, dxi = tap % 3, n = (2 - dyi) * COUT + co;
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(w + ((size_t)tap * COUT + co) * CIN + kg * 8));
        const int off = Cf::WSW ? dxi * Cf::WDX + n * 128 + ((kg ^ (n & 7)) * 16)
                                : (dxi * Cf::KG + kg) * Cf::WGS + n * 16;
        *reinterpret_cast<uint4*>(s_w + off) = v;
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    after_previous_grid();  // (the weights and biases are older: see ConvArgs)
    // instruction descriptor: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9,
    // 10-12 = 1), both K-major (bits 15, 16 = 0), M >> 4 (bits 24-28); N >> 3
    // (bits 17-22) is added per MMA
    const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TC_TW >> 4) << 24);
    const uint32_t s_in_addr = smem_u32(s_in), s_w_addr = smem_u32(s_w);
    // descriptors of the weights and of ring slot 0; an operand inside them is
    // the same descriptor with its start moved by a constant (the 14-bit
    // start field stays below 2^14 for any shared-memory address)
    const uint64_t b_desc0 = Cf::WSW ? sdesc_sw128(s_w_addr) : sdesc(s_w_addr, Cf::WGS, 128);
    const uint64_t a_desc0 = Cf::ASW ? sdesc_sw128(s_in_addr) : sdesc(s_in_addr, Cf::GS, 128);
    const int tiles_x = (W + TC_TW - 1) / TC_TW;
    const long long rows_total = (long long)N * tiles_x * H;
    const long long r_begin = rows_total * blockIdx.x / gridDim.x;
    const long long r_end = rows_total * (blockIdx.x + 1) / gridDim.x;
    uint32_t parity = 0;   // bit b: phase parity awaited next on bar[b]
    uint32_t pending = 0;  // bit b: a commit to bar[b] not yet waited for
    bool ok = true;

    // epilogue geometry of this thread: pixel = TMEM lane, a share of the columns
    const int pix = 32 * (warp % 4) + lane;
    const int col0 = (warp / 4) * Cf::EPI_COLS;
    const uint32_t t_lane = tmem + ((uint32_t)(32 * (warp % 4)) << 16);
    float* tiles = reinterpret_cast<float*>(s_out);

    for (long long r = r_begin; r < r_end && ok;) {
        const int y0 = (int)(r % H);
        const long long strip = r / H;
        const int x0 = (int)(strip % tiles_x) * TC_TW, n = (int)(strip / tiles_x);
        const int L = (int)((long long)(H - y0) < r_end - r ? (long long)(H - y0) : r_end - r);
        const int nvalid = W - x0 < TC_TW ? W - x0 : TC_TW;  // output pixels of this strip
        r += L;
        const __nv_bfloat16* img = in + (size_t)n * H * W * CIN;
        // this thread's vectors of a halo'd row: global element offset within
        // an input row (periodic in x) and byte offset within a slot, fixed
        // for the run
        int src_off[Cf::VPT], dst_off[Cf::VPT];
#pragma unroll
        for (int i = 0; i < Cf::VPT; ++i) {
            const int e = tid + i * TC_EPI_THREADS;
            const int kg = e % Cf::KG, px = e / Cf::KG;
            int gx = x0 - 1 + px;
            gx = gx < 0 ? gx + W : gx;
            gx = gx >= W ? gx % W : gx;
            src_off[i] = gx * CIN + kg * 8;
            dst_off[i] = Cf::ASW ? px * 128 + ((kg ^ (px & 7)) * 16) : kg * Cf::GS + px * 16;
        }
        // halo'd input row li of this run (input row y0 - 1 + li, periodic)
        // into ring slot li % TC_NSLOT; one commit group per row, empty for
        // rows the run does not need, so that group counts stay uniform
        auto copy_row = [&](int li) {
            if (li <= L + 1) {
                int gy = y0 - 1 + li;
                gy = gy < 0 ? gy + H : (gy >= H ? gy - H : gy);
                const __nv_bfloat16* row = img + (size_t)gy * W * CIN;
                unsigned char* slot = s_in + (li % TC_NSLOT) * Cf::SLOT_BYTES;
#pragma unroll
                for (int i = 0; i < Cf::VPT; ++i)
                    if (tid + i * TC_EPI_THREADS < Cf::ROW_VECS) cp_async16(slot + dst_off[i], row + src_off[i]);
            }
            cp_async_commit();
        };
        // ReLU in place on the vectors this thread copied (after they landed)
        auto relu_row = [&](int li) {
            if (!in_relu || li > L + 1) return;
            unsigned char* slot = s_in + (li % TC_NSLOT) * Cf::SLOT_BYTES;
#pragma unroll
            for (int i = 0; i < Cf::VPT; ++i) {
                if (tid + i * TC_EPI_THREADS < Cf::ROW_VECS) {
                    uint4* v = reinterpret_cast<uint4*>(slot + dst_off[i]);
                    *v = relu8(*v);
                }
            }
        };
        // MMAs of input row li (in ring slot li % TC_NSLOT): it feeds output rows
        // li - 2 (tap dy = +1), li - 1 (dy = 0) and li (dy = -1), those of them in
        // the run. One MMA per (dx, channel chunk) step covers the rows whose
        // accumulator blocks are adjacent; the first step starts row li's
        // accumulator in an MMA of its own.
        auto issue = [&](int li) {
            const int tlo = li - 2 > 0 ? li - 2 : 0, thi = li < L - 1 ? li : L - 1;
            // The cut of the rows into MMA segments is the same for every step but
            // the first, so it is worked out once per row and the steps only add
            // constant offsets (worked out per MMA, the issuing thread's scalar
            // code took longer than the MMAs). Cut points in (tlo, thi], thi + 1
            // where there is none: wr, the row whose block index wraps to 0 (at
            // most one in three rows); sp, row li where it starts its accumulator
            // after other rows of the step.
            int wr = thi + 1;
            for (int t = tlo + 1; t <= thi; ++t)
                if ((t & (TC_NBLK - 1)) == 0) wr = t;
            const int sp = li > tlo && li <= thi ? li : thi + 1;
            const int q1 = wr < sp ? wr : sp, q2 = wr < sp ? sp : (sp < wr ? wr : thi + 1);
            // one MMA segment, output rows a .. b: tensor-memory column, offset of
            // the weight block (16-byte units) and instruction descriptor
            auto seg = [&](int a, int b, uint32_t& d, uint32_t& bo, uint32_t& id) {
                d = tmem + (uint32_t)((a & (TC_NBLK - 1)) * COUT);
                bo = (uint32_t)(((a - li + 2) * COUT * (Cf::WSW ? 128 : 16)) >> 4);
                id = idesc0 | ((uint32_t)(((b - a + 1) * COUT) >> 3) << 17);
            };
            uint32_t f0d, f0b, f0i, f1d = 0, f1b = 0, f1i = 0, f2d = 0, f2b = 0, f2i = 0;  // first step
            uint32_t g0d, g0b, g0i, g1d = 0, g1b = 0, g1i = 0;                           // the others
            seg(tlo, q1 - 1, f0d, f0b, f0i);
            if (q1 <= thi) seg(q1, q2 - 1, f1d, f1b, f1i);
            if (q2 <= thi) seg(q2, thi, f2d, f2b, f2i);
            seg(tlo, wr - 1, g0d, g0b, g0i);
            if (wr <= thi) seg(wr, thi, g1d, g1b, g1i);
            const uint64_t a_row = a_desc0 + (uint64_t)(((li % TC_NSLOT) * Cf::SLOT_BYTES) >> 4);
#pragma unroll
            for (int dxi = 0; dxi < 3; ++dxi) {
#pragma unroll
                for (int kc = 0; kc < CIN / 16; ++kc) {
                    // swizzled: the window of tap dx starts dx + 1 pixels (128-byte rows)
                    // in and the K step moves the start 32 bytes along the rows; the
                    // swizzle follows the address bits, so the base offset stays 0
                    const uint64_t ad = a_row + (uint64_t)((Cf::ASW ? dxi * 128 + kc * 32
                                                                    : dxi * 16 + 2 * kc * Cf::GS) >> 4);
                    // swizzled: the K step moves the start 32 bytes along the 128-byte rows
                    const uint64_t bs = b_desc0 + (uint64_t)((Cf::WSW ? dxi * Cf::WDX + kc * 32
                                                                      : (dxi * Cf::KG + 2 * kc) * Cf::WGS) >> 4);
                    if (dxi == 0 && kc == 0) {
                        tc_mma(f0d, ad, bs + f0b, f0i, tlo == li ? 0u : 1u);
                        if (q1 <= thi) tc_mma(f1d, ad, bs + f1b, f1i, q1 == li ? 0u : 1u);
                        if (q2 <= thi) tc_mma(f2d, ad, bs + f2b, f2i, q2 == li ? 0u : 1u);
                    } else {
                        tc_mma(g0d, ad, bs + g0b, g0i, 1u);
                        if (wr <= thi) tc_mma(g1d, ad, bs + g1b, g1i, 1u);
                    }
                }
            }
            tc_commit(&bar[li & 1]);
        };
        // the mask and residual chunks of output row t this thread stores
        uint4 mreg[Cf::O16], rreg[Cf::O16];
        auto prefetch_epi = [&](int t) {
            if (!out16 || t >= L) return;
            const size_t row0 = ((size_t)n * H + y0 + t) * W + x0;
#pragma unroll
            for (int j = 0; j < Cf::O16; ++j) {
                const int i = tid + j * TC_EPI_THREADS;
                const int p = i / (COUT / 8), g8 = i % (COUT / 8);
                if (i < Cf::N16 && p < nvalid) {
                    const size_t o = (row0 + p) * COUT + g8 * 8;
                    if (mask) mreg[j] = *reinterpret_cast<const uint4*>(mask + o);
                    if (res16) rreg[j] = *reinterpret_cast<const uint4*>(res16 + o);
                }
            }
        };

        // staging tile -> global, coalesced 16-byte chunks of output row tr
        // of the run, applying mask and residual (loaded by prefetch_epi(tr))
        auto copy_out = [&](int tr, const float* tile) {
            const int y = y0 + tr;
            const size_t row0 = ((size_t)n * H + y) * W + x0;
            if (out16) {
#pragma unroll
                for (int j = 0; j < Cf::O16; ++j) {
                    const int i = tid + j * TC_EPI_THREADS;
                    const int p = i / (COUT / 8), g8 = i % (COUT / 8);
                    if (i >= Cf::N16 || p >= nvalid) continue;
                    // the two FP32 chunks 2 g8 and 2 g8 + 1, read first the one that puts the
                    // 8 threads of a shared-memory phase on 8 different bank groups
                    const int c1 = 2 * g8 + (g8 >> 2) % 2, c2 = 2 * g8 + 1 - (g8 >> 2) % 2;
                    const float4 q1 = *reinterpret_cast<const float4*>(tile + p * COUT + 4 * (c1 ^ (p & Cf::SWZ)));
                    const float4 q2 = *reinterpret_cast<const float4*>(tile + p * COUT + 4 * (c2 ^ (p & Cf::SWZ)));
                    const float4 lo = c1 < c2 ? q1 : q2, hi = c1 < c2 ? q2 : q1;
                    float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                    if (mask) {
                        const __nv_bfloat16* mh = reinterpret_cast<const __nv_bfloat16*>(&mreg[j]);
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            if (!(__bfloat162float(mh[q]) > 0.f)) v[q] = 0.f;
                    }
                    if (res16) {
                        const __nv_bfloat16* rh = reinterpret_cast<const __nv_bfloat16*>(&rreg[j]);
#pragma unroll
                        for (int q = 0; q < 8; ++q) v[q] += __bfloat162float(rh[q]);
                    }
                    uint4 ov;
                    __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&ov);
#pragma unroll
                    for (int q = 0; q < 4; ++q) oh[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
                    *reinterpret_cast<uint4*>(out16 + (row0 + p) * COUT + g8 * 8) = ov;
                }
            } else {
                // the first four channels, one 16-byte chunk per pixel
                if (tid < TC_TW && tid < nvalid) {
                    const size_t p = row0 + tid;
                    float4 v = *reinterpret_cast<const float4*>(tile + tid * COUT + 4 * (0 ^ (tid & Cf::SWZ)));
                    if (res32) {
                        const float4 x = *reinterpret_cast<const float4*>(res32 + p * 4);
                        v.x += x.x;
                        v.y += x.y;
                        v.z += x.z;
                        v.w += x.w;
                    }
                    *reinterpret_cast<float4*>(out32 + p * 4) = v;
                }
            }
        };

        if (is_epi) {
            // prologue: every slot's row in flight; input row 0 in place for its MMAs
#pragma unroll 1
            for (int li = 0; li < TC_NSLOT; ++li) copy_row(li);
            cp_async_wait<TC_NSLOT - 1>();
            relu_row(0);
            fence_proxy_async();
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == TC_EPI_THREADS) issue(0);
        pending |= 1u;
        bool timed_out = false;
        // iteration j: issue input row j + 1, then (epilogue) wait for input row
        // j, whose MMAs complete output row j - 2, and write that row out
        for (int j = 0; j < L + 2; ++j) {
            if (j + 1 < L + 2) {
                if (is_epi) {
                    cp_async_wait<TC_NSLOT - 2>();
                    relu_row(j + 1);
                    fence_proxy_async();
                }
                tc_fence_before();
                // also: every thread has left the staging tile that row j - 2 takes
                // (and tensor-memory blocks of rows read out are free long before
                // they come round again)
                if (__syncthreads_or(timed_out)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (tid == TC_EPI_THREADS) issue(j + 1);
                pending |= 1u << ((j + 1) & 1);
            }
            if (!is_epi) continue;
            const uint32_t b = (uint32_t)(j & 1);
            if (!bar_wait(&bar[b], (parity >> b) & 1u)) timed_out = true;
            parity ^= 1u << b;
            pending &= ~(1u << b);
            tc_fence_after();
            // input row j's MMAs are done: its slot takes row j + TC_NSLOT
            copy_row(j + TC_NSLOT);
            const int t = j - 2;
            if (t < 0) continue;
            // accumulator + bias -> FP32 staging tile t & 1 (on the run's last row
            // no block barrier has separated this from the tile's previous readers)
            if (j + 1 >= L + 2) epi_sync();
            float* tile = tiles + (t & 1) * Cf::TILE;
            const uint32_t blk = (uint32_t)((t % TC_NBLK) * COUT);
#pragma unroll
            for (int ch = 0; ch < Cf::EPI_CH; ++ch) {
                if (warp >= Cf::TW_WARPS) break;
                const int c = col0 + Cf::NC * ch;
                float v[16];
                tc_ld<Cf::NC>(t_lane + blk + (uint32_t)c, v);
#pragma unroll
                for (int q = 0; q < Cf::NC / 4; ++q) {
                    const int k = c / 4 + q;
                    const float4 bb = *reinterpret_cast<const float4*>(s_bias + 4 * k);
                    *reinterpret_cast<float4*>(tile + pix * COUT + 4 * (k ^ (pix & Cf::SWZ))) =
                        make_float4(v[4 * q] + bb.x, v[4 * q + 1] + bb.y, v[4 * q + 2] + bb.z, v[4 * q + 3] + bb.w);
                }
            }
            // row t - 1 leaves from the other tile (written in the previous
            // iteration, one block barrier ago)
            if (t >= 1) copy_out(t - 1, tiles + ((t - 1) & 1) * Cf::TILE);
            prefetch_epi(t);  // row t's mask and residual, for its copy-out
        }
        // the run's last row (after a timeout every thread has left the loop together)
        if (ok && is_epi) {
            epi_sync();
            copy_out(L - 1, tiles + ((L - 1) & 1) * Cf::TILE);
        }
        // copies still in flight (rows the run does not need) land before the slots are reused
        if (is_epi) cp_async_wait<0>();
        tc_fence_before();
        if (__syncthreads_or(timed_out)) ok = false;
        tc_fence_after();
    }
    if (!ok) {
        // let MMAs still in flight finish (bounded) before the memory is released
        if (is_epi)
            for (uint32_t b = 0; b < 2; ++b)
                if (pending & (1u << b)) bar_wait(&bar[b], (parity >> b) & 1u);
        if (tid == 0) atomicOr(status, 1);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)Cf::TMEM_COLS)
                     : "memory");
    }
}

template <int CIN, int COUT>
cudaError_t conv_tc_t(const ConvArgs& a, cudaStream_t s, int sms, int* status) {
    using Cf = TcCfg<CIN, COUT>;
    static bool set = false;
    if (!set) {
        cudaError_t e = cudaFuncSetAttribute(k_conv_tc<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cf::BYTES);
        if (e != cudaSuccess) return e;
        set = true;
    }
    const long long rows = (long long)a.N * a.H * ((a.W + TC_TW - 1) / TC_TW);
    const int grid = rows < sms ? (int)rows : sms;
    return launch_early(k_conv_tc<CIN, COUT>, grid, TC_THREADS, Cf::BYTES, s, a.in, a.w, a.bias, a.N, a.H, a.W, a.in_relu, a.mask,
                        a.res16, a.res32, a.out16, a.out32, status);
}

}  // namespace

cudaError_t launch_conv_tc(int cin, int cout, const ConvArgs& a, cudaStream_t s, int sms, int* status) {
    if (a.N < 1 || a.H < 1 || a.W < 16 || a.W % 16 != 0 || !status || sms < 1) return cudaErrorInvalidValue;
    if (cin == 16 && cout == 64) return conv_tc_t<16, 64>(a, s, sms, status);
    if (cin == 64 && cout == 16) return conv_tc_t<64, 16>(a, s, sms, status);
    return cudaErrorInvalidValue;
}

}  // namespace lbm
