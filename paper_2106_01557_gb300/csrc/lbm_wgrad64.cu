// Weight and bias gradients of the surrogate's convolutions (64 -> 64, 16 -> 64,
// 64 -> 16) on the tensor cores, warp-specialised:
// dW[tap (dy, dx)][co][ci] = sum over pixels p of dOut[p][co] In[p + (dy, dx)][ci]
// (In after the ReLU the forward applied) and db[co] = sum of dOut[p][co].
//
// A CTA takes a contiguous run of the input rows of all 128-pixel strips (one
// partial sum per CTA, added by k_wgrad_sum in a fixed order). Input row y
// meets dOut rows y - 1, y and y + 1 (taps dy = +1, 0, -1), which lie next to
// each other in a ring of shared-memory rows, so that they are one operand of
// N = 3 x 64; the pixel is the K index of both operands (MN-major, 128-byte
// rows per pixel, 128-byte swizzle). Per 16 pixels one MMA takes as its two
// 64-row halves of M the input from pixel k - 1 (dx = -1) and from pixel k
// (dx = 0), a second one those from k and k + 1 (dx = +1; its first half
// repeats dx = 0 and is not read). The accumulators (2 x 192 columns of tensor
// memory) live for all of the CTA's rows.
//   warp 0       tensor copies of input rows (128 pixels and 8 more on each
//                side) and dOut rows into their rings
//   warp 1       issues the MMAs
//   warps 4-7    ReLU of an input row in place, where the layer wants it
//   warps 8-11   sum the dOut rows over the pixels for the bias gradient
//   warps 12-15  (with a 16-channel operand) copy its rows, 16 bytes at a time,
//                into the first two chunks of 128-byte rows whose other 48
//                channels stay zero: the MMAs and layouts are the 64 -> 64
//                layers', three quarters of one operand idle
//
// What bounds it (8 x 256 x 256, 38.7 GFLOP, 134 MB): 21 us of MMAs at the
// tensor rate, a quarter of it spent on the repeated dx = 0, and 20 us at the
// copy bandwidth; it takes 41 us (bias included) where the kernel before it, which
// read every dOut row three times, took 79 and the bias sums another 23: it ran
// a block per filter row with block barriers per 128 pixels. The lift and the
// projection take 43 and 44 us where that kernel and separate bias sums took 81
// and 102.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_conv.h"
#include "lbm_conv64.cuh"
#include "lbm_launch.cuh"
#include "lbm_ptx.cuh"
#include "lbm_tc.cuh"

namespace lbm {
namespace {

constexpr int W6_XS = 4;                 // input-row ring
constexpr int W6_DS = 6;                 // dOut-row ring
template <int CIN, int COUT>
constexpr int W6_THREADS = CIN == 64 && COUT == 64 ? 384 : 512;
constexpr int W6_AHEAD = 3;              // 16-channel rows in flight
// Row q is handed over once row q + W6_AHEAD is issued, for which row q +
// W6_AHEAD - (ring) has to be free: an earlier step than the first that needs
// row q (for dOut, step q - 2) frees it.
static_assert(W6_AHEAD < W6_XS && W6_AHEAD + 2 < W6_DS, "rings");
constexpr int W6_OFF_D = W6_XS * C6_SLOT;
constexpr int W6_BYTES = W6_OFF_D + W6_DS * C6_ROW + 1024;
static_assert(W6_BYTES <= 227 * 1024 && C6_SLOT % 1024 == 0, "shared memory");

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, int src_bytes) {  // src_bytes 0: zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(W6_THREADS<CIN, COUT>, 1)
    k_wgrad_tc(const __grid_constant__ CUtensorMap tx, const __grid_constant__ CUtensorMap tx8,
               const __grid_constant__ CUtensorMap td, const __nv_bfloat16* in, const __nv_bfloat16* dout, int N, int H, int W,
               int in_relu, float* __restrict__ part, float* __restrict__ bpart, int* __restrict__ status) {
    constexpr int THREADS = W6_THREADS<CIN, COUT>;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t xfull[W6_XS], xready[W6_XS], xempty[W6_XS], dfull[W6_DS], dempty[W6_DS], done;
    __shared__ uint32_t tmem_base;
    __shared__ float s_b[16][64];
    __shared__ int dead_flag;
    volatile int* dead = &dead_flag;
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid / 32, 0), lane = tid % 32;

    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < W6_XS; ++s) {
            mbar_init(&xfull[s], 1);
            mbar_init(&xready[s], 4);
            mbar_init(&xempty[s], 1);
        }
        for (int s = 0; s < W6_DS; ++s) {
            mbar_init(&dfull[s], COUT == 64 ? 1 : 4);
            mbar_init(&dempty[s], 5);  // the MMAs and the four bias warps
        }
        mbar_init(&done, 1);
        fence_mbar_init();
        dead_flag = 0;
    }
    // pixels past a narrow strip meet dOut zeros, but have to be finite; 16-channel rows leave the other 48 channels zero
    for (int e = tid; e < (COUT == 64 ? W6_OFF_D : W6_OFF_D + W6_DS * C6_ROW) / 16; e += THREADS)
        reinterpret_cast<uint4*>(smem)[e] = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;
    if (warp >= 4 && warp < 8) {
#pragma unroll 1
        for (int c = 0; c < 384; c += 32) tc_st_zero32(tmem + ((uint32_t)(32 * (warp % 4)) << 16) + (uint32_t)c);
        tc_wait_st();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    after_previous_grid();

    const StripRuns R(N, H, W);
    const long long r_begin = R.rows * blockIdx.x / gridDim.x, r_end = R.rows * (blockIdx.x + 1) / gridDim.x;

    if (warp == 0) {
        if (lane == 0) {
            unsigned qx = 0, qd = 0;  // input and dOut rows issued
            bool ok = true;
            for (long long r = r_begin; r < r_end && ok;) {
                const StripRun u = R.at(r, r_end);
                r += u.L;
                const int xl = u.x0 == 0 ? W - 8 : u.x0 - 8, xr = u.x0 + u.nv == W ? 0 : u.x0 + u.nv;
                for (int j = 0; j < u.L + 2; ++j) {
                    if constexpr (COUT == 64) {
                        const unsigned s = qd % W6_DS;
                        if (qd >= W6_DS && !role_wait(&dempty[s], (qd / W6_DS - 1) & 1u, dead)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_expect_tx(&dfull[s], C6_ROW);
                        tma_load_rows(sbase + W6_OFF_D + s * C6_ROW, &td, u.x0, u.n * H + R.wrap(u.y0 - 1 + j), &dfull[s]);
                        ++qd;
                    }
                    if (CIN == 16 || j < 2) continue;
                    const unsigned s = qx % W6_XS;
                    if (qx >= W6_XS && !role_wait(&xempty[s], (qx / W6_XS - 1) & 1u, dead)) {
                        ok = false;
                        break;
                    }
                    const int row = u.n * H + u.y0 + j - 2;
                    const uint32_t dst = sbase + s * C6_SLOT;
                    mbar_arrive_expect_tx(&xfull[s], (uint32_t)(u.nv + 16) * 128u);
                    tma_load_rows(dst, &tx8, xl, row, &xfull[s]);
                    if (u.nv == C6_W) {
                        tma_load_rows(dst + 1024, &tx, u.x0, row, &xfull[s]);
                    } else {
                        for (int x = 0; x < u.nv; x += 8) tma_load_rows(dst + 1024 + x * 128, &tx8, u.x0 + x, row, &xfull[s]);
                    }
                    tma_load_rows(dst + 1024 + u.nv * 128, &tx8, xr, row, &xfull[s]);
                    ++qx;
                }
            }
            // every copy issued lands before the shared memory is given up
            for (unsigned j = 0; j < W6_XS && j < qx; ++j) land(&xfull[(qx - 1 - j) % W6_XS], ((qx - 1 - j) / W6_XS) & 1u);
            for (unsigned j = 0; j < W6_DS && j < qd; ++j) land(&dfull[(qd - 1 - j) % W6_DS], ((qd - 1 - j) / W6_DS) & 1u);
        }
    } else if (warp == 1) {
        // D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9, 10-12 = 1), both MN-major (bits 15, 16 = 1), M = 128
        const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((128u >> 4) << 24);
        const uint64_t ad = sdesc_mn_sw128(sbase + 1024 - 128, 128), bd = sdesc_mn_sw128(sbase + W6_OFF_D, C6_ROW);
        const uint32_t ahi = (uint32_t)(ad >> 32), bhi = (uint32_t)(bd >> 32);
        unsigned qx = 0, qd = 0;
        bool ok = true;
        for (long long r = r_begin; r < r_end && ok;) {
            const StripRun u = R.at(r, r_end);
            r += u.L;
            for (int li = 0; li < u.L; ++li, ++qx) {
                const unsigned s = qx % W6_XS;
                // dOut rows li .. li + 2 of the run
                for (unsigned j = li == 0 ? 0 : 2; j < 3; ++j) {
                    const unsigned d = qd + li + j;
                    ok = ok && role_wait_warp(&dfull[d % W6_DS], (d / W6_DS) & 1u, dead);
                }
                ok = ok && role_wait_warp(CIN == 16 || in_relu ? &xready[s] : &xfull[s], (qx / W6_XS) & 1u, dead);
                if (!ok) break;
                tc_fence_after();
                const unsigned d0 = (qd + li) % W6_DS;
                const unsigned n0 = W6_DS - d0 < 3 ? W6_DS - d0 : 3;  // rows before the ring wraps
                const uint32_t i0 = idesc0 | ((n0 * 64u >> 3) << 17), i1 = idesc0 | (((3 - n0) * 64u >> 3) << 17);
                const uint32_t a0 = (uint32_t)ad + ((s * C6_SLOT) >> 4), b0 = (uint32_t)bd + ((d0 * C6_ROW) >> 4);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < C6_W / 16; ++kk) {
                        tc_mma_acc(tmem, a0 + ((kk * 2048) >> 4), ahi, b0 + ((kk * 2048) >> 4), bhi, i0);
                        tc_mma_acc(tmem + 192, a0 + ((kk * 2048 + 128) >> 4), ahi, b0 + ((kk * 2048) >> 4), bhi, i0);
                    }
                    if (n0 < 3) {
#pragma unroll
                        for (int kk = 0; kk < C6_W / 16; ++kk) {
                            tc_mma_acc(tmem + n0 * 64, a0 + ((kk * 2048) >> 4), ahi, (uint32_t)bd + ((kk * 2048) >> 4), bhi, i1);
                            tc_mma_acc(tmem + 192 + n0 * 64, a0 + ((kk * 2048 + 128) >> 4), ahi, (uint32_t)bd + ((kk * 2048) >> 4),
                                       bhi, i1);
                        }
                    }
                    tc_commit(&xempty[s]);
                    tc_commit(&dempty[d0]);
                    if (li == u.L - 1) {
                        tc_commit(&dempty[(qd + li + 1) % W6_DS]);
                        tc_commit(&dempty[(qd + li + 2) % W6_DS]);
                    }
                }
                __syncwarp();
            }
            qd += u.L + 2;
        }
        if (elect_one()) tc_commit(&done);
        __syncwarp();
    } else if (warp >= 4 && warp < 8) {
        if (CIN == 64 && in_relu) {
            const int rt = tid - 4 * 32;
            unsigned q = 0;
            bool ok = true;
            for (long long r = r_begin; r < r_end && ok;) {
                const StripRun u = R.at(r, r_end);
                r += u.L;
                const int nvec = (u.nv + 2) * 8;  // pixels -1 .. nv of the strip, 8 vectors each
                for (int li = 0; li < u.L; ++li, ++q) {
                    const unsigned s = q % W6_XS;
                    if (!role_wait_warp(&xfull[s], (q / W6_XS) & 1u, dead)) {
                        ok = false;
                        break;
                    }
                    uint4* v = reinterpret_cast<uint4*>(smem + s * C6_SLOT + 1024 - 128);
#pragma unroll 4
                    for (int e = rt; e < nvec; e += 128) v[e] = relu8(v[e]);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&xready[s]);
                }
            }
        }
    } else if (warp >= 12) {
        // the rows of the 16-channel operand, 16 bytes a copy
        const int rt = tid - 12 * 32;
        uint64_t *const given = COUT == 16 ? dfull : xready, *const taken = COUT == 16 ? dempty : xempty;
        constexpr unsigned RING = COUT == 16 ? W6_DS : W6_XS;
        unsigned q = 0;  // rows issued
        bool ok = true;
        auto hand_over = [&](unsigned j) {  // row j has landed
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&given[j % RING]);
        };
        for (long long r = r_begin; r < r_end && ok;) {
            const StripRun u = R.at(r, r_end);
            r += u.L;
            for (int j = 0; j < (COUT == 16 ? u.L + 2 : u.L); ++j) {
                const unsigned s = q % RING;
                if (q >= RING && !role_wait_warp(&taken[s], (q / RING - 1) & 1u, dead)) {
                    ok = false;
                    break;
                }
                if constexpr (COUT == 16) {  // zeros past a narrow strip
                    const __nv_bfloat16* row = dout + ((size_t)u.n * H + R.wrap(u.y0 - 1 + j)) * W * 16;
                    const uint32_t dst = sbase + W6_OFF_D + s * C6_ROW;
                    for (int e = rt; e < C6_W * 2; e += 128) {
                        const int kg = e & 1, px = e >> 1;
                        cp16(dst + px * 128 + ((kg ^ (px & 7)) * 16), row + (size_t)(u.x0 + (px < u.nv ? px : 0)) * 16 + kg * 8,
                             px < u.nv ? 16 : 0);
                    }
                } else {  // pixels -1 .. nv
                    const __nv_bfloat16* row = in + ((size_t)u.n * H + u.y0 + j) * W * 16;
                    const uint32_t dst = sbase + s * C6_SLOT + 1024 - 128;
                    for (int e = rt; e < (u.nv + 2) * 2; e += 128) {
                        const int kg = e & 1, px = e >> 1;
                        int gx = u.x0 - 1 + px;
                        gx = gx < 0 ? gx + W : (gx >= W ? gx - W : gx);
                        cp16(dst + px * 128 + ((kg ^ ((px + 7) & 7)) * 16), row + (size_t)gx * 16 + kg * 8, 16);
                    }
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
                ++q;
                if (q > W6_AHEAD) {
                    asm volatile("cp.async.wait_group %0;" ::"n"(W6_AHEAD) : "memory");
                    hand_over(q - 1 - W6_AHEAD);
                }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (ok)
            for (unsigned j = q > W6_AHEAD ? q - W6_AHEAD : 0; j < q; ++j) hand_over(j);
    } else if (warp >= 8) {
        // 8 channels of pixels sub, sub + 16, ... (those past a narrow strip are zero)
        const int bt = tid - 8 * 32, c8 = bt % 8, sub = bt / 8;
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        unsigned q = 0;
        bool ok = true;
        for (long long r = r_begin; r < r_end && ok;) {
            const StripRun u = R.at(r, r_end);
            r += u.L;
            for (int j = 0; j < u.L + 2; ++j, ++q) {
                const unsigned s = q % W6_DS;
                if (!role_wait_warp(&dfull[s], (q / W6_DS) & 1u, dead)) {
                    ok = false;
                    break;
                }
                if (j >= 1 && j <= u.L) {  // rows of the run itself
                    const unsigned char* row = smem + W6_OFF_D + s * C6_ROW;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int px = sub + 16 * i;
                        const uint4 v = *reinterpret_cast<const uint4*>(row + px * 128 + ((c8 ^ (px & 7)) * 16));
                        const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&v);
#pragma unroll
                        for (int c = 0; c < 8; ++c) acc[c] += __bfloat162float(h[c]);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&dempty[s]);
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) s_b[sub][c8 * 8 + c] = acc[c];
        group_sync(2);
        if (bt < 64) {
            float t = 0.f;
            for (int j = 0; j < 16; ++j) t += s_b[j][bt];
            bpart[(size_t)blockIdx.x * 64 + bt] = t;
        }
    }
    // the accumulators: rows m = (dx, ci) of D1 (dx = -1, 0) and the upper half of D2 (dx = +1); columns (dy = +1, 0, -1; co)
    __syncwarp();
    bool ok = true;
    if (warp >= 4 && warp < 8) {
        ok = role_wait_warp(&done, 0u, dead);
        if (!ok) land(&done, 0u);
        __syncwarp();
    }
    tc_fence_after();
    if (warp >= 4 && warp < 8) {
        const int m = 32 * (warp % 4) + lane, ci = m % 64;
        const uint32_t tl = tmem + ((uint32_t)(32 * (warp % 4)) << 16);
        float* pb = part + (size_t)blockIdx.x * 9 * COUT * CIN;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && warp % 4 < 2) continue;
            const int dxi = m / 64 + h;  // 0, 1, 2 for dx = -1, 0, +1
#pragma unroll 1
            for (int c = 0; c < 192; c += COUT == 64 ? 32 : 64) {
                float v[32];
                __syncwarp();
                tc_ld32(tl + h * 192 + c, v);
                tc_wait_ld(v);
                const int by = 2 - c / 64;
                float* o = pb + ((size_t)(by * 3 + dxi) * COUT + c % 64) * CIN + ci;
                if (CIN == 64 || ci < CIN) {
#pragma unroll
                    for (int j = 0; j < (COUT < 32 ? COUT : 32); ++j) o[j * CIN] = ok ? v[j] : 0.f;
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && dead_flag) atomicOr(status, 1);
    if (warp == 2) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

}  // namespace

namespace {

template <int CIN, int COUT>
cudaError_t wgrad_tc_t(const __nv_bfloat16* in, const __nv_bfloat16* dout, int N, int H, int W, int in_relu, float* dw, float* db,
                       float* part, cudaStream_t s, int sms, int* status) {
    const long long rows = (long long)N * H;
    if (rows >= (1ll << 31)) return cudaErrorInvalidValue;
    CUtensorMap tx{}, tx8{}, td{};
    cudaError_t e = cudaSuccess;
    if (CIN == 64) {
        e = encode_rows64(in, rows, W, C6_W, &tx);
        if (e == cudaSuccess) e = encode_rows64(in, rows, W, 8, &tx8);
    }
    if (e == cudaSuccess && COUT == 64) e = encode_rows64(dout, rows, W, C6_W, &td);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_wgrad_tc<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, W6_BYTES);
    if (e != cudaSuccess) return e;
    const int grid = wgrad_blocks(N, H, W, sms);
    float* bpart = part + (size_t)grid * 9 * COUT * CIN;
    e = launch_early(k_wgrad_tc<CIN, COUT>, grid, W6_THREADS<CIN, COUT>, W6_BYTES, s, tx, tx8, td, in, dout, N, H, W, in_relu, part,
                     bpart, status);
    return e != cudaSuccess ? e : launch_wgrad_sum(part, grid, COUT * CIN, dw, bpart, db, COUT, s);
}

}  // namespace

cudaError_t launch_wgrad_tc(int cin, int cout, const __nv_bfloat16* in, const __nv_bfloat16* dout, int N, int H, int W,
                            int in_relu, float* dw, float* db, float* part, cudaStream_t s, int sms, int* status) {
    if (N < 1 || H < 1 || W < 16 || W % 16 != 0 || !status || sms < 1) return cudaErrorInvalidValue;
    if (cin == 64 && cout == 64) return wgrad_tc_t<64, 64>(in, dout, N, H, W, in_relu, dw, db, part, s, sms, status);
    if (cin == 16 && cout == 64 && !in_relu) return wgrad_tc_t<16, 64>(in, dout, N, H, W, in_relu, dw, db, part, s, sms, status);
    if (cin == 64 && cout == 16) return wgrad_tc_t<64, 16>(in, dout, N, H, W, in_relu, dw, db, part, s, sms, status);
    return cudaErrorInvalidValue;
}

}  // namespace lbm
