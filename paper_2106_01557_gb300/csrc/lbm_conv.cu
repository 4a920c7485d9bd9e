// BF16 tensor-core kernels of the learned surrogate (a 3x3 convolutional
// neural operator that advances (rho, u_x, u_y, T) by K lattice steps), with
// FP32 accumulation:
//   k_conv       implicit-GEMM 3x3 convolution, periodic padding, NHWC BF16
//                activations; the whole weight tensor and a halo'd input tile
//                sit in shared memory; fused epilogue: bias, ReLU mask of
//                another tensor, residual add (BF16 or FP32), BF16 or FP32
//                output. Also serves the input gradient (flipped weights).
//   k_wgrad      weight gradient: per filter row a GEMM over pixels; each
//                block writes its partial sums, which k_wgrad_sum adds in a
//                fixed order
//   k_bgrad      bias gradient (per-block partials, summed in a fixed order).
// (These three on mma.sync; conv_path 0 takes the tcgen05 kernels of
// lbm_conv_tc.cu and lbm_wgrad64.cu, which sum in the same order.)
// No reduction uses atomics: the order of every sum is fixed, so training
// is bit-for-bit reproducible.
//   k_mse        loss and its gradient.
//   k_adam_refresh  optimiser step on FP32 master weights of all layers, and
//                the BF16 forward and flipped copies.
//   k_pack / k_unpack  fields <-> normalised network tensors.
// The MMA is mma.sync m16n8k16 (BF16 in, FP32 accumulate).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_conv.h"
#include "lbm_launch.cuh"
#include "lbm_ptx.cuh"

namespace lbm {
namespace {

__device__ __forceinline__ void mma_bf16(float& c0, float& c1, float& c2, float& c3, uint32_t a0, uint32_t a1,
                                         uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c0), "+f"(c1), "+f"(c2), "+f"(c3)
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t ld32(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ __nv_bfloat16 relu_bf(__nv_bfloat16 v) {
    return __hgt(v, __float2bfloat16(0.f)) ? v : __float2bfloat16(0.f);
}

constexpr int TW = 128;          // output pixels along x per tile
constexpr int TH = 2;            // output rows per tile
constexpr int CT = 512;          // threads: 16 warps, one 16-pixel m-tile each

template <int CIN, int COUT>
struct ConvSmem {
    static constexpr int PS = CIN + 8;                       // padded pixel stride (bank spread)
    static constexpr int IN_ELEMS = (TH + 2) * (TW + 2) * PS;
    static constexpr int W_ELEMS = 9 * COUT * PS;
    static constexpr int BYTES = 2 * (IN_ELEMS + W_ELEMS);
};

// Persistent: each CTA stages all weights once, then walks tiles of TH rows x
// TW pixels of one image.
template <int CIN, int COUT>
__global__ void __launch_bounds__(CT, 1)
    k_conv(const __nv_bfloat16* __restrict__ in, const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias,
           int N, int H, int W, int in_relu, const __nv_bfloat16* __restrict__ mask,
           const __nv_bfloat16* __restrict__ res16, const float* __restrict__ res32,
           __nv_bfloat16* __restrict__ out16, float* __restrict__ out32) {
    using SMc = ConvSmem<CIN, COUT>;
    constexpr int PS = SMc::PS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __nv_bfloat16* s_in = reinterpret_cast<__nv_bfloat16*>(smem_raw);
    __nv_bfloat16* s_w = s_in + SMc::IN_ELEMS;
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int g = lane / 4, t = lane % 4;

    // weights [9][COUT][CIN] -> shared [9][COUT][PS], 8 channels per copy
    for (int e = tid; e < 9 * COUT * (CIN / 8); e += CT) {
        const int row = e / (CIN / 8), c8 = e % (CIN / 8);
        *reinterpret_cast<uint4*>(s_w + row * PS + c8 * 8) = *reinterpret_cast<const uint4*>(w + row * CIN + c8 * 8);
    }
    const int tiles_x = (W + TW - 1) / TW, tiles_y = (H + TH - 1) / TH;
    const int ntiles = N * tiles_y * tiles_x;
    constexpr int NT8 = COUT / 8;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int tx = tile % tiles_x, ty = (tile / tiles_x) % tiles_y, n = tile / (tiles_x * tiles_y);
        const int x0 = tx * TW, y0 = ty * TH;
        __syncthreads();  // previous tile's reads of s_in done (and weights staged)
        // halo'd input tile: rows y0-1 .. y0+TH, pixels x0-1 .. x0+TW (periodic)
        for (int e = tid; e < (TH + 2) * (TW + 2) * (CIN / 8); e += CT) {
            const int c8 = e % (CIN / 8), px = (e / (CIN / 8)) % (TW + 2), r = e / ((CIN / 8) * (TW + 2));
            int gy = y0 - 1 + r, gx = x0 - 1 + px;
            gy = (gy % H + H) % H;
            gx = (gx % W + W) % W;
            uint4 v = *reinterpret_cast<const uint4*>(in + (((size_t)n * H + gy) * W + gx) * CIN + c8 * 8);
            if (in_relu) {
                __nv_bfloat16* h = reinterpret_cast<__nv_bfloat16*>(&v);
#pragma unroll
                for (int j = 0; j < 8; ++j) h[j] = relu_bf(h[j]);
            }
            *reinterpret_cast<uint4*>(s_in + (r * (TW + 2) + px) * PS + c8 * 8) = v;
        }
        __syncthreads();
        const int orow = warp / (TW / 16), px0 = (warp % (TW / 16)) * 16;
        float acc[NT8][4];
#pragma unroll
        for (int j = 0; j < NT8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
#pragma unroll 1
        for (int tap = 0; tap < 9; ++tap) {
            const int dy = tap / 3 - 1, dx = tap % 3 - 1;
            const __nv_bfloat16* arow = s_in + ((orow + 1 + dy) * (TW + 2) + px0 + 1 + dx) * PS;
            const __nv_bfloat16* wt = s_w + tap * COUT * PS;
#pragma unroll
            for (int kc = 0; kc < CIN / 16; ++kc) {
                const __nv_bfloat16* a = arow + kc * 16 + 2 * t;
                const uint32_t a0 = ld32(a + g * PS), a1 = ld32(a + (g + 8) * PS);
                const uint32_t a2 = ld32(a + g * PS + 8), a3 = ld32(a + (g + 8) * PS + 8);
#pragma unroll
                for (int j = 0; j < NT8; ++j) {
                    const __nv_bfloat16* b = wt + (j * 8 + g) * PS + kc * 16 + 2 * t;
                    mma_bf16(acc[j][0], acc[j][1], acc[j][2], acc[j][3], a0, a1, a2, a3, ld32(b), ld32(b + 8));
                }
            }
        }
        // epilogue
        const int oy = y0 + orow;
        if (oy < H) {
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int ox = x0 + px0 + g + 8 * half;
                if (ox >= W) continue;
                const size_t p = ((size_t)n * H + oy) * W + ox;
#pragma unroll
                for (int j = 0; j < NT8; ++j) {
                    const int co = j * 8 + 2 * t;
                    float v0 = acc[j][2 * half], v1 = acc[j][2 * half + 1];
                    if (bias) { v0 += bias[co]; v1 += bias[co + 1]; }
                    if (mask) {
                        const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162*>(mask + p * COUT + co);
                        if (!(__bfloat162float(m.x) > 0.f)) v0 = 0.f;
                        if (!(__bfloat162float(m.y) > 0.f)) v1 = 0.f;
                    }
                    if (res16) {
                        const __nv_bfloat162 r = *reinterpret_cast<const __nv_bfloat162*>(res16 + p * COUT + co);
                        v0 += __bfloat162float(r.x);
                        v1 += __bfloat162float(r.y);
                    }
                    if (out32) {
                        if (co >= 4) continue;
                        if (res32) {
                            v0 += res32[p * 4 + co];
                            v1 += res32[p * 4 + co + 1];
                        }
                        out32[p * 4 + co] = v0;
                        out32[p * 4 + co + 1] = v1;
                    } else {
                        *reinterpret_cast<__nv_bfloat162*>(out16 + p * COUT + co) = __floats2bfloat162_rn(v0, v1);
                    }
                }
            }
        }
    }
}

// Weight gradient dW[tap][co][ci] += sum_p dOut[p][co] * act(in[p + off(tap)][ci]).
// A CTA owns one filter row dy (its three taps dx = -1, 0, 1) and every
// output and input channel, over a run of 128-pixel row chunks: the chunk's
// dOut row [128 px][COUT] and the input row y + dy [130 px][CIN] (periodic
// halo) are copied with cp.async into padded shared tiles (two stages), and
// ldmatrix.trans forms the MMA fragments straight from these pixel-major
// tiles: A = dOut^T (co x pixels), B = input (pixels x ci, shifted by dx).
// One A fragment serves the three taps. Warp w owns the 16-channel output
// block w % (COUT/16) and a contiguous group of 8-channel input blocks; its
// FP32 sums are the block's partial, added by k_wgrad_sum in a fixed order.
constexpr int WT = 256;      // threads (8 warps)
constexpr int WCH = 128;     // pixels per chunk

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t addr, uint32_t& r0, uint32_t& r1) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r0), "=r"(r1) : "r"(addr));
}
// 16-byte async copy; src_bytes = 0 fills the destination with zeros
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

template <int CIN, int COUT>
struct WgCfg {
    static constexpr int RSD = COUT * 2 + 16;          // padded row bytes of the dOut tile (ldmatrix: no conflicts)
    static constexpr int RSX = CIN * 2 + 16;           // padded row bytes of the input tile
    static constexpr int D_BYTES = WCH * RSD;
    static constexpr int X_BYTES = (WCH + 2) * RSX;
    static constexpr int STAGE = D_BYTES + X_BYTES;
    static constexpr int MT = COUT / 16;               // 16-channel output blocks
    static constexpr int NG = 8 / MT;                  // warps per output block
    static constexpr int NPW = (CIN / 8) / NG;         // 8-channel input blocks per warp
    static_assert(COUT % 16 == 0 && COUT <= 128 && 8 % MT == 0 && (CIN / 8) % NG == 0 && NPW >= 1, "warp split");
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(WT)
    k_wgrad(const __nv_bfloat16* in, const __nv_bfloat16* dout, int N, int H, int W,
            int in_relu, float* __restrict__ part) {
    after_previous_grid();
    using Cf = WgCfg<CIN, COUT>;
    extern __shared__ __align__(16) unsigned char wg_smem[];
    const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
    const int g = lane / 4, t = lane % 4;
    const int dy = (int)blockIdx.y - 1;
    const int tiles_x = (W + WCH - 1) / WCH;
    // this block's run of the input rows of all strips, strip after strip
    const long long rows = (long long)N * H * tiles_x;
    const long long r_begin = rows * blockIdx.x / gridDim.x, r_end = rows * (blockIdx.x + 1) / gridDim.x;
    const int mt = warp % Cf::MT, nt0 = (warp / Cf::MT) * Cf::NPW;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(wg_smem);
    float acc[3][Cf::NPW][4];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int j = 0; j < Cf::NPW; ++j) acc[a][j][0] = acc[a][j][1] = acc[a][j][2] = acc[a][j][3] = 0.f;

    // copy chunk ch into stage st (one commit group per call, empty past the end)
    auto load = [&](long long ch, int st) {
        if (ch < r_end) {
            const int yy = (int)(ch % H);  // input row
            const long long strip = ch / H;
            const int x0 = (int)(strip % tiles_x) * WCH, n = (int)(strip / tiles_x);
            int y = yy - dy;  // dOut row
            y = y < 0 ? y + H : (y >= H ? y - H : y);
            const uint32_t sd = sbase + st * Cf::STAGE, sx = sd + Cf::D_BYTES;
            const __nv_bfloat16* drow = dout + ((size_t)n * H + y) * W * COUT;
            const __nv_bfloat16* xrow = in + ((size_t)n * H + yy) * W * CIN;
            for (int e = tid; e < WCH * (COUT / 8); e += WT) {
                const int px = e / (COUT / 8), c8 = e % (COUT / 8);
                const int x = x0 + px;
                cp16(sd + px * Cf::RSD + c8 * 16, drow + (size_t)(x < W ? x : 0) * COUT + c8 * 8, x < W ? 16 : 0);
            }
            for (int e = tid; e < (WCH + 2) * (CIN / 8); e += WT) {
                const int px = e / (CIN / 8), c8 = e % (CIN / 8);
                int x = x0 - 1 + px;
                x = x < 0 ? x + W : (x >= W ? x % W : x);
                cp16(sx + px * Cf::RSX + c8 * 16, xrow + (size_t)x * CIN + c8 * 8, 16);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // ReLU in place on the input vectors this thread copied
    auto relu_tile = [&](int st) {
        unsigned char* sx = wg_smem + st * Cf::STAGE + Cf::D_BYTES;
        for (int e = tid; e < (WCH + 2) * (CIN / 8); e += WT) {
            const int px = e / (CIN / 8), c8 = e % (CIN / 8);
            uint4* v = reinterpret_cast<uint4*>(sx + px * Cf::RSX + c8 * 16);
            uint4 u = *v;
            __nv_bfloat16* h = reinterpret_cast<__nv_bfloat16*>(&u);
#pragma unroll
            for (int q = 0; q < 8; ++q) h[q] = relu_bf(h[q]);
            *v = u;
        }
    };

    long long ch = r_begin;
    load(ch, 0);
    for (int it = 0; ch < r_end; ++ch, ++it) {
        const int st = it & 1;
        load(ch + 1, st ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        if (in_relu) relu_tile(st);
        __syncthreads();
        const uint32_t sd = sbase + st * Cf::STAGE, sx = sd + Cf::D_BYTES;
#pragma unroll 2
        for (int k0 = 0; k0 < WCH; k0 += 16) {
            // A = dOut^T: rows co (mt*16 ..), columns pixels k0 .. k0+15
            const int q = lane / 8;
            uint32_t a0, a1, a2, a3;
            ldsm_x4_t(sd + (k0 + (q >= 2 ? 8 : 0) + lane % 8) * Cf::RSD + (mt * 16 + (q & 1) * 8) * 2, a0, a1, a2, a3);
#pragma unroll
            for (int tap = 0; tap < 3; ++tap) {
                // B = input pixels k0 + dx .. (tile pixel index + 1 for the halo)
#pragma unroll
                for (int j = 0; j < Cf::NPW; ++j) {
                    uint32_t b0, b1;
                    const int l = lane % 16;
                    ldsm_x2_t(sx + (k0 + tap + (l >= 8 ? 8 : 0) + l % 8) * Cf::RSX + (nt0 + j) * 16, b0, b1);
                    mma_bf16(acc[tap][j][0], acc[tap][j][1], acc[tap][j][2], acc[tap][j][3], a0, a1, a2, a3, b0, b1);
                }
            }
        }
        __syncthreads();  // the stage is refilled by the next iteration's load
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // accumulator (row co, column ci) of filter column dx = tap - 1 -> this
    // block's partial [blockIdx.x][dy + 1][tap][co][ci]
    float* pb = part + ((size_t)blockIdx.x * 3 + blockIdx.y) * 3 * COUT * CIN;
#pragma unroll
    for (int tap = 0; tap < 3; ++tap) {
#pragma unroll
        for (int j = 0; j < Cf::NPW; ++j) {
            const int co = mt * 16 + g, ci = (nt0 + j) * 8 + 2 * t;
            float* d = pb + ((size_t)tap * COUT + co) * CIN + ci;
            d[0] = acc[tap][j][0];
            d[1] = acc[tap][j][1];
            d[8 * CIN] = acc[tap][j][2];
            d[8 * CIN + 1] = acc[tap][j][3];
        }
    }
}

// dw[tp][co][ci] = the sum over blocks of the partials, tap tp = 3 (dy + 1) +
// dx + 1, four weights per thread: thread row ty adds blocks ty, ty + 8, ... in
// that order, then the eight rows are added in order (a fixed order).
// The last block, where there is a bias gradient, adds its partials [nblk][64]
// the same way: row j of four adds blocks j, j + 4, ...
__global__ void __launch_bounds__(256) k_wgrad_sum(const float4* part, int nblk, int n4, float4* __restrict__ dw,
                                                   const float* bpart, float* __restrict__ db, int nb) {
    after_previous_grid();
    __shared__ float4 s[8][32];
    if (db && blockIdx.x == gridDim.x - 1) {
        float* t = reinterpret_cast<float*>(s);
        const int c = threadIdx.x % 64, j = threadIdx.x / 64;
        float a = 0.f;
#pragma unroll 4
        for (int b = j; b < nblk; b += 4) a += __ldcg(bpart + (size_t)b * 64 + c);
        t[threadIdx.x] = a;
        __syncthreads();
        if (j == 0 && c < nb) db[c] = ((a + t[64 + c]) + t[128 + c]) + t[192 + c];
        return;
    }
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
    const int e = blockIdx.x * 32 + tx;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (e < n4) {
#pragma unroll 8
        for (int b = ty; b < nblk; b += 8) {
            const float4 v = __ldcg(part + (size_t)b * n4 + e);
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
    }
    s[ty][tx] = a;
    __syncthreads();
    if (ty == 0 && e < n4) {
#pragma unroll
        for (int j = 1; j < 8; ++j) {
            const float4 v = s[j][tx];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
        dw[e] = a;
    }
}

// Bias gradient db[c] = sum_p dOut[p][c]: the block's partial sums over the
// blocks' runs of rows, in the order in which k_wgrad_tc sums them (128 threads:
// 8 channels of pixels sub, sub + 16, ...; [64] per block, zeros past C).
template <int C>
__global__ void __launch_bounds__(128) k_bgrad(const __nv_bfloat16* __restrict__ dout, int N, int H, int W, float* __restrict__ part) {
    __shared__ float s[16][64];
    const int c8 = threadIdx.x % 8, sub = threadIdx.x / 8;
    const int tiles_x = (W + WCH - 1) / WCH;
    const long long rows = (long long)N * H * tiles_x;
    const long long r_end = rows * (blockIdx.x + 1) / gridDim.x;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    // A row's loads are issued before any is used, two rows at a time: one after
    // another they cost the gradients of 8 x 256 x 256 0.6 ms of 8.3.
#pragma unroll 2
    for (long long r = rows * blockIdx.x / gridDim.x; r < r_end; ++r) {
        const long long strip = r / H;
        const int x0 = (int)(strip % tiles_x) * WCH;
        const __nv_bfloat16* row = dout + ((strip / tiles_x * H + r % H) * W + x0) * C + c8 * 8;
        uint4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int px = sub + 16 * i;
            v[i] = make_uint4(0, 0, 0, 0);
            if (x0 + px < W && c8 * 8 < C) v[i] = *reinterpret_cast<const uint4*>(row + (size_t)px * C);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&v[i]);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] += __bfloat162float(h[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) s[sub][c8 * 8 + c] = acc[c];
    __syncthreads();
    if (threadIdx.x < 64) {
        float t = 0.f;
        for (int j = 0; j < 16; ++j) t += s[j][threadIdx.x];
        part[(size_t)blockIdx.x * 64 + threadIdx.x] = t;
    }
}

// *out = sum over i = 0 .. n-1 of part[i], by one warp in a fixed order
// (lane l: i = l, l + 32, ...; then a butterfly)
__global__ void k_sum_in_order(const double* part, int n, double* __restrict__ out) {
    after_previous_grid();
    const int lane = threadIdx.x;
    if (blockIdx.x != 0 || lane >= 32) return;
    double t = 0.0;
    for (int i = lane; i < n; i += 32) t += part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) *out = t;
}

// loss = mean over P pixels and 4 channels of (out - target)^2; dout = d loss / d out.
// With the mass-conserving output layer (sums not null) out_rho is first
// shifted by -sums[n] / HW (image n), and the density gradient is projected:
// minus its per-image mean, which equals 2 (mean(x_rho) - mean(target_rho)) /
// (4 P); sums[N + n] = sum over image n of (x_rho - target_rho), HW pixels per
// image. Grid y: images. Bound by memory (P x 64 bytes); with 64-bit divisions
// and 2-byte stores per pixel it took 47 us on 8 x 256 x 256.
__global__ void k_mse(const float4* out, const float4* target, int N, long long HW,
                      uint4* __restrict__ dout, double* __restrict__ part, const double* sums) {
    after_previous_grid();
    __shared__ double s[256];
    double acc = 0.0;
    const long long P = HW * N;
    const float scale = 2.0f / (float)(P * 4);
    auto square = [](float d) { const double w = widen(d); return w * w; };
    __shared__ double means[2];
    for (int n = blockIdx.y; n < N; n += gridDim.y) {
    __syncthreads();
    if (threadIdx.x < 2) means[threadIdx.x] = sums ? sums[threadIdx.x * N + n] / (double)HW : 0.0;
    __syncthreads();
    const double mean = means[0];
    const float shift = (float)means[1];
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < HW; q += (long long)gridDim.x * blockDim.x) {
        const long long p = n * HW + q;
        const float4 o = out[p], t = target[p];
        const float d0 = (sums ? narrow(widen(o.x) - mean) : o.x) - t.x, d1 = o.y - t.y, d2 = o.z - t.z, d3 = o.w - t.w;
        acc += square(d0);
        acc += square(d1);
        acc += square(d2);
        acc += square(d3);
        const __nv_bfloat162 a = __floats2bfloat162_rn(scale * (d0 - shift), scale * d1), b = __floats2bfloat162_rn(scale * d2, scale * d3);
        uint4 v = make_uint4(0, 0, 0, 0);
        memcpy(&v.x, &a, 4);
        memcpy(&v.y, &b, 4);
        dout[2 * p] = v;
        dout[2 * p + 1] = make_uint4(0, 0, 0, 0);
    }
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = s[0] / (double)(P * 4);
}

// Adam on FP32 master weights of all layers in one launch (grid y = layers):
// the update, then the BF16 forward copy and the flipped, transposed copy used
// for the input gradient: wf[8 - tap][ci][co] = w[tap][co][ci]. Without
// `update` only the copies. (42 launches of one layer's update or copy took 95 + 69 us.)
__global__ void k_adam_refresh(const LayerDesc* __restrict__ layers, float* __restrict__ w, float* __restrict__ m,
                               float* __restrict__ v, const float* g, __nv_bfloat16* __restrict__ w16,
                               __nv_bfloat16* __restrict__ wflip, int update, float lr, float b1, float b2, float eps,
                               float c1, float c2) {
    after_previous_grid();
    const LayerDesc d = layers[blockIdx.y];
    const int nw = 9 * d.cout * d.cin;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw + d.cout; i += gridDim.x * blockDim.x) {
        const long long e = d.off + i;  // the layer's weights, then its biases
        float wi = w[e];
        if (update) {
            const float gi = g[e];
            const float mi = b1 * m[e] + (1.f - b1) * gi;
            const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
            m[e] = mi;
            v[e] = vi;
            wi -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
            w[e] = wi;
        }
        if (i < nw) {
            const int ci = i % d.cin, co = (i / d.cin) % d.cout, tap = i / (d.cin * d.cout);
            const float val = (ci < d.cin_real && co < d.cout_real) ? wi : 0.f;  // padding stays zero
            const __nv_bfloat16 b = __float2bfloat16(val);
            w16[d.off16 + i] = b;
            wflip[d.off16 + ((long long)(8 - tap) * d.cin + ci) * d.cout + co] = b;
        }
    }
}

// fields -> normalised network input: 16 BF16 channels (4 used; x16 may be
// null) and an FP32 copy of the 4 channels. One pixel per thread, 16-byte
// stores (with 2-byte stores: 100 us at 1024 x 1024; 26.5 with the conversions
// to FP32 on the FP64 unit, 21.4 in integer arithmetic; memory alone 12).
__global__ void k_pack(const double* rho, const double* ux, const double* uy,
                       const double* T, long long P, NormConsts nc, uint4* __restrict__ x16,
                       float4* __restrict__ x32) {
    after_previous_grid();
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        const float4 v = make_float4(narrow((rho[p] - nc.off[0]) * nc.inv_scale[0]), narrow((ux[p] - nc.off[1]) * nc.inv_scale[1]),
                                     narrow((uy[p] - nc.off[2]) * nc.inv_scale[2]), narrow((T[p] - nc.off[3]) * nc.inv_scale[3]));
        x32[p] = v;
        if (x16) {
            const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
            uint4 o = make_uint4(0, 0, 0, 0);
            memcpy(&o.x, &a, 4);
            memcpy(&o.y, &b, 4);
            x16[2 * p] = o;
            x16[2 * p + 1] = make_uint4(0, 0, 0, 0);
        }
    }
}

// network output [P][4] -> fields, the density of image n (HW pixels; grid y =
// images) first shifted by -sums[n] / HW (sums not null)
__global__ void k_unpack(const float4* y, long long HW, const double* sums, NormConsts nc,
                         int N, double* __restrict__ rho, double* __restrict__ ux, double* __restrict__ uy,
                         double* __restrict__ T) {
    after_previous_grid();
    __shared__ double s_mean;
    for (int n = blockIdx.y; n < N; n += gridDim.y) {
    __syncthreads();
    if (threadIdx.x == 0) s_mean = sums ? sums[n] / (double)HW : 0.0;  // (FP64 divisions are slow here: one per block)
    __syncthreads();
    const double mean = s_mean;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < HW; q += (long long)gridDim.x * blockDim.x) {
        const long long p = n * HW + q;
        const float4 v = y[p];
        const float r = sums ? narrow(widen(v.x) - mean) : v.x;
        rho[p] = nc.off[0] + widen(r) * nc.scale[0];
        ux[p] = nc.off[1] + widen(v.y) * nc.scale[1];
        uy[p] = nc.off[2] + widen(v.z) * nc.scale[2];
        T[p] = nc.off[3] + widen(v.w) * nc.scale[3];
    }
    }
}

// Mass-conserving output layer: per image n, sums[n] = sum of
// (y_rho - x_rho) and, with a target, sums[N + n] = sum of (x_rho - t_rho);
// its readers shift y_rho by -sums[n] / HW. y, x, t: [P][4]; grid y = images.
// Each block writes its two partial sums to part[n][block][2];
// k_mass_sums adds them in block order.
__global__ void k_mass_stats(const float4* y, const float4* x, const float4* t,
                             int N, long long HW, double* __restrict__ part) {
    after_previous_grid();
    __shared__ double s[2][256];
    const int n = blockIdx.y;
    double a = 0.0, b = 0.0;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < HW; q += (long long)gridDim.x * blockDim.x) {
        const long long p = n * HW + q;
        const double xr = (double)x[p].x;
        a += (double)y[p].x - xr;
        if (t) b += xr - (double)t[p].x;
    }
    s[0][threadIdx.x] = a;
    s[1][threadIdx.x] = b;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s[0][threadIdx.x] += s[0][threadIdx.x + o];
            s[1][threadIdx.x] += s[1][threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double* pp = part + ((size_t)n * gridDim.x + blockIdx.x) * 2;
        pp[0] = s[0][0];
        pp[1] = s[1][0];
    }
}

// one warp per image: lane l adds blocks l, l + 32, ..., then a butterfly
// (a fixed order)
__global__ void k_mass_sums(const double* part, int N, int nblk, int with_t, double* __restrict__ sums) {
    after_previous_grid();
    const int n = (int)((blockIdx.x * blockDim.x + threadIdx.x) / 32), lane = threadIdx.x % 32;
    if (n >= N) return;
    double a = 0.0, b = 0.0;
    for (int k = lane; k < nblk; k += 32) {
        a += part[((size_t)n * nblk + k) * 2];
        b += part[((size_t)n * nblk + k) * 2 + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
        sums[n] = a;
        if (with_t) sums[N + n] = b;
    }
}

// counts over a field set [4][P] of one W-wide periodic image: cnt[0] nodes
// with rho > mid (liquid), cnt[1] nodes that are non-finite or have rho <= 0
// or T <= 0, cnt[2] liquid-vapour edges between x- and y-neighbours (the
// interface length on the lattice's staircase), cnt[3] nodes whose phase
// differs from that in the field set prev (if not null)
__global__ void k_field_check(const double* __restrict__ f, const double* __restrict__ prev, long long P, int W,
                              double mid, unsigned long long* __restrict__ cnt) {
    unsigned long long liq = 0, bad = 0, edge = 0, flip = 0;
    const long long H = P / W;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
        const double r = f[p], u = f[P + p], v = f[2 * P + p], T = f[3 * P + p];
        const bool l = r > mid;
        liq += l;
        bad += !(isfinite(r) && isfinite(u) && isfinite(v) && isfinite(T) && r > 0.0 && T > 0.0);
        const long long yy = p / W, xx = p % W;
        const long long px = yy * W + (xx + 1 == W ? 0 : xx + 1);
        const long long py = (yy + 1 == H ? 0 : yy + 1) * W + xx;
        edge += (l != (f[px] > mid)) + (l != (f[py] > mid));
        if (prev) flip += l != (prev[p] > mid);
    }
    for (int o = 16; o > 0; o >>= 1) {
        liq += __shfl_down_sync(0xffffffffu, liq, o);
        bad += __shfl_down_sync(0xffffffffu, bad, o);
        edge += __shfl_down_sync(0xffffffffu, edge, o);
        flip += __shfl_down_sync(0xffffffffu, flip, o);
    }
    if (threadIdx.x % 32 == 0) {
        atomicAdd(&cnt[0], liq);
        atomicAdd(&cnt[1], bad);
        atomicAdd(&cnt[2], edge);
        atomicAdd(&cnt[3], flip);
    }
}

// Largest per-node change between two field sets [4][P] (a, b) for the
// density (plane 0) and the temperature (plane 3), and the largest |b| of
// each: out[0] max |a_rho - b_rho|, out[1] max |b_rho|, out[2], out[3] the
// same for T, as the bit patterns of non-negative doubles (their order is the
// order of the values, so an integer maximum is exact and independent of the
// order of the nodes; a NaN difference compares above every number).
__global__ void k_field_change(const double* __restrict__ a, const double* __restrict__ b, long long P,
                               unsigned long long* __restrict__ out) {
    double m[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < P; p += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const long long q = (k == 0 ? 0 : 3) * P + p;
            const double d = fabs(a[q] - b[q]), v = fabs(b[q]);
            m[2 * k] = (d > m[2 * k] || d != d) ? d : m[2 * k];
            m[2 * k + 1] = (v > m[2 * k + 1] || v != v) ? v : m[2 * k + 1];
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        unsigned long long u = (unsigned long long)__double_as_longlong(m[k]);
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long w = __shfl_down_sync(0xffffffffu, u, o);
            u = w > u ? w : u;
        }
        if (threadIdx.x % 32 == 0) atomicMax(&out[k], u);
    }
}

template <int CIN, int COUT>
cudaError_t conv_t(const ConvArgs& a, cudaStream_t s, int sms) {
    using SMc = ConvSmem<CIN, COUT>;
    static bool set = false;
    if (!set) {
        cudaError_t e = cudaFuncSetAttribute(k_conv<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMc::BYTES);
        if (e != cudaSuccess) return e;
        set = true;
    }
    const int tiles = a.N * ((a.H + TH - 1) / TH) * ((a.W + TW - 1) / TW);
    const int grid = tiles < sms ? tiles : sms;
    k_conv<CIN, COUT><<<grid, CT, SMc::BYTES, s>>>(a.in, a.w, a.bias, a.N, a.H, a.W, a.in_relu, a.mask, a.res16,
                                                   a.res32, a.out16, a.out32);
    return cudaGetLastError();
}

template <int CIN, int COUT>
cudaError_t wgrad_t(const __nv_bfloat16* in, const __nv_bfloat16* dout, int N, int H, int W, int in_relu, float* dw,
                    float* part, cudaStream_t s, int sms) {
    using Cf = WgCfg<CIN, COUT>;
    static bool set = false;
    if (!set) {
        cudaError_t e = cudaFuncSetAttribute(k_wgrad<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * Cf::STAGE);
        if (e != cudaSuccess) return e;
        set = true;
    }
    const int gx = wgrad_blocks(N, H, W, sms);  // the rows are split as the tcgen05 path splits them
    const cudaError_t e = launch_early(k_wgrad<CIN, COUT>, dim3((unsigned)gx, 3), WT, 2 * Cf::STAGE, s, in, dout, N, H, W, in_relu, part);
    return e != cudaSuccess ? e : launch_wgrad_sum(part, gx, COUT * CIN, dw, nullptr, nullptr, 0, s);
}

}  // namespace

cudaError_t launch_field_check(const double* f, const double* prev, long long P, int W, double mid,
                               unsigned long long* cnt, cudaStream_t s) {
    if (W < 1 || P % W != 0) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(cnt, 0, 4 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    long long g = (P + 255) / 256;
    if (g > 2048) g = 2048;
    k_field_check<<<(unsigned)g, 256, 0, s>>>(f, prev, P, W, mid, cnt);
    return cudaGetLastError();
}

cudaError_t launch_field_change(const double* a, const double* b, long long P, unsigned long long* out,
                                cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, 4 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    long long g = (P + 255) / 256;
    if (g > 2048) g = 2048;
    k_field_change<<<(unsigned)g, 256, 0, s>>>(a, b, P, out);
    return cudaGetLastError();
}

cudaError_t launch_mass_layer(const float* y, const float* x, const float* t, int N, long long HW, double* sums,
                              double* part, cudaStream_t s) {
    if (N < 1 || HW < 1) return cudaErrorInvalidValue;
    long long gx = (HW + 255) / 256;
    if (gx > MASS_BLOCKS) gx = MASS_BLOCKS;
    const cudaError_t e = launch_early(k_mass_stats, dim3((unsigned)gx, (unsigned)N), 256, 0, s, reinterpret_cast<const float4*>(y),
                                       reinterpret_cast<const float4*>(x), reinterpret_cast<const float4*>(t), N, HW, part);
    return e != cudaSuccess ? e : launch_early(k_mass_sums, (32 * N + 127) / 128, 128, 0, s, part, N, (int)gx, (int)(t != nullptr), sums);
}

cudaError_t launch_conv(int cin, int cout, const ConvArgs& a, cudaStream_t s, int sms) {
    if (a.W % 16 != 0) return cudaErrorInvalidValue;
    if (cin == 16 && cout == 64) return conv_t<16, 64>(a, s, sms);
    if (cin == 64 && cout == 64) return conv_t<64, 64>(a, s, sms);
    if (cin == 64 && cout == 16) return conv_t<64, 16>(a, s, sms);
    return cudaErrorInvalidValue;
}

size_t grad_scratch_floats(int sms) {
    return (size_t)sms * (9 * 64 * 64 + 64);
}

cudaError_t launch_wgrad(int cin, int cout, const __nv_bfloat16* in, const __nv_bfloat16* dout, int N, int H, int W,
                         int in_relu, float* dw, float* part, cudaStream_t s, int sms) {
    if (cin == 16 && cout == 64) return wgrad_t<16, 64>(in, dout, N, H, W, in_relu, dw, part, s, sms);
    if (cin == 64 && cout == 64) return wgrad_t<64, 64>(in, dout, N, H, W, in_relu, dw, part, s, sms);
    if (cin == 64 && cout == 16) return wgrad_t<64, 16>(in, dout, N, H, W, in_relu, dw, part, s, sms);
    return cudaErrorInvalidValue;
}

cudaError_t launch_wgrad_sum(const float* part, int nblk, int cc, float* dw, const float* bpart, float* db, int nb, cudaStream_t s) {
    if (nblk < 1 || cc < 0 || cc % 4 != 0 || (cc == 0 && !db)) return cudaErrorInvalidValue;
    const int n4 = 9 * cc / 4;
    return launch_early(k_wgrad_sum, (n4 + 31) / 32 + (db ? 1 : 0), 256, 0, s, reinterpret_cast<const float4*>(part), nblk, n4,
                        reinterpret_cast<float4*>(dw), bpart, db, nb);
}

int wgrad_blocks(int N, int H, int W, int sms) {
    const long long rows = (long long)N * H * ((W + WCH - 1) / WCH);
    return rows < sms ? (int)rows : sms;
}

cudaError_t launch_bgrad(const __nv_bfloat16* dout, int N, int H, int W, int C, float* db, float* part, cudaStream_t s, int sms) {
    const int g = wgrad_blocks(N, H, W, sms);
    if (C == 64) k_bgrad<64><<<g, 128, 0, s>>>(dout, N, H, W, part);
    else if (C == 16) k_bgrad<16><<<g, 128, 0, s>>>(dout, N, H, W, part);
    else return cudaErrorInvalidValue;
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_wgrad_sum(part, g, 0, nullptr, part, db, C, s);
}

cudaError_t launch_mse(const float* out, const float* target, int N, long long HW, __nv_bfloat16* dout, double* loss,
                       const double* sums, double* part, cudaStream_t s) {
    if (N < 1 || HW < 1) return cudaErrorInvalidValue;
    const int ny = N < MSE_BLOCKS ? N : MSE_BLOCKS;
    long long g = (HW + 255) / 256;
    if (g > MSE_BLOCKS / ny) g = MSE_BLOCKS / ny;
    const cudaError_t e = launch_early(k_mse, dim3((unsigned)g, (unsigned)ny), 256, 0, s, reinterpret_cast<const float4*>(out),
                                       reinterpret_cast<const float4*>(target), N, HW, reinterpret_cast<uint4*>(dout), part, sums);
    return e != cudaSuccess ? e : launch_early(k_sum_in_order, 1, 32, 0, s, part, (int)g * ny, loss);
}

cudaError_t launch_adam_refresh(const LayerDesc* layers, int nlayers, float* w, float* m, float* v, const float* g,
                                __nv_bfloat16* w16, __nv_bfloat16* wflip, int update, float lr, float b1, float b2, float eps,
                                float c1, float c2, cudaStream_t s) {
    if (nlayers < 1) return cudaErrorInvalidValue;
    return launch_early(k_adam_refresh, dim3(36, (unsigned)nlayers), 256, 0, s, layers, w, m, v, g, w16, wflip, update, lr, b1, b2, eps, c1, c2);
}

cudaError_t launch_pack(const double* rho, const double* ux, const double* uy, const double* T, long long P,
                        const NormConsts& nc, __nv_bfloat16* x16, float* x32, cudaStream_t s) {
    long long g = (P + 255) / 256;
    if (g > 4096) g = 4096;
    return launch_early(k_pack, (unsigned)g, 256, 0, s, rho, ux, uy, T, P, nc, reinterpret_cast<uint4*>(x16), reinterpret_cast<float4*>(x32));
}

cudaError_t launch_unpack(const float* y, int N, long long HW, const double* sums, const NormConsts& nc, double* rho,
                          double* ux, double* uy, double* T, cudaStream_t s) {
    if (N < 1 || HW < 1) return cudaErrorInvalidValue;
    const int ny = N < 1024 ? N : 1024;
    long long g = (HW + 255) / 256;
    if (g > 1216) g = 1216;
    return launch_early(k_unpack, dim3((unsigned)g, (unsigned)ny), 256, 0, s, reinterpret_cast<const float4*>(y), HW, sums, nc, N, rho, ux, uy, T);
}

}  // namespace lbm
