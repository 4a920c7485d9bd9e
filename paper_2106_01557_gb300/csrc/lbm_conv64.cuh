// What the surrogate's warp-specialised kernels share: the cut of an image into
// strips of rows, tensor copies of pixel rows, and the bounded waits of roles.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "lbm_ptx.cuh"
#include "lbm_tc.cuh"

namespace lbm {

constexpr int C6_W = 128;                   // pixels per row segment
constexpr int C6_SLOT = (C6_W + 16) * 128;  // a row with 8 more pixels on each side
constexpr int C6_ROW = C6_W * 128;          // a row without

// a run of rows y0 .. y0 + L - 1 of the strip that starts at pixel x0 and has
// nv pixels, in image n
struct StripRun {
    int y0, L, x0, nv, n;
};

// the rows of all strips of N images, strip after strip
struct StripRuns {
    int H, W, tiles_x;
    long long rows;
    __device__ __forceinline__ StripRuns(int N, int h, int w) : H(h), W(w), tiles_x((w + C6_W - 1) / C6_W) {
        rows = (long long)N * tiles_x * H;
    }
    __device__ __forceinline__ StripRun at(long long r, long long r_end) const {
        StripRun u;
        u.y0 = (int)(r % H);
        const long long strip = r / H;
        u.x0 = (int)(strip % tiles_x) * C6_W;
        u.n = (int)(strip / tiles_x);
        u.L = (int)((long long)(H - u.y0) < r_end - r ? (long long)(H - u.y0) : r_end - r);
        u.nv = W - u.x0 < C6_W ? W - u.x0 : C6_W;
        return u;
    }
    __device__ __forceinline__ int wrap(int y) const { return y < 0 ? y + H : (y >= H ? y - H : y); }
};

// pixels x, x + 1, ... of a row into shared memory (the map's box wide)
__device__ __forceinline__ void tma_load_rows(uint32_t dst, const CUtensorMap* tm, int x, int row, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tm)), "r"(0), "r"(x), "r"(row), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_store_rows(const CUtensorMap* tm, int x, int row, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(tm)),
                 "r"(0), "r"(x), "r"(row), "r"(src)
                 : "memory");
}

// Wait for a phase of bar, bounded; false after the bound, or once another
// role has given up (dead is set for all). For a single lane: lanes of a warp
// that wait each for itself can part when the bound is near, and the ones that go
// on would wait without a bound at the next instruction of the whole warp.
__device__ __forceinline__ bool role_wait(uint64_t* bar, uint32_t parity, volatile int* dead) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (*dead || globaltimer_ns() - t0 > WAIT_NS) {
            *dead = 1;
            return false;
        }
    }
    return true;
}
// the same for a converged warp: one outcome for all lanes. (Warps of a group
// that meet at a barrier in between can still differ: the ones that give up go
// on to the barrier, group_any.)
__device__ __forceinline__ bool role_wait_warp(uint64_t* bar, uint32_t parity, volatile int* dead) {
    return __all_sync(0xffffffffu, role_wait(bar, parity, dead));
}
// a last wait, bounded, for copies or MMAs in flight
__device__ __forceinline__ void land(uint64_t* bar, uint32_t parity) {
    const uint64_t t0 = globaltimer_ns();
    while (!mbar_try_wait(bar, parity) && globaltimer_ns() - t0 < WAIT_NS) {}
}

// [rows][W][64] BF16: boxes of `px` pixels of one row, 128-byte swizzle
cudaError_t encode_rows64(const void* base, long long rows, int W, int px, CUtensorMap* m);

}  // namespace lbm
