// Batched time step: many independent cases of different size and
// temperature advance together, one launch per time step. Every warp marches
// the rows of its list of items (case, strip, rows) with the engine of
// lbm_march.cuh; the host deals the items so that the warps of one wave of
// resident blocks get equal work, neighbouring strips to neighbouring warps. A case's constants (temperature-dependent
// c, dt, c_s, G^2/c, rho_v/rho_l, C_ref, shift) and geometry are copied into
// the warp's shared memory when an item starts.
// Per-item partial sums of the conservation record go to a table from which
// per-case records are reduced on demand: FP32 sums cover 16 rows of a strip (21
// roundings; 500 rows and FP32 items were off by up to 7e-6 on uniform boxes),
// FP64 sums the rest. 256 boxes of 64 to 512 a side, FP16 storage: 334.7 us per
// step with FP32 items, 338.5 so.
#include "lbm_batch.h"
#include "lbm_march.cuh"

namespace lbm {

namespace {

// Warps per block and blocks per SM. A case's constants come from shared
// memory instead of the launch's constant bank, so a warp needs registers for
// them: with the 168 of three blocks per SM the 16-bit form spills (256 boxes
// of 64 to 512 a side, FP16 storage: 445 us per step with 12 warps per SM, 342
// with 8, 500 with 9 or 10, which share the four schedulers unevenly).
template <class S>
struct BatchCfg {
    static constexpr int W = 4;
    static constexpr int BPS = sizeof(S) == 2 ? 2 : 4;
};

template <class S>
__global__ void __launch_bounds__(32 * BatchCfg<S>::W, BatchCfg<S>::BPS) k_batch_step(const BatchLaunch B, int from, const S* arena_in, S* arena_out) {
    using Cf = MarchCfg<S>;
    using V = typename std::conditional<Cf::NPL == 2, F2, float>::type;
    constexpr int W = BatchCfg<S>::W;
    __shared__ BatchCase s_case[W];
    __shared__ double s_rec[W][7];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int gw = blockIdx.x * W + warp;
    if (gw >= B.warps) return;
    BatchCase& cs = s_case[warp];
    Strip<S, float> w;
    w.phi = nullptr;
    w.wait_ns = B.tile_wait_ns;
    w.sr = Store<S, float>::SHIFTED && B.rounding;
    w.steps = &B.steps[from];
    const int end = B.first[gw + 1];
    for (int item = B.first[gw]; item < end; ++item) {
        const BatchItem it = B.items[item];
        w.xs = it.xs;
        w.y0 = it.y0;
        w.y1 = it.y1;
        {
            const uint32_t* src = reinterpret_cast<const uint32_t*>(B.cases + it.c);
            uint32_t* dst = reinterpret_cast<uint32_t*>(&cs);
            __syncwarp();
            for (int j = lane; j < (int)(sizeof(BatchCase) / 4); j += 32) dst[j] = __ldg(src + j);
            __syncwarp();
        }
        w.in = arena_in + cs.off;
        w.out = arena_out + cs.off;
        Geometry G = cs.geo;
        G.lsw = Cf::NPL == 2 ? 6 : 5;  // (known here, so that the compiler knows them too; a batch's cases are periodic)
        G.walls = G.open = 0;
        const int q = lane / 4;
        const bool mine = lane % 4 == 0 && q < 7;  // this lane carries quantity q
        if (mine) s_rec[warp][q] = 0.0;
        const Rec<float> zero = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        Rec<float> acc = zero;
        auto flush = [&](Rec<float>& a) {
            const double v = (double)reduce_record(a, lane);
            if (mine) s_rec[warp][q] = q == 5 ? fmax(s_rec[warp][q], v) : s_rec[warp][q] + v;
            a = zero;
        };
        if (!march_rows<S, float, false, false, true>(cs.kf, march_constants<V>(cs), G, w, acc, flush)) {
            if (lane == 0) atomicOr(B.status, ST_TIMEOUT);
            break;
        }
        if (mine) {
            const double t = s_rec[warp][q], c = (double)cs.kf.c;
            if (q == 6 && t > 0.0) atomicOr(B.status, ST_NONFINITE);
            B.partials[(size_t)item * 8 + q] = q == 1 || q == 2 ? t * c : (q == 5 ? t * (c * c) : t);
        }
    }
    if (gw == 0 && lane == 0) {
        after_previous_grid();
        B.steps[1 - from] = __ldcg(&B.steps[from]) + 1.0;
    }
}

// Per-case conservation record from the per-item partials, FP64, items in
// list order (deterministic).
__global__ void k_batch_case_record(const BatchItem* __restrict__ items, int nitems, int c,
                                    const double* __restrict__ partials, double* __restrict__ out) {
    __shared__ double red[8][256];
    double t[7] = {0, 0, 0, 0, 0, 0, 0};
    for (int i = threadIdx.x; i < nitems; i += blockDim.x) {
        if (items[i].c != c) continue;
        for (int q = 0; q < 7; ++q) {
            const double v = partials[(size_t)i * 8 + q];
            t[q] = (q == 5) ? fmax(t[q], v) : t[q] + v;
        }
    }
    for (int q = 0; q < 7; ++q) red[q][threadIdx.x] = t[q];
    __syncthreads();
    if (threadIdx.x < 7) {
        const int q = threadIdx.x;
        double s = 0.0;
        for (int j = 0; j < (int)blockDim.x; ++j) s = (q == 5) ? fmax(s, red[q][j]) : s + red[q][j];
        out[q] = (q == 5) ? sqrt(s) : s;
    }
}

template <class S>
cudaError_t launch_bt(const BatchLaunch& B, int from, const void* in, void* out, cudaStream_t s) {
    return launch_early(k_batch_step<S>, (B.warps + BatchCfg<S>::W - 1) / BatchCfg<S>::W, 32 * BatchCfg<S>::W, 0, s, B, from,
                        static_cast<const S*>(in), static_cast<S*>(out));
}

}  // namespace

int batch_warps(int storage, int sms) {
    return sms * (storage == S_F32 ? BatchCfg<float>::W * BatchCfg<float>::BPS : BatchCfg<__half>::W * BatchCfg<__half>::BPS);
}

cudaError_t launch_batch_step(int storage, const BatchLaunch& B, int from, const void* in, void* out, cudaStream_t s) {
    switch (storage) {
        case S_F16: return launch_bt<__half>(B, from, in, out, s);
        case S_BF16: return launch_bt<__nv_bfloat16>(B, from, in, out, s);
        case S_F32: return launch_bt<float>(B, from, in, out, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_batch_case_record(const BatchLaunch& B, int c, double* out, cudaStream_t s) {
    k_batch_case_record<<<1, 256, 0, s>>>(B.items, B.nitems, c, B.partials, out);
    return cudaGetLastError();
}

}  // namespace lbm
