// The fused f+g step of a single lattice: the row-marching engine of
// lbm_march.cuh over strips and chunks of rows, one task per warp.
//
// The blocks of one chunk of rows cover adjacent strips, and all chunks run
// at once (one wave: as many chunks as there are resident blocks), so the
// sectors two strips share are in the L2 cache when the second one asks.
//
// The conservation record of a step (per-block FP64 partial sums) is combined
// by extra blocks of the next step's launch, off the critical path, or,
// where no step follows in the call, by the last block to finish.
#include "lbm_march.cuh"

namespace lbm {

namespace {

// stats[q] from the per-block partials [nblk][NQ]: warp w takes the
// quantities w, w + nw, ...; lane l takes blocks l, l + 32, ... (independent
// L2 loads), then a butterfly: a fixed order, so the record is the same on
// every run
__device__ __forceinline__ void combine_record(const double* partials, int nblk, double* stats, int warp, int nw, int lane) {
    for (int q = warp; q < 7; q += nw) {
        double t = 0.0;
        for (int b = lane; b < nblk; b += 32 * 8) {
            double pv[8];  // eight loads in flight
#pragma unroll
            for (int j = 0; j < 8; ++j) pv[j] = b + 32 * j < nblk ? __ldcg(partials + (size_t)(b + 32 * j) * NQ + q) : 0.0;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (b + 32 * j < nblk) t = (q == 5) ? fmax(t, pv[j]) : t + pv[j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double w = __shfl_xor_sync(0xffffffffu, t, o);
            t = (q == 5) ? fmax(t, w) : t + w;
        }
        if (lane == 0) stats[q] = (q == 5) ? sqrt(t) : t;
    }
}

// OPEN: the case has open sides; CUBIC: the cubic-term elimination, with
// phi = rho u_x^3, rho u_y^3 of the entering state (separate instantiations,
// so that the common path carries none of their code)
template <class S, class C, bool OPEN, bool CUBIC>
__global__ void __launch_bounds__(32 * MW, MarchCfg<S>::BPS)
    k_march(const S* in, S* out, const __grid_constant__ Launch L, const MarchGrid mg, double* __restrict__ partials,
            const double* prev, double* __restrict__ stats, const double* cnt_in,
            double* __restrict__ cnt_out, unsigned* __restrict__ counter, int* __restrict__ status,
            const double* phi) {
    using Cf = MarchCfg<S>;
    using V = typename std::conditional<Cf::NPL == 2, F2, C>::type;
    __shared__ C red[MW][7];
    __shared__ bool last;
    // 16-bit storage, which is short of issue slots, gains from a strip width
    // that the compiler knows (4096 x 1024 in FP16 82.2 -> 81.1 us when it came in); FP32 loses
    // (103.8 -> 104.2) by the copy that the calls for the edges then take
    typename std::conditional<Cf::NPL == 2, Geometry, const Geometry&>::type G = L.geo;
    if constexpr (Cf::NPL == 2) G.lsw = 6;
    const KC<C>& k = kc<C>(L);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = blockDim.x / 32;
    int block = blockIdx.x;
    if (mg.combine_prev) {
        // the first blocks: the record of the step before this one
        if (block < mg.combine_prev) {
            after_previous_grid();
            combine_record(prev, mg.groups * mg.chunks, stats, warp + block * nw, nw * mg.combine_prev, lane);
            return;
        }
        block -= mg.combine_prev;
    }
    const int group = block % mg.groups, chunk = block / mg.groups;
    Strip<S, C> w;
    w.in = in;
    w.out = out;
    w.phi = phi;
    w.xs = (group * nw + warp) * Cf::SW;
    w.y0 = (int)((long long)G.ny * chunk / mg.chunks);
    w.y1 = (int)((long long)G.ny * (chunk + 1) / mg.chunks);
    Rec<C> acc = {C(0), C(0), C(0), C(0), C(0), C(0), C(0)};
    if (w.xs < G.nx) {
        w.wait_ns = L.tile_wait_ns;
        w.sr = Store<S, C>::SHIFTED && L.rounding;
        w.steps = cnt_in;
        if (!march_rows<S, C, OPEN, CUBIC, OPEN || CUBIC>(k, march_constants<V>(L), G, w, acc) && lane == 0) atomicOr(status, ST_TIMEOUT);
    } else {
        after_previous_grid();
    }
    if (block == 0 && threadIdx.x == 0) *cnt_out = __ldcg(cnt_in) + 1.0;

    // ---- block reduction: compute type within warps, FP64 across warps -----
    const C v = reduce_record(acc, lane);
    if (lane % 4 == 0 && lane < 28) red[warp][lane / 4] = v;
    __syncthreads();
    if (threadIdx.x < 7) {
        const int q = threadIdx.x;
        double t = 0.0;
        for (int j = 0; j < nw; ++j) t = (q == 5) ? fmax(t, (double)red[j][q]) : t + (double)red[j][q];
        const double cc = (double)k.c;
        if (q == 1 || q == 2) t *= cc;
        if (q == 5) t *= cc * cc;
        partials[(size_t)block * NQ + q] = t;
        if (q == 6 && t > 0.0) atomicOr(status, ST_NONFINITE);
    }
    if (!mg.combine_here) return;
    __syncthreads();
    const unsigned nblocks = (unsigned)(mg.groups * mg.chunks);
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(counter, 1u) == nblocks - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    combine_record(partials, (int)nblocks, stats, warp, nw, lane);
    if (threadIdx.x == 0) *counter = 0u;
}

__global__ void k_record_finish(const double* __restrict__ partials, int nblk, double* __restrict__ stats) {
    combine_record(partials, nblk, stats, threadIdx.x / 32, blockDim.x / 32, threadIdx.x % 32);
}

template <class S, class C>
cudaError_t march_t(const Launch& L, const void* in, void* out, const MarchGrid& mg,
                    double* partials, const double* prev, double* stats, const double* cnt_in, double* cnt_out,
                    unsigned* counter, int* status, cudaStream_t s, const double* phi) {
    const dim3 grid((unsigned)(mg.groups * mg.chunks + mg.combine_prev)), blk((unsigned)(32 * mg.warps));
    const S* i = static_cast<const S*>(in);
    S* o = static_cast<S*>(out);
    auto* const kernel = L.geo.open ? k_march<S, C, true, false> : (L.cubic ? k_march<S, C, false, true> : k_march<S, C, false, false>);
    return launch_early(kernel, grid, blk, 0, s, i, o, L, mg, partials, prev, stats, cnt_in, cnt_out, counter, status, phi);
}

}  // namespace

int march_strip(int storage) {
    return storage == S_F64 ? MarchCfg<double>::SW : (storage == S_F32 ? MarchCfg<float>::SW : MarchCfg<__half>::SW);
}

// Blocks of w warps that combine a record, a warp per quantity: with one block, and
// one load at a time, they ran longer than the step of a lattice of up to about
// 300 x 300 (FP32: 300 x 300 9.1 -> 6.5 us per step, 224 x 224 8.4 -> 4.8, 128 x
// 128 4.23 -> 3.92, 40 x 40 7.3 -> 3.6, 96 x 500 17.3 -> 5.4).
static int combine_blocks(int w) { return (7 + w - 1) / w; }

MarchGrid march_grid(int storage, const Geometry& g) {
    const int sw = march_strip(storage);
    const int bps = storage == S_F64 ? MarchCfg<double>::BPS : (storage == S_F32 ? MarchCfg<float>::BPS : MarchCfg<__half>::BPS);
    const int strips = (g.nx + sw - 1) / sw;
    // Blocks of w adjacent strips, and as many chunks of rows as fill one wave of
    // resident blocks, which the blocks that combine the last record are part of.
    // w is the largest for which the longest chunk is shortest: with 4 warps, 22
    // strips leave 2 of 24 idle, and 5 strips a quarter of every SM's, as blocks
    // of 3 count as blocks of 4 (1363 x 777 in BF16 27.4 -> 25.8 us per step, 900 x
    // 2000 43.2 -> 41.1, 160 x 900 in FP32 13.3 -> 7.7, 40 x 3000 in FP16 24.6 ->
    // 11.0).
    MarchGrid m{};
    int chunks = 0, rows = 0;
    for (int w = MW; w >= 2; --w) {
        const int groups = (strips + w - 1) / w, warps = (strips + groups - 1) / groups;
        int n = (bps * MW / w * g.sms - combine_blocks(warps)) / groups;
        n = n > g.ny ? g.ny : (n < 1 ? 1 : n);
        const int longest = (g.ny + n - 1) / n;
        if (rows == 0 || longest < rows) {
            rows = longest;
            chunks = n;
            m.groups = groups;
            m.warps = warps;
        }
    }
    // In FP32, which waits for memory, as few chunks as keep the longest as it
    // is: fewer rows read twice (512 x 512: 10.5 us per step with 151 chunks of 3
    // or 4 rows, 9.6 with 128 of 4). In 16-bit storage and FP64 the warps of the
    // shorter chunks leave the arithmetic to the others (512 x 512 in FP16 10.45
    // and 10.8 us, 1363 x 777 in BF16 27.5 and 28.0).
    if (storage == S_F32) chunks = (g.ny + rows - 1) / rows;
    m.chunks = chunks;
    m.combine_prev = combine_blocks(m.warps);
    return m;
}

cudaError_t launch_march(int storage, const Launch& L, const void* in, void* out,
                         const MarchGrid& mg, double* partials, const double* prev, double* stats, const double* cnt_in,
                         double* cnt_out, unsigned* counter, int* status, cudaStream_t s, const double* phi) {
    if (L.cubic && !phi) return cudaErrorInvalidValue;
    switch (storage) {
        case S_F64: return march_t<double, double>(L, in, out, mg, partials, prev, stats, cnt_in, cnt_out, counter, status, s, phi);
        case S_F32: return march_t<float, float>(L, in, out, mg, partials, prev, stats, cnt_in, cnt_out, counter, status, s, phi);
        case S_F16: return march_t<__half, float>(L, in, out, mg, partials, prev, stats, cnt_in, cnt_out, counter, status, s, phi);
        case S_BF16: return march_t<__nv_bfloat16, float>(L, in, out, mg, partials, prev, stats, cnt_in, cnt_out, counter, status, s, phi);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_record_finish(const double* partials, int nblk, double* stats, cudaStream_t s) {
    k_record_finish<<<1, 224, 0, s>>>(partials, nblk, stats);
    return cudaGetLastError();
}

}  // namespace lbm
