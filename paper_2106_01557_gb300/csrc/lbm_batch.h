// Device-side tables and launchers of the batched step (lbm_batch.cu).
#pragma once

#include <cuda_runtime.h>

#include "lbm_internal.h"

namespace lbm {

// One case of a batch, as the kernels see it (device table).
struct BatchCase {
    Geometry geo;   // lattice and layout
    long long off;  // element offset of the case in each arena buffer
    KC<float> kf;   // its constants
    KC<float2> kp;  // in both lanes, for 16-bit storage
};

struct BatchItem {
    int c;       // case
    int xs;      // first column of the strip
    int y0, y1;  // rows
};

struct BatchLaunch {
    const BatchItem* items;   // warp w takes items first[w] .. first[w + 1] - 1
    const int* first;
    int nitems, warps;
    const BatchCase* cases;
    double* partials;         // [nitems][8]
    int* status;
    double* steps;            // [2] by buffer: steps executed (keys stochastic rounding)
    int rounding;             // 16-bit storage: 0 nearest, 1 stochastic
    unsigned long long tile_wait_ns;  // bound on a warp's wait for its first rows; 0: no waiting
};

// Rows of an item of the second split (lbm_batch_select shape 1), whose items go
// to the warps in turn: at most 32, and at most a warp's equal share of the `rows`
// rows of strips (with 32 always, two boxes of 64 x 64 in FP16 took 38 us per step
// on four warps, and 9 on tiles of 32 x 16 nodes before).
inline int batch_item_rows(long long rows, int warps) {
    const long long r = (rows + warps - 1) / warps;
    return (int)(r < 1 ? 1 : (r < 32 ? r : 32));
}
// warps of one wave of resident blocks
int batch_warps(int storage, int sms);
cudaError_t launch_batch_step(int storage, const BatchLaunch& B, int from, const void* in, void* out, cudaStream_t s);
cudaError_t launch_batch_case_record(const BatchLaunch& B, int c, double* out, cudaStream_t s);

}  // namespace lbm
