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

// warps of one wave of resident blocks
int batch_warps(int storage, int sms);
cudaError_t launch_batch_step(int storage, const BatchLaunch& B, int from, const void* in, void* out, cudaStream_t s);
cudaError_t launch_batch_case_record(const BatchLaunch& B, int c, double* out, cudaStream_t s);

}  // namespace lbm
