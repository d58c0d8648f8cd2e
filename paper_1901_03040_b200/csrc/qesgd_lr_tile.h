// The epoch or gradient that qesgd_lr_epoch.cu hands to qesgd_lr_tile.cu where it is the faster kernel.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct QesgdTileCall {
    const float *X, *y;
    uint64_t n_local, d, nsteps;
    uint32_t K, m;               // workers; rows of a full minibatch
    float lr;
    const float *u;
    float *dst;
    bool gradient;
    uint64_t u_stride;
    int copy;                    // bytes per copy that X's rows allow: 16 (TMA, and u by vectors), 8, 4
    uint32_t *header;            // the workspace of qesgd_lr_epoch.cu
    unsigned long long *acc, *wide;
    uint32_t *status;
    int device;
    uint32_t sms;                // SMs that the call may take
    uint64_t wait_ns;
    uint32_t drop_cta;
    cudaStream_t stream;
};
// 0 = launched (`plan`: see qesgd_debug_lr_plan), -1 = not covered, or the other kernel is modelled to be faster
// (`other_us` a step), > 0 = cudaError_t.
int qesgd_launch_lr_tile(const QesgdTileCall &q, uint32_t smem_limit, float other_us, int *launched,
                         uint32_t (&plan)[8]);
