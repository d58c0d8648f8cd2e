// Internal declarations shared by the translation units of libqesgd.so.
// Nothing here is part of the public ABI (that is include/qesgd.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "qesgd.h"

// Debug build: an index is checked against its limit; outside it the status word receives
// QESGD_STATUS_RANGE and the caller skips the access.  Release build: always true, no code.
#ifdef QESGD_DEBUG
#define QESGD_IN_RANGE(status, cond) ((cond) ? true : (atomicOr((status), QESGD_STATUS_RANGE), false))
#else
#define QESGD_IN_RANGE(status, cond) true
#endif

struct qesgd_ctx {
    int device;
    cudaStream_t stream;
    uint32_t *d_status;     // device status word (bit set by kernels)
    float *d_lr_work;       // logistic-regression partial margins
    uint64_t lr_work_floats;
    float *d_lr_epoch;      // inter-CTA accumulators of the persistent kernel, behind d_lr_work
    uint64_t launches;
    int last_cuda_error;
    int sm_count;
    uint64_t wait_ns;       // limit of each wait inside the local-epoch kernel
    uint32_t drop_cta;      // give-up-path test hook of the local-epoch kernels (none: ~0)
    uint32_t lr_plan[8];    // qesgd_debug_lr_plan
};
static const uint64_t QESGD_DEFAULT_WAIT_NS = 1000000000ull;
static const uint64_t QESGD_MAX_WAIT_NS = 10000000000ull;

// Workspace (4 MiB): partial margins of the two-pass steps, K * P * m floats, and behind them what the
// persistent kernel's CTAs exchange: a header of 16 words per group of CTAs, then for each of 8 ring
// slots the accumulators (four 64-bit words and three of space per row) of up to
// QESGD_LR_EPOCH_ROWS rows of all groups.  With all 2^20 floats for the partial margins no step is faster
// (64 workers, minibatches of 1024 rows of 4096 columns, 11 parts a worker or 14: 306 and 304 us; 8 workers,
// 98 parts or 126: 90.1 and 90.1).
static const uint32_t QESGD_LR_EPOCH_ROWS = 2048;
static const uint64_t QESGD_LR_EPOCH_FLOATS = QESGD_MAX_WORKERS * 16ull + 8ull * QESGD_LR_EPOCH_ROWS * 14ull;
static const uint64_t QESGD_LR_WORK_FLOATS = (1ull << 20) - QESGD_LR_EPOCH_FLOATS;

// Kernels that go through qesgd_launch may be set up while the kernel before them in the stream drains
// (programmatic dependent launch), and begin with qesgd_wait_for_previous: nothing is read or written
// before that one is done and its writes are visible (qesgd_lr_tile.cu launches its clusters and its grids of one
// minibatch the same way).  The cooperative local-epoch kernels and the debug build's range self-test do not: they are
// launched plainly, start when all before them is done and contain
// no such wait, so they must not be given the attribute without one (in the epoch kernel ahead of the
// producers' first copy and the consumers' loads of u).  No kernel lets its successor
// start earlier than at its own end: a waiting grid would take resident slots.  Without the overlap a
// kernel costs a whole number of about 2.05 us in a stream: encode + decode-average-apply of 4 x 30000
// 11.3 -> 5.9 us, of 8 x 10^6 18.5 -> 14.4, decode of 2^24 13.9 -> 11.3, a logistic step of 64 x 2^22
// 319 -> 311, and no grid was found that is slower.  (With griddepcontrol.launch_dependents at the top of
// every kernel the successor's CTAs come early: 461 instead of 353 us for an encode of 400 000 CTAs.)
template <typename... Params, typename... Args>
inline cudaError_t qesgd_launch(void (*kernel)(Params...), dim3 grid, dim3 block, cudaStream_t stream, const Args &...args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, Params(args)...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void qesgd_wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

struct EncodeArgs {
    const float *local;
    uint64_t local_stride;  // elements between workers
    const float *anchor;    // may be null
    uint64_t d;             // elements per worker
    uint64_t padded;        // nb * bucket
    uint32_t log2_bucket;
    uint32_t s;
    float fixed_scale;      // fl32(s * delta), FIXED mode only
    uint32_t round_key[10][2];  // Philox round keys: seed + r * Weyl constants
    uint32_t worker0, epoch;
    uint32_t K;             // workers in this launch
    uint32_t *codes;
    uint64_t code_stride;   // bytes between workers
    float *scales;
    uint64_t scale_stride;  // elements between workers
    uint32_t *status;
    float *u_out;           // per-step QESGD: receives anchor + Q(z) (same layout as local); else null
    float *zsum;            // per-step QESGD: running sum of Q(z), may be null
};

// One inner step of QESGD on logistic regression in two launches: the margin pass of the
// plain step, then one kernel that forms the updated parameter of a tile in shared memory
// and requantises it there.
struct QstepArgs {
    EncodeArgs e;           // the requantisation of u (K = 1, u_out = local = u)
    const float *X, *y;     // the minibatch, m rows of d columns
    uint32_t m;
    float rate;             // lr / m
    const float *margins;   // the m margins, as the margin pass left them
    uint32_t reverse;       // tiles from the last to the first (see qesgd_second_pass_reversed)
    uint32_t wide;          // X and its rows, u, anchor and running sum 32-byte aligned
};

struct DecodeArgs {
    float *param;           // decode-average-apply: in/out; decode: out
    uint64_t d;
    uint64_t nb;
    uint32_t K;
    float avg_scale;        // alpha / K applied to the sum over workers (1/K for the plain average)
    uint32_t log2_bucket;
    uint32_t s;
    const uint32_t *codes;
    uint64_t code_stride;   // bytes
    const float *scales;
    uint64_t scale_stride;  // elements
    uint32_t *status;
};
int qesgd_launch_range_selftest(uint32_t *status, cudaStream_t stream);

// Launchers.  Return a cudaError_t as int.  qesgd_codec.cu is compiled once per code width
// and defines the *_2, *_4, *_8 functions; the width-dispatching wrappers are inline here.
#define QESGD_DECLARE_WIDTH(B)                                                                  \
    int qesgd_launch_encode_##B(const EncodeArgs &a, uint32_t K, uint32_t scale_mode, bool vec, \
                                int sm_count, cudaStream_t stream);                             \
    int qesgd_launch_decode_##B(const DecodeArgs &a, bool vec, cudaStream_t stream);            \
    int qesgd_launch_decode_average_apply_##B(const DecodeArgs &a, bool vec, cudaStream_t stream);
int qesgd_launch_lr_qstep_2(const QstepArgs &a, uint32_t scale_mode, cudaStream_t stream);
int qesgd_launch_lr_qstep_4(const QstepArgs &a, uint32_t scale_mode, cudaStream_t stream);
int qesgd_launch_lr_qstep_8(const QstepArgs &a, uint32_t scale_mode, cudaStream_t stream);
QESGD_DECLARE_WIDTH(2)
QESGD_DECLARE_WIDTH(4)
QESGD_DECLARE_WIDTH(8)
#undef QESGD_DECLARE_WIDTH

inline int qesgd_launch_encode(const EncodeArgs &a, uint32_t K, uint32_t bits, uint32_t scale_mode,
                               bool vec, int sm_count, cudaStream_t stream)
{
    switch (bits) {
        case 2: return qesgd_launch_encode_2(a, K, scale_mode, vec, sm_count, stream);
        case 4: return qesgd_launch_encode_4(a, K, scale_mode, vec, sm_count, stream);
        default: return qesgd_launch_encode_8(a, K, scale_mode, vec, sm_count, stream);
    }
}
inline int qesgd_launch_decode(const DecodeArgs &a, uint32_t bits, bool vec, cudaStream_t stream)
{
    switch (bits) {
        case 2: return qesgd_launch_decode_2(a, vec, stream);
        case 4: return qesgd_launch_decode_4(a, vec, stream);
        default: return qesgd_launch_decode_8(a, vec, stream);
    }
}
inline int qesgd_launch_decode_average_apply(const DecodeArgs &a, uint32_t bits, bool vec,
                                             cudaStream_t stream)
{
    switch (bits) {
        case 2: return qesgd_launch_decode_average_apply_2(a, vec, stream);
        case 4: return qesgd_launch_decode_average_apply_4(a, vec, stream);
        default: return qesgd_launch_decode_average_apply_8(a, vec, stream);
    }
}
// One minibatch step for K workers; returns the number of kernels launched in *launched.
int qesgd_launch_lr_step(const float *Xb, uint64_t x_worker_stride, const float *yb,
                         uint64_t y_worker_stride, uint32_t m, uint64_t d, uint32_t K, float lr,
                         float *u, uint64_t u_stride, float *work, uint64_t work_floats,
                         cudaStream_t stream, int *launched);
// A minibatch that does not fit L2 is read a second time from its end: what the margin pass, which walks
// the workers and their columns upwards, read last is still there.  Measured (second pass included): 64 x 2^22
// sgd_step 324 -> 318 us, qstep 343 -> 337; 64 x 2^19 54 -> 50; where the minibatch fits, the plain order is the
// better one (16 x 2^20, 67 MB: 31.8 against 33.8).  Several workers, m the rows of all of them, against the
// columns alone turned round: K = 4, n = 256, d = 160000, minibatches of 64 258 -> 233 us, K = 8, n = 64,
// d = 400000, of 16 374 -> 347, K = 16, n = 600, d = 20000, of 300 302 -> 298; K = 32, n = 512, of 512 404 -> 409.
inline bool qesgd_second_pass_reversed(uint64_t m, uint64_t d) { return m * d * 4u > (96ull << 20); }
// The margin pass alone (pass 1 of a step) for one worker; *parts_out receives the number of
// partial margins per row that the pass leaves in `work` ([parts][m]).
int qesgd_launch_lr_margins(const float *Xb, const float *yb, uint32_t m, uint64_t d, const float *u,
                            float *work, uint64_t work_floats, cudaStream_t stream, const float **margins_out);
// Minibatch mean gradient at w into g (same two passes; the second writes instead of updating).
int qesgd_launch_lr_gradient(const float *Xb, const float *yb, uint32_t m, uint64_t d,
                             const float *w, float *g, float *work, uint64_t work_floats,
                             cudaStream_t stream, int *launched);
// A whole local epoch of K workers (or, with K = 1, n_local = batch and lr = -1, the mean gradient of
// one minibatch at u) as one persistent kernel that reads X once.  Returns 0 = launched (one kernel),
// -1 = shape not covered (the caller falls back to the two-pass steps), > 0 = cudaError_t.  `work`
// (QESGD_LR_EPOCH_FLOATS floats) holds the inter-CTA accumulators: zero before the first launch, and
// every launch leaves it at zero.
int qesgd_launch_lr_epoch_fused(const float *X, const float *y, uint64_t n_local, uint64_t d,
                                uint32_t K, uint32_t batch, float lr, const float *u, float *dst,
                                bool gradient, uint64_t u_stride, float *work, uint32_t *status, int device,
                                int sm_count, uint64_t wait_ns, uint32_t drop_cta, cudaStream_t stream,
                                int *launched, uint32_t (&plan)[8]);
