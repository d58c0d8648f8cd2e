// What the logistic-regression kernels that keep a minibatch on chip share: barriers, copies, the sum over a
// warp, and the exchange of margins between CTAs through global memory.
#pragma once

#include <cuda.h>

#include "qesgd_internal.h"

// Row-major float matrix [rows][d] as a tensor map, of floats or of pairs of them, with boxes of SUB rows of box_cols
// columns (qesgd_lr_epoch.cu).
bool qesgd_lr_tensor_map(CUtensorMap *map, const float *X, uint64_t rows, uint64_t d, uint32_t box_cols, bool pairs);

namespace {

constexpr int SUB = 8;               // rows per sub-tile
constexpr int EP_RING = 8;           // accumulator slots; a slot is cleared RING/2 tiles before its use
constexpr uint64_t DRAIN_LIMIT_NS = 2000000000ull;   // the producers' last wait for their own copies
constexpr uint64_t COARSE_TIMER_NS = 1024ull;        // limits below this mean "one look, then give up"
constexpr uint32_t EP_HEADER_WORDS = 16;             // per group: [0] abort flag, [1] CTAs that have read their last margins
constexpr uint32_t EP_ACC_PITCH = 32;                // 64-bit words from one 8-row group of accumulators to the next
constexpr uint32_t EP_WIDE_WORDS = 3;                // rarely used 64-bit words per accumulator row
constexpr float FX_SCALE = 268435456.0f;             // 2^28: unit of the first word
constexpr float FX_LIMIT = 131072.0f;                // 2^17: partials below go to the first word
constexpr float FX_WIDE_SCALE = 64.0f;               // 2^6: unit of the second word
constexpr float FX_WIDE_LIMIT = 562949953421312.0f;  // 2^49: partials below go to the second word
constexpr unsigned long long FX_BIAS = 1ull << 45;   // makes every contribution to the first word positive
constexpr unsigned long long FX_ONE = 1ull << 55;    // one contribution counted
constexpr unsigned long long FX_SPECIAL = 1ull << 54;   // one of the row's other words is in use


// ------------------------------------------------------------- primitives ----
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t now_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0u;
}
// Has a wait that began at t0 used up `limit`?  The global timer may tick as coarsely as a
// microsecond, so a smaller limit is read as "give up after one round of looks".
__device__ __forceinline__ bool expired(uint64_t t0, uint64_t limit)
{
    return limit < COARSE_TIMER_NS || now_ns() - t0 > limit;
}
// Bounded wait for phase `parity` of a barrier; gives up early when `*stop` is set.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, const volatile uint32_t *stop,
                                          uint64_t limit)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = now_ns();
    for (;;) {
        for (int n = 0; n < 32; ++n)
            if (mbar_try_wait(bar, parity)) return true;
        if (*stop != 0u || expired(t0, limit)) return false;
    }
}
// Bounded wait until the counter *flag, which another warp of this CTA advances, exceeds `value`.
__device__ __forceinline__ bool flag_above(const volatile uint32_t *flag, uint32_t value,
                                           const volatile uint32_t *stop, uint64_t limit)
{
    if (*flag > value) return true;
    const uint64_t t0 = now_ns();
    for (;;) {
        for (int n = 0; n < 32; ++n)
            if (*flag > value) return true;
        if (*stop != 0u || expired(t0, limit)) return false;
    }
}
// One 2-D box of a tensor map: elements from x on, rows [y, y + SUB).  x is a multiple of 16 bytes; dst is 128-byte
// aligned.  The copy goes to this CTA alone.
__device__ __forceinline__ void tma_load_box(float *dst, const CUtensorMap *map, uint32_t x, uint32_t y,
                                             uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Barrier `id` of `count` threads that also answers one question the same way for all of them:
// has any of them seen `flag` set?  (Each thread reads the flag for itself; a plain barrier
// followed by separate reads could send the threads different ways while another warp sets it,
// and the ones that stay would then wait at the next barrier for the ones that left.)
__device__ __forceinline__ bool sync_any(uint32_t id, uint32_t count, uint32_t flag)
{
    uint32_t r;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 q, %1, 0;\n"
        "bar.red.or.pred p, %2, %3, q;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}"
        : "=r"(r)
        : "r"(flag), "r"(id), "r"(count)
        : "memory");
    return r != 0u;
}

// EB bytes from global to shared memory, asynchronously; zeros where `inside` does not hold (then
// nothing is read).
template <int EB>
__device__ __forceinline__ void copy_elements(uint32_t dst, const float *src, bool inside)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(EB == 8 ? 8 : 4),
                 "r"(inside ? (EB == 8 ? 8 : 4) : 0)
                 : "memory");
}
// One arrival on the barrier when all copies of this thread so far have landed.
__device__ __forceinline__ void arrive_when_copied(uint64_t *bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Sum over the 32 lanes of 8 per-lane values at once: three halving exchanges leave one
// value per lane, two plain butterflies finish.  Lane L ends with the total of value
// 4*bit4(L) + 2*bit3(L) + bit2(L); the order of the additions is fixed.
__device__ __forceinline__ float reduce8(float (&v)[8], uint32_t lane)
{
    const bool h4 = lane & 16u, h3 = lane & 8u, h2 = lane & 4u;
    float a[4], b[2];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float keep = h4 ? v[r + 4] : v[r], send = h4 ? v[r] : v[r + 4];
        a[r] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 16);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float keep = h3 ? a[r + 2] : a[r], send = h3 ? a[r] : a[r + 2];
        b[r] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 8);
    }
    const float keep = h2 ? b[1] : b[0], send = h2 ? b[0] : b[1];
    float c = keep + __shfl_xor_sync(0xFFFFFFFFu, send, 4);
    c += __shfl_xor_sync(0xFFFFFFFFu, c, 2);
    c += __shfl_xor_sync(0xFFFFFFFFu, c, 1);
    return c;
}
__device__ __forceinline__ uint32_t reduce8_row(uint32_t lane)
{
    return ((lane >> 4) & 1u) * 4u + ((lane >> 3) & 1u) * 2u + ((lane >> 2) & 1u);
}

// Where row j's accumulator lies within its ring slot: eight rows in a row, the eights 256 bytes apart.
__device__ __forceinline__ uint32_t acc_index(uint32_t j) { return (j / SUB) * EP_ACC_PITCH + j % SUB; }

// A row's partial margin onto its accumulator; `wide` are the row's rarely used words.
__device__ __forceinline__ void exchange_add(unsigned long long *r, unsigned long long *wide, float tot)
{
    if (fabsf(tot) < FX_LIMIT) {
        atomicAdd(r, FX_ONE + FX_BIAS + (unsigned long long)__float2ll_rn(tot * FX_SCALE));
    } else {
        // rare: the special bit and the row's other words first, visible before the count
        atomicOr(r, FX_SPECIAL);
        if (fabsf(tot) < FX_WIDE_LIMIT)
            atomicAdd(wide, (unsigned long long)__float2ll_rn(tot * FX_WIDE_SCALE));
        else if (tot != tot)
            atomicAdd(wide + 1, 1ull);                               // NaN
        else
            atomicAdd(wide + 2, tot > 0.0f ? (1ull << 32) : 1ull);   // +-Inf, or beyond the wide word
        __threadfence();
        atomicAdd(r, FX_ONE + FX_BIAS);
    }
}
// The margin that a complete accumulator word of P contributions stands for.
__device__ __forceinline__ float exchange_margin(unsigned long long v, const unsigned long long *wide, uint32_t P)
{
    const long long fine = (long long)((v & (FX_SPECIAL - 1ull)) - (unsigned long long)P * FX_BIAS);
    float margin = (float)((double)fine * (1.0 / (double)FX_SCALE));
    if ((v & FX_SPECIAL) != 0ull) {
        __threadfence();
        const unsigned long long w0 = ld_relaxed(wide), w1 = ld_relaxed(wide + 1), w2 = ld_relaxed(wide + 2);
        margin = (float)((double)fine * (1.0 / (double)FX_SCALE) + (double)(long long)w0 * (1.0 / (double)FX_WIDE_SCALE));
        if (w2 != 0ull) {   // +Inf count << 32 + -Inf count
            const bool pos = (w2 >> 32) != 0ull, neg = (w2 & 0xFFFFFFFFull) != 0ull;
            margin = pos && neg ? __int_as_float(0x7FC00000) : __int_as_float(pos ? 0x7F800000 : (int)0xFF800000);
        }
        if (w1 != 0ull) margin = __int_as_float(0x7FC00000);
    }
    return margin;
}

}  // namespace
