// Local epoch of logistic-regression minibatch SGD as ONE persistent kernel for sm_100a
// (paper Sec. 1: f_i(w) = log(1 + exp(-y_i x_i^T w)); Eq. 2: u <- u - (lr/m) sum_j grad f_j(u);
// worker task of Algorithm 3: consecutive minibatches of the worker's shard).
//
// A step needs the minibatch twice -- once for the margins x_j . u, once for the update
// sum_j c_j x_j -- with a reduction over all columns in between.  The K workers are dealt out to
// G groups of P CTAs; a group runs the epochs of its workers, and each of its CTAs owns a slice
// of `cols` columns for the whole epoch.  The slice of a minibatch (a "tile") passes through the
// SM once, so X is read from HBM exactly once:
//
//   producer warps  fetch sub-tiles (8 rows of the slice) by TMA (2-D boxes of at most 256
//                   columns, cp.async.bulk.tensor global -> shared, completion on an mbarrier
//                   per slot) into a ring of slots, as far ahead as the ring reaches.  Several
//                   warps, one thread of each, take the slots in turn: looking at the slot, arming
//                   its barrier and issuing two to four boxes takes a thread about 650 clocks, which
//                   with one producer bounded the whole kernel at 27 bytes per clock and SM.  Two are best:
//                   K = 4, n = 2048, d = 65536: 441 us with one, 329, 337 and 341 with two, three and
//                   four; K = 8, n = 1010, d = 10000: 127, 81, 87, 88; K = 8, n = 512, d = 65536: 224, 167,
//                   177, 175 (more requests at once delay the exchange between the CTAs); only the widest
//                   slices do better with one (K = 4, n = 512, d = 131072: 236, 240, 237, 247).
//                   For the same reason a producer leaves a pause between two copies: the CTAs free
//                   their slots in step, right after the exchange, and refilled at once by all of them
//                   the copies of one SM queue behind another's, the slowest of which everybody then
//                   waits for.  At 0.6 of the interval at which HBM can serve every SM the first
//                   shape takes 329 us, the HBM time of X (343 without a pause; 327 at 0.5, 362 at 0.7,
//                   394 at 0.8); K = 8, n = 512, d = 65536: 179 -> 168.  The pause is kept by the global
//                   timer (32 ns a tick), not in clocks: under the power cap the SM clock falls by a
//                   quarter, and a pause that grew with it would hold HBM back (whole rounds of the first
//                   shape, repeated for a second, were 1 % slower than without a pause by clocks, 1 %
//                   faster by the timer)
//   consumer chain  eight warps; tile i = minibatch i / Kg of the group's worker i % Kg:
//     M(i)  warp w takes the sub-tiles w, w + 8, ...: partial margins of the rows over the slice;
//           the values it reads go to tensor memory on the way (tcgen05.st), so the slot returns
//           to the producer at once; the partial margins go out to the group's other CTAs
//     W(i)  wait for the partial margins of all P CTAs; coefficients (lr/m) y_j / (1 + exp(y_j m_j))
//     U(i)  every warp reads back what it stored (tcgen05.ld), forms coef_j x_j summed over its
//           rows, the eight warps' sums meet in shared memory and are added to the slice of u,
//           which stays in shared memory from the first minibatch to the last
//
// What bounds it.  X is read once, so HBM bounds large minibatches; below, every step is a chain
// M - exchange - U - M of dependent latencies (2 to 3 us through global memory).  Workers are
// independent, so groups run side by side (G > 1 divides the number of chained tiles by G), and
// where one group holds several workers two chains (NC = 2) alternate over its tiles, one
// computing while the other waits.  The tensor memory (256 KB) holds what waits for its
// coefficients: 64 rows x 512 columns for each of two chains or x 1024 columns for one.
// Epochs of few columns per CTA, where that chain is all the time there is, go to qesgd_lr_tile.cu.
// Measured against the kernel this one replaces (one group, u in global memory, tiles kept in two
// shared-memory buffers, at most 512 columns per SM): K = 8, n = 1010, d = 10000, batch 50:
// 434 -> 81 us; K = 4, n = 128, d = 4096, batch 32: 37.6 -> 14.4; K = 4, n = 512, d = 131072 (two
// passes before): 426 -> 240; K = 4, n = 2048, d = 65536: 460 -> 329; K = 64, n = 64, d = 65536: 255 -> 253.
//
// Exchange through global memory: each row's partial margin is added, as a fixed-point integer,
// to the row's accumulator acc[i % RING][row] by one 64-bit reduction that also counts the
// contribution in the word's top bits.  Integer addition is exact and commutes, so the sum over
// the CTAs needs no order, no second pass over the partials and -- the count travelling in the
// same word as the sum -- no fence between data and signal; the result is the same in every run.
// A word is count << 55 | special << 54 | sum, every contribution adds 1 << 55 plus 2^45 +
// round(partial * 2^28) (the 2^45 keeps it positive; |partial| < 2^17; up to 256 CTAs fit below
// bit 54).  A larger finite partial goes, in units of 2^-6 (the spacing of fp32 at 2^17), into a
// second word of the row; a NaN is counted in the third word and makes the margin NaN; an infinite
// partial, or one of 2^49 or more, is counted by sign in the fourth and makes the margin that
// infinity (NaN if both signs occur), which the step coefficient saturates on as it would on the
// number itself.  These rare kinds set the special bit, and fence before they count themselves in
// the first word, so a reader looks at the other words only where the bit is set: one round trip
// to L2 in place of two.  Every thread that owns a row polls that row's word itself; the eight
// rows of a sub-tile lie in 64 bytes, so a warp's reduction touches two sectors, and the sub-tiles
// 256 bytes apart: they then fall into different parts of L2, whose atomic units and read ports
// 148 CTAs otherwise queue at (an exchange of 64 rows, nothing else running: all rows in 512 bytes
// 3590 clocks at 148 CTAs and 2250 at 74; 256 bytes apart 2375 and 1570; every row 256 bytes from
// the next 2470 and 1970; one reader per row that hands the margin on 3640 and 3020).
// The slot that tile i + RING/2 will use is cleared by one CTA after M(i), while it waits: every
// CTA has read it by then (it has taken part in tile i-2, hence finished tile i-4) and none adds
// to it before it has seen that CTA's contributions to tile i+2.  The CTA of a group that reads its
// last margins last clears what is left, so every launch finds the accumulators at zero.
//
// The CTAs wait on one another, so the kernel is launched cooperatively (all CTAs are
// resident by construction: at most one per SM).  Every wait the kernel itself loops on is
// bounded by the context's wait limit: a wait that runs out sets QESGD_STATUS_TIMEOUT and an
// abort word that the group's other CTAs poll, and the CTA's consumer warps leave.  The producer
// warps are the last to go on every path: they wait (on a bound of its own) for each copy they have
// requested and nobody has consumed, so no CTA ends with a copy still writing its shared
// memory.  The one wait without a bound is the tensor-memory allocation at the start, which
// blocks while another kernel resident on the same SM holds tensor memory (until that kernel
// ends).
#include <mutex>

#include "qesgd_lr_device.cuh"
#include "qesgd_lr_tile.h"

namespace {

constexpr int EP_WARPS = 8;                       // consumer warps of a chain
constexpr int EP_CHAIN = EP_WARPS * 32;
constexpr int EP_BOX_COLS = 256;     // widest TMA box; element-wise copies keep whole rows together
constexpr int EP_MAX_M = EP_CHAIN;   // rows per minibatch: a thread of the chain per row
constexpr int EP_MAX_SLOTS = 64;     // ring slots
constexpr uint32_t EP_FLAG_BYTES = (16 + EP_MAX_SLOTS) * 4;
constexpr float EP_HBM_BYTES_PER_NS = 6500.0f;   // what HBM delivers to all SMs together
constexpr int EP_PRODUCERS = 2;      // producer warps with TMA
constexpr int EP_LOADERS = 8;        // producer warps with element-wise copies
constexpr int EP_UNITS = 8;          // 8 x 128 blocks of a tile that the tensor memory holds per warp
constexpr float EP_CHAIN_US = 2.5f, EP_UNIT_US = 0.25f;   // a tile's latency: exchange, and per block of a warp
struct EpochArgs {
    const float *X;         // element-wise copies only
    const float *y;
    uint64_t n_local;       // rows per worker
    uint64_t d;
    uint32_t K, G, P;       // workers, groups, CTAs per group
    uint32_t batch, nsteps;
    uint32_t m_last;        // rows of the last minibatch
    uint32_t nsub_max, nsub_last;
    uint32_t cols, nit;     // columns per CTA (a multiple of 4), blocks of 128 columns
    uint32_t nslots;        // sub-tiles the ring holds
    uint32_t pace;          // ns between two copies of a producer, at least
    uint32_t off_u, off_part, off_coef, off_bars, off_flags;   // shared-memory layout, bytes
    float rate, rate_last;  // lr / rows of a minibatch, of the last one (lr = -1 for the mean gradient)
    const float *u;         // where the epoch starts
    float *dst;             // where its result goes: u, or the place for a mean gradient
    uint32_t gradient;      // != 0: one minibatch, dst = sum_j coef_j x_j instead of u + that
    uint64_t u_stride;
    uint32_t *header;       // [G][EP_HEADER_WORDS]
    unsigned long long *acc;    // [G][EP_RING][nsub_max][EP_ACC_PITCH] margin accumulators, zero between launches
    unsigned long long *wide;   // [G][EP_RING][8 * nsub_max][EP_WIDE_WORDS]
    uint32_t *status;
    uint64_t wait_ns;       // limit of every wait on another CTA, chain or copy
    uint32_t poll_mask;     // the clock is read every (poll_mask + 1) looks at a counter
    uint32_t drop_cta;      // test hook: this CTA does not count itself for tile 0 (none: ~0)
};

// ---- tensor memory as a stash for a tile between its two uses --------------------------
// The SM's 256 KB of tensor memory (128 lanes x 512 columns of 32 bits) is not needed for
// any matrix product here, so it holds a chain's tile while the chain waits for the
// other CTAs: thread t of a warp owns lane 32 * (warp % 4) + t and reads back exactly what it
// stored, so no ordering between threads is involved.  One access moves 32 registers of
// every thread of the warp (the 8 rows x 4 columns a thread takes of an 8 x 128 block).
__device__ __forceinline__ void tmem_alloc_all(uint32_t *smem_result)   // one whole warp
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(smem_result))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free_all(uint32_t taddr)           // the same warp
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float4 (&v)[8])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "f"(v[0].x), "f"(v[0].y), "f"(v[0].z), "f"(v[0].w), "f"(v[1].x), "f"(v[1].y), "f"(v[1].z), "f"(v[1].w),
        "f"(v[2].x), "f"(v[2].y), "f"(v[2].z), "f"(v[2].w), "f"(v[3].x), "f"(v[3].y), "f"(v[3].z), "f"(v[3].w),
        "f"(v[4].x), "f"(v[4].y), "f"(v[4].z), "f"(v[4].w), "f"(v[5].x), "f"(v[5].y), "f"(v[5].z), "f"(v[5].w),
        "f"(v[6].x), "f"(v[6].y), "f"(v[6].z), "f"(v[6].w), "f"(v[7].x), "f"(v[7].y), "f"(v[7].z), "f"(v[7].w)
        : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float4 (&v)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[0].z), "=f"(v[0].w), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[1].z),
          "=f"(v[1].w), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[2].z), "=f"(v[2].w), "=f"(v[3].x), "=f"(v[3].y),
          "=f"(v[3].z), "=f"(v[3].w), "=f"(v[4].x), "=f"(v[4].y), "=f"(v[4].z), "=f"(v[4].w), "=f"(v[5].x),
          "=f"(v[5].y), "=f"(v[5].z), "=f"(v[5].w), "=f"(v[6].x), "=f"(v[6].y), "=f"(v[6].z), "=f"(v[6].w),
          "=f"(v[7].x), "=f"(v[7].y), "=f"(v[7].z), "=f"(v[7].w)
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// A tile of a group: minibatch t of the group's worker kk; `first` is the number of its first
// sub-tile.  Stepped, not divided out: an integer division takes 240 clocks, a small step 3500.
struct Tile {
    uint32_t t, kk, m, nsub, first;
    __device__ __forceinline__ void start(const EpochArgs &a)
    {
        t = kk = first = 0u;
        size(a);
    }
    __device__ __forceinline__ void size(const EpochArgs &a)
    {
        m = t == a.nsteps - 1u ? a.m_last : a.batch;
        nsub = t == a.nsteps - 1u ? a.nsub_last : a.nsub_max;
    }
    __device__ __forceinline__ void next(const EpochArgs &a, uint32_t kg)
    {
        first += nsub;
        if (++kk == kg) {
            kk = 0u;
            ++t;
            size(a);
        }
    }
};

// The warps' sums of a tile (minibatch t of `worker`) onto the worker's slice of u, which goes out with the
// last minibatch.
template <int EB>
__device__ __forceinline__ void add_to_u(const EpochArgs &a, float *us, const float *part, uint32_t ucols, uint32_t tg,
                                         uint32_t c0, uint32_t worker, uint32_t nsub, uint32_t t_step)
{
    if (tg < ucols / 4u) {
        const uint32_t c = tg * 4u;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f), t = o;
        if (!a.gradient) o = *reinterpret_cast<const float4 *>(us + c);
#pragma unroll
        for (uint32_t w = 0; w < (uint32_t)EP_WARPS; ++w) {
            if (w < nsub) {
                const float4 v = *reinterpret_cast<const float4 *>(part + (size_t)w * ucols + c);
                t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
            }
        }
        t.x += o.x; t.y += o.y; t.z += o.z; t.w += o.w;
        *reinterpret_cast<float4 *>(us + c) = t;
        if (t_step == a.nsteps - 1u && c < a.cols && (uint64_t)c0 + c < a.d) {   // the worker's last minibatch
            float *const to = a.dst + (uint64_t)worker * a.u_stride + c0 + c;
            if (EB == 16) {
                *reinterpret_cast<float4 *>(to) = t;
            } else {
                const uint64_t have = a.d - c0 - c;
                to[0] = t.x;
                if (have > 1u) to[1] = t.y;
                if (have > 2u) to[2] = t.z;
                if (have > 3u) to[3] = t.w;
            }
        }
    }
}

extern __shared__ __align__(1024) unsigned char ep_smem[];

// Shared memory: the ring of slots of SUB x cols floats (a slot holds its boxes of 256 columns one
// after the other, the last one narrower), the slices of u of the group's workers, the warps'
// partial updates, the step coefficients, the barriers, a few flag words.
// EB = 16: rows of X start on 16-byte boundaries and TMA fetches them.  EB = 4 or 8: they do not (d no
// multiple of 4, or unaligned vectors); eight producer warps copy 4 or 8 bytes at a time instead
// (cp.async, completion on the same barriers, elements outside the matrix as zeros) and u is read and
// written element by element.  One chain.  Bound by the copies' instructions (128 or 256 bytes each),
// but against two passes of scalar loads per minibatch: K = 4, n = 512, d = 16383: 193 -> 45 us; K = 8,
// n = 1010, d = 10001: 465 -> 132; one minibatch of 64 x 65537: 19.6 -> 10.3; K = 4, n = 2048, d = 65538:
// 1173 -> 670.
template <int NC, int EB>
__global__ void __launch_bounds__(NC * EP_CHAIN + (EB == 16 ? EP_PRODUCERS : EP_LOADERS) * 32, 1)
    qesgd_lr_epoch_kernel(const EpochArgs a, const __grid_constant__ CUtensorMap map_full,
                          const __grid_constant__ CUtensorMap map_rest)
{
    constexpr uint32_t BOX = EB == 16 ? EP_BOX_COLS : 1024u, BOX_UNITS = BOX / 128u;   // columns that lie together in a slot
    constexpr uint32_t PRODUCERS = EB == 16 ? EP_PRODUCERS : EP_LOADERS;
    const uint32_t slot_floats = SUB * a.cols, ucols = a.nit * 128u;
    float *const ring = reinterpret_cast<float *>(ep_smem);
    float *const s_u = reinterpret_cast<float *>(ep_smem + a.off_u);
    float *const s_part = reinterpret_cast<float *>(ep_smem + a.off_part);
    float *const s_coef = reinterpret_cast<float *>(ep_smem + a.off_coef);
    uint64_t *const full = reinterpret_cast<uint64_t *>(ep_smem + a.off_bars);
    uint64_t *const empty = full + a.nslots;
    // [0] a wait ran out in this CTA, [3] always zero, [4], [5] tiles completed by chain 0, 1,
    // [8] base address of the tensor memory
    volatile uint32_t *const s_flag = reinterpret_cast<volatile uint32_t *>(ep_smem + a.off_flags);
    volatile uint32_t *const s_turn = s_flag + 16;         // copies requested into each slot so far

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t grp = blockIdx.x / a.P, rank = blockIdx.x - grp * a.P;
    const uint32_t kg = (a.K - grp + a.G - 1u) / a.G;      // workers of this group
    const uint32_t c0 = rank * a.cols;
    const uint32_t ntiles = a.nsteps * kg;

    if (tid < 2u * a.nslots) {
        mbar_init(&full[tid], EB == 16 || tid >= a.nslots ? 1u : 32u);   // element-wise: every lane of the loader
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 16u + EP_MAX_SLOTS) s_flag[tid] = 0u;
    __syncthreads();

    // ----------------------------------------------------------- producers ----
    if (warp >= NC * EP_WARPS) {
        // The sub-tiles go round the ring in the order in which the chains take them.  Warp p serves
        // the slots p, p + EP_PRODUCERS, ... and each of them turn by turn: a slot that several warps
        // refilled could be looked at two turns early, where a barrier's parity reads the same.
        const uint32_t p = warp - NC * EP_WARPS;
        if ((EB != 16 || lane == 0) && p < a.nslots) {
            uint32_t i = 0u, s = p, slot = p, turn = 0u;
            Tile T;
            T.start(a);
            uint32_t issued = (uint32_t)now_ns() - a.pace;
            for (;;) {
                while (s >= T.nsub && i < ntiles) {
                    s -= T.nsub;
                    T.next(a, kg);
                    ++i;
                }
                if (i >= ntiles) break;
                while (EB == 16 && (uint32_t)now_ns() - issued < a.pace) __nanosleep(20);
                // the slot's previous sub-tile has been taken
                bool ok = turn == 0u || mbar_wait(&empty[slot], (turn - 1u) & 1u, &s_flag[0], a.wait_ns);
                if (EB != 16) ok = __all_sync(0xFFFFFFFFu, ok) != 0;
                if (!ok) {
                    s_flag[0] = 1u;
                    atomicOr(a.status, QESGD_STATUS_TIMEOUT);
                    break;
                }
                const uint32_t row = (uint32_t)((uint64_t)(grp + T.kk * a.G) * a.n_local + (uint64_t)T.t * a.batch) + s * SUB;
                float *dst = ring + (size_t)slot * slot_floats;
                if (EB == 16) {
                    issued = (uint32_t)now_ns();
                    mbar_arrive_expect_tx(&full[slot], slot_floats * 4u);
                    uint32_t c = 0u;
                    for (; c + EP_BOX_COLS <= a.cols; c += EP_BOX_COLS, dst += SUB * EP_BOX_COLS)
                        tma_load_box(dst, &map_full, c0 + c, row, &full[slot]);
                    if (c < a.cols) tma_load_box(dst, &map_rest, c0 + c, row, &full[slot]);
                } else {
                    constexpr uint32_t N = EB / 4;
                    const uint32_t rows = min(T.m - s * SUB, (uint32_t)SUB);
                    const float *const src = a.X + (uint64_t)row * a.d + c0;
                    for (uint32_t r = 0; r < rows; ++r) {
                        const float *const line = src + (uint64_t)r * a.d;
                        const uint32_t to = smem_u32(dst + r * a.cols);
#pragma unroll 4
                        for (uint32_t c = lane * N; c < a.cols; c += 32u * N)
                            copy_elements<EB>(to + c * 4u, line + c, (uint64_t)c0 + c < a.d);
                    }
                    arrive_when_copied(&full[slot]);
                }
                if (lane == 0) s_turn[slot] = turn + 1u;
                if (slot + PRODUCERS < a.nslots) {
                    slot += PRODUCERS;
                    s += PRODUCERS;
                } else {
                    s += a.nslots - slot + p;
                    slot = p;
                    ++turn;
                }
            }
        }
        __syncwarp();
        // Last out, on every path: each slot's latest copy has been consumed (then it has
        // landed) or is waited for here, so that the CTA does not end -- and its shared memory
        // is not handed to another CTA -- while a copy is still writing it.  After a normal
        // epoch these waits end with the consumers' last tiles.
        for (uint32_t q = p + PRODUCERS * lane; q < a.nslots; q += PRODUCERS * 32u)
            if (s_turn[q] != 0u) mbar_wait(&full[q], (s_turn[q] - 1u) & 1u, &s_flag[3], DRAIN_LIMIT_NS);
        // The first producer warp then waits until the chains have read their last margins and counts
        // the CTA, while they update for the last time.  Counted last of the group: nobody adds or
        // reads any more, and it clears the accumulators.
        if (p == 0u) {
            __syncwarp();
#pragma unroll
            for (int c = 0; c < NC; ++c) asm volatile("bar.sync %0, 64;" ::"r"(4 + c) : "memory");
            const uint32_t mpad = SUB * a.nsub_max;
            unsigned long long *const acc_g = a.acc + (size_t)grp * EP_RING * a.nsub_max * EP_ACC_PITCH;
            unsigned long long *const wide_g = a.wide + (size_t)grp * EP_RING * mpad * EP_WIDE_WORDS;
            uint32_t *const header = a.header + grp * EP_HEADER_WORDS;
            uint32_t before = 0u;
            if (lane == 0) {
                if (s_flag[0] != 0u) atomicExch(header, 1u);   // gave up: so shall the others
                asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(header + 1) : "memory");
            }
            if (__shfl_sync(0xFFFFFFFFu, before, 0) == a.P - 1u) {
                for (uint32_t j = lane; j < EP_RING * mpad; j += 32u) {
                    acc_g[acc_index(j)] = 0ull;   // slots follow one another at the same pitch
#pragma unroll
                    for (uint32_t w = 0; w < EP_WIDE_WORDS; ++w) wide_g[(size_t)j * EP_WIDE_WORDS + w] = 0ull;
                }
                if (lane < 2u) header[lane] = 0u;
            }
        }
        return;
    }

    // ----------------------------------------------------------- consumers ----
    const uint32_t g = NC == 2 ? warp / EP_WARPS : 0u, wg = warp % EP_WARPS, tg = tid % EP_CHAIN;
    float *const coef = s_coef + g * EP_MAX_M;
    float *const part = s_part + (size_t)g * EP_WARPS * ucols;
    auto chain_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1u + g), "n"(EP_CHAIN) : "memory"); };
    const uint32_t mpad = SUB * a.nsub_max;
    unsigned long long *const acc_g = a.acc + (size_t)grp * EP_RING * a.nsub_max * EP_ACC_PITCH;
    unsigned long long *const wide_g = a.wide + (size_t)grp * EP_RING * mpad * EP_WIDE_WORDS;
    uint32_t *const header = a.header + grp * EP_HEADER_WORDS;

    if (warp == 0) tmem_alloc_all(const_cast<uint32_t *>(&s_flag[8]));
    // the slices of u of the group's workers, zeros past the slice
    for (uint32_t q = tid; q < kg * (ucols / 4u); q += NC * EP_CHAIN) {
        const uint32_t kk = q / (ucols / 4u), c = (q - kk * (ucols / 4u)) * 4u;
        const float *const from = a.u + (uint64_t)(grp + kk * a.G) * a.u_stride + c0 + c;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (EB == 16) {
            if (c < a.cols && (uint64_t)c0 + c < a.d) v = *reinterpret_cast<const float4 *>(from);
        } else if (c < a.cols) {
            const uint64_t left = (uint64_t)c0 + c < a.d ? a.d - c0 - c : 0u;
            if (left > 0u) v.x = from[0];
            if (left > 1u) v.y = from[1];
            if (left > 2u) v.z = from[2];
            if (left > 3u) v.w = from[3];
        }
        reinterpret_cast<float4 *>(s_u)[q] = v;
    }
    // (the producers are under way meanwhile)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    asm volatile("bar.sync 3, %0;" ::"n"(NC * EP_CHAIN) : "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = s_flag[8];
    // this thread's lane of the tensor memory, this warp's columns
    const uint32_t taddr = tmem_base + ((32u * (wg & 3u)) << 16) +
                           (NC == 2 ? 256u * g + 128u * (wg >> 2) : 256u * (wg >> 2));

    Tile T;
    T.start(a);
    if (g == 1u) T.next(a, kg);
    uint32_t base = 0u, turn0 = 0u, first0 = 0u;           // the tile's first sub-tile: its slot and turn in the ring, its number
    // With one chain the next tile, if it is another worker's, does not need this tile's update: its
    // margins go out first, and the warps' sums are added up while they travel, off the chain of
    // dependent steps and with one barrier less.  K = 4, n = 512, d = 131072: 246 -> 239 us; K = 3,
    // n = 640, d = 100000: 152 -> 147.5; K = 4, n = 512, d = 40000, batch 128: 83.5 -> 80.  With two chains the
    // other one's work lies there already.
    uint32_t due_kk = 0u, due_nsub = 0u, due_t = 0u;       // the tile whose sums are still to be added (none: no sub-tiles)
    bool read_all = false;                                 // the producer warp knows that this chain needs no margins any more
    for (uint32_t i = g; i < ntiles; i += NC) {
        for (base += T.first - first0; base >= a.nslots; base -= a.nslots) ++turn0;
        first0 = T.first;
        const uint32_t worker = grp + T.kk * a.G;
        float *const us = s_u + (size_t)T.kk * ucols;

        // The worker's previous minibatch is tile i-kg.  With two chains and an odd kg it belonged
        // to the other chain: wait until that chain has stored its update.
        if (NC == 2 && i >= kg && ((i - kg) & 1u) != g) {
            const uint32_t need = ((i - kg) >> 1) + 1u;
            if (tg == 0) {
                if (!flag_above(&s_flag[4u + (g ^ 1u)], need - 1u, &s_flag[0], a.wait_ns)) s_flag[0] = 1u;
                __threadfence_block();
            }
            if (sync_any(1u + g, EP_CHAIN, s_flag[0])) break;
        }

        // the label of the row this thread will finish, requested before it is needed
        const float yj = tg < T.m ? __ldg(a.y + (uint64_t)worker * a.n_local + (uint64_t)T.t * a.batch + tg) : 0.0f;

        // ---- M(i): margins over this CTA's columns, the values to tensor memory ----
        unsigned long long *const acc_t = acc_g + (size_t)(i % EP_RING) * a.nsub_max * EP_ACC_PITCH;
        unsigned long long *const wide_t = wide_g + (size_t)(i % EP_RING) * mpad * EP_WIDE_WORDS;
        const bool signal = i != 0u || blockIdx.x != a.drop_cta;
        uint32_t unit = 0u;      // 8 x 128 blocks stored so far
        for (uint32_t s = wg; s < T.nsub; s += EP_WARPS) {
            uint32_t slot = base + s, turn = turn0;
            for (; slot >= a.nslots; slot -= a.nslots) ++turn;
            // a barrier's parity tells neighbouring turns apart and no more, so see this turn begin first
            if (__all_sync(0xFFFFFFFFu, flag_above(&s_turn[slot], turn, &s_flag[0], a.wait_ns) &&
                                            mbar_wait(&full[slot], turn & 1u, &s_flag[0], a.wait_ns)) == 0) {
                s_flag[0] = 1u;
                break;
            }
            const float *const xs = ring + (size_t)slot * slot_floats;
            const uint32_t rows = T.m - s * SUB;     // rows of the minibatch in this sub-tile, if below 8
            float acc[SUB];
#pragma unroll
            for (int r = 0; r < SUB; ++r) acc[r] = 0.0f;
            if constexpr (NC == 1 && EB == 16) {
                // Two blocks are requested at a time: one chain has the registers, and where slices are wide the time
                // until a slot is free again is what the last sub-tiles of a minibatch wait for (six slots for eight
                // sub-tiles: the margins of the six take 2330 clocks for 2940).  K = 4, n = 512, d = 131072 238.6 ->
                // 230.8 us, n = 256, d = 140000, batch 32 138.4 -> 132.3; with element-wise copies, whose blocks have
                // 128 registers a thread, 152.8 -> 164.2 (K = 3, n = 300, d = 131073).
                auto load = [&](uint32_t it, float4 (&x)[SUB]) {
                    const uint32_t b0 = it / BOX_UNITS * BOX, c = it * 128u + lane * 4u;
                    const uint32_t pitch = min(a.cols - b0, BOX);
                    const float *const from = xs + SUB * b0 + (c - b0);
                    if (rows >= (uint32_t)SUB && it * 128u + 128u <= a.cols) {
#pragma unroll
                        for (uint32_t r = 0; r < (uint32_t)SUB; ++r) x[r] = *reinterpret_cast<const float4 *>(from + r * pitch);
                    } else {
#pragma unroll
                        for (uint32_t r = 0; r < (uint32_t)SUB; ++r)
                            x[r] = (c < a.cols && r < rows) ? *reinterpret_cast<const float4 *>(from + r * pitch)
                                                            : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                };
                auto margins = [&](const float4 uu, const float4 (&x)[SUB]) {
#pragma unroll
                    for (int r = 0; r < SUB; ++r) {
                        acc[r] = fmaf(x[r].x, uu.x, acc[r]);
                        acc[r] = fmaf(x[r].y, uu.y, acc[r]);
                        acc[r] = fmaf(x[r].z, uu.z, acc[r]);
                        acc[r] = fmaf(x[r].w, uu.w, acc[r]);
                    }
                };
                const float *const ul = us + lane * 4u;
                float4 x0[SUB], x1[SUB];
                uint32_t it = 0u;
#pragma unroll 1
                for (; it + 1u < a.nit; it += 2u) {
                    load(it, x0);
                    const float4 u0 = *reinterpret_cast<const float4 *>(ul + it * 128u);
                    load(it + 1u, x1);
                    const float4 u1 = *reinterpret_cast<const float4 *>(ul + it * 128u + 128u);
                    margins(u0, x0);
                    margins(u1, x1);
                    tmem_st32(taddr + 32u * unit, x0);
                    tmem_st32(taddr + 32u * (unit + 1u), x1);
                    unit += 2u;
                }
                if (it < a.nit) {
                    load(it, x0);
                    margins(*reinterpret_cast<const float4 *>(ul + it * 128u), x0);
                    tmem_st32(taddr + 32u * unit, x0);
                    ++unit;
                }
            } else {
#pragma unroll 1
                for (uint32_t it = 0; it < a.nit; ++it) {
                    const uint32_t b0 = it / BOX_UNITS * BOX, c = it * 128u + lane * 4u;
                    const uint32_t pitch = min(a.cols - b0, BOX);
                    const float *const base = xs + SUB * b0 + (c - b0);
                    const float4 uu = *reinterpret_cast<const float4 *>(us + c);
                    float4 x[SUB];
#pragma unroll
                    for (uint32_t r = 0; r < (uint32_t)SUB; ++r)
                        x[r] = (c < a.cols && r < rows) ? *reinterpret_cast<const float4 *>(base + r * pitch)
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int r = 0; r < SUB; ++r) {
                        acc[r] = fmaf(x[r].x, uu.x, acc[r]);
                        acc[r] = fmaf(x[r].y, uu.y, acc[r]);
                        acc[r] = fmaf(x[r].z, uu.z, acc[r]);
                        acc[r] = fmaf(x[r].w, uu.w, acc[r]);
                    }
                    tmem_st32(taddr + 32u * unit, x);
                    ++unit;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[slot]);
            const float tot = reduce8(acc, lane);
            const uint32_t jj = s * SUB + reduce8_row(lane);
            // (exchange_add and exchange_margin of qesgd_lr_device.cuh written out: through the functions K = 3, n = 300,
            // d = 131073 takes 154.5 us instead of 152.8, K = 4, n = 2048, d = 65536 330.5 instead of 329.8)
            if ((lane & 3u) == 0u && jj < T.m && signal) {
                unsigned long long *const r = acc_t + acc_index(jj);
                if (fabsf(tot) < FX_LIMIT) {
                    atomicAdd(r, FX_ONE + FX_BIAS + (unsigned long long)__float2ll_rn(tot * FX_SCALE));
                } else {
                    // rare: the special bit and the row's other words first, visible before the count
                    unsigned long long *const w = wide_t + (size_t)jj * EP_WIDE_WORDS;
                    atomicOr(r, FX_SPECIAL);
                    if (fabsf(tot) < FX_WIDE_LIMIT)
                        atomicAdd(w, (unsigned long long)__float2ll_rn(tot * FX_WIDE_SCALE));
                    else if (tot != tot)
                        atomicAdd(w + 1, 1ull);                               // NaN
                    else
                        atomicAdd(w + 2, tot > 0.0f ? (1ull << 32) : 1ull);   // +-Inf, or beyond the wide word
                    __threadfence();
                    atomicAdd(r, FX_ONE + FX_BIAS);
                }
            }
        }
        tmem_wait_st();
        if (NC == 1 && due_nsub != 0u) {
            chain_sync();
            add_to_u<EB>(a, s_u + (size_t)due_kk * ucols, part, ucols, tg, c0, grp + due_kk * a.G, due_nsub, due_t);   // complete for all at the barrier in W(i)
            due_nsub = 0u;
        }

        // ---- W(i): all CTAs' partial margins -> step coefficients in shared memory ----
        if (rank == i % a.P) {   // this CTA clears the slot that tile i + RING/2 will add into
            const uint32_t zs = (i + EP_RING / 2) % EP_RING;
            unsigned long long *const az = acc_g + (size_t)zs * a.nsub_max * EP_ACC_PITCH;
            unsigned long long *const wz = wide_g + (size_t)zs * mpad * EP_WIDE_WORDS;
            for (uint32_t j = EP_CHAIN - 1u - tg; j < mpad; j += EP_CHAIN) {
                az[acc_index(j)] = 0ull;
#pragma unroll
                for (uint32_t w = 0; w < EP_WIDE_WORDS; ++w) wz[(size_t)j * EP_WIDE_WORDS + w] = 0ull;
                __threadfence();     // cleared for every CTA before this thread goes on
            }
        }
        if (tg < SUB * T.nsub) {
            float cj = 0.0f;
            if (tg < T.m) {
                const unsigned long long *const r = acc_t + acc_index(tg);
                unsigned long long v = ld_relaxed(r);
                if ((v >> 55) < a.P) {
                    const uint64_t t0 = now_ns();
                    uint32_t n = 0u;
                    while (((v = ld_relaxed(r)) >> 55) < a.P) {
                        if ((++n & a.poll_mask) == 0u &&
                            (s_flag[0] != 0u || ld_acquire(header) != 0u || expired(t0, a.wait_ns))) {
                            s_flag[0] = 1u;
                            break;
                        }
                    }
                }
                const long long fine = (long long)((v & (FX_SPECIAL - 1ull)) - (unsigned long long)a.P * FX_BIAS);
                float margin = (float)((double)fine * (1.0 / (double)FX_SCALE));
                if ((v & FX_SPECIAL) != 0ull) {
                    const unsigned long long *const w = wide_t + (size_t)tg * EP_WIDE_WORDS;
                    __threadfence();
                    const unsigned long long w0 = ld_relaxed(w), w1 = ld_relaxed(w + 1), w2 = ld_relaxed(w + 2);
                    margin = (float)((double)fine * (1.0 / (double)FX_SCALE) +
                                     (double)(long long)w0 * (1.0 / (double)FX_WIDE_SCALE));
                    if (w2 != 0ull) {   // +Inf count << 32 + -Inf count
                        const bool pos = (w2 >> 32) != 0ull, neg = (w2 & 0xFFFFFFFFull) != 0ull;
                        margin = pos && neg ? __int_as_float(0x7FC00000)
                                            : __int_as_float(pos ? 0x7F800000 : (int)0xFF800000);
                    }
                    if (w1 != 0ull) margin = __int_as_float(0x7FC00000);
                }
                // -(lr/m) * c_j with c_j = -y_j / (1 + exp(y_j m_j))
                cj = (T.t == a.nsteps - 1u ? a.rate_last : a.rate) * yj / (1.0f + expf(yj * margin));
            }
            coef[tg] = cj;
        }
        if (sync_any(1u + g, EP_CHAIN, s_flag[0])) break;

        if (i + NC >= ntiles && wg == 0u) {
            asm volatile("bar.arrive %0, 64;" ::"r"(4u + g) : "memory");
            read_all = true;
        }

        // ---- U(i): coef_j x_j summed over the warp's rows, then over the warps, onto u ----
        if (wg < T.nsub) {
            // one chain has the registers for two blocks at a time
            for (uint32_t it = 0; it < a.nit; it += 3u - NC) {
                const bool two = NC == 1 && it + 1u < a.nit;
                float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0;
                uint32_t q = it;
                for (uint32_t s = wg; s < T.nsub; s += EP_WARPS, q += a.nit) {
                    float4 x0[SUB], x1[SUB];
                    tmem_ld32(taddr + 32u * q, x0);
                    if (NC == 1 && two) tmem_ld32(taddr + 32u * (q + 1u), x1);
                    const float4 ca = *reinterpret_cast<const float4 *>(coef + s * SUB);
                    const float4 cb = *reinterpret_cast<const float4 *>(coef + s * SUB + 4u);
                    const float cs[SUB] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
                    tmem_wait_ld();
#pragma unroll
                    for (int r = 0; r < SUB; ++r) {
                        s0.x = fmaf(cs[r], x0[r].x, s0.x);
                        s0.y = fmaf(cs[r], x0[r].y, s0.y);
                        s0.z = fmaf(cs[r], x0[r].z, s0.z);
                        s0.w = fmaf(cs[r], x0[r].w, s0.w);
                    }
                    if (NC == 1 && two) {
#pragma unroll
                        for (int r = 0; r < SUB; ++r) {
                            s1.x = fmaf(cs[r], x1[r].x, s1.x);
                            s1.y = fmaf(cs[r], x1[r].y, s1.y);
                            s1.z = fmaf(cs[r], x1[r].z, s1.z);
                            s1.w = fmaf(cs[r], x1[r].w, s1.w);
                        }
                    }
                }
                float *const pw = part + (size_t)wg * ucols + it * 128u + lane * 4u;
                *reinterpret_cast<float4 *>(pw) = s0;
                if (NC == 1 && two) *reinterpret_cast<float4 *>(pw + 128) = s1;
            }
        }
        if constexpr (NC == 1) {
            if (kg > 1u) {
                due_kk = T.kk;
                due_nsub = T.nsub;
                due_t = T.t;
            } else {
                chain_sync();
                add_to_u<EB>(a, us, part, ucols, tg, c0, worker, T.nsub, T.t);
                chain_sync();                                 // u complete for the next minibatch
            }
        } else {
            // add_to_u written out: through the function K = 4, n = 2048, d = 65536 takes 333.6 us instead of
            // 329.5, K = 8, n = 512 171.0 instead of 167.5
            static_assert(NC == 1 || EB == 16, "two chains are fed by TMA");
            chain_sync();
            if (tg < ucols / 4u) {
                const uint32_t c = tg * 4u;
                float4 o = make_float4(0.f, 0.f, 0.f, 0.f), t = o;
                if (!a.gradient) o = *reinterpret_cast<const float4 *>(us + c);
#pragma unroll
                for (uint32_t w = 0; w < (uint32_t)EP_WARPS; ++w) {
                    if (w < T.nsub) {
                        const float4 v = *reinterpret_cast<const float4 *>(part + (size_t)w * ucols + c);
                        t.x += v.x; t.y += v.y; t.z += v.z; t.w += v.w;
                    }
                }
                t.x += o.x; t.y += o.y; t.z += o.z; t.w += o.w;
                *reinterpret_cast<float4 *>(us + c) = t;
                if (T.t == a.nsteps - 1u && c < a.cols && (uint64_t)c0 + c < a.d)   // the worker's last minibatch
                    *reinterpret_cast<float4 *>(a.dst + (uint64_t)worker * a.u_stride + c0 + c) = t;
            }
            chain_sync();                                     // u complete for the next minibatch
        }
        if (NC == 2 && tg == 0) {
            __threadfence_block();
            s_flag[4u + g] = (i >> 1) + 1u;               // this chain's tiles completed
        }
        for (uint32_t n = 0; n < (uint32_t)NC && i + n + 1u < ntiles; ++n) T.next(a, kg);
    }
    if (NC == 1 && due_nsub != 0u) {
        chain_sync();
        add_to_u<EB>(a, s_u + (size_t)due_kk * ucols, part, ucols, tg, c0, grp + due_kk * a.G, due_nsub, due_t);
    }
    if (!read_all && wg == 0u)                             // a chain without tiles, or one that gave up
        asm volatile("bar.arrive %0, 64;" ::"r"(4u + g) : "memory");

    // All chains meet here, whether they finished or gave up.
    asm volatile("bar.sync 3, %0;" ::"n"(NC * EP_CHAIN) : "memory");
    if (warp == 0) tmem_free_all(tmem_base);              // on every path out of the kernel
    // A wait ran out: tell the host.  The copies still in flight are the producer warps' to wait for.
    if (s_flag[0] != 0u && tid == 0) atomicOr(a.status, QESGD_STATUS_TIMEOUT);
}

// ------------------------------------------------------------------ host ----
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

// one and two chains with TMA, one chain with copies of 8 and 4 bytes
const void *const EPOCH_KERNELS[4] = {(const void *)qesgd_lr_epoch_kernel<1, 16>, (const void *)qesgd_lr_epoch_kernel<2, 16>,
                                      (const void *)qesgd_lr_epoch_kernel<1, 8>, (const void *)qesgd_lr_epoch_kernel<1, 4>};

// Per-device set-up: shared-memory limit of the kernels, the driver's tensor-map encoder.
constexpr int MAX_DEVICES = 64;
std::mutex g_epoch_mutex;
int g_epoch_smem_limit[MAX_DEVICES] = {0};   // 0 = not queried, -1 = unsupported
EncodeTiledFn g_encode_tiled = nullptr;

int epoch_smem_limit(int device)
{
    if (device < 0 || device >= MAX_DEVICES) return -1;
    std::lock_guard<std::mutex> lock(g_epoch_mutex);
    if (g_epoch_smem_limit[device] == 0) {
        int coop = 0, optin = 0;
        cudaError_t e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device);
        if (e == cudaSuccess)
            e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
        for (const void *kernel : EPOCH_KERNELS)
            if (e == cudaSuccess && coop && optin > 0)
                e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        if (e == cudaSuccess && !g_encode_tiled) {
            void *fn = nullptr;
            cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
            e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q);
            if (e == cudaSuccess && q == cudaDriverEntryPointSuccess) g_encode_tiled = (EncodeTiledFn)fn;
        }
        g_epoch_smem_limit[device] =
            (e == cudaSuccess && coop && optin > 0 && g_encode_tiled) ? optin : -1;
        if (e != cudaSuccess) cudaGetLastError();
    }
    return g_epoch_smem_limit[device];
}

// Row-major float matrix [rows][d] seen as a 2-D tensor; a box is SUB rows of box_cols columns.  As a tensor of pairs of
// floats (d and box_cols are even) the widest box, 256 elements, is 512 columns.  Elements outside the matrix read as zero.
}  // namespace
bool qesgd_lr_tensor_map(CUtensorMap *map, const float *X, uint64_t rows, uint64_t d, uint32_t box_cols, bool pairs)
{
    const uint32_t n = pairs ? 2u : 1u;
    const cuuint64_t dims[2] = {d / n, rows};
    const cuuint64_t strides[1] = {d * sizeof(float)};
    const cuuint32_t box[2] = {box_cols / n, (cuuint32_t)SUB};
    const cuuint32_t elem[2] = {1u, 1u};
    return g_encode_tiled(map, pairs ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2u, const_cast<float *>(X), dims, strides, box,
                          elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
namespace {

// One way to deal the epoch out: G groups of P CTAs, NC chains per CTA.
struct Split {
    uint32_t G, P, NC, cols, nit, nslots;
    uint32_t off_u, off_part, off_coef, off_bars, off_flags, bytes;
    float us;            // modelled time of a step of all workers
};

// Fills in the rest of a split with G groups and P CTAs each; false where it does not fit.
bool complete_split(Split &s, uint64_t d, uint32_t K, uint32_t m, uint32_t nsub, bool tma, uint32_t limit)
{
    const uint64_t cols = ((d + s.P - 1) / s.P + 3) / 4 * 4;
    if (cols > 1024) return false;
    s.cols = (uint32_t)cols;
    s.P = (uint32_t)((d + cols - 1) / cols);
    s.nit = (s.cols + 127u) / 128u;
    const uint32_t kg = (K + s.G - 1u) / s.G;
    const uint32_t units = (nsub + EP_WARPS - 1u) / EP_WARPS * s.nit;    // tensor-memory blocks per warp
    if (units > (uint32_t)EP_UNITS) return false;
    s.NC = tma && kg >= 2u && units <= (uint32_t)EP_UNITS / 2u ? 2u : 1u;
    const uint32_t slot = SUB * s.cols * 4u, ubytes = s.nit * 512u;
    const uint32_t fixed = kg * ubytes + s.NC * EP_WARPS * ubytes + s.NC * EP_MAX_M * 4u + 2u * EP_MAX_SLOTS * 8u + EP_FLAG_BYTES;
    if (fixed + 2u * slot > limit) return false;
    s.nslots = (limit - fixed) / slot;
    if (s.nslots > (uint32_t)EP_MAX_SLOTS) s.nslots = EP_MAX_SLOTS;
    s.off_u = s.nslots * slot;                   // slots are multiples of 128 bytes
    s.off_part = s.off_u + kg * ubytes;
    s.off_coef = s.off_part + s.NC * EP_WARPS * ubytes;
    s.off_bars = s.off_coef + s.NC * EP_MAX_M * 4u;
    s.off_flags = s.off_bars + 2u * EP_MAX_SLOTS * 8u;
    s.bytes = s.off_flags + EP_FLAG_BYTES;
    const float hbm = (float)((double)K * m * d * 4.0 / (1000.0 * EP_HBM_BYTES_PER_NS));   // us
    const float chain = EP_CHAIN_US + EP_UNIT_US * (float)units;
    const float chained = chain * (float)kg / (float)s.NC;
    s.us = hbm > chained ? hbm : chained;
    return true;
}

// The modelled time picks the split; ties go to fewer groups.
bool choose_split(Split &best, uint64_t d, uint32_t K, uint32_t m, uint32_t nsub, bool tma, uint32_t sm_count,
                  uint32_t limit)
{
    bool any = false;
    for (uint32_t G = 1; G <= K && G <= sm_count; ++G) {
        if (G * nsub * SUB > QESGD_LR_EPOCH_ROWS) break;     // accumulators of all groups
        if (G > 1u && (K + G - 1u) / G == (K + G - 2u) / (G - 1u)) continue;   // no fewer workers per group than before
        Split s;
        s.G = G;
        s.P = sm_count / G;
        const uint64_t most = (d + 127u) / 128u;              // a warp takes 128 columns at a time
        if (s.P > most) s.P = (uint32_t)most;
        if (!complete_split(s, d, K, m, nsub, tma, limit)) continue;
        if (!any || s.us < 0.99f * best.us) best = s;
        any = true;
    }
    return any;
}

}  // namespace

// Returns 0 = launched, -1 = shape not covered by the fused kernel (caller uses the
// two-pass steps), > 0 = cudaError_t.
// A single minibatch's mean gradient is an epoch of one step with lr = -1 that does not add u: minibatches
// of 64 x 65536 out of HBM 10.3 us instead of 16.5 for the margin pass and the update pass, of 256 x 35584
// 13.1 instead of 37.7 (two launches, and most SMs idle in the first).
int qesgd_launch_lr_epoch_fused(const float *X, const float *y, uint64_t n_local, uint64_t d,
                                uint32_t K, uint32_t batch, float lr, const float *u, float *dst,
                                bool gradient, uint64_t u_stride, float *work, uint32_t *status, int device, int sm_count, uint64_t wait_ns,
                                uint32_t drop_cta, cudaStream_t stream, int *launched, uint32_t (&plan)[8])
{
    *launched = 0;
    for (uint32_t &v : plan) v = 0u;          // two passes, unless a kernel is launched here
    const uint32_t m_full = (uint32_t)(n_local < batch ? n_local : batch);
    if (m_full > (uint32_t)EP_MAX_M) return -1;
    const uint64_t nsteps64 = (n_local + m_full - 1) / m_full;
    if (nsteps64 * K > (1u << 20)) return -1;
    if ((uint64_t)K * n_local + EP_MAX_M >= (1ull << 31)) return -1;   // TMA row coordinates
    const bool tma = d % 4 == 0 && u_stride % 4 == 0 && ((uintptr_t)X | (uintptr_t)u | (uintptr_t)dst) % 16 == 0;
    const bool pairs = d % 2 == 0 && (uintptr_t)X % 8 == 0;
    if (sm_count < 1 || d > 1024ull * (uint64_t)sm_count) return -1;
    const int limit = epoch_smem_limit(device);
    if (limit <= 0) return -1;
    const uint32_t nsub = (m_full + SUB - 1) / SUB;
    Split s;
    // A CTA takes a whole SM and none starts before all can, so a call that takes every SM waits for any
    // kernel of another stream that holds one.  A single step leaves one SM in sixteen free, which costs it
    // nothing (148, 140, 132 and 128 SMs: 64 x 65536 8.4, 8.3, 8.5, 8.3 us; 64 x 131072 out of HBM 12.4, 12.4,
    // 12.4, 12.5).  A gradient never takes more: where it only fits all SMs (256 x 37888: 14.4 us), two passes
    // of small kernels (28.9) run on whatever is free.  The accumulator word counts up to 256 contributions.
    const uint32_t sms = (uint32_t)(sm_count < 256 ? sm_count : 256);
    bool fits = nsteps64 * K == 1u && choose_split(s, d, K, m_full, nsub, tma, sms - sms / 16u, (uint32_t)limit);
    if (!fits && !gradient) fits = choose_split(s, d, K, m_full, nsub, tma, sms, (uint32_t)limit);
    // workspace, all zero between launches: headers | accumulators | their rarely used words
    uint32_t *const header = reinterpret_cast<uint32_t *>(work);
    unsigned long long *const acc = reinterpret_cast<unsigned long long *>(work + QESGD_MAX_WORKERS * EP_HEADER_WORDS);
    unsigned long long *const wide = acc + (size_t)EP_RING * (QESGD_LR_EPOCH_ROWS / SUB) * EP_ACC_PITCH;
    {
        const QesgdTileCall q = {X, y, n_local, d, nsteps64, K, m_full, lr, u, dst, gradient, u_stride, tma ? 16 : (pairs ? 8 : 4),
                                 header, acc, wide, status, device, nsteps64 * K == 1u ? sms - sms / 16u : sms, wait_ns, drop_cta, stream};
        const int e = qesgd_launch_lr_tile(q, (uint32_t)limit, fits ? s.us : 1e30f, launched, plan);
        if (e >= 0) return e;
    }
    if (!fits) return -1;

    EpochArgs a;
    a.X = X; a.y = y; a.n_local = n_local;
    a.d = d; a.K = K; a.G = s.G; a.P = s.P;
    a.batch = m_full; a.nsteps = (uint32_t)nsteps64;
    a.m_last = (uint32_t)(n_local - (nsteps64 - 1) * m_full);
    a.nsub_max = nsub;
    a.nsub_last = (a.m_last + SUB - 1) / SUB;
    a.cols = s.cols; a.nit = s.nit; a.nslots = s.nslots;
    a.off_u = s.off_u; a.off_part = s.off_part; a.off_coef = s.off_coef; a.off_bars = s.off_bars; a.off_flags = s.off_flags;
    // Pause between a producer's copies, in parts of the interval at which HBM serves all SMs (see the head of
    // the file).  One group with one chain is late for the next tile whenever it was for this one, and gains
    // from copies spread a little wider: 0.6 -> 0.8, K = 4, n = 512, d = 131072 251.9 -> 238.8 us, K = 8,
    // n = 128 132.5 -> 125.4, K = 1, d = 65536 36.3 -> 35.0, minibatches of 128, d = 75776 35.0 -> 33.9 (K = 4:
    // 120.0 -> 112.6); only where all of X stays in L2 from call to call is it slower (K = 1, d = 50000,
    // minibatches of 128 24.7 -> 26.7).  A single tile is late for none: 128 x 75776 11.2 us against 12.4.
    // Two chains whose ring holds no more than half a minibatch (many workers: their slices of u take the
    // room) leave no slot free for long and wait for one another's copies: 0.6 -> 0.9, K = 64, n = 64,
    // d = 65536 (four slots) 261 -> 253 us, d = 75776 (three) 334 -> 330; with five slots the copies already
    // run ahead and a wider pace only costs (K = 48, d = 75776 176 -> 201, K = 56, d = 65536 200 -> 217).
    const float pace = s.G == 1u && s.NC == 1u && nsteps64 * K > 1u ? 0.8f : s.NC == 2u && 2u * s.nslots <= nsub ? 0.9f : 0.6f;
    a.pace = (uint32_t)(pace * (float)(SUB * s.cols * 4u * EP_PRODUCERS) * (float)(s.G * s.P) / EP_HBM_BYTES_PER_NS);
    a.rate = lr / (float)m_full;
    a.rate_last = lr / (float)a.m_last;
    a.u = u; a.dst = dst; a.gradient = gradient ? 1u : 0u; a.u_stride = u_stride;
    a.status = status;
    a.wait_ns = wait_ns;
    a.poll_mask = wait_ns < COARSE_TIMER_NS ? 0u : 31u;
    a.drop_cta = drop_cta;
    a.header = header;
    a.acc = acc;
    a.wide = wide;

    CUtensorMap map_full = {}, map_rest = {};
    const uint32_t wide_box = s.cols < (uint32_t)EP_BOX_COLS ? s.cols : (uint32_t)EP_BOX_COLS;
    const uint32_t rest = s.cols % EP_BOX_COLS;
    if (tma && !qesgd_lr_tensor_map(&map_full, X, (uint64_t)K * n_local, d, wide_box, false)) return -1;
    if (tma && !qesgd_lr_tensor_map(&map_rest, X, (uint64_t)K * n_local, d, rest ? rest : wide_box, false)) return -1;

    void *params[] = {(void *)&a, (void *)&map_full, (void *)&map_rest};
    const void *const kernel = EPOCH_KERNELS[tma ? s.NC - 1u : (pairs ? 2u : 3u)];
    const uint32_t threads = s.NC * EP_CHAIN + (tma ? EP_PRODUCERS : EP_LOADERS) * 32u;
    const cudaError_t e = cudaLaunchCooperativeKernel(kernel, dim3(s.G * s.P), dim3(threads), params, s.bytes, stream);
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources ||
        e == cudaErrorInvalidConfiguration || e == cudaErrorNotSupported) {
        cudaGetLastError();   // the device cannot hold all CTAs at once as configured: two-pass steps
        return -1;
    }
    if (e != cudaSuccess) return (int)e;
    *launched = 1;
    const uint32_t shape[8] = {QESGD_LR_PERSISTENT, s.P, s.cols, s.NC, s.nslots, tma ? 16u : (pairs ? 8u : 4u), s.G * s.P,
                               (K + s.G - 1u) / s.G};
    for (int i = 0; i < 8; ++i) plan[i] = shape[i];
    return 0;
}
