// Local epochs and mean gradients of logistic regression whose minibatch slice fits the registers of a CTA.
//
// The persistent kernel of qesgd_lr_epoch.cu hides the chain of a step -- margins, exchange, coefficients,
// update -- behind copies of many columns and behind a second chain.  With few columns per CTA nothing hides
// it, and the chain itself is the time: there every phase goes through shared or tensor memory with four
// barriers a step, about 3500 clocks of which the exchange is 400 to 1000.  Here a worker has its own CTAs
// (one cluster of up to 16, a group of the cooperative grid, or for one minibatch a grid launched plainly), and a
// warp its own eight rows of U x 128 columns: the rows live in registers from the margins to the update, a lane
// always holds the same columns, and the row whose sum a lane ends up with is the row it exchanges and finishes, so
// between the margins and the update nothing crosses the warp.  Two barriers a step are left, around the sum of the
// warps' updates.
//
//   M  partial margins of the warp's rows from registers and the slice of u (shared memory); sum over the lanes
//   X  the sums go out; the slot they came from is refilled (TMA, or element-wise copies); wait for all P
//      partials of the rows; coefficients; handed to the lanes by shuffle
//   U  the warp's update of its columns to shared memory; the next rows into the registers, while
//   A  the block adds the warps' updates to the slice of u.
//
// Exchange in a cluster: each CTA stores {partial, tile number + 1} as one 64-bit word into every CTA's shared
// memory; the reader polls its own.  The number says that the value beside it is there, so there is no barrier
// and nothing in flight that the cluster's barrier would not cover.  The sum over the ranks carries every
// addition's error along (two_sum) and is rounded once, in a fixed order.  Exchange in a group or a plain grid: the
// accumulators in global memory described in qesgd_lr_epoch.cu, by the functions of qesgd_lr_device.cuh.
//
// Every wait is bounded by the context's limit.  A wait that runs out sets QESGD_STATUS_TIMEOUT and the block
// leaves at its next barrier, together; it then waits for the copies it has requested, and in a cluster until the
// others have left or ended too, since they may still be storing margins here.
#include <mutex>

#include "qesgd_lr_device.cuh"
#include "qesgd_lr_tile.h"

namespace {

constexpr uint32_t TL_MAX_SLOTS = 64;

struct TileArgs {
    const float *X, *y;
    uint64_t n_local, d;
    uint32_t P;                  // CTAs per worker
    uint32_t batch, nsteps, m_last, nsub, nsub_last;
    uint32_t nslots;
    uint32_t off_u, off_part, off_x, off_bars, off_flags;   // shared memory, bytes
    uint32_t x_pitch;            // words of the exchange from one rank to the next
    float rate, rate_last;
    const float *u;
    float *dst;
    uint32_t gradient;
    uint64_t u_stride;
    uint32_t *header;
    unsigned long long *acc, *wide;
    uint32_t *status;
    uint64_t wait_ns;
    uint32_t poll_mask, drop_cta;
    uint32_t *claims;            // one minibatch, plain launch: [P] Claim of each slice; else null
    uint32_t off_claims;         // shared memory: the coefficients, then how many slices this CTA took over and which
};
constexpr uint64_t TL_STEAL_NS = 20000ull;   // a wait longer than this looks for slices that nobody has begun
constexpr uint64_t TL_BEGIN_NS = 2000000000ull;   // by then every slice has been begun
// A slice is BEGUN by a CTA that runs, or its margins are out; TAKEN: another CTA does it, they are not out yet.
enum Claim { FREE = 0, BEGUN = 1, TAKEN = 2 };
constexpr uint32_t TL_ROWS = 128;            // coefficients kept for them

__device__ __forceinline__ uint32_t cluster_address(uint32_t addr, uint32_t rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, float v, uint32_t tag)
{
    asm volatile("{\n.reg .b64 w;\nmov.b64 w, {%1, %2};\nst.relaxed.cluster.shared::cluster.b64 [%0], w;\n}" ::"r"(addr),
                 "f"(v), "r"(tag)
                 : "memory");
}
__device__ __forceinline__ void cluster_store2(uint32_t addr, float v0, float v1, uint32_t tag)
{
    asm volatile("{\n.reg .b64 w, x;\nmov.b64 w, {%1, %3};\nmov.b64 x, {%2, %3};\n"
                 "st.relaxed.cluster.shared::cluster.v2.b64 [%0], {w, x};\n}" ::"r"(addr),
                 "f"(v0), "f"(v1), "r"(tag)
                 : "memory");
}
__device__ __forceinline__ void cluster_load(uint32_t addr, float &v, uint32_t &tag)
{
    asm volatile("{\n.reg .b64 w;\nld.relaxed.cluster.shared::cta.b64 w, [%2];\nmov.b64 {%0, %1}, w;\n}"
                 : "=f"(v), "=r"(tag)
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// A warp's eight totals (lanes 4r to 4r + 3 hold row r's) to every CTA of the cluster: 32 / P lanes a CTA (two and more
// of them for small clusters, where some lanes have nothing to do), the rows dealt out among them.
__device__ __forceinline__ uint32_t send_rank(uint32_t P, uint32_t lane)
{
    return P == 16u ? lane >> 1 : (P == 8u ? lane >> 2 : lane >> 3);
}
__device__ __forceinline__ uint32_t send_row(uint32_t P, uint32_t lane)
{
    return P == 16u ? (lane & 1u) * 4u : (P == 8u ? (lane & 3u) * 2u : lane & 7u);
}
__device__ __forceinline__ void cluster_send(uint32_t to, uint32_t row, float tot, uint32_t tag, uint32_t P, uint32_t lane)
{
    const float v0 = __shfl_sync(0xFFFFFFFFu, tot, 4u * row), v1 = __shfl_sync(0xFFFFFFFFu, tot, 4u * row + 4u);
    if (P == 16u) {
        const float v2 = __shfl_sync(0xFFFFFFFFu, tot, 4u * row + 8u);
        const float v3 = __shfl_sync(0xFFFFFFFFu, tot, 4u * row + 12u);
        cluster_store2(to, v0, v1, tag);
        cluster_store2(to + 16u, v2, v3, tag);
    } else if (P == 8u) {
        cluster_store2(to, v0, v1, tag);
    } else if ((lane >> 3) < P) {
        cluster_store(to, v0, tag);
    }
}
// a + b = s + e exactly, for finite sums (the error-free addition of Knuth and of Moller)
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

template <int N>
__device__ __forceinline__ void load_n(const float *p, float (&v)[N])
{
    if (N == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x; v[1 % N] = q.y; v[2 % N] = q.z; v[3 % N] = q.w;
    } else if (N == 2) {
        const float2 q = *reinterpret_cast<const float2 *>(p);
        v[0] = q.x; v[1 % N] = q.y;
    } else {
        v[0] = *p;
    }
}

extern __shared__ __align__(1024) unsigned char tl_smem[];

// A kernel argument that the loop uses, in a register: read from the constant bank at each use it costs the chain
// 40 clocks.
__device__ __forceinline__ uint32_t kept(uint32_t v)
{
    asm volatile("" : "+r"(v));
    return v;
}

// Slices that nobody has begun.  The grid of one minibatch is launched like any other kernel, so that it is set up
// while the one before it drains (a cooperative launch is not, and occupies the stream for a whole number of 2.05 us:
// 64 x 65536 from L2 8.2 us, launched plainly 6.2, from HBM 10.2 and 8.0; 64 x 20000 8.2 and 5.1; 16 x 80000 8.1 and
// 5.0).  Then nothing promises that all its CTAs are resident at once: beside other streams' kernels some may start
// late.  So a CTA never waits for one that has not started: each claims its slice when it starts, a wait longer than
// 20 us claims one that is still free and does its margins here, by the same operations in the same order, and after
// its own update the CTA does theirs.  A CTA that finds its slice claimed has nothing left to do.  64 x 65536 beside
// 24, 64, 100 and 130 held SMs: 95, 131, 156 and 194 us; a cooperative launch waits for those SMs.
//
// The wait limit is about CTAs that run and do not answer.  Time in which slices have not been begun, because other
// streams' kernels hold the SMs, or are being made up for, does not count: a limit of 100 us is no reason to give up
// a call that takes 180 us beside such kernels.  It counts from when a look finds every slice BEGUN.
//
// A warp looks whether every slice has been begun (then true); where that is `due` it takes a free one and adds its
// partial margins to the rows' accumulators.
template <int U>
__device__ __noinline__ bool take_over(const TileArgs &a, uint32_t *list, bool due, uint32_t lane)
{
    uint32_t slice = ~0u;
    bool begun = true;
    for (uint32_t b = 0; b < a.P && slice == ~0u; b += 32u) {
        const uint32_t claim = b + lane < a.P ? ld_acquire(a.claims + b + lane) : (uint32_t)BEGUN;
        if (__any_sync(0xFFFFFFFFu, claim != BEGUN)) begun = false;
        const uint32_t free = __ballot_sync(0xFFFFFFFFu, claim == FREE);
        if (free == 0u || !due) continue;
        const uint32_t first = b + (uint32_t)__ffs((int)free) - 1u;
        uint32_t before = BEGUN;
        if (lane == 0) before = atomicCAS(a.claims + first, (uint32_t)FREE, (uint32_t)TAKEN);
        if (__shfl_sync(0xFFFFFFFFu, before, 0) == FREE) slice = first;
    }
    if (slice == ~0u) return begun;
    if (lane == 0) list[1u + atomicAdd(list, 1u)] = slice;
    const uint32_t m = a.m_last, nsub = a.nsub_last;
    const float *const X = a.X, *const u = a.u;
    const uint64_t d = a.d, c0 = (uint64_t)slice * (U * 128u) + lane * 4u;
    for (uint32_t s = 0; s < nsub; ++s) {
        float acc[SUB];
        // Two rows at a time: what this needs of registers the kernel saves around the call, and for sixteen warps of two
        // blocks all eight at once cost the way without it too (gradient of 100 x 30001 8.4 us, so 7.5).
#pragma unroll 1
        for (uint32_t g = 0; g < 4u; ++g) {
            const float *line = X + (uint64_t)(s * SUB + g * 2u) * d + c0;
            float p[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) p[r] = 0.0f;
#pragma unroll 1
            for (uint32_t c = 0; c < U * 128u; c += 128u)
#pragma unroll
                for (uint32_t e = 0; e < 4u; ++e) {
                    const float w = c0 + c + e < d ? u[c0 + c + e] : 0.0f;
#pragma unroll
                    for (uint32_t r = 0; r < 2u; ++r)
                        p[r] = fmaf(s * SUB + g * 2u + r < m && c0 + c + e < d ? line[r * d + c + e] : 0.0f, w, p[r]);
                }
#pragma unroll
            for (uint32_t r = 0; r < (uint32_t)SUB; ++r)
                if (r / 2u == g) acc[r] = p[r % 2u];
        }
        const float tot = reduce8(acc, lane);
        const uint32_t row = s * SUB + (lane >> 2);
        if ((lane & 3u) == 0u && row < m)
            exchange_add(a.acc + acc_index(row), a.wide + (size_t)row * EP_WIDE_WORDS, tot);
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) atomicExch(a.claims + slice, (uint32_t)BEGUN);
    return false;
}
// One more CTA of the group that neither adds margins nor reads them any more; how many were before it.
__device__ __forceinline__ uint32_t count_out(uint32_t *header)
{
    uint32_t before;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(header + 1) : "memory");
    return before;
}
// Counted last of the group: nobody adds or reads any more.  By a warp; the accumulators that the epoch has used.
__device__ __noinline__ void leave_clear(const TileArgs &a, uint32_t lane)
{
    const uint32_t worker = blockIdx.x / a.P, mpad = SUB * a.nsub, used = min(a.nsteps, (uint32_t)EP_RING);
    uint32_t *const header = a.header + worker * EP_HEADER_WORDS;
    unsigned long long *const acc = a.acc + (size_t)worker * EP_RING * a.nsub * EP_ACC_PITCH;
    unsigned long long *const wide = a.wide + (size_t)worker * EP_RING * mpad * EP_WIDE_WORDS;
    for (uint32_t j = lane; j < used * mpad; j += 32u) {
        acc[acc_index(j)] = 0ull;    // slots follow one another at the same pitch
#pragma unroll
        for (uint32_t v = 0; v < EP_WIDE_WORDS; ++v) wide[(size_t)j * EP_WIDE_WORDS + v] = 0ull;
    }
    if (a.claims != nullptr)
        for (uint32_t j = lane; j < a.P; j += 32u) a.claims[j] = 0u;
    if (lane < 2u) header[lane] = 0u;
}
// The update of a slice that this CTA has taken over, by all its threads.
template <int U, int W>
__device__ __noinline__ void finish_slice(const TileArgs &a, uint32_t slice, const float *coef)
{
    for (uint32_t q = threadIdx.x; q < U * 128u; q += W * 32u) {
        const uint64_t c = (uint64_t)slice * (U * 128u) + q;
        if (c >= a.d) continue;
        float s = 0.0f;
        for (uint32_t v = 0; v < a.nsub_last; ++v) {
            float p = 0.0f;
            for (uint32_t r = 0; r < (uint32_t)SUB; ++r) {
                const uint32_t row = v * SUB + r;
                p = fmaf(coef[row], row < a.m_last ? a.X[(uint64_t)row * a.d + c] : 0.0f, p);
            }
            s += p;
        }
        if (a.gradient == 0u) s += a.u[c];
        a.dst[c] = s;
    }
}

// U blocks of 128 columns, W warps of eight rows each.  Shared memory: a ring of slots of eight rows (boxes of 512
// columns one after the other, the last one narrower), the slice of u, the warps' updates, the exchange's words, a
// barrier per slot, flags.  The sub-tiles (eight rows) of the epoch go round the ring; the warp that has taken one into
// registers requests the one that the slot serves next, whoever will read it.
// EX: how a worker's CTAs meet -- a group of a cooperative grid, a cluster, or a plain grid of one minibatch.
enum Exchange { GROUP = 0, CLUSTER = 1, PLAIN = 2 };
template <int U, int W, int EB, int EX>
__global__ void __launch_bounds__(W * 32, U == 1 && W == 8 ? 2 : 1)
    qesgd_lr_tile_kernel(const __grid_constant__ TileArgs a, const __grid_constant__ CUtensorMap map,
                         const __grid_constant__ CUtensorMap map_rest)
{
    constexpr bool CL = EX == CLUSTER, plain = EX == PLAIN;
    constexpr uint32_t COLS = U * 128u, SLOT = SUB * COLS;
    // The slot of the warp's own sub-tile, once that is in the registers, takes the next copy: right away where blocks
    // are wide and the ring holds little more than a minibatch, else while the margins travel.
    constexpr bool EARLY = U >= 3 && EX != PLAIN;
    float *const ring = reinterpret_cast<float *>(tl_smem);
    float *const us = reinterpret_cast<float *>(tl_smem + a.off_u);
    float *const part = reinterpret_cast<float *>(tl_smem + a.off_part);
    uint64_t *const full = reinterpret_cast<uint64_t *>(tl_smem + a.off_bars);
    // [0] a wait ran out in this CTA, [1] always zero, [2] warps that have read their last margins, [3] the CTA is
    // counted, [4 + slot] bits: 1 the slot's copy did not land in time, 2 nor did its very first one (either way no
    // other is requested)
    volatile uint32_t *const flag = reinterpret_cast<volatile uint32_t *>(tl_smem + a.off_flags);

    const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
    const uint32_t P = kept(a.P), nsteps = plain ? 1u : kept(a.nsteps), batch = kept(a.batch);
    const uint32_t nsub = kept(a.nsub), nslots = kept(a.nslots);
    const uint32_t worker = blockIdx.x / P, rank = blockIdx.x - worker * P;
    const uint32_t c0 = rank * COLS;

    if (tid < nslots) {
        mbar_init(&full[tid], EB == 16 ? 1u : 32u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid < 4u + TL_MAX_SLOTS) flag[tid] = 0u;
    if (CL)                      // no word of the exchange carries a tile's number yet
        for (uint32_t q = tid; q < 2u * P * a.x_pitch; q += W * 32u)
            reinterpret_cast<unsigned long long *>(tl_smem + a.off_x)[q] = 0ull;
    float *const kept_coef = reinterpret_cast<float *>(tl_smem + a.off_claims);
    uint32_t *const list = reinterpret_cast<uint32_t *>(kept_coef + TL_ROWS);
    if (plain && tid == 0) list[0] = 0u;
    __syncthreads();
    if (CL) cluster_arrive();    // waited for before the first store into another CTA
    if (CL || plain) qesgd_wait_for_previous();
    uint32_t taken = 0u;
    if (plain && tid == 0) taken = atomicCAS(a.claims + rank, (uint32_t)FREE, (uint32_t)BEGUN);

    const uint32_t row0 = (uint32_t)((uint64_t)worker * a.n_local);
    auto rows_of = [&](uint32_t t) { return t + 1u == nsteps ? a.m_last : batch; };
    auto subs_of = [&](uint32_t t) { return t + 1u == nsteps ? a.nsub_last : nsub; };
    // sub-tile s of minibatch t into a slot, by one warp
    auto request = [&](uint32_t slot, uint32_t t, uint32_t s) {
        const uint32_t row = row0 + t * batch + s * SUB;
        float *const dst = ring + slot * SLOT;
        if (EB == 16) {
            if (lane == 0) {
                mbar_arrive_expect_tx(&full[slot], SLOT * 4u);
#pragma unroll
                for (uint32_t b = 0; b < COLS; b += 512u)
                    tma_load_box(dst + SUB * b, b + 512u <= COLS || COLS < 512u ? &map : &map_rest, (c0 + b) / 2u, row,
                                 &full[slot]);
            }
        } else {
            constexpr uint32_t N = EB / 4;
            const uint32_t rows = min(rows_of(t) - s * SUB, (uint32_t)SUB);
            for (uint32_t r = 0; r < rows; ++r) {
                const float *const line = a.X + (uint64_t)(row + r) * a.d + c0;
#pragma unroll
                for (uint32_t e0 = 0; e0 < COLS; e0 += 32u * N) {
                    const uint32_t b = e0 & ~511u, pitch = COLS - b < 512u ? COLS - b : 512u, e = e0 + lane * N;
                    copy_elements<EB>(smem_u32(dst + SUB * b + r * pitch + (e - b)), line + e, (uint64_t)c0 + e < a.d);
                }
            }
            arrive_when_copied(&full[slot]);
        }
    };
    // a warp's rows of a landed slot into registers, zeros past the minibatch
    // (`late` in the slot's flag word if the copy did not land in time)
    float4 x[U][SUB];
    auto take = [&](bool landed, uint32_t slot, uint32_t parity, uint32_t rows, uint32_t late) {
        if (!landed && __builtin_expect(!mbar_wait(&full[slot], parity, &flag[0], a.wait_ns), 0)) {
            flag[0] = 1u;
            flag[4u + slot] = flag[4u + slot] | late;
        }
        const float *const from = ring + slot * SLOT + lane * 4u;
#pragma unroll
        for (uint32_t it = 0; it < U; ++it) {
            const uint32_t b = it * 128u & ~511u, pitch = COLS - b < 512u ? COLS - b : 512u;
#pragma unroll
            for (uint32_t r = 0; r < (uint32_t)SUB; ++r)
                x[it][r] = *reinterpret_cast<const float4 *>(from + SUB * b + (it * 128u - b) + r * pitch);
        }
        if (rows < (uint32_t)SUB) {
#pragma unroll
            for (uint32_t r = 0; r < (uint32_t)SUB; ++r)
                if (r >= rows)
#pragma unroll
                    for (int it = 0; it < U; ++it) x[it][r] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };

    // The first turn of the ring: slot n holds sub-tile n.  The warp's first two now, the rest once the first step is
    // under way.
    uint32_t slot = w, parity = 0u;
    if (w < subs_of(0u)) request(w, 0u, w);
    // and which sub-tile follows the warp's own of minibatch t in its slot: sub-tile next_s of minibatch t + next_t
    uint32_t next_s = w + nslots % nsub, next_t = nslots / nsub;
    if (next_s >= nsub) {
        next_s -= nsub;
        ++next_t;
    }
    const uint32_t my_row = w * SUB + (lane >> 2);         // of the minibatch; lanes 4r to 4r + 3 end with row r's sum
    const float *label = a.y + (uint64_t)row0 + my_row;
    float yj = w < nsub && my_row < rows_of(0u) ? __ldg(label) : 0.0f;
    constexpr uint32_t UPT = (COLS + W * 32u - 1u) / (W * 32u);
    float u0[UPT];
#pragma unroll
    for (uint32_t e = 0; e < UPT; ++e) {
        const uint64_t c = (uint64_t)c0 + tid + e * W * 32u;
        u0[e] = tid + e * W * 32u < COLS && c < a.d ? a.u[(uint64_t)worker * a.u_stride + c] : 0.0f;
    }
    if (w < nsub && w + nsub < nslots && nsteps > 1u && w < subs_of(1u)) request(w + nsub, 1u, w);
#pragma unroll
    for (uint32_t e = 0; e < UPT; ++e)
        if (tid + e * W * 32u < COLS) us[tid + e * W * 32u] = u0[e];
    if (CL) cluster_wait();
    if (w < subs_of(0u)) take(false, slot, 0u, rows_of(0u) - w * SUB, 2u);
    if (!plain) {
        __syncthreads();
    } else if (__syncthreads_or((int)taken) != 0) {               // another CTA does this slice
        // every copy requested has been taken, or was late and is waited for here as at the end
        if (tid < nslots && flag[4u + tid] != 0u) mbar_wait(&full[tid], 0u, &flag[1], DRAIN_LIMIT_NS);
        uint32_t before = 0u;
        if (tid == 0) before = count_out(a.header);
        if (w == 0u && __shfl_sync(0xFFFFFFFFu, before, 0) == P - 1u) leave_clear(a, lane);
        return;
    }

    const uint32_t mpad = SUB * nsub;
    unsigned long long *const acc_g = a.acc + (size_t)worker * EP_RING * nsub * EP_ACC_PITCH + acc_index(my_row);
    unsigned long long *const wide_g = a.wide + ((size_t)worker * EP_RING * mpad + my_row) * EP_WIDE_WORDS;
    uint32_t *const header = a.header + worker * EP_HEADER_WORDS;
    // the exchange's words: where this lane's go in another CTA, and where it reads (minibatches of odd number: + odd)
    const uint32_t pitch = kept(a.x_pitch * 8u), words = smem_u32(tl_smem + a.off_x), odd = kept(P * pitch);
    const uint32_t send_r = send_row(P, lane), to_rank = send_rank(P, lane);
    const uint32_t send_to =
        !CL || to_rank >= P ? 0u : cluster_address(words + rank * pitch + (w * SUB + send_r) * 8u, to_rank);
    const uint32_t read_at = words + (lane & 3u) * pitch + my_row * 8u;
    auto refill = [&](uint32_t t, uint32_t late) {
        __syncwarp();            // every lane's rows are in its registers
        if ((!EARLY || (flag[4u + slot] & late) == 0u) && t + next_t < nsteps && next_s < subs_of(t + next_t))
            request(slot, t + next_t, next_s);
    };
    if (EARLY && w < subs_of(0u)) refill(0u, 2u);          // (bit 1 here would be the next turn's, by another warp)
    bool gave_up = false;
    uint32_t gave_up_at = 0u, clears = 0u;
    uint32_t counted = ~0u;                                // by the warp that counted the CTA: how many were before it
    const uint32_t m_last = kept(a.m_last), nsub_last = kept(a.nsub_last);
    uint32_t t = 0u, m = nsteps == 1u ? m_last : batch, subs = nsteps == 1u ? nsub_last : nsub;
    float ry = (nsteps == 1u ? a.rate_last : a.rate) * yj;
    bool signal = blockIdx.x != a.drop_cta;
    // The first copy is not there: nothing goes out, the block leaves this step.  (The hint is worth 4 % to clusters fed
    // by TMA, K = 7, n = 1075, d = 1228, batch 100 26.3 -> 25.3 us, and costs the others 2 to 8: K = 3, n = 530,
    // d = 1611, batch 128 15.8 -> 17.7, gradient of 64 x 24780 5.08 -> 5.26.)
    const bool missing = (flag[4u + slot] & 2u) != 0u;
    if (CL && EB == 16 ? __builtin_expect(missing, 0) : missing) {
        signal = false;
        if (!EARLY) next_t = nsteps;       // no refill (EARLY: refused above)
    }

    for (;;) {
        const bool last = t + 1u == nsteps;
        unsigned long long *const acc_t = acc_g + (size_t)(t % EP_RING) * nsub * EP_ACC_PITCH;
        unsigned long long *const wide_t = wide_g + (size_t)(t % EP_RING) * mpad * EP_WIDE_WORDS;
        const uint32_t side = t & 1u ? odd : 0u;
        if (w < subs) {
            // ---- M
            float acc[SUB];
#pragma unroll
            for (int r = 0; r < SUB; ++r) acc[r] = 0.0f;
#pragma unroll
            for (int it = 0; it < U; ++it) {
                const float4 uu = *reinterpret_cast<const float4 *>(us + it * 128 + lane * 4u);
#pragma unroll
                for (int r = 0; r < SUB; ++r) {
                    acc[r] = fmaf(x[it][r].x, uu.x, acc[r]);
                    acc[r] = fmaf(x[it][r].y, uu.y, acc[r]);
                    acc[r] = fmaf(x[it][r].z, uu.z, acc[r]);
                    acc[r] = fmaf(x[it][r].w, uu.w, acc[r]);
                }
            }
            const float tot = reduce8(acc, lane);
            // ---- X
            if (CL) {
                if (signal) cluster_send(send_to + side, send_r, tot, t + 1u, P, lane);
            } else if ((lane & 3u) == 0u && my_row < m && signal) {
                exchange_add(acc_t, wide_t, tot);
            }
            if (!EARLY) refill(t, 0u);
            if (t == 0u)         // the rest of the ring's first turn
                for (uint32_t n = w + 2u * nsub, v = 2u; n < nslots && v < nsteps; n += nsub, ++v)
                    if (w < subs_of(v)) request(n, v, w);
        }
        // the next minibatch, as far as it can be seen to now
        uint32_t next_slot = slot + nsub, next_parity = parity;
        if (next_slot >= nslots) {
            next_slot -= nslots;
            next_parity ^= 1u;
        }
        const uint32_t next_m = t + 2u == nsteps ? m_last : batch, next_subs = t + 2u == nsteps ? nsub_last : nsub;
        const bool more = !last && w < next_subs;
        const float next_y = more && my_row < next_m ? __ldg(label + batch) : 0.0f;
        const bool landed = more && mbar_try_wait(&full[next_slot], next_parity);
        if (!CL && rank == clears && t + EP_RING / 2 < nsteps) {     // clears what minibatch t + RING/2 will add to
            const uint32_t zs = (t + EP_RING / 2) % EP_RING;
            unsigned long long *const az = a.acc + ((size_t)worker * EP_RING + zs) * nsub * EP_ACC_PITCH;
            unsigned long long *const wz = a.wide + ((size_t)worker * EP_RING + zs) * mpad * EP_WIDE_WORDS;
            for (uint32_t j = W * 32u - 1u - tid; j < mpad; j += W * 32u) {
                az[acc_index(j)] = 0ull;
#pragma unroll
                for (uint32_t v = 0; v < EP_WIDE_WORDS; ++v) wz[(size_t)j * EP_WIDE_WORDS + v] = 0ull;
                __threadfence();     // cleared for every CTA before this thread goes on
            }
        }
        if (w < subs) {
            float margin = 0.0f;
            uint32_t looks = 0u;
            uint64_t t0 = 0u;
            auto give_up = [&]() {   // asked after every look that did not find everything
                if (looks == 0u) t0 = now_ns();
                if ((++looks & a.poll_mask) == 0u &&
                    (flag[0] != 0u || (!CL && ld_acquire(header) != 0u) || expired(t0, a.wait_ns))) {
                    flag[0] = 1u;
                    return true;
                }
                return false;
            };
            if (CL) {
                // lane 4r + q reads row r's words of the ranks q, q + 4, q + 8, q + 12
                float v[4];
                for (;;) {
                    bool all = true;
#pragma unroll
                    for (uint32_t e = 0; e < 4u; ++e) {
                        uint32_t tag = t + 1u;
                        v[e] = 0.0f;
                        if ((lane & 3u) + 4u * e < P) cluster_load(read_at + side + e * 4u * pitch, v[e], tag);
                        all &= tag == t + 1u;
                    }
                    if (all || give_up()) break;
                }
                // every addition with its error, so that the sum is rounded once
                float s, e, s1, e1, d;
                two_sum(v[0], v[1], s, e);
                two_sum(v[2], v[3], s1, e1);
                e += e1;
                two_sum(s, s1, s, d);
                e += d;
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    s1 = __shfl_xor_sync(0xFFFFFFFFu, s, o);
                    e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
                    two_sum(s, s1, s, d);
                    e += d;
                }
                margin = fabsf(s) <= 3.402823466e38f ? s + e : s;   // the errors of an infinite sum are NaN
            } else if (!plain) {
                if ((lane & 3u) == 0u && my_row < m) {
                    unsigned long long v;
                    while (((v = ld_relaxed(acc_t)) >> 55) < P)
                        if (give_up()) break;
                    margin = exchange_margin(v, wide_t, P);
                }
            } else {
                // the warp together, so that it can take over a slice
                unsigned long long v = 0ull;
                bool done = (lane & 3u) != 0u || my_row >= m;
                const bool reads = !done;
                bool begun = false;          // every slice: from then on the limit counts
                for (;;) {
                    for (uint32_t n = 0; !done && n <= a.poll_mask; ++n) done = ((v = ld_relaxed(acc_t)) >> 55) >= P;
                    if (__all_sync(0xFFFFFFFFu, done)) break;
                    if (looks++ == 0u) t0 = now_ns();
                    const bool stop = flag[0] != 0u || ld_acquire(header) != 0u || (begun && expired(t0, a.wait_ns));
                    if (__any_sync(0xFFFFFFFFu, stop)) {
                        flag[0] = 1u;
                        break;
                    }
                    const bool due = __any_sync(0xFFFFFFFFu, now_ns() - t0 > TL_STEAL_NS) != 0;
                    if (!begun && (due || __any_sync(0xFFFFFFFFu, expired(t0, a.wait_ns)) != 0)) {
                        begun = take_over<U>(a, list, due, lane) ||
                                __any_sync(0xFFFFFFFFu, now_ns() - t0 > TL_BEGIN_NS) != 0;
                        if (begun) t0 = now_ns();
                    }
                }
                if (reads) margin = exchange_margin(v, wide_t, P);
            }
            // -(lr/m) * c_j with c_j = -y_j / (1 + exp(y_j m_j))
            const float cj = my_row < m ? ry / (1.0f + expf(yj * margin)) : 0.0f;
            if (plain && (lane & 3u) == 0u) kept_coef[my_row] = cj;
            __syncwarp();
            if (!CL && last && lane == 0) {                // the last warp counts the CTA
                __threadfence_block();
                if (atomicAdd(const_cast<uint32_t *>(&flag[2]), 1u) == subs - 1u) {
                    flag[3] = 1u;
                    if (flag[0] != 0u) atomicExch(header, 1u);   // gave up: so shall the others
                    counted = count_out(header);
                }
            }
            // ---- U
            float cs[SUB];
#pragma unroll
            for (int r = 0; r < SUB; ++r) cs[r] = __shfl_sync(0xFFFFFFFFu, cj, 4 * r);
#pragma unroll
            for (int it = 0; it < U; ++it) {
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int r = 0; r < SUB; ++r) {
                    s.x = fmaf(cs[r], x[it][r].x, s.x);
                    s.y = fmaf(cs[r], x[it][r].y, s.y);
                    s.z = fmaf(cs[r], x[it][r].z, s.z);
                    s.w = fmaf(cs[r], x[it][r].w, s.w);
                }
                *reinterpret_cast<float4 *>(part + w * COLS + it * 128 + lane * 4u) = s;
            }
        }
        slot = next_slot;
        parity = next_parity;
        if (more) {
            take(landed, slot, parity, next_m - w * SUB, 1u);
            if (EARLY) refill(t + 1u, 3u);
        }
        if (sync_any(1u, W * 32u, flag[0])) {
            gave_up = true;
            gave_up_at = t;
            break;
        }
        // ---- A (N columns a thread, so that the block needs one round)
        constexpr uint32_t N = COLS <= W * 32u ? 1u : (COLS <= W * 64u ? 2u : 4u);
        const uint32_t c = tid * N;
        if (c < COLS) {
            float s[N];
#pragma unroll
            for (uint32_t e = 0; e < N; ++e) s[e] = 0.0f;
#pragma unroll
            for (uint32_t v = 0; v < (uint32_t)W; ++v)
                if (v < subs) {
                    float p[N];
                    load_n<N>(part + v * COLS + c, p);
#pragma unroll
                    for (uint32_t e = 0; e < N; ++e) s[e] += p[e];
                }
#pragma unroll
            for (uint32_t e = 0; e < N; ++e) {
                if (a.gradient == 0u) s[e] += us[c + e];
                us[c + e] = s[e];
                if (last && (uint64_t)c0 + c + e < a.d) a.dst[(uint64_t)worker * a.u_stride + c0 + c + e] = s[e];
            }
        }
        if (last) {
            if constexpr (plain)
                for (uint32_t n = 0; n < list[0]; ++n) finish_slice<U, W>(a, list[1u + n], kept_coef);
            break;
        }
        asm volatile("bar.sync 2, %0;" ::"n"(W * 32) : "memory");   // u complete for the next minibatch
        ++t;
        m = next_m;
        subs = next_subs;
        yj = next_y;
        ry = (t + 1u == nsteps ? a.rate_last : a.rate) * yj;
        label += batch;
        signal = true;
        if (!CL && ++clears == P) clears = 0u;
    }

    if (gave_up) {
        if (tid == 0) atomicOr(a.status, QESGD_STATUS_TIMEOUT);
        // Every slot's last copy has landed before the block ends, so that none is on its way into memory that another
        // block then owns.  Sub-tile n goes to slot n % nslots, and all below `requested` have been requested, but for
        // those that would have followed a late one: `next` is the minibatch taken last.
        const uint32_t total = (nsteps - 1u) * nsub + nsub_last, next = min(gave_up_at + EARLY, nsteps - 1u);
        const uint32_t requested = min(total, (gave_up_at + EARLY) * nsub + subs_of(next) + nslots);
        for (uint32_t q = tid; q < nslots && q < requested; q += W * 32u) {
            const uint32_t late = flag[4u + q];
            const uint32_t before = EARLY && late != 0u ? next * nsub + nslots - 1u - q : requested - 1u - q;
            const uint32_t turn = late & 2u ? 0u : before / nslots;
            mbar_wait(&full[q], turn & 1u, &flag[1], DRAIN_LIMIT_NS);
        }
        if (CL) {
            cluster_arrive();
            cluster_wait();
        } else if (tid == 0 && flag[3] == 0u) {
            atomicExch(header, 1u);
            counted = count_out(header);
        }
    }
    if (CL) return;
    __syncwarp();
    if (__shfl_sync(0xFFFFFFFFu, counted, 0) == P - 1u) leave_clear(a, lane);
}

// ------------------------------------------------------------------ host ----
typedef void (*TileKernel)(TileArgs, CUtensorMap, CUtensorMap);
struct Variant {
    uint32_t U, W;
    TileKernel kernel[3][3];     // by Exchange; copies of 16 (TMA), 8, 4 bytes
};
#define TL_COPIES(U, W, EX) \
    {qesgd_lr_tile_kernel<U, W, 16, EX>, qesgd_lr_tile_kernel<U, W, 8, EX>, qesgd_lr_tile_kernel<U, W, 4, EX>}
#define TL_VARIANT(U, W) {U, W, {TL_COPIES(U, W, GROUP), TL_COPIES(U, W, CLUSTER), TL_COPIES(U, W, PLAIN)}}
// Registers: 32 U for the rows.  A block of eight warps has 255 a thread, one of sixteen 128.  (Six blocks of columns
// spill: a gradient of 64 x 100000 10.4 us against 10.3 for the other kernel.)
const Variant VARIANTS[] = {TL_VARIANT(1, 8), TL_VARIANT(2, 8), TL_VARIANT(3, 8), TL_VARIANT(4, 8),
                            TL_VARIANT(5, 8), TL_VARIANT(1, 16), TL_VARIANT(2, 16)};
constexpr uint32_t NVARIANTS = sizeof(VARIANTS) / sizeof(VARIANTS[0]);

constexpr int MAX_DEVICES = 64;
std::mutex g_tile_mutex;
bool g_tile_ready[MAX_DEVICES] = {false};
uint32_t g_room[MAX_DEVICES][NVARIANTS][5];      // clusters of 1, 2, 4, 8, 16 CTAs that are resident at once

cudaLaunchConfig_t cluster_config(uint32_t ctas, uint32_t P, uint32_t threads, uint32_t bytes, cudaStream_t stream,
                                  cudaLaunchAttribute (&at)[2])
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(ctas);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = bytes;
    c.stream = stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = P;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 2;
    return c;
}

// Shared memory of a block; a block of one unit and eight warps takes less than half of an SM's.
uint32_t budget(const Variant &v, uint32_t limit) { return v.U == 1u && v.W == 8u ? limit / 2u - 2048u : limit; }

struct Plan {
    const Variant *v;
    uint32_t P, exchange, nslots, bytes, x_pitch;
    uint32_t off_u, off_part, off_x, off_bars, off_flags, off_claims;
};
bool lay_out(Plan &p, uint32_t nsub, uint64_t subtiles, uint32_t limit)
{
    const uint32_t cols = p.v->U * 128u, slot = SUB * cols * 4u;
    p.x_pitch = SUB * nsub + (nsub % 2u ? 12u : 4u);
    const uint32_t xbytes = p.exchange == CLUSTER ? 2u * p.P * p.x_pitch * 8u : 0u;
    const uint32_t cbytes = p.exchange == PLAIN ? (TL_ROWS + 1u + 256u) * 4u : 0u;
    const uint32_t fixed =
        cols * 4u + p.v->W * cols * 4u + xbytes + TL_MAX_SLOTS * 8u + (4u + TL_MAX_SLOTS) * 4u + cbytes;
    const uint32_t have = budget(*p.v, limit);
    if (fixed + nsub * slot > have) return false;
    p.nslots = (have - fixed) / slot;
    if (p.nslots > TL_MAX_SLOTS) p.nslots = TL_MAX_SLOTS;
    if (p.nslots > subtiles) p.nslots = (uint32_t)(subtiles < nsub ? nsub : subtiles);
    p.off_u = p.nslots * slot;
    p.off_part = p.off_u + cols * 4u;
    p.off_x = p.off_part + p.v->W * cols * 4u;
    p.off_bars = p.off_x + xbytes;
    p.off_flags = p.off_bars + TL_MAX_SLOTS * 8u;
    p.off_claims = p.off_flags + (4u + TL_MAX_SLOTS) * 4u;
    p.bytes = p.off_claims + cbytes;
    return true;
}

bool prepare_device(int device, uint32_t limit)
{
    if (device < 0 || device >= MAX_DEVICES) return false;
    std::lock_guard<std::mutex> lock(g_tile_mutex);
    if (g_tile_ready[device]) return true;
    for (uint32_t i = 0; i < NVARIANTS; ++i) {
        for (uint32_t j = 0; j < 9u; ++j) {
            const void *const k = (const void *)VARIANTS[i].kernel[j / 3u][j % 3u];
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess ||
                (j / 3u == CLUSTER &&
                 cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
                cudaGetLastError();
                return false;
            }
        }
        for (uint32_t l = 0; l < 5u; ++l) {
            cudaLaunchAttribute at[2];
            const cudaLaunchConfig_t c =
                cluster_config(1u << l, 1u << l, VARIANTS[i].W * 32u, budget(VARIANTS[i], limit), nullptr, at);
            int n = 0, least = 1 << 30;
            for (const TileKernel k : VARIANTS[i].kernel[CLUSTER]) {
                if (cudaOccupancyMaxActiveClusters(&n, k, &c) != cudaSuccess) {
                    cudaGetLastError();
                    n = 0;
                }
                least = n < least ? n : least;
            }
            g_room[device][i][l] = (uint32_t)least;
        }
    }
    g_tile_ready[device] = true;
    return true;
}

// Modelled time of an epoch in us (measured over some 20 shapes, see below): a step's chain, the copies, the launch.
// A chain costs 0.85 us in a cluster and 1.3 through global memory, and for each block of 128 columns 0.03 and 0.026
// for each eight rows; element-wise copies are issued by the warps themselves, and sixteen warps meet later than eight.
// HBM is not reached where the ring holds little more than a minibatch (U > 2).  A cluster is launched with the kernel
// before it still draining; a cooperative grid is not.  Clusters that take turns cost a fifth more than a turn each.
float modelled_us(const Plan &p, const QesgdTileCall &q, uint32_t nsub, uint32_t waves)
{
    const float hbm = (float)((double)q.K * q.m * q.d * 4.0 / 6.5e6), U = (float)p.v->U, rows = (float)nsub;
    const float copy = q.copy == 16 ? 0.0f : (q.copy == 8 ? 0.045f : 0.085f) * U * rows;
    const float turn =
        (p.exchange == CLUSTER ? 0.85f : 1.3f) + U * (0.03f + 0.026f * rows) + copy + (p.v->W == 16u ? 0.3f : 0.0f);
    const float chain = (waves > 1u ? 1.2f * (float)waves : 1.0f) * turn;
    const float fetch = hbm * (p.v->U > 2u ? 1.3f : 1.1f);
    const float start = p.exchange != GROUP ? 2.0f * (float)waves - 0.5f : (p.v->U > 2u ? 5.0f : 4.0f);
    return (float)q.nsteps * (chain > fetch ? chain : fetch) + start;
}

}  // namespace

// Which kernel.  Both times are modelled (the other kernel's by qesgd_lr_epoch.cu, within a quarter of what it takes).
// Measured, whole epochs back to back, other kernel -> this one:
//   K = 4, n = 128, d = 4096, batch 32 (cluster of 16, two blocks): 14.4 -> 7.0 us
//   K = 4, n = 1000, d = 1000, batch 32 (8, one): 71.8 -> 34.1
//   K = 2, n = 800, d = 300, batch 64 (4, one): 41.0 -> 16.6
//   K = 8, n = 500, d = 2000, batch 100 (8, two, sixteen warps): 28.7 -> 12.4
//   K = 8, n = 2000, d = 128, batch 16 (one CTA): 271 -> 126;  one gradient of 64 x 4096 (16, two): 6.7 -> 3.5
//   gradients of 64 x 65536 (128 CTAs, four): 8.2 -> 6.2
//   K = 1, n = 1010, d = 10000, batch 50 (79 CTAs of a group, one): 44.7 -> 36.9
//   K = 8 of them (16, five): 80.8 -> 71.1
//   K = 4, n = 1000, d = 16384, batch 32 (32 CTAs, four): 89.5 -> 72.3
// Where it loses and is not taken: more clusters than the device holds at once (K = 16, n = 200, d = 8000, batch 64:
// 32.5 in three turns against 28.7); element-wise copies of many columns (K = 6, n = 700, d = 8003, batch 50: 57
// against 49).
// A cluster starts when one GPC has its SMs free: one of 16 beside up to 48 held SMs at once, beside 64 after them (one
// of 8 beside 100, not beside 130).
int qesgd_launch_lr_tile(const QesgdTileCall &q, uint32_t smem_limit, float other_us, int *launched,
                         uint32_t (&plan)[8])
{
    const uint32_t nsub = (q.m + SUB - 1u) / SUB, W = nsub <= 8u ? 8u : 16u;
    if (nsub > 16u || !prepare_device(q.device, smem_limit)) return -1;
    Plan p = {};
    float best = other_us * (float)q.nsteps + 4.0f;
    for (uint32_t i = 0; i < NVARIANTS; ++i) {
        const Variant &v = VARIANTS[i];
        if (v.W != W) continue;
        const uint64_t need = (q.d + v.U * 128u - 1u) / (v.U * 128u);        // CTAs that hold a row
        for (const uint32_t exchange : {(uint32_t)CLUSTER, (uint32_t)(q.nsteps * q.K == 1u ? PLAIN : GROUP)}) {
            Plan c = {};
            c.v = &v;
            c.exchange = exchange;
            uint32_t waves = 1u;
            if (exchange == CLUSTER) {
                uint32_t l = 0;
                while ((1u << l) < need && l < 5u) ++l;
                if (l > 4u || g_room[q.device][i][l] == 0u) continue;
                c.P = 1u << l;
                waves = (q.K + g_room[q.device][i][l] - 1u) / g_room[q.device][i][l];
            } else {
                // all CTAs at once, the accumulators of all groups in the workspace; a lone CTA exchanges nothing
                if (need * q.K > q.sms || q.K * nsub * SUB > QESGD_LR_EPOCH_ROWS || need < 2u) continue;
                c.P = (uint32_t)need;
            }
            const float us = modelled_us(c, q, nsub, waves);
            if (us < best && lay_out(c, nsub, q.nsteps * nsub, smem_limit)) {
                best = us;
                p = c;
            }
        }
    }
    if (!p.v) return -1;

    TileArgs a = {};
    a.X = q.X; a.y = q.y; a.n_local = q.n_local; a.d = q.d;
    a.P = p.P;
    a.batch = q.m; a.nsteps = (uint32_t)q.nsteps;
    a.m_last = (uint32_t)(q.n_local - (q.nsteps - 1) * q.m);
    a.nsub = nsub; a.nsub_last = (a.m_last + SUB - 1u) / SUB;
    a.nslots = p.nslots;
    a.off_u = p.off_u; a.off_part = p.off_part; a.off_x = p.off_x; a.off_bars = p.off_bars; a.off_flags = p.off_flags;
    a.x_pitch = p.x_pitch;
    a.rate = q.lr / (float)q.m; a.rate_last = q.lr / (float)a.m_last;
    a.u = q.u; a.dst = q.dst; a.gradient = q.gradient ? 1u : 0u; a.u_stride = q.u_stride;
    a.header = q.header; a.acc = q.acc; a.wide = q.wide;
    a.status = q.status; a.wait_ns = q.wait_ns; a.poll_mask = q.wait_ns < COARSE_TIMER_NS ? 0u : 31u;
    a.drop_cta = q.drop_cta;
    // in the headers of other workers' groups, of which there are none
    a.claims = p.exchange == PLAIN ? q.header + EP_HEADER_WORDS : nullptr;
    a.off_claims = p.off_claims;
    static_assert(QESGD_MAX_WORKERS * EP_HEADER_WORDS >= EP_HEADER_WORDS + 256u, "a word for each CTA");
    CUtensorMap map = {}, map_rest = {};
    const uint32_t cols = p.v->U * 128u, rest = cols > 512u ? cols - 512u : cols;
    const uint64_t rows = (uint64_t)q.K * q.n_local;
    if (q.copy == 16 && !qesgd_lr_tensor_map(&map, q.X, rows, q.d, cols < 512u ? cols : 512u, true)) return -1;
    if (q.copy == 16 && cols > 512u && !qesgd_lr_tensor_map(&map_rest, q.X, rows, q.d, rest, true)) return -1;
    const TileKernel kernel = p.v->kernel[p.exchange][q.copy == 16 ? 0 : (q.copy == 8 ? 1 : 2)];
    const uint32_t threads = W * 32u;
    cudaError_t err;
    if (p.exchange == CLUSTER) {
        cudaLaunchAttribute at[2];
        const cudaLaunchConfig_t c = cluster_config(q.K * p.P, p.P, threads, p.bytes, q.stream, at);
        err = cudaLaunchKernelEx(&c, kernel, a, map, map_rest);
    } else if (p.exchange == PLAIN) {
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t c = cluster_config(p.P, 1u, threads, p.bytes, q.stream, at);
        at[0] = at[1];           // no cluster
        c.numAttrs = 1;
        err = cudaLaunchKernelEx(&c, kernel, a, map, map_rest);
    } else {
        void *params[] = {(void *)&a, (void *)&map, (void *)&map_rest};
        err = cudaLaunchCooperativeKernel((const void *)kernel, dim3(q.K * p.P), dim3(threads), params, p.bytes,
                                          q.stream);
    }
    if (err == cudaErrorCooperativeLaunchTooLarge || err == cudaErrorLaunchOutOfResources ||
        err == cudaErrorInvalidConfiguration || err == cudaErrorNotSupported || err == cudaErrorInvalidClusterSize) {
        cudaGetLastError();
        return -1;
    }
    if (err != cudaSuccess) return (int)err;
    *launched = 1;
    const uint32_t kind =
        p.exchange == PLAIN ? QESGD_LR_PLAIN : (p.exchange == CLUSTER ? QESGD_LR_CLUSTER : QESGD_LR_GROUP);
    const uint32_t shape[8] = {kind, p.P, cols, W, p.nslots, (uint32_t)q.copy, q.K * p.P, 1u};
    for (int i = 0; i < 8; ++i) plan[i] = shape[i];
    return 0;
}
