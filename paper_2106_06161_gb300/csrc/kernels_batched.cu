// Many independent shuffles in one persistent launch.
//
// Every instance t (its own input, output, length n_t and seed) is cut into
// tiles of the same size as the plain element kernel's.  The tiles of all
// instances form one global sequence, instance after instance, handed out by
// a global ticket to a grid of persistent CTAs (a few per SM).  A CTA maps its
// ticket to (instance, tile) by a warp-cooperative search of the tile prefix
// table, derives the instance's round keys from its seed, and runs the same
// fused pipeline as the plain kernel: bijection, gather, in-tile scan, and a
// decoupled look-back that stops at the instance's first tile.  The output of
// each instance is exactly that of a plain call with the same arguments.
//
// A small planning kernel (one CTA) runs first: it validates the descriptors,
// computes every instance's domain exponent and tile count, and scans the
// tile counts.
#include <atomic>
#include <cstdint>

#include "bshuffle_device.cuh"
#include "bshuffle_internal.h"

namespace bsh {
namespace {

using dev::kFull;

// CTA shape of the persistent kernel (overridable at build time for tuning
// experiments): threads, domain indices per thread, and the resident CTAs
// per SM that the register budget targets for elements of up to 4 bytes
// (8- and 16-byte elements hold more live data and target fewer).
#ifndef BSHUFFLE_BATCH_BLOCK
#define BSHUFFLE_BATCH_BLOCK 256
#endif
#ifndef BSHUFFLE_BATCH_ITEMS
#define BSHUFFLE_BATCH_ITEMS 8
#endif
#ifndef BSHUFFLE_BATCH_MIN_CTAS
#define BSHUFFLE_BATCH_MIN_CTAS 5
#endif
constexpr int kBBlock = BSHUFFLE_BATCH_BLOCK;
constexpr int kBItems = BSHUFFLE_BATCH_ITEMS;
constexpr int kBMinCtas = BSHUFFLE_BATCH_MIN_CTAS;
constexpr int min_ctas_for(unsigned elem_bytes)
{
    return elem_bytes <= 4 ? kBMinCtas : (elem_bytes == 8 ? (kBMinCtas > 3 ? 3 : kBMinCtas) : 2);
}
constexpr uint32_t kTile = kBBlock * kBItems;
constexpr uint32_t kRingShift = 16;
constexpr uint64_t kRingWords = uint64_t{1} << kRingShift;
constexpr int kPlanThreads = 1024;
// Tags are 31 bits, and a launch uses at most 2^16 (2^32 tiles) past its first.
constexpr uint32_t kMaxBatchTag = 0x7ffe0000u;
constexpr int kErrInvalid = -10;
constexpr int kErrAlign = -6;

__device__ __forceinline__ uint32_t domain_bits_dev(uint64_t n)
{
    if (n == 0) return 0;
    const uint32_t k = 64u - static_cast<uint32_t>(__clzll(n - 1));  // ceil(log2 n) for n >= 2
    return n == 1 ? 4u : (k < 4u ? 4u : k);
}

// Checks one descriptor and returns its tiles (0 for an empty or bad one).
__device__ __forceinline__ uint32_t plan_instance(const BatchArgs &a, uint32_t t, uint32_t &k)
{
    const BatchDesc d = a.descs[t];
    k = domain_bits_dev(d.n);
    if (d.n > 4294967295ull) {
        dev::record_error(a.ws, kErrInvalid, t);
        k = 0;
    } else if (d.n > 0 && (d.in == nullptr || d.out == nullptr)) {
        dev::record_error(a.ws, kErrInvalid, t);
        k = 0;
    } else if (d.n > 0) {
        const uint64_t al = a.elem_bytes < 16u ? a.elem_bytes : 16u;
        if (reinterpret_cast<uintptr_t>(d.in) % al != 0 || reinterpret_cast<uintptr_t>(d.out) % al != 0) {
            dev::record_error(a.ws, kErrAlign, t);
            k = 0;
        }
    }
    return k == 0 ? 0u : static_cast<uint32_t>(((uint64_t{1} << k) + a.tile - 1) / a.tile);
}

// One CTA; each warp owns a run of consecutive instances and walks it 32 at a
// time (coalesced): once for the tile counts, and, with the warps' totals
// scanned, once more for the prefixes.  Bound by latency: 4,096 instances
// 23 -> 12 us (clearing the look-back ring here and a 20-barrier scan
// took most of it), 100,000 instances 363 -> 225 us.
__global__ void __launch_bounds__(kPlanThreads) batch_plan_kernel(const __grid_constant__ BatchArgs a)
{
    constexpr uint32_t kWarps = kPlanThreads / 32;
    __shared__ uint64_t s_sums[kWarps];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t rows = (a.count + 31u) / 32u;  // of 32 instances
    const uint32_t per = (rows + kWarps - 1u) / kWarps;
    const uint32_t row0 = warp * per < rows ? warp * per : rows;
    const uint32_t row1 = row0 + per < rows ? row0 + per : rows;
    uint64_t sum = 0;
#pragma unroll 4
    for (uint32_t row = row0; row < row1; ++row) {
        const uint32_t t = row * 32u + lane;
        if (t < a.count) {
            uint32_t k;
            const uint32_t tiles = plan_instance(a, t, k);
            a.plan[t].k = k;
            a.plan[t].tiles = tiles;
            sum += tiles;
        }
    }
    const uint64_t incl = dev::warp_inclusive_scan64(sum);
    if (lane == 31u) s_sums[warp] = incl;
    __syncthreads();
    if (warp == 0u) {
        const uint64_t mine = s_sums[lane];
        const uint64_t all = dev::warp_inclusive_scan64(mine);
        s_sums[lane] = all - mine;
        if (lane == 31u) {
            uint64_t total = all;
            if (total > 0xfff00000ull) {  // tickets are 32-bit
                dev::record_error(a.ws, kErrInvalid, total);
                total = 0;
            }
            a.tile_prefix[a.count] = total;
            *a.total_tiles = total;
        }
    }
    __syncthreads();
    uint64_t run = s_sums[warp];
    for (uint32_t row = row0; row < row1; ++row) {
        const uint32_t t = row * 32u + lane;
        const uint64_t tiles = t < a.count ? a.plan[t].tiles : 0u;  // written by this thread
        const uint64_t upto = dev::warp_inclusive_scan64(tiles);
        if (t < a.count) {
            a.plan[t].first_tile = run + upto - tiles;
            a.tile_prefix[t] = run + upto - tiles;
        }
        run += __shfl_sync(kFull, upto, 31);
    }
}

// The look-back ring of a launch: its passes over the ring carry the tags
// after the ones of the launches before it on the stream, so nothing is
// cleared per launch.
__device__ __forceinline__ dev::StatusRing batch_ring(const BatchArgs &a)
{
    return dev::StatusRing{a.status, kRingWords - 1, kRingShift, dev::ld_relaxed_gpu(&a.ws->batch_tag)};
}

// Called by one thread per CTA once the CTA no longer uses the ring: the last
// one readies the header for the next launch and steps the tags past this
// launch's (and clears the ring before they would run out).
__device__ __forceinline__ void finish_batch(const BatchArgs &a, const dev::StatusRing &ring, uint64_t total)
{
    __threadfence();
    const uint32_t d = atomicAdd(&a.ws->batch_done, 1u);
    if (d != gridDim.x - 1u) return;
    __threadfence();
    uint32_t tag = ring.base_tag + static_cast<uint32_t>(total >> kRingShift) + 1u;
    if (tag > kMaxBatchTag) {
        for (uint64_t w = 0; w < kRingWords; ++w) dev::st_relaxed_gpu(a.status + w, 0ull);
        tag = 1u;
    }
    atomicExch(&a.ws->batch_ticket, 0u);
    atomicExch(&a.ws->batch_done, 0u);
    atomicExch(&a.ws->batch_tag, tag);
    __threadfence();
}

// The instance owning global tile g: the largest t in [lo, hi) with
// tile_prefix[t] <= g, given tile_prefix[lo] <= g.  Warp-cooperative.  The
// first probe reads the 32 entries after lo (one coalesced load): a CTA's
// successive tickets are a grid's width apart, so the owner of its next
// ticket is usually among the next few instances.  Wider ranges are then
// split into 32 parts per pass.
__device__ __forceinline__ uint32_t find_instance(const uint64_t *prefix, uint32_t lo, uint32_t hi, uint64_t g)
{
    const uint32_t lane = threadIdx.x & 31u;
    {
        const uint32_t m = lo + lane;
        const bool le = m < hi && prefix[m] <= g;
        const uint32_t ball = __ballot_sync(kFull, le);
        const uint32_t top = 31u - static_cast<uint32_t>(__clz(ball));  // lane 0 always qualifies
        if (top < 31u || lo + 32u >= hi) return lo + top;
        lo += 31u;
    }
    while (hi - lo > 32u) {
        const uint32_t span = hi - lo;
        const uint32_t m = lo + static_cast<uint32_t>((static_cast<uint64_t>(span) * lane) / 32u);
        const bool le = prefix[m] <= g;
        const uint32_t ball = __ballot_sync(kFull, le);
        const int top = 31 - __clz(ball);  // lane 0 always qualifies (prefix[lo] <= g)
        const uint32_t new_lo = lo + static_cast<uint32_t>((static_cast<uint64_t>(span) * top) / 32u);
        const uint32_t new_hi = top == 31 ? hi : lo + static_cast<uint32_t>((static_cast<uint64_t>(span) * (top + 1)) / 32u);
        lo = new_lo;
        hi = new_hi;
    }
    const uint32_t m = lo + lane;
    const bool le = m < hi && prefix[m] <= g;
    const uint32_t ball = __ballot_sync(kFull, le);
    return lo + static_cast<uint32_t>(31 - __clz(ball));
}

struct BatchJob {
    const void *in;
    void *out;
    uint64_t first;  // global index of the instance's first tile
    uint64_t end;    // one past its last tile
    Geometry g;
    uint32_t instance;
    uint32_t ticket;
};
static_assert(sizeof(BatchJob) % 4 == 0 && sizeof(BatchJob) <= 128, "copied by a warp, one word a lane");

// CTA state, double-buffered: the job of the CTA's next ticket is resolved
// into one buffer while the tile of the other is still being stored.
template <int ENTRIES>
struct BatchShared {
    dev::TileShared<ENTRIES> st[2];
    uint32_t keys[2][kMaxRounds];
    BatchJob job[2];
};

// Run by one full warp: turns ticket `ticket` into its job (instance,
// geometry, round keys) in slot `nb`.  `prev` is the slot of the CTA's
// previous ticket (-1 before the first one); a CTA's tickets grow, so the
// owner is `prev`'s instance or a later one.
template <class SH>
__device__ __forceinline__ void resolve_job(const BatchArgs &a, uint32_t ticket, uint64_t total, int prev, SH &sh,
                                            int nb)
{
    const uint32_t lane = threadIdx.x & 31u;
    BatchJob &job = sh.job[nb];
    if (ticket >= total) {
        if (lane == 0) job.ticket = ticket;
        return;
    }
    if (prev >= 0 && ticket < sh.job[prev].end) {  // the same instance: its job and keys again
        if (lane < sizeof(BatchJob) / 4)
            reinterpret_cast<uint32_t *>(&job)[lane] = reinterpret_cast<const uint32_t *>(&sh.job[prev])[lane];
        for (uint32_t r = lane; r < a.rounds; r += 32) sh.keys[nb][r] = sh.keys[prev][r];
        __syncwarp();
        if (lane == 0) job.ticket = ticket;
    } else {
        const uint32_t lo = prev >= 0 ? sh.job[prev].instance + 1u : 0u;
        const uint32_t t = find_instance(a.tile_prefix, lo, a.count, ticket);
        const BatchDesc d = a.descs[t];
        const BatchPlan p = a.plan[t];
        if (lane == 0) {
            const uint32_t k = p.k;
            job.in = d.in;
            job.out = d.out;
            job.first = p.first_tile;
            job.end = p.first_tile + p.tiles;
            job.g.n = static_cast<uint32_t>(d.n);
            job.g.k = k;
            job.g.L = k / 2;
            job.g.R = k - k / 2;
            job.g.lmask = (1u << (k / 2)) - 1u;
            job.g.rmask = (k - k / 2) >= 32 ? 0xffffffffu : ((1u << (k - k / 2)) - 1u);
            job.g.domain = uint64_t{1} << k;
            job.g.odd_mul = 1u << (31u - k / 2);
            job.g.lift_mul = 1u << (k / 2);
            job.instance = t;
            job.ticket = ticket;
        }
        for (uint32_t r = lane; r < a.rounds; r += 32) sh.keys[nb][r] = dev::splitmix_key(d.seed, r);
    }
}

// One tile of job `b`, then the CTA's next ticket.  The next ticket is taken
// only after the look-back: a CTA that held a ticket while its current tile
// still waited on other tiles would make every later tile wait for it.  Warp
// 1 takes it and resolves it into buffer b ^ 1 while the other warps store.
template <class T, bool ODD, int ITEMS, int ENTRIES, bool UNROLL>
__device__ __forceinline__ void batch_tile(const BatchArgs &a, const BatchJob &job, BatchShared<ENTRIES> &sh, int b,
                                           const dev::StatusRing &ring, uint64_t total)
{
    constexpr int WARPS = kBBlock / 32;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    const Geometry &g = job.g;
    const uint64_t tile = job.ticket;
    const uint32_t base = static_cast<uint32_t>(tile - job.first) * kTile;
    dev::TileShared<ENTRIES> &st = sh.st[b];

    uint32_t left[ITEMS], right[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t i = base + static_cast<uint32_t>(j * kBBlock) + threadIdx.x;
        left[j] = i >> g.R;
        right[j] = i & g.rmask;
    }
    if constexpr (UNROLL)
        dev::cipher_items<ODD, ITEMS>(left, right, sh.keys[b], a.rounds, g);
    else
        dev::cipher_items_loop<ODD, ITEMS>(left, right, sh.keys[b], a.rounds, g);
    uint32_t src[ITEMS];
    bool keep[ITEMS];
    T val[ITEMS];
    const T *in = static_cast<const T *>(job.in);
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t i = base + static_cast<uint32_t>(j * kBBlock) + threadIdx.x;
        src[j] = (left[j] << g.R) | right[j];
        keep[j] = static_cast<uint64_t>(i) < g.domain && src[j] < g.n;
        if (keep[j]) val[j] = __ldg(in + src[j]);
    }
    uint32_t mask[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) mask[j] = __ballot_sync(kFull, keep[j]);
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) st.counts[j * WARPS + warp] = __popc(mask[j]);
    }
    __syncthreads();
    if (warp == 0)
        dev::tile_scan_lookback<ENTRIES>(st, ring, tile, job.first, a.timeout_ns, a.skip_publish_tile, a.ws);
    __syncthreads();
    uint32_t next = 0;
    if (threadIdx.x == 32) next = atomicAdd(&a.ws->batch_ticket, 1u);
    if (st.ok != 0u) {
        const uint32_t prefix = st.prefix;
        const uint32_t lt = dev::lanemask_lt();
        T *out = static_cast<T *>(job.out);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t dst = prefix + st.counts[j * WARPS + warp] + __popc(mask[j] & lt);
            if (keep[j]) {
                if (dst < g.n) out[dst] = val[j];
                else dev::record_error(a.ws, dev::kErrDeviceBounds, dst);
            }
        }
    }
    if (warp == 1) resolve_job(a, __shfl_sync(kFull, next, 0), total, b, sh, b ^ 1);
    __syncthreads();
}

// Persistent CTAs, a few per SM, take tickets in order and only when they
// are ready to start the tile, so the smallest unfinished ticket always
// belongs to a running CTA whose look-back depends only on smaller tickets:
// every wait ends.
// UNROLL: for the default 24 rounds; other counts have an instance of their
// own, without the 24-round forms, whose registers made it spill (512 uneven
// instances of 1-byte elements with 10 rounds 540 -> 485 us).
template <class T, bool UNROLL>
__global__ void __launch_bounds__(kBBlock, min_ctas_for(sizeof(T))) batch_tile_kernel(const __grid_constant__ BatchArgs a)
{
    constexpr int ENTRIES = kBItems * (kBBlock / 32);
    __shared__ BatchShared<ENTRIES> sh;
    const dev::StatusRing ring = batch_ring(a);
    const uint64_t total = *reinterpret_cast<volatile const uint64_t *>(a.total_tiles);
    const uint32_t warp = threadIdx.x >> 5;

    if (warp == 1) {
        uint32_t t0 = 0;
        if ((threadIdx.x & 31u) == 0) t0 = atomicAdd(&a.ws->batch_ticket, 1u);
        resolve_job(a, __shfl_sync(kFull, t0, 0), total, -1, sh, 0);
    }
    __syncthreads();
    for (int b = 0;; b ^= 1) {
        const BatchJob job = sh.job[b];
        if (job.ticket >= total) break;
        if (job.g.k & 1u)
            batch_tile<T, true, kBItems, ENTRIES, UNROLL>(a, job, sh, b, ring, total);
        else
            batch_tile<T, false, kBItems, ENTRIES, UNROLL>(a, job, sh, b, ring, total);
    }
    if (threadIdx.x == 0) finish_batch(a, ring, total);
}

// ------------------------------------------------------------------ pipelined
// The batched shuffle with the look-back, the tickets and the lookup of their
// instances taken off the compute warps.  A persistent CTA holds NW compute
// warps and one look-back warp:
//
//   compute warps, tile i (buffer i % 2, job slot i % 4): wait for its job,
//     and SUB times evaluate the bijection over 32 * ITEMS consecutive
//     indices of their own and start copying the kept elements, packed, into
//     their part of the buffer with cp.async; publish the tile aggregate (the
//     last warp to add its count does it); then store tile i - 1 once it is
//     ranked: a warp's kept elements are SUB runs of consecutive slots.
//   look-back warp, tile i: wait for the counts, form the parts' offsets,
//     look back, publish the inclusive prefix, hand the prefix over; then
//     take the ticket of tile i + 2 and resolve its instance, while the
//     compute warps are in tile i + 1.
//
// The compute warps share no barrier: each passes on as soon as the job and
// the rank that it needs are there, up to a tile ahead of the slowest.  A
// ticket is taken only when the CTA's latest look-back is over, and no
// aggregate waits on a later look-back, so the smallest unfinished ticket
// always makes progress.  (The second ticket of a CTA is taken once its first
// tile is published, so a batch with fewer tiles than CTAs spreads over all.)
// Every wait is bounded.  Used for 4-, 8- and 16-byte elements.
//
// What bounds it: the ALU pipe (cipher, ballots: 6.5 ms of the figure below
// with the gathers, look-backs and stores taken out), then the serial chain of
// the look-back warp.  Steps measured on GB300 with 4,096 uneven int32
// instances (8.3e8 elements, 1.2e9 evaluations), from 9.58 ms: the job kept in
// shared memory instead of 25 registers (56 registers a thread, 4 CTAs) 8.67;
// tickets and lookups by the look-back warp, no barrier 8.52; then that warp
// was busy 17 of a tile's 18.6 thousand cycles (a poll takes a thousand
// cycles behind the gathers), and four rounds of 4 indices per thread a tile
// instead of one of 8 gave 7.50 (16 indices in registers 8.94; a third buffer
// 8.62; images in shared memory and plain loads at the store instead of
// cp.async 8.38).  8-byte elements 2.13 ms for 1,024 instances (2.71 before),
// 16-byte 2.23 (2.70).
// Shapes (kBatchConfigs): NW compute warps, SUB * ITEMS indices per thread,
// MINB resident CTAs per SM targeted, UNROLL the default 24 rounds unrolled.
// Shape 0 is the default.
constexpr int DEPTH = 2;  // tile buffers of a CTA

template <int NW, int SUB>
struct BatchPipeShared {
    uint64_t full[DEPTH];            // compute -> look-back: counts of the buffer's tile written
    uint64_t ranked[DEPTH];          // look-back -> compute: offsets and prefix ready
    uint64_t ready[DEPTH];           // look-back -> compute: job of the tile resolved
    unsigned long long aggc[DEPTH];  // (compute warps done << 32) | kept count
    BatchJob job[DEPTH + 2];
    uint32_t keys[DEPTH + 2][kMaxRounds];
    uint32_t counts[DEPTH][NW * SUB];  // kept indices per (round, compute warp)
    uint32_t offs[DEPTH][NW * SUB];    // their exclusive sums
    uint32_t prefix[DEPTH];
    uint32_t ok[DEPTH];
    uint32_t abort;
};

template <class T, int NW, int ITEMS, int SUB, int MINB, bool UNROLL>
__global__ void __launch_bounds__((NW + 1) * 32, MINB) batch_pipe_kernel(const __grid_constant__ BatchArgs a)
{
    constexpr uint32_t kWarpTile = 32 * ITEMS;  // domain indices of one compute warp and round
    constexpr uint32_t kPTile = NW * SUB * kWarpTile;
    constexpr int SLOTS = DEPTH + 2;
    static_assert(NW * SUB <= 32, "one lane of the look-back warp per count");
    __shared__ BatchPipeShared<NW, SUB> sh;
    extern __shared__ __align__(16) unsigned char batch_dyn[];
    T *vals = reinterpret_cast<T *>(batch_dyn);  // [DEPTH][kPTile]
    const dev::StatusRing ring = batch_ring(a);
    const uint64_t total = *reinterpret_cast<volatile const uint64_t *>(a.total_tiles);
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    const uint64_t role_limit = 2 * a.timeout_ns + 1000000000ull;
    volatile uint32_t *abort = &sh.abort;

    if (threadIdx.x == 0) {
        for (int b = 0; b < DEPTH; ++b) {
            dev::mbar_init(&sh.full[b], NW);
            dev::mbar_init(&sh.ranked[b], 1);
            dev::mbar_init(&sh.ready[b], 1);
            sh.aggc[b] = 0ull;
        }
        sh.abort = 0u;
    }
    __syncthreads();

    if (warp < NW) {
        // ---------------------------------------------------------- compute
        const uint32_t lt = dev::lanemask_lt();
        // stores this warp's part of the tile in buffer `b` (job slot `slot`)
        // once it is ranked; its copies have landed
        const auto store = [&](int b, uint32_t phase, int slot) {
            const bool ranked = dev::mbar_wait(&sh.ranked[b], phase, role_limit, abort);
            if (!ranked) {
                if (lane == 0) dev::record_error(a.ws, dev::kErrLookbackTimeout, static_cast<uint64_t>(slot));
                *abort = 1u;
            }
            __syncwarp();  // every lane's copies have landed
            if (!ranked || sh.ok[b] == 0u) return;
            const uint32_t n = sh.job[slot].g.n;
#pragma unroll 1
            for (int q = 0; q < SUB; ++q) {
                const uint32_t part = static_cast<uint32_t>(q * NW) + warp;
                const T *buf = vals + static_cast<size_t>(b) * kPTile + part * kWarpTile;
                const uint32_t count = sh.counts[b][part];
                const uint32_t dst = sh.prefix[b] + sh.offs[b][part];
                T *out = static_cast<T *>(sh.job[slot].out) + dst;
                if (count <= n && dst <= n - count) {
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t e = static_cast<uint32_t>(j * 32) + lane;
                        if (e < count) out[e] = buf[e];
                    }
                } else if (lane == 0) {  // impossible; kept as a guard, and nothing is written
                    dev::record_error(a.ws, dev::kErrDeviceBounds, dst + count - 1u);
                }
            }
        };
        int b = 0, slot = 0;
        uint32_t phase = 0;
        for (uint32_t iter = 0;; ++iter) {
            const bool ready = __all_sync(kFull, dev::mbar_wait(&sh.ready[b], phase, role_limit, abort));
            if (!ready) {
                if (lane == 0) dev::record_error(a.ws, dev::kErrLookbackTimeout, iter);
                *abort = 1u;
            }
            const BatchJob &job = sh.job[slot];  // stays in shared memory: fewer registers, more CTAs
            const uint32_t tile = job.ticket;
            if (!ready || tile >= total) {
                // the tiles not stored yet, oldest first
                dev::cp_async_wait_all();
                for (int t = DEPTH - 1; t > 0; --t)
                    if (iter >= static_cast<uint32_t>(t))
                        store(b >= t ? b - t : b - t + DEPTH, b >= t ? phase : phase ^ 1u,
                              slot >= t ? slot - t : slot - t + SLOTS);
                break;
            }
            const Geometry &g = job.g;
            const uint64_t tile_base = uint64_t{tile - static_cast<uint32_t>(job.first)} * kPTile;
            const uint32_t shift = g.R, rmask = g.rmask;
            const uint32_t n = g.n, last = static_cast<uint32_t>(g.domain - 1u);
            const T *in = static_cast<const T *>(job.in);
            uint32_t total_count = 0;
#pragma unroll 1
            for (int q = 0; q < SUB; ++q) {
                const uint32_t part = static_cast<uint32_t>(q * NW) + warp;
                const uint64_t start = tile_base + part * kWarpTile;
                const uint32_t base = static_cast<uint32_t>(start) + lane;
                uint32_t count = 0;
                if (start <= last) {  // the domain ends inside its last tile
                    uint32_t left[ITEMS], right[ITEMS];
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t i = base + static_cast<uint32_t>(j * 32);
                        left[j] = i >> shift;
                        right[j] = i & rmask;
                    }
                    if constexpr (UNROLL) {
                        if (g.k & 1u)
                            dev::cipher_items<true, ITEMS>(left, right, sh.keys[slot], a.rounds, g);
                        else
                            dev::cipher_items<false, ITEMS>(left, right, sh.keys[slot], a.rounds, g);
                    } else {
                        if (g.k & 1u)
                            dev::cipher_items_loop<true, ITEMS>(left, right, sh.keys[slot], a.rounds, g);
                        else
                            dev::cipher_items_loop<false, ITEMS>(left, right, sh.keys[slot], a.rounds, g);
                    }
                    T *buf = vals + static_cast<size_t>(b) * kPTile + part * kWarpTile;
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t i = base + static_cast<uint32_t>(j * 32);
                        const uint32_t src = (left[j] << shift) | right[j];
                        const bool keep = i <= last && src < n;
                        const uint32_t m = __ballot_sync(kFull, keep);
                        if (keep) dev::cp_async<sizeof(T)>(buf + count + __popc(m & lt), in + src);
                        count += __popc(m);
                    }
                }
                if (lane == 0) sh.counts[b][part] = count;
                total_count += count;
            }
            if (lane == 0) {
                const unsigned long long v = atomicAdd(&sh.aggc[b], (1ull << 32) | total_count);
                if ((v >> 32) == NW - 1 && static_cast<int64_t>(tile) != a.skip_publish_tile) {
                    const uint32_t sum = static_cast<uint32_t>(v) + total_count;
                    dev::st_relaxed_gpu(ring.slot(tile), dev::status_word(ring.tag(tile), tile == job.first, sum));
                }
            }
            dev::cp_async_commit();
            __syncwarp();
            if (lane == 0) dev::mbar_arrive(&sh.full[b]);
            if (iter >= static_cast<uint32_t>(DEPTH - 1)) {
                dev::cp_async_wait_groups<DEPTH - 1>();  // this thread's copies of the oldest tile
                store(b == DEPTH - 1 ? 0 : b + 1, b == DEPTH - 1 ? phase : phase ^ 1u,
                      slot >= DEPTH - 1 ? slot - (DEPTH - 1) : slot - (DEPTH - 1) + SLOTS);
            }
            slot = slot == SLOTS - 1 ? 0 : slot + 1;
            if (++b == DEPTH) {
                b = 0;
                phase ^= 1u;
            }
        }
    } else {
        // -------------------------------------------------------- look-back
        // the next ticket into slot `to` (`from`: the slot of the ticket
        // before it), for the compute warps' tile of buffer `rb`
        const auto take = [&](int from, int to, int rb) {
            uint32_t t = 0xffffffffu;
            if (lane == 0 && *abort == 0u) t = atomicAdd(&a.ws->batch_ticket, 1u);
            resolve_job(a, __shfl_sync(kFull, t, 0), total, from, sh, to);
            __syncwarp();
            if (lane == 0) dev::mbar_arrive(&sh.ready[rb]);
        };
        take(-1, 0, 0);
        int b = 0, slot = 0;
        uint32_t phase = 0;
        for (uint32_t iter = 0;; ++iter) {
            const uint32_t tile = sh.job[slot].ticket;
            if (tile >= total) break;
            // lane 0 waits, so that the warp leaves the loop as one
            bool full = false;
            if (lane == 0) {
                full = dev::mbar_wait(&sh.full[b], phase, role_limit, abort);
                if (!full) {
                    dev::record_error(a.ws, dev::kErrLookbackTimeout, iter);
                    *abort = 1u;
                }
            }
            if (!__shfl_sync(kFull, full, 0)) break;
            (void)dev::mbar_test(&sh.full[b], phase);  // completed phase: every lane acquires it
            if (iter == 0u) take(0, 1, 1);
            const uint64_t first = sh.job[slot].first;
            const uint32_t mine = lane < NW * SUB ? sh.counts[b][lane] : 0u;
            const uint32_t incl = dev::warp_inclusive_scan(mine);
            if (lane < NW * SUB) sh.offs[b][lane] = incl - mine;
            const uint32_t aggregate = __shfl_sync(kFull, incl, 31);
            uint32_t prefix = 0;
            bool ok = true;
            if (tile > first) {
                prefix = dev::lookback(ring, tile, first, a.timeout_ns, ok);
                if (lane == 0 && static_cast<int64_t>(tile) != a.skip_publish_tile)
                    dev::st_relaxed_gpu(ring.slot(tile), dev::status_word(ring.tag(tile), true, prefix + aggregate));
                if (lane == 0 && !ok) dev::record_error(a.ws, dev::kErrLookbackTimeout, tile);
            }
            if (lane == 0) {
                sh.prefix[b] = prefix;
                sh.ok[b] = ok ? 1u : 0u;
                sh.aggc[b] = 0ull;
            }
            __syncwarp();
            if (lane == 0) dev::mbar_arrive(&sh.ranked[b]);
            const int next = slot == SLOTS - 1 ? 0 : slot + 1;
            if (sh.job[next].ticket < total)
                take(next, next == SLOTS - 1 ? 0 : next + 1, b + 2 < DEPTH ? b + 2 : b + 2 - DEPTH);
            slot = next;
            if (++b == DEPTH) {
                b = 0;
                phase ^= 1u;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) finish_batch(a, ring, total);
}

template <class T, int NW, int ITEMS, int SUB, int MINB, bool UNROLL>
cudaError_t launch_pipe_typed(const BatchArgs &a, cudaStream_t stream)
{
    constexpr int THREADS = (NW + 1) * 32;
    constexpr uint32_t TILE = NW * 32 * ITEMS * SUB;
    constexpr size_t DYN = DEPTH * sizeof(T) * TILE;
    const auto kernel = batch_pipe_kernel<T, NW, ITEMS, SUB, MINB, UNROLL>;
    static std::atomic<int> per_sm[64];  // CTAs to launch per device, 0 until first use
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    int ctas_cached = per_sm[device].load(std::memory_order_acquire);
    if (ctas_cached == 0) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(DYN));
        if (e != cudaSuccess) return e;
        int blocks = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, THREADS, DYN);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return e;
        ctas_cached = (blocks > 0 ? blocks : 1) * sms;
        per_sm[device].store(ctas_cached, std::memory_order_release);
    }
    BatchArgs b = a;
    b.grid = static_cast<uint32_t>(ctas_cached);
    b.tile = TILE;
    batch_plan_kernel<<<1, kPlanThreads, 0, stream>>>(b);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    kernel<<<b.grid, THREADS, DYN, stream>>>(b);
    return cudaGetLastError();
}

template <class T, bool UNROLL>
cudaError_t launch_rounds(const BatchArgs &a, cudaStream_t stream)
{
    static std::atomic<int> per_sm[64];  // CTAs to launch per device, 0 until first use
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    int ctas_cached = per_sm[device].load(std::memory_order_acquire);
    if (ctas_cached == 0) {
        int blocks = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, batch_tile_kernel<T, UNROLL>, kBBlock, 0);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return e;
        ctas_cached = (blocks > 0 ? blocks : 1) * sms;
        per_sm[device].store(ctas_cached, std::memory_order_release);
    }
    BatchArgs b = a;
    b.grid = static_cast<uint32_t>(ctas_cached);
    b.tile = kTile;
    batch_plan_kernel<<<1, kPlanThreads, 0, stream>>>(b);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    batch_tile_kernel<T, UNROLL><<<b.grid, kBBlock, 0, stream>>>(b);
    return cudaGetLastError();
}

template <class T>
cudaError_t launch_typed(const BatchArgs &a, cudaStream_t stream)
{
    return a.rounds == dev::kUnrolledRounds ? launch_rounds<T, true>(a, stream) : launch_rounds<T, false>(a, stream);
}

template <class T>
cudaError_t launch_pipe_config(const BatchArgs &a, int config, cudaStream_t stream)
{
    static_assert(kNumBatchConfigs == 6, "shapes instantiated here");
    // 8- and 16-byte elements: at most three rounds of 4 indices (a larger
    // buffer takes L1 away from the gathers: 2.13 -> 3.23 ms for 1,024
    // instances of 8-byte elements with four)
    constexpr int most = sizeof(T) == 4 ? 4 : 3;
    switch (config) {
    case 0: return launch_pipe_typed<T, 8, 4, most, 3, true>(a, stream);
    case 1: return launch_pipe_typed<T, 12, 4, 2, 3, true>(a, stream);
    case 2: return launch_pipe_typed<T, 8, 4, 2, 4, true>(a, stream);
    case 3: return launch_pipe_typed<T, 6, 4, most, 4, true>(a, stream);
    case 4: return launch_pipe_typed<T, 16, 4, 2, 2, true>(a, stream);
    case 5: return launch_pipe_typed<T, 8, 4, most, 3, false>(a, stream);
    default: return cudaErrorInvalidValue;
    }
}

std::atomic<int> g_batch_selected[3];  // 4, 8, 16 bytes

int batch_slot(uint32_t elem_bytes) { return elem_bytes == 4 ? 0 : elem_bytes == 8 ? 1 : elem_bytes == 16 ? 2 : -1; }

}  // namespace

const PipeConfig kBatchConfigs[kNumBatchConfigs] = {
    {8, 16, 3, 1}, {12, 8, 3, 1}, {8, 8, 4, 1}, {6, 16, 4, 1}, {16, 8, 2, 1}, {8, 16, 3, 0},
};

int select_batch_config(uint32_t elem_bytes, int config)
{
    const int slot = batch_slot(elem_bytes);
    if (slot < 0 || config < 0 || config >= kNumBatchConfigs) return -1;
    g_batch_selected[slot].store(config);
    return 0;
}

int selected_batch_config(uint32_t elem_bytes)
{
    const int slot = batch_slot(elem_bytes);
    return slot < 0 ? 0 : g_batch_selected[slot].load();
}

uint64_t batch_ring_words() { return kRingWords; }

cudaError_t launch_batched(const BatchArgs &a, cudaStream_t stream)
{
    const int config = selected_batch_config(a.elem_bytes);
    switch (a.elem_bytes) {
    case 1: return launch_typed<unsigned char>(a, stream);
    case 2: return launch_typed<unsigned short>(a, stream);
    case 4: return launch_pipe_config<unsigned int>(a, config, stream);
    case 8: return launch_pipe_config<unsigned long long>(a, config, stream);
    case 16: return launch_pipe_config<uint4>(a, config, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace bsh
