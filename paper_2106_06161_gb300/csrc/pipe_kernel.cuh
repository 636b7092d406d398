// Pipelined single pass of Algorithm 1 (gather and scatter of 1- to 16-byte
// elements, and the index output): the same output as the fused tile
// kernel, with the inter-tile look-back taken off the compute warps' path.
//
// In the plain fused kernel every warp of a tile waits while one warp looks
// back, and under a full load of random gathers a look-back takes several
// L2 round trips.  Here a persistent CTA holds NW compute warps and one
// look-back warp, and the compute warps run one tile ahead of their stores:
//
//   compute warps, tile i (buffer i % 2): wait for its ticket, and SUB times
//     evaluate the bijection over 32 * ITEMS consecutive indices of their own
//     and start copying the kept elements X[f(i)], packed, into their part of
//     the buffer with cp.async (one copy group per thread and tile; the index
//     and scatter modes store the images themselves); publish the tile
//     aggregate (the last compute warp to add its count does it); then store
//     tile i - 1: wait for its rank (look-back warp) and this thread's copy
//     group of that tile, and write each part's kept entries to consecutive
//     slots (scatter: read those slots and write them to the images).
//   look-back warp, tile i: wait for the counts, form the parts' offsets,
//     look back, publish the inclusive prefix and hand the prefix to the
//     compute warps; then take the ticket of tile i + 2 (the second ticket,
//     once the first tile is published).  Launches over kTicketsAheadBytes: the
//     last compute warp takes the ticket of tile i + 1 instead, when the stores
//     of tile i - 1 are done; the look-back of tile i may still be running.
//
// The compute warps share no barrier and pass on as soon as the ticket and
// the rank that they need are there.  When a ticket is taken, nothing is left
// that its tile's aggregate would have to wait for: ahead, the compute warps
// are at most in tile i + 1, whose stores of tile i need the look-back that is
// over; else they are at the end of tile i.  They publish the aggregate right
// after the tile's counts, so every ticket's aggregate comes without waiting
// for a look-back of any CTA, a look-back waits for aggregates of smaller
// tickets only, and the smallest unfinished ticket always makes progress.
// Every wait is bounded.
//
// What bounds it: up to the L2's size the ALU pipe (cipher) and, below some
// 2^20 indices, the latency of one tile's steps; beyond, the random-access
// rate of the memory behind the gathers.  A tile of several rounds spares the
// look-back warp, whose polls queue behind the gathers: see pipe_rounds.
// Against the form with a barrier and a ticket between two tiles and the
// kept elements at their natural places (GB300, calls replayed from a graph,
// n = 15/16 of the domain, domains of 2^20, 2^22 and 2^24): 4-byte gathers
// 17.6 -> 14.8, 40.6 -> 31.6 and 137 -> 109 us, 8-byte 16.0 -> 14.3, 40.5 ->
// 34.6 and 186 -> 186, 64-bit indices 14.4 -> 13.5, 33.3 -> 29.6 and 107 -> 90,
// with the cipher's share of it.  A scatter reads its input as a stream
// (__ldcs), which leaves the L2 to the writes: 8-byte at 2^24 - 5 385 -> 312 us,
// 16-byte at 2^23 + 1 239 -> 192, 4-byte at 2^25 + 1 680 -> 579.
//
// The kernel template and its launch, shared by the translation units that
// instantiate its shapes (kernels_pipe.cu: the default shapes for every mode;
// kernels_pipe_tuned.cu: the other shapes of the gather, for the autotuner).
#pragma once

#include <atomic>
#include <cstdint>
#include <type_traits>

#include "bshuffle_device.cuh"
#include "bshuffle_internal.h"

namespace bsh {
namespace pipe {

using dev::kFull;

template <int NW, int SUB>
struct PipeShared {
    uint64_t full[2];            // compute -> look-back: counts of the buffer's tile written
    uint64_t ranked[2];          // look-back -> compute: offsets and prefix of that tile ready
    uint64_t ready[2];           // look-back -> compute: ticket of the tile taken
    unsigned long long aggc[2];  // (compute warps done << 32) | kept count, per buffer
    uint32_t counts[2][NW * SUB];  // kept indices per (round, compute warp)
    uint32_t offs[2][NW * SUB];    // their exclusive sums
    uint32_t prefix[2];          // exclusive prefix of the tile over all earlier tiles
    uint32_t ok[2];              // look-back finished in time
    uint32_t ticket[4];
    uint32_t stored;  // compute warps done with their stores (tickets not taken ahead)
    uint32_t tag;
    uint32_t abort;
};

// Launches that move fewer bytes take their tickets ahead.  Measured on GB300
// ahead / not: 8-byte gathers at 2^25 - 5 538 / 528 us, 16-byte gathers at 2^26
// + 1 1508 / 1467, 16-byte scatters at 2^24 + 1 583 / 581 and 2^26 + 1 2756 /
// 2679; at the L2's sizes the ticket's latency shows instead (indices at 2^24
// 90 us ahead, 107 in the form with a barrier).
constexpr uint64_t kTicketsAheadBytes = uint64_t{96} << 20;

// Whether the gathers run with cp.async while the tile waits for its rank: it
// copies 4, 8 or 16 bytes.  Narrower elements are read when they are stored.
// (Copying the aligned word around each, with its bit offset in a byte beside
// it, was no faster: 2-byte gathers at 2^26 + 1 1126 / 1134 us, at 2^27 - 5
// 1909 / 1770.)
template <class T, Mode MODE>
constexpr bool kAsyncGather = MODE == Mode::Gather && sizeof(T) >= 4;

// What a tile buffer holds per kept index: the gathered element, or the image
// itself, which the store writes (indices), reads from (1- and 2-byte gathers)
// or writes the element that it reads then to (scatter: out[f(i_j)] = in[j]).
template <class T, Mode MODE>
using PipeSlot = typename std::conditional<kAsyncGather<T, MODE>, T, uint32_t>::type;

// MINB: resident CTAs per SM the register budget targets; UNROLL: the
// default round count runs fully unrolled (else every count runs in a loop).
// RANGE: Algorithm 1 restricted to the domain indices [range_first,
// range_end) (tiles counted from range_first), writing the range's kept
// elements to out[0 .. count), at most range_cap of them.
template <class T, Mode MODE, bool ODD, int NW, int ITEMS, int SUB, int MINB, bool UNROLL, bool RANGE = false>
__global__ void __launch_bounds__((NW + 1) * 32, MINB) pipe_tile_kernel(const __grid_constant__ TileArgs a)
{
    using S = PipeSlot<T, MODE>;
    constexpr bool ASYNC = kAsyncGather<T, MODE>;
    constexpr uint32_t kWarpTile = 32 * ITEMS;  // domain indices of one compute warp and round
    constexpr uint32_t TILE = NW * SUB * kWarpTile;
    static_assert(NW * SUB <= 32, "one lane of the look-back warp per count");
    __shared__ PipeShared<NW, SUB> sh;
    const long long c_start = dev::clock_mark();
    extern __shared__ __align__(16) unsigned char pipe_dyn[];
    S *vals = reinterpret_cast<S *>(pipe_dyn);  // [2][TILE], each part's kept entries packed

    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    // a wait for the other role gets room for one full look-back timeout
    const uint64_t role_limit = 2 * a.timeout_ns + 1000000000ull;
    // Tickets one tile ahead, or only when a tile's stores are done: data that
    // the L2 does not hold is moved faster with fewer tiles open at a time.
    const bool ahead =
        MODE == Mode::Index32 || MODE == Mode::Index64 || uint64_t{a.g.n} * sizeof(T) < kTicketsAheadBytes;
    // slots a launch may write
    const uint32_t limit = RANGE && a.range_cap < a.g.n ? static_cast<uint32_t>(a.range_cap) : a.g.n;

    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            dev::mbar_init(&sh.full[b], NW);
            dev::mbar_init(&sh.ranked[b], 1);
            dev::mbar_init(&sh.ready[b], 1);
            sh.aggc[b] = 0ull;
        }
        sh.stored = 0u;
        sh.tag = dev::ld_relaxed_gpu(&a.ws->tag);
        sh.abort = 0u;
    }
    __syncthreads();
    const uint32_t tag = sh.tag;
    const dev::StatusRing ring{a.status, ~0ull, 63u, tag};
    volatile uint32_t *abort = &sh.abort;
    // takes the ticket of the compute warps' iteration `it` (one thread)
    const auto take = [&](uint32_t it) {
        sh.ticket[it & 3u] = *abort == 0u ? atomicAdd(&a.ws->ticket, 1u) : 0xffffffffu;
        dev::mbar_arrive(&sh.ready[it & 1u]);
    };

    if (warp < NW) {
        // ---------------------------------------------------------- compute
        const uint32_t lt = dev::lanemask_lt();
        const T *in = static_cast<const T *>(a.in);
        T *out = static_cast<T *>(a.out);
        // stores this warp's parts of the tile in buffer `b` once it is
        // ranked; its copies have landed
        const auto store = [&](int b, uint32_t phase) {
            const long long w0 = dev::clock_mark();
            const bool ranked = dev::mbar_wait(&sh.ranked[b], phase, role_limit, abort);
            if (threadIdx.x == 0) dev::clock_add(&a.ws->lookback_cycles, w0);  // the compute warps wait on the rank
            if (!ranked) {
                if (lane == 0) dev::record_error(a.ws, dev::kErrLookbackTimeout, static_cast<uint64_t>(b));
                *abort = 1u;
            }
            __syncwarp();  // every lane's copies have landed
            if (!ranked || sh.ok[b] == 0u) return;
#pragma unroll 1
            for (int q = 0; q < SUB; ++q) {
                const uint32_t part = static_cast<uint32_t>(q * NW) + warp;
                const S *buf = vals + static_cast<size_t>(b) * TILE + part * kWarpTile;
                const uint32_t dst = sh.prefix[b] + sh.offs[b][part];
                uint32_t count = sh.counts[b][part];
                if (count > limit || dst > limit - count) {
                    // past a range's output capacity (impossible otherwise)
                    if (lane == 0) dev::record_error(a.ws, dev::kErrDeviceBounds, uint64_t{dst} + count - 1u);
                    count = dst < limit ? limit - dst : 0u;
                }
                if constexpr (MODE == Mode::Gather && !ASYNC) {
                    T v[ITEMS];
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t e = static_cast<uint32_t>(j * 32) + lane;
                        if (e < count) v[j] = __ldg(in + buf[e]);
                    }
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t e = static_cast<uint32_t>(j * 32) + lane;
                        if (e < count) out[uint64_t{dst} + e] = v[j];
                    }
                } else if constexpr (MODE == Mode::Scatter) {
                    // coalesced reads of this tile's slots, then the random writes
                    T v[ITEMS];
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t e = static_cast<uint32_t>(j * 32) + lane;
                        if (e < count) v[j] = __ldcs(in + dst + e);  // read once: the L2 is the writes'
                    }
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t e = static_cast<uint32_t>(j * 32) + lane;
                        if (e < count) out[buf[e]] = v[j];
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t e = static_cast<uint32_t>(j * 32) + lane;
                        if (e < count) out[uint64_t{dst} + e] = buf[e];
                    }
                }
            }
        };
        for (uint32_t iter = 0;; ++iter) {
            const int b = static_cast<int>(iter & 1u);
            const uint32_t phase = (iter >> 1) & 1u;
            const bool ready = __all_sync(kFull, dev::mbar_wait(&sh.ready[b], phase, role_limit, abort));
            if (!ready) {
                if (lane == 0) dev::record_error(a.ws, dev::kErrLookbackTimeout, iter);
                *abort = 1u;
            }
            const uint32_t tile = sh.ticket[iter & 3u];
            if (!ready || tile >= a.num_tiles) {
                if constexpr (ASYNC) dev::cp_async_wait_all();
                if (iter > 0) store(b ^ 1, b == 0 ? phase ^ 1u : phase);
                break;
            }
            const uint64_t tile_base = (RANGE ? uint64_t{a.range_first} : 0ull) + uint64_t{tile} * TILE;
            const uint64_t end = RANGE ? a.range_end : a.g.domain;
            uint32_t total = 0;
#pragma unroll 1
            for (int q = 0; q < SUB; ++q) {
                const uint32_t part = static_cast<uint32_t>(q * NW) + warp;
                const uint64_t start = tile_base + part * kWarpTile;
                uint32_t count = 0;
                if (start < end) {  // the domain may end inside its last tile
                    const uint32_t base = static_cast<uint32_t>(start) + lane;
                    // indices of the part inside the domain
                    const uint32_t live = end - start < kWarpTile ? static_cast<uint32_t>(end - start) : kWarpTile;
                    uint32_t left[ITEMS], right[ITEMS];
                    if constexpr (UNROLL && !RANGE) {  // a range may start anywhere
                        dev::cipher_run<ODD, ITEMS, 32>(left, right, base, a.keys, a.rounds, a.g);
                    } else {
                        dev::split_items<ITEMS, 32>(left, right, base, a.g);
                        if constexpr (UNROLL)
                            dev::cipher_items<ODD, ITEMS>(left, right, a.keys, a.rounds, a.g);
                        else
                            dev::cipher_items_loop<ODD, ITEMS>(left, right, a.keys, a.rounds, a.g);
                    }
                    S *buf = vals + static_cast<size_t>(b) * TILE + part * kWarpTile;
#pragma unroll
                    for (int j = 0; j < ITEMS; ++j) {
                        const uint32_t src = (left[j] << a.g.R) | right[j];
                        const bool keep = static_cast<uint32_t>(j * 32) + lane < live && src < a.g.n;
                        const uint32_t m = __ballot_sync(kFull, keep);
                        if (keep) {
                            S *slot = buf + count + __popc(m & lt);
                            if constexpr (ASYNC)
                                dev::cp_async<sizeof(T)>(slot, in + src);
                            else
                                *slot = src;
                        }
                        count += __popc(m);
                    }
                }
                if (lane == 0) sh.counts[b][part] = count;
                total += count;
            }
            if (lane == 0) {
                const unsigned long long v = atomicAdd(&sh.aggc[b], (1ull << 32) | total);
                if ((v >> 32) == NW - 1 && static_cast<int64_t>(tile) != a.skip_publish_tile) {
                    const uint32_t sum = static_cast<uint32_t>(v) + total;
                    dev::st_relaxed_gpu(ring.slot(tile), dev::status_word(tag, tile == 0u, sum));
                }
            }
            if constexpr (ASYNC) dev::cp_async_commit();
            __syncwarp();
            if (lane == 0) dev::mbar_arrive(&sh.full[b]);
            if (iter > 0) {
                if constexpr (ASYNC) dev::cp_async_wait_prior();  // the previous tile's copies
                store(b ^ 1, b == 0 ? phase ^ 1u : phase);
            }
            if (!ahead && lane == 0 && atomicAdd(&sh.stored, 1u) == NW - 1) {  // the last warp
                sh.stored = 0u;
                take(iter + 1u);
            }
        }
    } else {
        // -------------------------------------------------------- look-back
        // lane 0 waits, so that the warp leaves the loop as one
        const auto wait = [&](uint64_t *bar, uint32_t phase, uint32_t iter) {
            bool done = false;
            if (lane == 0) {
                done = dev::mbar_wait(bar, phase, role_limit, abort);
                if (!done) {
                    dev::record_error(a.ws, dev::kErrLookbackTimeout, iter);
                    *abort = 1u;
                }
            }
            if (!__shfl_sync(kFull, done, 0)) return false;
            (void)dev::mbar_test(bar, phase);  // completed phase: every lane acquires it
            return true;
        };
        if (lane == 0) take(0);
        __syncwarp();
        for (uint32_t iter = 0;; ++iter) {
            const int b = static_cast<int>(iter & 1u);
            const uint32_t phase = (iter >> 1) & 1u;
            if (!ahead && iter > 0u && !wait(&sh.ready[b], phase, iter)) break;
            const uint32_t tile = sh.ticket[iter & 3u];
            if (tile >= a.num_tiles) break;
            if (!wait(&sh.full[b], phase, iter)) break;
            if (ahead && iter == 0u) {
                if (lane == 0) take(1);
                __syncwarp();
            }
            const uint32_t mine = lane < NW * SUB ? sh.counts[b][lane] : 0u;
            const uint32_t incl = dev::warp_inclusive_scan(mine);
            if (lane < NW * SUB) sh.offs[b][lane] = incl - mine;
            const uint32_t aggregate = __shfl_sync(kFull, incl, 31);
            uint32_t prefix = 0;
            bool ok = true;
            if (tile > 0u) {
                prefix = dev::lookback(ring, tile, 0, a.timeout_ns, ok);
                if (lane == 0 && static_cast<int64_t>(tile) != a.skip_publish_tile)
                    dev::st_relaxed_gpu(ring.slot(tile), dev::status_word(tag, true, prefix + aggregate));
                if (lane == 0 && !ok) dev::record_error(a.ws, dev::kErrLookbackTimeout, tile);
            }
            if (lane == 0) {
                sh.prefix[b] = prefix;
                sh.ok[b] = ok ? 1u : 0u;
                sh.aggc[b] = 0ull;
            }
            __syncwarp();
            if (lane == 0) dev::mbar_arrive(&sh.ranked[b]);
            if (ahead && sh.ticket[(iter + 1u) & 3u] < a.num_tiles) {
                if (lane == 0) take(iter + 2u);
                __syncwarp();
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        dev::clock_add(&a.ws->cta_cycles, c_start);
        dev::finish_launch(a.ws, tag, gridDim.x);
    }
}

// Launch one shape: persistent CTAs, as many as fit on the device (cached
// per device and parity on first use), never more than the tiles.
template <class T, Mode MODE, int NW, int ITEMS, int SUB, int MINB, bool UNROLL, bool RANGE = false>
cudaError_t launch_shape(const TileArgs &a, cudaStream_t stream)
{
    constexpr int THREADS = (NW + 1) * 32;
    constexpr size_t DYN = sizeof(PipeSlot<T, MODE>) * 2 * (NW * 32 * ITEMS * SUB);
    static std::atomic<int> per_sm[64][2];  // CTAs to launch per device and parity, 0 until first use
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    const bool odd = (a.g.k & 1u) != 0u;
    auto kernel = odd ? pipe_tile_kernel<T, MODE, true, NW, ITEMS, SUB, MINB, UNROLL, RANGE>
                      : pipe_tile_kernel<T, MODE, false, NW, ITEMS, SUB, MINB, UNROLL, RANGE>;
    std::atomic<int> &slot = per_sm[device][odd ? 1 : 0];
    int ctas = slot.load(std::memory_order_acquire);
    if (ctas == 0) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(DYN));
        if (e != cudaSuccess) return e;
        int blocks = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, THREADS, DYN);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return e;
        ctas = (blocks > 0 ? blocks : 1) * sms;
        slot.store(ctas, std::memory_order_release);
    }
    const uint32_t grid = a.num_tiles < static_cast<uint32_t>(ctas) ? a.num_tiles : static_cast<uint32_t>(ctas);
    kernel<<<grid, THREADS, DYN, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace pipe
}  // namespace bsh
