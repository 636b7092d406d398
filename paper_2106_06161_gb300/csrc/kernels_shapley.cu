// Shapley values of a weighted voting game by permutation sampling (an
// application named in Sec. 1), fused with the shuffle.
//
// Game [q; w_0 .. w_{n-1}]: a coalition wins when its weight reaches q.
// Sample s orders the players by the shuffle of Algorithm 1 with seed
// seed0 + s (slot j holds player f(i_j)).  The player whose weight takes the
// running total of the players before it from below q to at least q is
// pivotal; counts[player] is incremented.  counts / samples estimates the
// Shapley values.  One warp owns one sample at a time: it walks the sample's
// domain in chunks of 32 * ITEMS indices in increasing order, carries the
// running weight from chunk to chunk (no block barrier, no inter-warp
// communication), and stops once the total reaches q.  The order itself never
// leaves registers.
//
// Only the chunk that holds the pivot needs the order of its players: every
// earlier one adds its weight by two warp reductions, where an ordered 64-bit
// scan of each 32 players (ten shuffles) took a quarter of the time.  The
// kernel is bound by the ALU pipe (81 % busy, the cipher's rounds).  10,000
// players, 100,000 orders on GB300: 4.63 -> 3.04 ms, and 3.04 -> 2.93 with the
// first round shared (cipher_run).
#include <atomic>
#include <cstdint>

#include "bshuffle_device.cuh"
#include "bshuffle_internal.h"

namespace bsh {
namespace {

using dev::kFull;

constexpr int kSvBlock = 256;
constexpr int kSvWarps = kSvBlock / 32;
constexpr int kSvItems = 8;
constexpr int kSvGroup = 4;  // indices that share the cipher's first round (from 8,193 players on)
constexpr uint32_t kSvChunk = 32 * kSvItems;

template <bool ODD, CipherForm FORM>
__global__ void __launch_bounds__(kSvBlock, 5) shapley_voting_kernel(const __grid_constant__ ShapleyArgs a)
{
    __shared__ uint32_t s_keys[kSvWarps][kMaxRounds];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t warp = threadIdx.x >> 5;
    const Geometry &g = a.g;
    const uint32_t last = static_cast<uint32_t>(g.domain - 1u);
    uint32_t *keys = s_keys[warp];

    for (uint64_t smp = static_cast<uint64_t>(blockIdx.x) * kSvWarps + warp; smp < a.samples;
         smp += static_cast<uint64_t>(gridDim.x) * kSvWarps) {
        for (uint32_t r = lane; r < a.rounds; r += 32) keys[r] = dev::splitmix_key(a.seed0 + smp, r);
        __syncwarp();
        uint64_t carry = 0;  // weight of every kept player of the earlier chunks
        for (uint64_t base = 0; base < g.domain && carry < a.quota; base += kSvChunk) {
            uint32_t left[kSvItems], right[kSvItems];
            dev::cipher_run<ODD, kSvItems, 32, kSvGroup, FORM>(left, right, static_cast<uint32_t>(base) + lane, keys,
                                                        a.rounds, g);
            uint32_t player[kSvItems], wt[kSvItems];
            uint64_t mine = 0;  // this lane's weights of the chunk
#pragma unroll
            for (int j = 0; j < kSvItems; ++j) {
                const uint32_t i = static_cast<uint32_t>(base) + static_cast<uint32_t>(j * 32) + lane;
                player[j] = (left[j] << g.R) | right[j];
                wt[j] = i <= last && player[j] < g.n ? a.w[player[j]] : 0u;
                mine += wt[j];
            }
            // mine < 2^35: two warp sums of 24 and 11 bits are exact
            const uint64_t total = __reduce_add_sync(kFull, static_cast<uint32_t>(mine) & 0xffffffu) +
                                   (static_cast<uint64_t>(__reduce_add_sync(kFull, static_cast<uint32_t>(mine >> 24)))
                                    << 24);
            if (carry + total < a.quota) {  // no pivot in this chunk: no order within it is needed
                carry += total;
                continue;
            }
            for (int j = 0; j < kSvItems; ++j) {
                const uint64_t incl = dev::warp_inclusive_scan64(wt[j]);
                const uint64_t before = carry + incl - wt[j];
                // a player that is not kept has weight 0 and cannot reach the quota
                if (before < a.quota && before + wt[j] >= a.quota)
                    atomicAdd(reinterpret_cast<unsigned long long *>(a.counts + player[j]), 1ull);
                carry += __shfl_sync(kFull, incl, 31);
            }
        }
        __syncwarp();  // every lane is done with the keys before the next sample's
    }
}

}  // namespace

cudaError_t launch_shapley_voting(const ShapleyArgs &a, cudaStream_t stream)
{
    static std::atomic<int> per_sm[64];  // CTAs to launch per device, 0 until first use
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    int ctas_cached = per_sm[device].load(std::memory_order_acquire);
    if (ctas_cached == 0) {
        int blocks = 0, sms = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, shapley_voting_kernel<true, CipherForm::Float>, kSvBlock, 0);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e != cudaSuccess) return e;
        ctas_cached = (blocks > 0 ? blocks : 1) * sms;
        per_sm[device].store(ctas_cached, std::memory_order_release);
    }
    const uint64_t cap = static_cast<uint64_t>(ctas_cached);
    const uint64_t want = (a.samples + kSvWarps - 1) / kSvWarps;  // one warp per sample
    const unsigned grid = static_cast<unsigned>(want < cap ? want : cap);
    const bool odd = (a.g.k & 1u) != 0u;
    auto kernel = odd ? shapley_voting_kernel<true, CipherForm::Float> : shapley_voting_kernel<false, CipherForm::Float>;
    switch (cipher_run_form(a.g, kSvGroup * 32)) {
    case CipherForm::Float: break;
    case CipherForm::Short:
        kernel = odd ? shapley_voting_kernel<true, CipherForm::Short> : shapley_voting_kernel<false, CipherForm::Short>;
        break;
    case CipherForm::Mixed:
        kernel = odd ? shapley_voting_kernel<true, CipherForm::Mixed> : shapley_voting_kernel<false, CipherForm::Mixed>;
        break;
    default: kernel = odd ? shapley_voting_kernel<true, CipherForm::Wide> : shapley_voting_kernel<false, CipherForm::Wide>;
    }
    kernel<<<grid, kSvBlock, 0, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace bsh
