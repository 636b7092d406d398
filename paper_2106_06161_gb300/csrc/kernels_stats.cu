// The GPU side of the MMD test of Sec. 5 (Mallows kernel): permutations
// sampled as ranks, Kendall discordant-pair counts of their pairs, and the
// inversion of slot orders.
//
// For each pair p of permutations (s, t) = (perms[2p], perms[2p + 1]) of
// [0, n), n_dis = #{i < j : (s_i < s_j) != (t_i < t_j)}.  Ordered by s, the
// pair becomes one sequence c (c[s_i] = t_i) and n_dis its inversions.  One
// warp owns one pair at a time and walks c 32 elements a step: the inversions
// with earlier steps are the set bits above the element in a shared-memory
// bitmap of the values seen (a count of the words above it and a population
// count of its own word), those inside the step come from one ballot per
// value bit.  A step recounts the bitmap, a word a lane: n / 32 steps and about
// n^2 / 1024 word counts a pair, where comparing every pair in shared memory
// took n^2 / 2 comparisons and was bound by the shared-memory loads (96 %
// busy): 50,000 pairs of length 1000 on GB300: 5.53 -> 0.47 ms.
// Rows that are not permutations of [0, n) have no such sequence: their pairs
// are marked and counted by the all-pairs kernel, a CTA per pair at a time,
// which also serves few short rows (all_pairs_by_default).
#include <atomic>
#include <cstdint>

#include "bshuffle_device.cuh"

#include "bshuffle_internal.h"

namespace bsh {
namespace {

using dev::kFull;

constexpr int kKBlock = 256;
constexpr int kKWarps = kKBlock / 32;
constexpr uint32_t kMaxN = 4096;
constexpr uint64_t kNotPermutations = ~uint64_t{0};  // above every count (n_dis < 2^23)

// Shared memory of one warp of the inversion count: the sequence c (16-bit),
// the bitmap of the values seen and the set bits above each of its words.
__host__ __device__ constexpr uint32_t kendall_words(uint32_t n) { return (n + 1023u) / 1024u * 32u; }
__host__ __device__ constexpr uint32_t kendall_warp_bytes(uint32_t n)
{
    return (n + 31u) / 32u * 64u + 2u * kendall_words(n) * 4u;
}

__global__ void __launch_bounds__(kKBlock) kendall_inversions_kernel(const uint32_t *__restrict__ perms, uint32_t n,
                                                                     uint32_t value_bits, uint64_t pairs,
                                                                     uint64_t *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t lt = dev::lanemask_lt();
    const uint32_t words = kendall_words(n);
    unsigned char *mine = s_raw + warp * kendall_warp_bytes(n);
    uint32_t *bits = reinterpret_cast<uint32_t *>(mine);
    uint32_t *above = bits + words;
    uint16_t *c = reinterpret_cast<uint16_t *>(above + words);

    for (uint64_t p = uint64_t{blockIdx.x} * kKWarps + warp; p < pairs; p += uint64_t{gridDim.x} * kKWarps) {
        const uint32_t *a = perms + 2 * p * n;
        const uint32_t *b = a + n;
        for (uint32_t w = lane; w < words; w += 32) bits[w] = 0u;
        __syncwarp();
        bool ok = true;
#pragma unroll 4
        for (uint32_t i = lane; i < n; i += 32) {
            const uint32_t s = a[i], t = b[i];
            if (s < n && t < n) {
                const uint32_t old = atomicOr(&bits[s >> 5], 1u << (s & 31u));
                ok = ok && ((old >> (s & 31u)) & 1u) == 0u;
                c[s] = static_cast<uint16_t>(t);
            } else {
                ok = false;
            }
        }
        if (!__all_sync(kFull, ok)) {
            if (lane == 0) out[p] = kNotPermutations;
            __syncwarp();
            continue;
        }
        __syncwarp();
        for (uint32_t w = lane; w < words; w += 32) {
            bits[w] = 0u;
            above[w] = 0u;
        }
        __syncwarp();
        uint32_t count = 0;
        for (uint32_t first = 0; first < n; first += 32) {
            const bool live = first + lane < n;  // lanes past the end come after every live one
            const uint32_t v = live ? c[first + lane] : 0u;
            const uint32_t w = v >> 5;
            if (live) count += above[w] + static_cast<uint32_t>(__popc(bits[w] & (0xfffffffeu << (v & 31u))));
            // lanes whose value is greater: the first differing bit decides
            uint32_t greater = 0, equal = kFull;
            for (uint32_t bit = value_bits; bit-- > 0u;) {
                const bool one = (v >> bit) & 1u;
                const uint32_t ones = __ballot_sync(kFull, one);
                if (!one) greater |= equal & ones;
                equal &= one ? ones : ~ones;
            }
            if (live) count += static_cast<uint32_t>(__popc(greater & lt));
            __syncwarp();
            if (live) {
                const uint32_t old = atomicOr(&bits[w], 1u << (v & 31u));
                ok = ok && ((old >> (v & 31u)) & 1u) == 0u;
            }
            __syncwarp();
            uint32_t higher = 0;  // set bits of the words after these 32
            for (uint32_t q = words; q > 0u; q -= 32u) {
                const uint32_t pc = static_cast<uint32_t>(__popc(bits[q - 32u + lane]));
                uint32_t sum = pc;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t u = __shfl_down_sync(kFull, sum, d);
                    if (lane + static_cast<uint32_t>(d) < 32u) sum += u;
                }
                above[q - 32u + lane] = higher + sum - pc;
                higher += __shfl_sync(kFull, sum, 0);
            }
            __syncwarp();
        }
        count = __reduce_add_sync(kFull, count);
        ok = __all_sync(kFull, ok);
        if (lane == 0) out[p] = ok ? count : kNotPermutations;
    }
}

// Every pair i < j compared: all pairs of rows (ALL), or those marked as no
// permutations.
// CTA c owns the pairs c, c + gridDim.x, ..., so that marked pairs which follow
// one another (all of them, where the rows have ties) run on as many CTAs; one
// strided load per thread finds the marks of 256 of them at a time.  (With 256
// consecutive pairs a CTA, 256 marked ones of length 1000 took 6.0 ms.)
struct KendallShared {
    uint32_t a[kMaxN];
    uint32_t b[kMaxN];
    unsigned long long sum[kKWarps];
    uint32_t marked[kKWarps];  // a bit per pair of 256
};

// Pair p by the whole CTA.
__device__ __forceinline__ void count_all_pairs(const uint32_t *__restrict__ perms, uint32_t n, uint64_t p,
                                                uint64_t *__restrict__ out, KendallShared &sh)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t *a = perms + 2 * p * n;
    const uint32_t *b = a + n;
    for (uint32_t i = tid; i < n; i += kKBlock) {
        sh.a[i] = a[i];
        sh.b[i] = b[i];
    }
    __syncthreads();
    unsigned long long count = 0;
    // rows i and n-1-i together keep the work per thread balanced
    for (uint32_t i = tid; i < (n + 1) / 2; i += kKBlock) {
        for (uint32_t r = 0; r < 2; ++r) {
            const uint32_t row = r == 0 ? i : n - 1 - i;
            if (r == 1 && row == i) break;
            const uint32_t ai = sh.a[row], bi = sh.b[row];
            uint32_t c = 0;
            for (uint32_t j = row + 1; j < n; ++j) c += ((ai < sh.a[j]) != (bi < sh.b[j])) ? 1u : 0u;
            count += c;
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) count += __shfl_down_sync(kFull, count, d);
    if (lane == 0) sh.sum[warp] = count;
    __syncthreads();
    if (tid == 0) {
        unsigned long long total = 0;
        for (int w = 0; w < kKWarps; ++w) total += sh.sum[w];
        out[p] = total;
    }
    __syncthreads();
}

template <bool ALL>
__global__ void __launch_bounds__(kKBlock) kendall_pairs_kernel(const uint32_t *__restrict__ perms, uint32_t n,
                                                                uint64_t pairs, uint64_t *__restrict__ out)
{
    __shared__ KendallShared sh;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint64_t step = gridDim.x;
    if constexpr (ALL) {
        for (uint64_t p = blockIdx.x; p < pairs; p += step) count_all_pairs(perms, n, p, out, sh);
        return;
    }
    for (uint64_t p0 = blockIdx.x; p0 < pairs; p0 += kKBlock * step) {
        const uint64_t mine = p0 + tid * step;
        const bool marked = mine < pairs && out[mine] == kNotPermutations;
        const uint32_t ball = __ballot_sync(kFull, marked);
        if (lane == 0) sh.marked[warp] = ball;
        if (!__syncthreads_or(marked)) continue;
        // a word of marks and the bit taken from it: the same for the whole CTA
        uint32_t word = 0, bits = sh.marked[0];
        while (true) {
            while (bits == 0u && ++word < kKWarps) bits = sh.marked[word];
            if (bits == 0u) break;
            count_all_pairs(perms, n, p0 + (word * 32u + static_cast<uint32_t>(__ffs(bits)) - 1u) * step, out, sh);
            bits &= bits - 1u;
        }
        __syncthreads();  // the marks are read before the next ones are written
    }
}

// Comparing every pair takes one launch and no bitmap: faster for few short
// rows.  Calls replayed from a graph on GB300, all pairs / inversions, us: n =
// 32, 600 pairs 2.6 / 3.9, 1,200 4.3 / 4.5, 2,500 7.1 / 5.2; n = 100, 600 3.7 /
// 6.4, 1,200 6.4 / 7.0; n = 200, 600 6.2 / 7.9, 1,200 10.4 / 8.6; n = 300, 300
// 6.6 / 10.0, 600 9.8 / 10.1, 1,200 16.7 / 10.7; n = 400, 100
// 6.9 / 11.8, 300 9.2 / 11.9, 600 15.1 / 12.0; n = 600 (a thread then has
// several rows), 16 15.5 / 16.3, 300 19.2 / 16.5.
bool all_pairs_by_default(uint32_t n, uint64_t pairs, uint64_t resident)
{
    return n <= 2 * kKBlock && pairs <= resident && pairs * n <= 180'000u;
}

// Row r of `sigma` = the ranks of the shuffle with seed seed0 + r:
// sigma[f(i_j)] = j (Sec. 2's convention), so a sample of permutations comes
// from the seeds alone.  One warp owns a row at a time: it walks the domain in
// chunks of 256 indices, ranks the kept ones with ballots and a running count,
// places each rank at its element in shared memory (16 bits, n <= 4096) and
// writes the row out in order.  Nothing but the ranks touches memory; the
// batched shuffle of copies of 0 .. n-1 and the inversion of its slot orders
// moved four times their bytes through five kernels and a table of
// descriptors.  Bound by the cipher (ALU pipe).  100,000 rows of 1000 on
// GB300: 0.39 ms (the five kernels 2.6 ms, behind 10 ms of host work for the
// descriptors).
constexpr int kRItems = 8;
constexpr uint32_t kRChunk = 32 * kRItems;
__host__ __device__ constexpr uint32_t ranks_warp_bytes(uint32_t n) { return (n + 7u) / 8u * 16u; }

struct RanksArgs {
    uint32_t *sigma;
    Geometry g;  // g.n = length of a row
    uint32_t rounds;
    uint32_t pad0;
    uint64_t seed0;
    uint64_t rows;
};

template <bool ODD>
__global__ void __launch_bounds__(kKBlock) sample_ranks_kernel(const __grid_constant__ RanksArgs a)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ uint32_t s_keys[kKWarps][kMaxRounds];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t lt = dev::lanemask_lt();
    const Geometry &g = a.g;
    const uint32_t last = static_cast<uint32_t>(g.domain - 1u);
    uint16_t *rank = reinterpret_cast<uint16_t *>(s_raw + warp * ranks_warp_bytes(g.n));
    uint32_t *keys = s_keys[warp];

    for (uint64_t r = uint64_t{blockIdx.x} * kKWarps + warp; r < a.rows; r += uint64_t{gridDim.x} * kKWarps) {
        for (uint32_t q = lane; q < a.rounds; q += 32) keys[q] = dev::splitmix_key(a.seed0 + r, q);
        __syncwarp();
        uint32_t running = 0;
        for (uint32_t base = 0; base <= last; base += kRChunk) {
            uint32_t left[kRItems], right[kRItems];
#pragma unroll
            for (int j = 0; j < kRItems; ++j) {
                const uint32_t i = base + static_cast<uint32_t>(j * 32) + lane;
                left[j] = i >> g.R;
                right[j] = i & g.rmask;
            }
            dev::cipher_items<ODD, kRItems, CipherForm::Float>(  // n <= 4096
                left, right, keys, a.rounds, g);
#pragma unroll
            for (int j = 0; j < kRItems; ++j) {
                const uint32_t i = base + static_cast<uint32_t>(j * 32) + lane;
                const uint32_t src = (left[j] << g.R) | right[j];
                const bool keep = i <= last && src < g.n;
                const uint32_t m = __ballot_sync(kFull, keep);
                if (keep) rank[src] = static_cast<uint16_t>(running + static_cast<uint32_t>(__popc(m & lt)));
                running += static_cast<uint32_t>(__popc(m));
            }
        }
        __syncwarp();
        uint32_t *row = a.sigma + r * g.n;
        for (uint32_t e = lane; e < g.n; e += 32) row[e] = rank[e];
        __syncwarp();  // the row is read before the next one is placed
    }
}

// sigma[r][idx[r][j]] = j for every row r: a shuffle's slot order (element
// idx[j] in slot j) turned into the rank of each element, the permutation
// convention of Sec. 2.
__global__ void __launch_bounds__(kKBlock) invert_rows_kernel(const uint32_t *__restrict__ idx, uint32_t n,
                                                              uint64_t rows, uint32_t *__restrict__ sigma)
{
    const uint64_t total = rows * n;
    for (uint64_t e = static_cast<uint64_t>(blockIdx.x) * kKBlock + threadIdx.x; e < total;
         e += static_cast<uint64_t>(gridDim.x) * kKBlock) {
        const uint64_t r = e / n;
        const uint32_t j = static_cast<uint32_t>(e - r * n);
        const uint32_t v = idx[e];
        if (v < n) sigma[r * n + v] = j;
    }
}

}  // namespace

uint32_t kendall_max_n() { return kMaxN; }

cudaError_t launch_sample_ranks(const Geometry &g, uint32_t rounds, uint64_t seed0, uint64_t rows, uint32_t *sigma,
                                cudaStream_t stream)
{
    if (g.n == 0u || g.n > kMaxN) return cudaErrorInvalidValue;
    int device = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    const auto odd = sample_ranks_kernel<true>, even = sample_ranks_kernel<false>;
    static std::atomic<bool> configured[64];  // attributes set on this device
    if (!configured[device].load(std::memory_order_acquire)) {
        const int most = static_cast<int>(kKWarps * ranks_warp_bytes(kMaxN));
        e = cudaFuncSetAttribute(odd, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(even, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
        configured[device].store(true, std::memory_order_release);
    }
    RanksArgs a{};
    a.sigma = sigma;
    a.g = g;
    a.rounds = rounds;
    a.seed0 = seed0;
    a.rows = rows;
    const uint64_t blocks = (rows + kKWarps - 1) / kKWarps;
    const uint64_t most = static_cast<uint64_t>(sms) * 16;
    const unsigned grid = static_cast<unsigned>(blocks < most ? blocks : most);
    ((g.k & 1u) ? odd : even)<<<grid, kKBlock, kKWarps * ranks_warp_bytes(g.n), stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_invert_rows(const uint32_t *idx, uint32_t n, uint64_t rows, uint32_t *sigma, cudaStream_t stream)
{
    int device = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    const uint64_t blocks = (rows * n + kKBlock - 1) / kKBlock;
    const uint64_t grid = blocks < static_cast<uint64_t>(sms) * 16 ? blocks : static_cast<uint64_t>(sms) * 16;
    invert_rows_kernel<<<static_cast<unsigned>(grid), kKBlock, 0, stream>>>(idx, n, rows, sigma);
    return cudaGetLastError();
}

cudaError_t launch_kendall_pairs(const uint32_t *perms, uint32_t n, uint64_t pairs, uint64_t *out,
                                 cudaStream_t stream)
{
    int device = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    const uint64_t most = static_cast<uint64_t>(sms) * 8;
    const unsigned grid = static_cast<unsigned>(pairs < most ? pairs : most);
    if (all_pairs_by_default(n, pairs, most)) {
        kendall_pairs_kernel<true><<<grid, kKBlock, 0, stream>>>(perms, n, pairs, out);
        return cudaGetLastError();
    }
    static std::atomic<bool> configured[64];  // attribute set on this device
    if (!configured[device].load(std::memory_order_acquire)) {
        e = cudaFuncSetAttribute(kendall_inversions_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 static_cast<int>(kKWarps * kendall_warp_bytes(kMaxN)));
        if (e != cudaSuccess) return e;
        configured[device].store(true, std::memory_order_release);
    }
    uint32_t value_bits = 0;
    while ((1u << value_bits) < n) ++value_bits;
    const uint64_t blocks = (pairs + kKWarps - 1) / kKWarps;
    kendall_inversions_kernel<<<static_cast<unsigned>(blocks < most ? blocks : most), kKBlock,
                                kKWarps * kendall_warp_bytes(n), stream>>>(perms, n, value_bits, pairs, out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // half of the CTAs that fit: 0.2 us a call that has nothing marked (0.7 with
    // all of them, 2,000 pairs of length 1000 31.7 and 32.3 us), and 2,000 pairs
    // with ties of length 1000 247 us (240)
    const unsigned check = static_cast<unsigned>(pairs < most / 2 ? pairs : most / 2);
    kendall_pairs_kernel<false><<<check, kKBlock, 0, stream>>>(perms, n, pairs, out);
    return cudaGetLastError();
}

}  // namespace bsh
