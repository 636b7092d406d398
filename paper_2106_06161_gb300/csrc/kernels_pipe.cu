// Pipelined single pass of Algorithm 1 (pipe_kernel.cuh): the default shapes
// for every mode and width, the table of shapes the gather of 4-, 8- and
// 16-byte elements can be tuned over, and the selection per width.
//
// Shape 0 is the default: eight compute warps of four indices a round, with
// the rounds per tile set by the call (pipe_rounds).  The other shapes are
// instantiated in kernels_pipe_tuned.cu and serve bshuffle_permute only.
#include <atomic>
#include <cstdint>

#include "bshuffle_internal.h"
#include "pipe_kernel.cuh"

namespace bsh {

const PipeConfig kPipeConfigs[kNumPipeConfigs] = {
    {8, 8, 4, 1}, {8, 4, 4, 1}, {8, 16, 3, 1}, {4, 8, 5, 1}, {16, 4, 2, 1}, {8, 8, 3, 0},
};

namespace {

std::atomic<int> g_pipe_selected[5];  // per width class: 1, 2, 4, 8, 16 bytes

int width_slot(uint32_t elem_bytes)
{
    switch (elem_bytes) {
    case 4: return 2;
    case 8: return 3;
    case 16: return 4;
    default: return -1;
    }
}

// Rounds of four indices per thread in a tile of the default shape.  Four (3
// CTAs per SM) where the kernel keeps the look-back warp busy: indices from
// 2^21 on, 4-byte gathers from there to 2^24, whose input the L2 holds, and
// narrower ones from 2^25 on.
// Two (4 CTAs per SM) elsewhere: smaller domains have too few tiles to fill
// the GPU with larger ones, larger gathers wait for memory, and the buffers
// of wider elements would take the L1 that the gathers in flight need.
// Measured on GB300, calls replayed from a graph, n = 15/16 of the domain,
// four rounds against two: indices 2^20 14.0 / 12.7 us, 2^22 29.5 / 29.6,
// 2^24 89.6 / 94.4; 4-byte gathers 2^20 15.2 / 14.8, 2^22 31.2 / 33.0, 2^24
// 103 / 109, 2^25 328 / 316; 8-byte gathers 2^22 46.6 / 35.6, 2^24 422 / 186;
// 8-byte scatters 2^22 39.4 / 39.2.  Two-byte gathers, four / two: 2^22 + 1
// 81.0 / 78.0, 2^24 + 1 263 / 269, 2^26 + 1 1087 / 1134, 2^28 + 1 4951 / 4955
// (in the plain fused kernel 84, 286, 1250 and 7099; two-byte scatters at 2^22
// + 1 81 against 88 there, at 2^26 + 1 1206 against 1454).
int pipe_rounds(uint32_t elem_bytes, Mode mode, uint32_t k)
{
    const bool index = mode == Mode::Index32 || mode == Mode::Index64;
    const bool gather4 = mode == Mode::Gather && elem_bytes == 4;
    const bool narrow = mode == Mode::Gather && elem_bytes < 4;
    return (index && k >= 21) || (gather4 && k >= 21 && k <= 24) || (narrow && k >= 25) ? 4 : 2;
}

template <class T, Mode MODE>
cudaError_t launch_default(const TileArgs &a, cudaStream_t stream)
{
    constexpr bool index = MODE == Mode::Index32 || MODE == Mode::Index64;
    if constexpr (index || (MODE == Mode::Gather && sizeof(T) <= 4))
        if (pipe_rounds(sizeof(T), MODE, a.g.k) == 4) return pipe::launch_shape<T, MODE, 8, 4, 4, 3, true>(a, stream);
    // one round of eight for scatters, and for 8-byte gathers that the L2 does
    // not hold: three CTAs of more accesses in flight each, instead of four
    // (8-byte gathers at 2^24 - 5 208 / 203 us, scatters at 2^22 + 1 of 4
    // bytes 76.4 / 74.6, 16-byte at 2^24 + 1 468 / 465)
    if constexpr (MODE == Mode::Scatter || (MODE == Mode::Gather && sizeof(T) == 8))
        if (MODE == Mode::Scatter || uint64_t{a.g.n} * sizeof(T) >= pipe::kTicketsAheadBytes)
            return pipe::launch_shape<T, MODE, 8, 8, 1, 3, true>(a, stream);
    return pipe::launch_shape<T, MODE, 8, 4, 2, 4, true>(a, stream);
}

}  // namespace

int pipe_config_for(uint32_t elem_bytes, Mode mode)
{
    const int slot = width_slot(elem_bytes);
    if (mode != Mode::Gather || slot < 0) return 0;
    return g_pipe_selected[slot].load();
}

int select_pipe_config(uint32_t elem_bytes, int config)
{
    const int slot = width_slot(elem_bytes);
    if (slot < 0 || config < 0 || config >= kNumPipeConfigs) return -1;
    g_pipe_selected[slot].store(config);
    return 0;
}

int selected_pipe_config(uint32_t elem_bytes)
{
    const int slot = width_slot(elem_bytes);
    return slot < 0 ? 0 : g_pipe_selected[slot].load();
}

uint32_t pipe_tile_size(uint32_t elem_bytes, int config, Mode mode, uint32_t k)
{
    if (config == 0) return 8u * 32u * 4u * static_cast<uint32_t>(pipe_rounds(elem_bytes, mode, k));
    const PipeConfig &c = kPipeConfigs[config >= 0 && config < kNumPipeConfigs ? config : 0];
    return static_cast<uint32_t>(c.warps * 32 * c.items);
}

bool pipe_supports(Mode mode, uint32_t elem_bytes)
{
    switch (mode) {
    case Mode::Gather:
    case Mode::Scatter:
        return elem_bytes == 1 || elem_bytes == 2 || elem_bytes == 4 || elem_bytes == 8 || elem_bytes == 16;
    case Mode::Index32:
    case Mode::Index64: return true;
    }
    return false;
}

cudaError_t launch_pipe(const TileArgs &a, Mode mode, uint32_t elem_bytes, int config, cudaStream_t stream)
{
    if (config != 0) {
        if (mode != Mode::Gather) return cudaErrorInvalidValue;
        return launch_pipe_tuned(a, elem_bytes, config, stream);
    }
    switch (mode) {
    case Mode::Index32: return launch_default<unsigned int, Mode::Index32>(a, stream);
    case Mode::Index64: return launch_default<unsigned long long, Mode::Index64>(a, stream);
    case Mode::Gather:
        switch (elem_bytes) {
        case 1: return launch_default<unsigned char, Mode::Gather>(a, stream);
        case 2: return launch_default<unsigned short, Mode::Gather>(a, stream);
        case 4: return launch_default<unsigned int, Mode::Gather>(a, stream);
        case 8: return launch_default<unsigned long long, Mode::Gather>(a, stream);
        case 16: return launch_default<uint4, Mode::Gather>(a, stream);
        default: return cudaErrorInvalidValue;
        }
    case Mode::Scatter:
        switch (elem_bytes) {
        case 1: return launch_default<unsigned char, Mode::Scatter>(a, stream);
        case 2: return launch_default<unsigned short, Mode::Scatter>(a, stream);
        case 4: return launch_default<unsigned int, Mode::Scatter>(a, stream);
        case 8: return launch_default<unsigned long long, Mode::Scatter>(a, stream);
        case 16: return launch_default<uint4, Mode::Scatter>(a, stream);
        default: return cudaErrorInvalidValue;
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace bsh
