"""A stream's workspace when it cannot grow: the library's host code linked
against a CUDA runtime made of host memory, whose allocations can be told to
fail, and a batched launch that only looks at the header and the look-back ring
it is given.  A word of the ring is a status of an earlier launch if its tag is
below the header's; any other one would be taken for a status of this launch."""
import os
import subprocess

import pytest

from paper_2106_06161_gb300 import build

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "bshuffle.h"
#include "bshuffle_internal.h"

static bool g_fail = false;
static int g_launches = 0, g_stale = 0;
static std::size_t g_live = 0;

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n)
{
    if (g_fail) return cudaErrorMemoryAllocation;
    *p = malloc(n);
    ++g_live;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { free(p); --g_live; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}

namespace bsh {
constexpr uint64_t kRing = 1024;
uint64_t batch_ring_words() { return kRing; }
uint32_t elem_tile_size(int) { return 2048; }
int elem_config_for(uint32_t, Mode, uint32_t) { return 0; }
bool pipe_supports(Mode, uint32_t) { return false; }
cudaError_t launch_elem(const TileArgs &, Mode, uint32_t, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_batched(const BatchArgs &a, cudaStream_t)
{
    ++g_launches;
    for (uint64_t w = 0; w < kRing; ++w)
        if (a.status[w] >= a.ws->batch_tag) ++g_stale;
    for (uint64_t w = 0; w < kRing; ++w) a.status[w] = a.ws->batch_tag;
    a.ws->batch_tag += 1;
    return cudaSuccess;
}
}  // namespace bsh

int main(int argc, char **argv)
{
    const bool fail = argc > 1 && atoi(argv[1]) != 0;
    static unsigned char out[64] __attribute__((aligned(16)));
    static bshuffle_desc desc;
    bshuffle_set_strategy(BSHUFFLE_STRATEGY_SINGLE_PASS);
    for (int i = 0; i < 3; ++i)
        if (bshuffle_batched(&desc, 1, 8, 24, nullptr) != BSHUFFLE_OK) return 2;
    g_fail = fail;
    // 2^16 status words, 16 times what the stream has
    if (bshuffle_indices(out, 8, uint64_t{1} << 27, 1, 24, nullptr) != (fail ? BSHUFFLE_ERR_CUDA : BSHUFFLE_OK)) return 3;
    g_fail = false;
    for (int i = 0; i < 3; ++i)
        if (bshuffle_batched(&desc, 1, 8, 24, nullptr) != BSHUFFLE_OK) return 4;
    if (bshuffle_release_workspaces() != BSHUFFLE_OK) return 5;
    std::printf("%d launches, %d stale words, %d buffers left\n", g_launches, g_stale, (int)g_live);
    return g_launches == 6 && g_stale == 0 && g_live == 0 ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp("host")
    (d / "main.cpp").write_text(MAIN)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    # the objects alone, without the CUDA runtime; what is not called stays undefined
    subprocess.run(["g++", "-std=c++17", "-I", f"{build.ROOT}/include", "-I", build.CSRC, "-I", cuda,
                    str(d / "main.cpp"), f"{build.BUILD_DIR}/bshuffle_api.cu.o", "-o", str(d / "main"),
                    "-Wl,--unresolved-symbols=ignore-all", "-lpthread"], check=True)
    return str(d / "main")


@pytest.mark.parametrize("fail", [0, 1])
def test_no_status_of_an_earlier_batch_is_taken_for_the_next_ones(program, fail):
    r = subprocess.run([program, str(fail)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
