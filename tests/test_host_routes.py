"""Host-side choice between the one-launch and the per-field read-back of evp_get_fields
(no GPU): evp_abi.cu compiled with the runtime's pointer queries replaced by a table of
allocations, so that buffers on other devices and at allocations' ends can be had."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, 'paper_1803_09563_gb300', 'csrc')

# arguments: the current device; then the state's arena and two destinations, each as
# device, offset in its allocation and the allocation's bytes.  Prints 1 for one launch.
PROGRAM = r'''
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>
#include <cstdlib>
static int cur = 0;
struct Alloc { uintptr_t base; size_t size; int dev; };
static Alloc table[3];
static const Alloc* find(uintptr_t p) {
    for (const Alloc& a : table)
        if (p >= a.base && p < a.base + a.size) return &a;
    return nullptr;
}
static cudaError_t t_device(int* d) { *d = cur; return cudaSuccess; }
static cudaError_t t_attr(cudaPointerAttributes* at, const void* p) {
    const Alloc* a = find((uintptr_t)p);
    *at = cudaPointerAttributes{};
    at->type = a ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    at->device = a ? a->dev : -2;
    return cudaSuccess;
}
static CUresult t_range(CUdeviceptr* base, size_t* size, CUdeviceptr p) {
    const Alloc* a = find((uintptr_t)p);
    if (!a) return CUDA_ERROR_INVALID_VALUE;
    *base = a->base;
    *size = a->size;
    return CUDA_SUCCESS;
}
static cudaError_t t_entry(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* r) {
    *f = reinterpret_cast<void*>(&t_range);
    *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
#define cudaGetDriverEntryPointByVersion t_entry
#define cudaGetDevice t_device
#define cudaPointerGetAttributes t_attr
#include "evp_abi.cu"
int main(int, char** v) {
    cur = atoi(v[1]);
    uintptr_t at[3];
    for (int q = 0; q < 3; ++q) {
        table[q] = {uintptr_t(q + 1) << 40, (size_t)atoll(v[4 + 3 * q]), atoi(v[2 + 3 * q])};
        at[q] = table[q].base + atoll(v[3 + 3 * q]);
    }
    evp_state_s* s = new evp_state_s{};
    s->arena = reinterpret_cast<char*>(at[0]);
    s->arena_bytes = 1 << 16;
    void* d[2] = {reinterpret_cast<void*>(at[1]), reinterpret_cast<void*>(at[2])};
    std::printf("%d\n", one_launch(s, 2, d, 4096) ? 1 : 0);
    return 0;
}
'''
ARENA, BUF = 1 << 16, 4096


@pytest.fixture(scope='module')
def route(tmp_path_factory):
    from paper_1803_09563_gb300 import build
    nvcc = build.nvcc()
    if shutil.which(nvcc) is None:
        pytest.skip('needs nvcc')
    d = tmp_path_factory.mktemp('routes')
    src, exe = d / 'routes.cu', d / 'routes'
    src.write_text(PROGRAM)
    subprocess.run([nvcc, '-std=c++17', '-O1', '-I', CSRC, '-I', os.path.join(ROOT, 'include'), str(src), '-o', str(exe),
                    '-Xlinker', '--unresolved-symbols=ignore-all'], check=True)

    def run(cur, arena, a, b):
        args = [cur, arena, 0, ARENA] + list(a) + list(b)
        return int(subprocess.run([str(exe)] + [str(x) for x in args], capture_output=True, text=True,
                                  check=True).stdout)
    return run


# current device, the arena's, the destinations'
@pytest.mark.parametrize("cur,arena,a,b,want", [
    (0, 0, 0, 0, 1), (1, 1, 1, 1, 1),
    (0, 1, 0, 0, 0),       # a state on device 1 read into buffers on the current device 0
    (1, 0, 1, 1, 0), (0, 0, 1, 1, 0), (0, 0, 0, 1, 0), (1, 0, 0, 0, 0)])
def test_one_launch_only_on_one_device(route, cur, arena, a, b, want):
    assert route(cur, arena, (a, 0, BUF), (b, 256, BUF + 256)) == want


# destinations that end with their allocation and one byte (or far) beyond it
@pytest.mark.parametrize("a,b,want", [
    ((0, BUF), (0, BUF), 1), ((512, BUF + 512), (0, BUF), 1), ((0, BUF - 1), (0, BUF), 0),
    ((0, BUF), (0, BUF // 2), 0), ((0, BUF), (512, BUF), 0)])
def test_one_launch_only_inside_the_allocations(route, a, b, want):
    assert route(0, 0, (0,) + a, (0,) + b) == want


# two buffers of one allocation, the second ending with it and beyond it
@pytest.mark.parametrize("extra,want", [(0, 1), (1, 0), (BUF, 0)])
def test_one_launch_with_two_buffers_of_one_allocation(route, extra, want):
    # the program puts allocation q at (q + 1) 2^40: the third buffer's offset reaches back
    assert route(0, 0, (0, 0, 2 * BUF), (0, BUF + extra - (1 << 40), BUF)) == want
