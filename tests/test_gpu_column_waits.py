"""The tile loop of the two-pass kernels (col_loop in csrc/colfft.cuh) when a load
never lands: every group gives up within the limit, the status word says
FLUSI_ETIMEOUT, the block ends, and the next launch runs as if nothing had been.
The loop runs here with jobs that move no data: a load is an arrival on its
barrier, and the withheld one announces bytes that nothing sends.
"""
import ctypes

import pytest

from device_code import shared_library

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "colfft.cuh"
using namespace flusi;
template <class X> struct Job {
    int tiles, withheld;
    int* worked;
    __device__ bool exists(int i) const { return i < tiles; }
    __device__ void issue(int i, int h, float2*, unsigned long long* bar) const
    {
        mbar_expect_tx(bar, i * X::CH + h == withheld ? 16 : 0);
    }
    __device__ void copy(int, int, float2*, int) const {}
    template <class Refill>
    __device__ void work(int i, const typename X::Tile&, int tid, int group, Refill refill) const
    {
        if (tid == 0 && i % X::GROUPS == group) atomicAdd(worked, 1);
        refill();
    }
};
template <class X> __global__ void __launch_bounds__(X::THREADS, 1)
loop(int tiles, int withheld, int tma, int* err, int* worked, long long limit)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ ColState state;
    float2* bufs = reinterpret_cast<float2*>(smem_raw + ((128 - (smem_u32(smem_raw) & 127)) & 127));
    Job<X> job{tiles, withheld, worked};
    col_loop<X>(bufs, state, tma != 0, err, job, limit);
}
template <class X> int go(int tiles, int withheld, int tma, int* err, int* worked, long long limit)
{
    const cudaError_t e = cudaFuncSetAttribute(loop<X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X::kSmem);
    if (e) return (int)e;
    loop<X><<<2, X::THREADS, X::kSmem>>>(tiles, withheld, tma, err, worked, limit);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run(int kind, int tiles, int withheld, int tma, int* err, int* worked, long long limit)
{
    if (kind == 0) return go<Col<16, 8, 16>>(tiles, withheld, tma, err, worked, limit);    // one group, one buffer
    if (kind == 1) return go<Col<32, 16, 16>>(tiles, withheld, tma, err, worked, limit);   // two groups, three buffers
    return go<Col<32, 32, 16>>(tiles, withheld, tma, err, worked, limit);                  // one group, tiles in halves
}
"""
TILES, LIMIT = 9, 2_000_000   # a millisecond of SM clocks
LOADS = {0: 1, 1: 1, 2: 2}    # per tile


@pytest.fixture(scope="module")
def loop(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    lib = ctypes.CDLL(shared_library(SOURCE, tmp_path_factory.mktemp("waits")))

    def run(kind, withheld, tma=1):
        """(status word, tiles worked on by the two blocks)"""
        out = torch.zeros(2, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        p = out.data_ptr()
        assert lib.run(kind, TILES, withheld, tma, ctypes.c_void_p(p), ctypes.c_void_p(p + 4), ctypes.c_longlong(LIMIT)) == 0
        return tuple(out.tolist())
    return run


@pytest.mark.parametrize("kind", [0, 1, 2])
def test_every_tile_once(loop, kind):
    assert loop(kind, -1) == (0, 2 * TILES)
    assert loop(kind, -1, tma=0) == (0, 2 * TILES)


@pytest.mark.parametrize("tile", [0, 1, 2, 3, 4, TILES - 1])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_a_load_that_never_lands(loop, kind, tile):
    for h in range(LOADS[kind]):
        err, worked = loop(kind, tile * LOADS[kind] + h)
        # the tiles before it are done and, where another group takes it, the one after
        assert err == 5 and worked == 2 * (tile + (kind == 1 and tile + 1 < TILES))
        assert loop(kind, -1) == (0, 2 * TILES)
