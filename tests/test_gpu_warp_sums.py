"""A warp's twelve force sums (warp_sums12 in csrc/xphys.cuh): those of FP32 values
are no further from the exact sums than the same tree in FP64, over ordinary,
cancelling, wide-ranging, tiny and huge values, and infinities and sums past the
FP32 range come out as FP64 gives them.  The bound is that of the FP64 tree: five
levels, each rounded once, 5 2^-53 of the sum of magnitudes, and one rounding of
the result.
"""
import ctypes
import fractions

import numpy as np
import pytest

from device_code import shared_library

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "xphys.cuh"
using namespace flusi;
template <class T> __global__ void sums(const float* v, double* w)   // v[warp][lane][12], w[warp][12]
{
    __shared__ double s[12];
    if (threadIdx.x < 12) s[threadIdx.x] = 0.0;
    __syncwarp();
    T a[12];
    for (int k = 0; k < 12; ++k) a[k] = T(v[((size_t)blockIdx.x * 32 + threadIdx.x) * 12 + k]);
    warp_sums12(a, s, threadIdx.x);
    __syncwarp();
    if (threadIdx.x < 12) w[(size_t)blockIdx.x * 12 + threadIdx.x] = s[threadIdx.x];
}
extern "C" int run(const float* v, double* w32, double* w64, int warps)
{
    sums<float><<<warps, 32>>>(v, w32);
    sums<double><<<warps, 32>>>(v, w64);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    lib = ctypes.CDLL(shared_library(SOURCE, tmp_path_factory.mktemp("sums")))

    def run(v):
        """(FP32 form, FP64 form) of the sums over axis 1 of v[warp][lane][12]."""
        d = torch.as_tensor(v).cuda()
        out = [torch.zeros(v.shape[0], 12, dtype=torch.float64, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        args = [ctypes.c_void_p(t.data_ptr()) for t in (d, *out)]
        assert lib.run(*args, v.shape[0]) == 0
        return [t.cpu().numpy() for t in out]
    return run


def _values(kind, warps=256):
    rng = np.random.default_rng(11)
    shape = (warps, 32, 12)
    v = rng.uniform(-1, 1, shape)
    if kind == "positive":
        v = rng.uniform(0, 1, shape)
    elif kind == "wide":
        v = v * 10.0 ** rng.uniform(-20, 20, shape)
    elif kind == "cancelling":   # large values that leave, in pairs some lanes apart, small ones
        for w in range(warps):
            p = rng.permutation(32)
            big = v[w, p[:16]] * 10.0 ** rng.uniform(0, 12, (16, 1))
            v[w, p[:16]], v[w, p[16:]] = big, np.nextafter(-big.astype(np.float32), np.float32(0))
    elif kind == "tiny":
        v = v * 1e-38
    elif kind == "few":          # one point of a warp, as at the edge of a part
        v[:, 1:] = 0
    elif kind == "huge":
        v = v * 3.4e38
    return v.astype(np.float32)


KINDS = ["uniform", "positive", "wide", "cancelling", "tiny", "few", "huge"]


@pytest.mark.parametrize("kind", KINDS)
def test_no_further_from_the_exact_sums_than_fp64(sums, kind):
    v = _values(kind)
    got, tree = sums(v)
    err, ref = [], []
    for w in range(v.shape[0]):
        for k in range(12):
            terms = [fractions.Fraction(float(x)) for x in v[w, :, k]]
            exact, size = sum(terms), sum(map(abs, terms))
            e = abs(fractions.Fraction(float(got[w, k])) - exact)
            assert e <= 5 * size * fractions.Fraction(1, 2 ** 53) + abs(exact) * fractions.Fraction(1, 2 ** 53), (kind, w, k)
            err.append(float(e))
            ref.append(float(abs(fractions.Fraction(float(tree[w, k])) - exact)))
    # over all sums: no larger than the FP64 tree's, but for the rounding of the result
    assert np.sum(err) <= np.sum(ref) + 2.0 ** -53 * np.sum(np.abs(tree))


def test_past_the_fp32_range(sums):
    big = np.float32(3e38)
    v = np.zeros((5, 32, 12), np.float32)
    v[0] = big                                   # 32 of them: 9.6e39
    v[1, 3], v[1, 9] = np.inf, 1.0
    v[2, 0], v[2, 31] = -np.inf, big
    v[3, 4], v[3, 20] = np.inf, -np.inf
    v[4, 5, ::2] = np.nan
    got, tree = sums(v)
    assert np.array_equal(got, tree, equal_nan=True)
    assert (tree[0] == 32.0 * float(big)).all() and (got[1] == np.inf).all() and (got[2] == -np.inf).all()
