"""dm_powf2 (the packed power of the FP32 pyramid): every lane has the bits of
the scalar recipe dm_powf.  All 2^23 mantissas at exponents over the whole
range, several lambdas, and the values at the ends of the packed path's range
(zeros, subnormals, infinity, NaN among them).  The scalar recipe itself is
compared with the oracle by the pyramid tests.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "dm_internal.cuh"
__global__ void k(const float* x, long long n, float lam, unsigned long long* bad) {
    const DmPow r = dm_pow_setup(lam);
    for (long long i = 2 * (blockIdx.x * (long long)blockDim.x + threadIdx.x); i + 1 < n; i += 2LL * gridDim.x * blockDim.x) {
        const float2 v = dm_powf2(make_float2(x[i], x[i + 1]), r);
        const float a = dm_powf(x[i], lam), b = dm_powf(x[i + 1], lam);
        if (__float_as_uint(v.x) != __float_as_uint(a) || __float_as_uint(v.y) != __float_as_uint(b)) atomicAdd(bad, 1ull);
    }
}
extern "C" int compare(const float* x, long long n, float lam, unsigned long long* bad) {
    k<<<1216, 256>>>(x, n, lam, bad);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build
    d = tmp_path_factory.mktemp("pow")
    src, lib = d / "pow.cu", d / "pow.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"),
                    "-shared", "-cudart", "static", "-o", str(lib), str(src)], check=True)
    fn = C.CDLL(str(lib)).compare
    fn.argtypes = [C.c_void_p, C.c_longlong, C.c_float, C.c_void_p]

    def run(bits, lam):
        x = torch.from_numpy(np.ascontiguousarray(bits, dtype=np.uint32).view(np.int32)).cuda()
        bad = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        assert fn(x.data_ptr(), x.numel(), lam, bad.data_ptr()) == 0
        return int(bad.item())

    return run


@pytest.mark.parametrize("lam", [1.4, 1.0, 0.5, 2.75])
def test_every_mantissa(compare, lam):
    m = np.arange(1 << 23, dtype=np.uint32)
    for e in (127, 126, 125, 124, 120, 111, 96, 64, 33, 2, 1):
        assert compare(m | np.uint32(e << 23), lam) == 0, f"exponent {e - 127}"


@pytest.mark.parametrize("lam", [1.4, 0.02, 37.0])
def test_range_ends(compare, lam):
    rng = np.random.default_rng(3)
    x = rng.integers(0, 1 << 32, size=1 << 20, dtype=np.uint64).astype(np.uint32)   # any bits: NaN, infinities, negatives
    x[:8] = np.array([0, 0x80000000, 1, 0x007fffff, 0x00800000, 0x7f7fffff, 0x3f800000, 0x3f7fffff], dtype=np.uint32)
    ok = np.isfinite(x.view(np.float32)) & (x.view(np.float32) <= 1.0)
    assert compare(x[ok][: ok.sum() // 2 * 2], lam) == 0


@pytest.mark.parametrize("lam", [1.4, 1.0, 0.5, 2.75, 0.02, 37.0])
def test_every_mantissa_above_one(compare, lam):
    """Unnormalised descriptor fields give maps above 1: up to the packed path's upper end 2^(100 / lam) and past it."""
    m = np.arange(1 << 23, dtype=np.uint32)
    top = int(min(100.0 / lam, 100.0))
    for e in sorted({0, 1, 2, top // 2, max(top - 1, 0), top, top + 1}):
        assert compare(m | np.uint32((e + 127) << 23), lam) == 0, f"exponent {e}"


@pytest.mark.parametrize("lam", [1.4, 0.02, 37.0, 0.005, 2.0e4])
def test_ends_and_mixed_pairs(compare, lam):
    """A few thousand ulp around both ends of the packed path's range, every finite and non-finite kind of value, and
    pairs of which one lane is inside the range and the other is not.  (The last two exponents have no packed path.)"""
    lo, hi = 2.0 ** max(-118.0 / lam, -126.0), 2.0 ** min(100.0 / lam, 100.0)
    near = np.arange(-3000, 3000)
    ends = np.concatenate([np.array([v], dtype=np.float32).view(np.int32).astype(np.int64) + near for v in (lo, hi, 2.4e-38)])
    ends = ends[(ends >= 0) & (ends < 0x7f800000)].astype(np.uint32)
    kinds = np.array([0, 0x80000000, 1, 0x80000001, 0x007fffff, 0x00800000, 0x3f800000, 0x3f7fffff, 0x7f7fffff, 0x7f800000,
                      0xff800000, 0x7fc00000, 0xffc00000, 0x7f800001, 0xbf800000, 0xff7fffff], dtype=np.uint32)
    rng = np.random.default_rng(9)
    inside = rng.uniform(0.1, 1.0, 4096).astype(np.float32).view(np.uint32)
    odd = np.concatenate([ends, kinds, rng.integers(0, 1 << 32, size=1 << 16, dtype=np.uint64).astype(np.uint32)])
    with_in = np.resize(inside, len(odd))
    for a, b in ((odd, with_in), (with_in, odd), (odd, odd[::-1])):
        assert compare(np.stack([a, b], 1).reshape(-1), lam) == 0
