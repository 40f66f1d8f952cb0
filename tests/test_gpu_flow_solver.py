"""DeepFlow's solver kernels where their split changes: levels at the edge of the
one-CTA kernel (1024 pairs of pixels; odd widths, whose last pair has one pixel)
and tiles that end inside, at and just past a 32x16 block, bit for bit against the
FP32 oracle; and the division by a kept reciprocal against the division itself."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1506_07656_gb300 import synth

pytestmark = pytest.mark.gpu

SRC = r"""
#include "k_deepflow.cu"
__global__ void k(const float* a, const float* d, long long n, float lo, unsigned long long* bad) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        if (__float_as_uint(df_div(a[i], d[i], __frcp_rn(d[i]), lo)) != __float_as_uint(__fdiv_rn(a[i], d[i]))) atomicAdd(bad, 1ull);
}
extern "C" int compare(const float* a, const float* d, long long n, float lo, unsigned long long* bad) {
    k<<<1216, 256>>>(a, d, n, lo, bad);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("W,H", [(64, 32), (63, 32), (65, 31), (66, 32), (33, 62), (48, 43), (97, 33), (34, 129)])
def test_level_sizes_bit_exact(torch_cuda, W, H):
    from paper_1506_07656_gb300 import dm
    pr = synth.make_pair_smooth(W, H, seed=W + H, max_disp=3.0)
    m, _, _ = oracle.match(pr.img1, pr.img2, "f32")
    kw = dict(n_fixed=3, n_sor=9, eta=0.8)
    want = oracle.deepflow(pr.img1, pr.img2, m, "f32", **kw)
    ctx = dm.Context(dm.DM_FP32)
    try:
        got = ctx.deepflow(pr.img1, pr.img2, m.astype(np.float32), **kw)
        for g, w in zip(got, want):
            np.testing.assert_array_equal(g.cpu().numpy(), w)
    finally:
        ctx.close()


def test_division_by_kept_reciprocal(torch_cuda, tmp_path):
    torch = torch_cuda
    from paper_1506_07656_gb300 import build
    src, lib = tmp_path / "div.cu", tmp_path / "div.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"),
                    "-shared", "-cudart", "static", "-o", str(lib), str(src), build.LIB], check=True)
    fn = C.CDLL(str(lib)).compare
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_longlong, C.c_float, C.c_void_p]
    g = torch.Generator(device="cuda").manual_seed(5)
    n = 1 << 24
    for lo_d, hi_d in ((1e-12, 1e12), (0.5, 2.0), (1.0, 1.0000002)):
        # any mantissa, exponents over the kernel's range; zeros, tiny and huge numerators
        d = torch.exp(torch.empty(n, device="cuda", dtype=torch.float64).uniform_(np.log(lo_d), np.log(hi_d), generator=g)).float()
        d = d.clamp(lo_d, hi_d)
        a = torch.exp(torch.empty(n, device="cuda", dtype=torch.float64).uniform_(np.log(1e-30), np.log(1e28), generator=g)).float()
        a = a * torch.where(torch.rand(n, device="cuda", generator=g) < 0.5, -1.0, 1.0)
        a[:: 1001] = 0.0
        bad = torch.zeros(1, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        assert fn(a.data_ptr(), d.data_ptr(), n, 1.0e-24, bad.data_ptr()) == 0
        assert int(bad.item()) == 0
