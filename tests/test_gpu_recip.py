"""The double reciprocal and inverse square root by Newton's iteration (kf_math.cuh) against CUDA's division and
square root: within one unit of the last place of the exact value (a step's rounding, the square of 2^-44), and
the same at zeros, infinities, NaNs and outside the float range, where they divide."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1702_06359_gb300 import build  # noqa: E402

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include "kf_math.cuh"
__global__ void k_eval(const double *x, int n, double *r, double *s, double *rd, double *sd)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = tkf::recip<double>(x[i]);
    s[i] = tkf::inv_sqrt<double>(x[i]);
    rd[i] = 1.0 / x[i];
    sd[i] = 1.0 / sqrt(x[i]);
}
extern "C" int eval(const double *x, int n, double *r, double *s, double *rd, double *sd)
{
    k_eval<<<(n + 127) / 128, 128>>>(x, n, r, s, rd, sd);
    return cudaDeviceSynchronize();
}
"""


def test_newton_reciprocals_equal_divisions_to_one_ulp(tmp_path):
    (tmp_path / "r.cu").write_text(PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", *build.FAST_MATH, "-Xcompiler", "-fPIC", "-shared", "-I",
                           build.CSRC, "-I", build.INCLUDE, str(tmp_path / "r.cu"), "-o", str(tmp_path / "libr.so")])
    rng = np.random.default_rng(2)
    n = 200_000
    x = np.concatenate([rng.uniform(1, 2, n) * 2.0 ** rng.integers(-140, 140, n), 10.0 ** rng.uniform(-300, 300, n),
                        np.array([1e-37, 1e37]).repeat(50) * (1 + np.linspace(-1e-6, 1e-6, 100)), 1 + np.arange(200) * 2.0 ** -52,
                        [0.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, np.finfo(float).max, 1.0, 4.0]])
    x = np.concatenate([x, -x])
    t = torch.as_tensor(x, device="cuda")
    out = [torch.empty_like(t) for _ in range(4)]
    torch.cuda.synchronize()
    fn = C.CDLL(str(tmp_path / "libr.so")).eval
    assert fn(C.c_void_p(t.data_ptr()), len(x), *(C.c_void_p(o.data_ptr()) for o in out)) == 0
    r, s, rd, sd = (o.cpu().numpy() for o in out)
    wide = x.astype(np.longdouble)
    with np.errstate(all="ignore"):
        exact = (1 / wide, 1 / np.sqrt(wide))  # (CUDA's division by a rounded root is itself up to 1.5 units off)
    for got, want, e in ((r, rd, exact[0]), (s, sd, exact[1])):
        fine = np.isfinite(want) & (want != 0)
        assert np.array_equal(got[~fine], want[~fine], equal_nan=True)
        in_float = fine & (np.abs(x) > 1.001e-37) & (np.abs(x) < 0.999e37)
        out = fine & ((np.abs(x) < 0.999e-37) | (np.abs(x) > 1.001e37))
        assert in_float.sum() > 100_000 and out.sum() > 10_000
        assert np.all(np.abs(got[in_float] - e[in_float]) <= np.spacing(np.abs(want[in_float])))
        assert np.array_equal(got[out], want[out])
