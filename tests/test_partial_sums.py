"""The FP32 shares of the resident solve's sums (Part<float> of gridsync.cuh),
compiled for the host."""
import ctypes
import math
import shutil
import subprocess

import numpy as np
import pytest

from paper_2206_06495_gb300 import build


@pytest.mark.parametrize("n", [1, 2, 4, 13])
def test_fp32_shares_lose_nothing_that_fp64_sums_keep(n, tmp_path):
    """Sums of products of widely spread sizes that nearly cancel: within 2^-40
    of the sum of magnitudes for up to 13 rows, the most a thread has (an FP32
    sum is off by 2^-24), and infinities stay visible."""
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src = open(build.CSRC + "/gridsync.cuh").read()
    body = src[src.index("template <typename T>\nstruct Part {"):src.index("// Ends a kernel")]
    (tmp_path / "p.cpp").write_text(
        "#define __device__\n#define __forceinline__ inline\n"
        "static float __fadd_rn(float a, float b) { return a + b; }\n"
        "static float __fsub_rn(float a, float b) { return a - b; }\n" + body +
        'extern "C" double total(const float* v, int n) {\n'
        "  Part<float> p;\n  for (int i = 0; i < n; ++i) p.add(v[i]);\n  return p.value();\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared",
                    str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p.so")], check=True)
    f = ctypes.CDLL(str(tmp_path / "p.so")).total
    f.restype = ctypes.c_double
    rng = np.random.default_rng(n)
    total = lambda v: f(v.ctypes.data_as(ctypes.c_void_p), v.size)  # noqa: E731
    for _ in range(2000):
        v = (rng.standard_normal(n) * 10.0 ** rng.uniform(-6, 6, n)).astype(np.float32)
        v[n // 2:2 * (n // 2)] = -v[:n // 2] * np.float32(1 + 1e-6)
        v = rng.permutation(v)
        assert abs(total(v) - math.fsum(v.tolist())) <= 2.0 ** -40 * np.abs(v).sum(dtype=float)
    v[0] = np.inf
    assert not math.isfinite(total(v))


def test_solve_scalars_are_correctly_rounded_quotients():
    """alpha, omega and beta of the resident solves are the compiler's divisions:
    no approximate FP64 instruction in their sources."""
    for f in ("gridsync.cuh", "psolve.cu", "dsolve.cu"):
        assert ".approx" not in open(build.CSRC + "/" + f).read(), f
