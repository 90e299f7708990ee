"""The weight kernel's reciprocal and square root against the correctly rounded
division and root, over the exponents their comments state and their edges."""
import ctypes
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2206_06495_gb300 import build  # noqa: E402

KERNEL = """
__global__ void eval(const double* a, double* r, double* s, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    r[i] = recip(a[i]);
    s[i] = root(fabs(a[i]));
  }
}
extern "C" int run(const double* a, double* r, double* s, long long n) {
  eval<<<1024, 256>>>(a, r, s, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    src = open(build.CSRC + "/weights.cu").read()
    d = tmp_path_factory.mktemp("recip")
    (d / "k.cu").write_text("#include <cmath>\n" +
                            src[src.index("// 1/a"):src.index("// a^2 + b^2")] + KERNEL)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-shared", "-Xcompiler", "-fPIC",
                    str(d / "k.cu"), "-o", str(d / "k.so")], check=True)
    f = ctypes.CDLL(str(d / "k.so")).run

    def call(a):
        r, s = torch.empty_like(a), torch.empty_like(a)
        torch.cuda.synchronize()
        assert f(*(ctypes.c_void_p(t.data_ptr()) for t in (a, r, s)),
                 ctypes.c_longlong(a.numel())) == 0
        return r, s
    return call


def _ulps(x, y):
    return (x.view(torch.int64) - y.view(torch.int64)).abs()


@pytest.mark.parametrize("span", [2, 1000])
def test_random_arguments(run, span):
    """2^27 arguments of either sign with exponents within +-span.  The seed's
    relative error of 2^-20 leaves 2^-80 before the rounding, within which two
    in 2^27 results are expected to lie at a rounding boundary: at most 16 may
    differ, by one unit."""
    g = torch.Generator(device="cuda").manual_seed(span)
    n = 1 << 27
    a = torch.rand(n, dtype=torch.float64, device="cuda", generator=g) + 1.0
    e = torch.randint(-span, span + 1, (n,), device="cuda", generator=g)
    a = torch.ldexp(a, e) * (1 - 2 * torch.randint(0, 2, (n,), device="cuda", generator=g))
    r, s = run(a)
    for got, ref in ((r, 1.0 / a), (s, a.abs().sqrt())):
        d = _ulps(got, ref)
        assert int(d.max()) <= 1 and int((d != 0).sum()) <= 16


def test_edges(run):
    """Powers of two and their neighbours, and for the root zero, subnormals and
    both sides of 2^-1000."""
    p = torch.ldexp(torch.ones(2001, dtype=torch.float64), torch.arange(-1000, 1001))
    bits = p.view(torch.int64)
    a = torch.cat([bits - 1, bits, bits + 1]).view(torch.float64).cuda()
    r, s = run(a)
    assert int(_ulps(r, 1.0 / a).max()) <= 1 and int(_ulps(s, a.sqrt()).max()) <= 1
    tiny = torch.tensor([0.0, 5e-324, 2.0 ** -1074 * 12345, 2.0 ** -1022, 2.0 ** -1000],
                        dtype=torch.float64)
    tiny = torch.cat([tiny, torch.nextafter(tiny[-1:], torch.zeros(1, dtype=torch.float64))]).cuda()
    assert torch.equal(run(tiny)[1], tiny.sqrt())
