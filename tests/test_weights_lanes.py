"""The weight kernel's warp under independent thread scheduling, on the CPU.

The kernel's own source is compiled for the host with the 32 lanes as
coroutines.  Each lane runs alone up to its next warp-wide primitive, in
ascending or descending order of lanes: both are schedules that CUDA's
execution model allows, and any shared-memory access that relies on lanes
moving together, instead of on a barrier, reads the wrong word in one of them.
"""
import ctypes
import re
import shutil
import subprocess

import numpy as np
import pytest

from oracle import rbffd_oracle as O
from paper_2206_06495_gb300 import build
from paper_2206_06495_gb300 import nodesets as ns

SHIM = r"""
#include <ucontext.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>
#define __device__
#define __global__
#define __shared__
#define __forceinline__ inline
#define __launch_bounds__(x)
struct int4 { int x, y, z, w; };
struct Dim { int x; };
static int4 make_int4(int a, int b, int c, int d) { return {a, b, c, d}; }
static Dim threadIdx, blockIdx{0}, blockDim{32}, gridDim{1};
static ucontext_t lanes[32], host;
static bool done[32];
static unsigned long long slot[2][32];
static int cur;
static void wait_warp() { swapcontext(&lanes[cur], &host); }
static void __syncwarp() { wait_warp(); }
template <typename T> static T __shfl_xor_sync(unsigned, T v, int o) {
  unsigned long long b = 0, r;
  std::memcpy(&b, &v, sizeof(T));
  slot[0][cur] = b;
  wait_warp();
  r = slot[0][cur ^ o];
  wait_warp();  // every lane has read before the next exchange writes
  std::memcpy(&v, &r, sizeof(T));
  return v;
}
static long long __double_as_longlong(double d) { long long v; std::memcpy(&v, &d, 8); return v; }
static double __longlong_as_double(long long v) { double d; std::memcpy(&d, &v, 8); return d; }
static int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
static int __double2loint(double d) { return (int)__double_as_longlong(d); }
static double __hiloint2double(int h, int l) {
  return __longlong_as_double(((long long)h << 32) | (unsigned)l);
}
static double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static double __dmul_rn(double a, double b) { return a * b; }
static void atomicMin(unsigned long long* p, unsigned long long v) { *p = std::min(*p, v); }
using std::fma;
static double smem_words[1 << 16];
#define smem smem_words_ref
static double* smem_words_ref = smem_words;
"""

MAIN = r"""
struct Call {
  const double *ax, *ay, *bx, *by; const int32_t* idx; int64_t na, ld;
  int n, m, q, nrhs, cond; double* w; unsigned long long* bad;
};
static Call C;
static void lane_main() {
  const int np = C.q < 0 ? 0 : (C.q + 1) * (C.q + 2) / 2, S = C.n + np, LD = S % 2 ? S : S + 1;
  if (C.cond)
    weights_kernel<true>(C.ax, C.ay, C.na, C.bx, C.by, C.idx, C.ld, C.n, C.m, C.q, 0,
                         make_int4(0, 0, 0, 0), LD, C.w, C.bad);
  else
    weights_kernel<false>(C.ax, C.ay, C.na, C.bx, C.by, C.idx, C.ld, C.n, C.m, C.q, C.nrhs,
                          make_int4(1, 2, 3, 0), LD, C.w, C.bad);
  done[cur] = true;
  swapcontext(&lanes[cur], &host);
}
extern "C" void run(const double* ax, const double* ay, const double* bx, const double* by,
                    const int32_t* idx, int64_t na, int64_t ld, int n, int m, int q, int nrhs,
                    int cond, int descending, double* w, unsigned long long* bad) {
  C = {ax, ay, bx, by, idx, na, ld, n, m, q, nrhs, cond, w, bad};
  std::vector<std::vector<char>> stacks(32, std::vector<char>(1 << 18));
  for (int l = 0; l < 32; ++l) {
    done[l] = false;
    getcontext(&lanes[l]);
    lanes[l].uc_stack.ss_sp = stacks[l].data();
    lanes[l].uc_stack.ss_size = stacks[l].size();
    lanes[l].uc_link = &host;
    makecontext(&lanes[l], lane_main, 0);
  }
  for (bool any = true; any;) {
    any = false;
    for (int t = 0; t < 32; ++t) {
      cur = descending ? 31 - t : t;
      if (done[cur]) continue;
      any = true;
      threadIdx.x = cur;
      swapcontext(&host, &lanes[cur]);
    }
  }
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src = open(build.CSRC + "/weights.cu").read()
    body = src[src.index("constexpr int kMaxWarpsPerBlock"):
               src.index("// shared memory of one warp")]
    # the hardware seeds: single-precision values serve as well
    body = re.sub(r'asm\("rcp\.approx.*?\);', "y = (float)(1.0 / a);", body)
    body = re.sub(r'asm\("rsqrt\.approx.*?\);', "y = (float)(1.0 / std::sqrt(a));", body)
    body = body.replace("extern __shared__ double smem[];", "")
    assert "asm(" not in body
    d = tmp_path_factory.mktemp("lanes")
    (d / "lanes.cpp").write_text(SHIM + body + MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared", "-w",
                    str(d / "lanes.cpp"), "-o", str(d / "lanes.so")], check=True)
    f = ctypes.CDLL(str(d / "lanes.so")).run
    P = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731

    def call(ax, ay, bx, by, idx, m, q, cond, descending):
        na, n = idx.shape
        ii = np.ascontiguousarray(idx.T.astype(np.int32))
        w = np.zeros(na if cond else 3 * n * na)
        bad = np.full(1, -1, np.int64)
        f(P(ax), P(ay), P(bx), P(by), P(ii), ctypes.c_int64(na), ctypes.c_int64(na), n, m, q, 3,
          int(cond), int(descending), P(w), P(bad))
        assert bad[0] == -1
        return w if cond else w.reshape(3, n, na)
    return call


@pytest.mark.parametrize("descending", [False, True])
@pytest.mark.parametrize("n,m,q", [(28, 7, 3), (21, 5, 2), (33, 7, 3)])
def test_lanes_need_no_lockstep(run, n, m, q, descending):
    """Weights within 1e-10 of the oracle's, the bar of the GPU tests; condition
    numbers within 1e-5 of numpy's (about 1e8, times the unit roundoff and S)."""
    nd = ns.jittered_cavity(12, 3)
    rows = np.arange(0, nd.N, 23)
    ax, ay = nd.vx[rows].copy(), nd.vy[rows].copy()
    idx, W = O.build_weights(ax, ay, nd.vx, nd.vy, n, m, q, (O.OP_DX, O.OP_DY, O.OP_LAP))
    got = run(ax, ay, nd.vx, nd.vy, idx, m, q, False, descending)
    for o, op in enumerate((O.OP_DX, O.OP_DY, O.OP_LAP)):
        assert (np.abs(got[o].T - W[op]).max(1) / np.abs(W[op]).max(1)).max() < 1e-10
    cond = run(ax, ay, nd.vx, nd.vy, idx, m, q, True, descending)
    for i in range(rows.size):
        X, Y = nd.vx[idx[i]] - ax[i], nd.vy[idx[i]] - ay[i]
        s = np.hypot(X, Y).max()
        X, Y = X / s, Y / s
        P = np.stack([X ** (d - b) * Y ** b for d in range(q + 1) for b in range(d + 1)], 1)
        A = np.hypot(X[:, None] - X, Y[:, None] - Y) ** m
        A = np.block([[A, P], [P.T, np.zeros((P.shape[1],) * 2)]])
        assert abs(cond[i] / np.linalg.cond(A, 1) - 1.0) < 1e-5
