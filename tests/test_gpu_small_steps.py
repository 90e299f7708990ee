"""Small FP64 flows enqueue up to 32 steps before the host looks at their
results: the run must not depend on how its steps are grouped into calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402
from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402


def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _flow(kind, **kw):
    from paper_2206_06495_gb300 import rbffd as R
    from paper_2206_06495_gb300 import wake
    ctx = R.Context(30 if kind == "21 n30" else 28, 7, 3)
    if kind == "wake":
        nd = ns.cylinder_wake(h_wall=0.06, h_wake=0.08, h_far=0.5, x0=-3.0, x1=6.0, y0=-3.0,
                              y1=3.0)
        flow = wake.wake_flow(ctx, nd, Re=100.0, dt=0.005, tol=1e-12, **kw)
        gu, gv = wake.wake_data(nd)
        u0 = torch.ones(nd.N, dtype=torch.float64, device="cuda")
        return R, ctx, flow, gu, gv, u0
    n = int(kind.split()[0])
    nd = ns.jittered_cavity(n, 3)
    flow = R.flow_from_nodes(ctx, nd, **{**dict(Re=100.0, dt=0.08 / (n - 1), tol=1e-12), **kw})
    gu, gv = (_d(g) for g in O.lid_bc(nd))
    return R, ctx, flow, gu, gv, torch.zeros(nd.N, dtype=torch.float64, device="cuda")


def _same(a, b):
    return all(torch.equal(torch.nan_to_num(x), torch.nan_to_num(y)) and
               torch.equal(x.isnan(), y.isnan())
               for x, y in ((a.u, b.u), (a.v, b.v), (a.pt, b.pt), (a.p, b.p)))


# 81 nodes: fewer than the SMs; 1,089 and 4,096 (the largest); a stencil of
# other than 28 nodes; an open flow
@pytest.mark.parametrize("kind", ["9", "33", "64", "21 n30", "wake"])
@pytest.mark.parametrize("steps", [1, 32, 33])
def test_grouping_of_steps(kind, steps):
    """One call of n steps gives the bits of n calls, and the launch by launch
    solves (a profiled flow) the same to 1e-9 relative: both solve to 1e-12,
    and a step amplifies what is left by less than 30 over these runs."""
    R, ctx, flow, gu, gv, u0 = _flow(kind)
    one, each = R.State.zeros(flow), R.State.zeros(flow)
    one.u.copy_(u0)
    each.u.copy_(u0)
    s1 = R.step(ctx, flow, one, gu, gv, steps)
    assert s1["steps"] == steps and one.j == steps and s1["poisson_relres"] <= 1e-12
    if steps == 1:
        R, c2, flow2, gu, gv, _ = _flow(kind, profile=1)
        R.step(c2, flow2, each, gu, gv, 1)
        for x, y in ((one.u, each.u), (one.v, each.v), (one.p, each.p)):
            assert (x - y).norm() <= 1e-9 * y.norm()
        return
    its = 0
    for _ in range(steps):
        its += R.step(ctx, flow, each, gu, gv, 1)["helm_iters"]
    assert each.j == steps and its == s1["helm_iters"]
    assert _same(one, each)


def test_a_step_that_fails_in_the_middle():
    """A run that overflows: the call ends at the failing step with the state,
    the step count and the statistics of the calls of one step."""
    out = []
    for group in (40, 1):
        R, ctx, flow, gu, gv, u0 = _flow("20", dt=50.0, Re=1e4)
        st = R.State.zeros(flow)
        done = 0
        with pytest.raises(R.RbffdError) as e:
            for _ in range(40 // group):
                done += R.step(ctx, flow, st, gu * 1e3, gv, group)["steps"]
        done += e.value.stats["steps"]
        assert e.value.code in (R.ERR_NONFINITE, R.ERR_NOT_CONVERGED)
        assert st.j == done and 1 <= done < 40
        out.append((done, e.value.code, st))
    assert out[0][:2] == out[1][:2]
    assert _same(out[0][2], out[1][2])
