"""The bounded wait of the direct and resident solves' grid barrier.  The test
hook rbffd_debug_set_barrier_limit has every wait give up after one poll: the
blocks return, the call reports it and the context stays usable.  No kernel
waits longer than that, and nothing faults or hangs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402
from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402


# 20: FP64 steps enqueued ahead, MIXED ones with the direct solve alone; 60: the
# direct solve behind a launched viscous one (10,502 V-nodes); 66: the resident
# solve.  "plan": the wait runs out in the dense inversion of the plan.
@pytest.mark.parametrize("n,when", [(20, "plan"), (20, "step"), (60, "step"), (66, "step")])
@pytest.mark.parametrize("precision", [0, 1])
def test_a_wait_that_runs_out_is_reported(n, when, precision):
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 3)
    gu, gv = (torch.as_tensor(g, device="cuda") for g in O.lid_bc(nd))
    got = []
    for fail in (True, False):
        ctx = R.Context(28, 7, 3)
        flow = R.flow_from_nodes(ctx, nd, Re=100.0, dt=0.08 / (n - 1), precision=precision,
                                 tol=1e-11 if precision else 1e-12)
        if when == "step":
            R.step(ctx, flow, R.State.zeros(flow), gu, gv, 1)  # builds the plan
        if fail:
            st = R.State.zeros(flow)
            R.debug_set_barrier_limit(ctx, 0)
            with pytest.raises(R.RbffdError) as e:
                R.step(ctx, flow, st, gu, gv, 3)
            assert e.value.code == R.ERR_CUDA and "bounded wait" in str(e.value)
            assert st.j == 0
            R.debug_set_barrier_limit(ctx, -1)
        st = R.State.zeros(flow)
        assert R.step(ctx, flow, st, gu, gv, 3)["steps"] == 3
        got.append(st)
    for x, y in zip((got[0].u, got[0].v, got[0].pt), (got[1].u, got[1].v, got[1].pt)):
        assert torch.equal(x, y)
