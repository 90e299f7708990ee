"""Either side of the limit up to which FP64 steps are enqueued ahead (8,192
V-nodes), and the largest share of rows a block of the resident viscous solve
has there."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402
from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402


def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _run(n, group, steps, **kw):
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 3)
    ctx = R.Context(28, 7, 3)
    flow = R.flow_from_nodes(ctx, nd, Re=100.0, dt=0.08 / (n - 1), tol=1e-12, **kw)
    gu, gv = (_d(g) for g in O.lid_bc(nd))
    st = R.State.zeros(flow)
    stats = [R.step(ctx, flow, st, gu, gv, group) for _ in range(steps // group)]
    assert st.j == steps
    return nd, st, sum(s["launches"] for s in stats), sum(s["helm_iters"] for s in stats)


# 52: 7,905 V-nodes, 53 rows a block (the others have 32); 53: 8,216 V-nodes;
# 40 with the exact projection, whose pressure rows are wider
@pytest.mark.parametrize("n,ahead,kw", [(52, True, {}), (53, False, {}),
                                        (40, True, dict(projection=1))])
def test_either_side_of_the_enqueued_steps(n, ahead, kw):
    """33 steps in one call give the bits of 33 calls; eight launches a step say
    that they were enqueued.  Three of them agree with the launched form to the
    bars of the forms elsewhere (velocities 1e-9, p~ 1e-8)."""
    nd, one, launches, its = _run(n, 33, 33, **kw)
    _, each, _, its1 = _run(n, 1, 33, **kw)
    assert its == its1
    for x, y in ((one.u, each.u), (one.v, each.v), (one.pt, each.pt), (one.p, each.p)):
        assert torch.equal(x, y)
    assert (launches == 8 * 33) == ahead, launches
    _, a, _, _ = _run(n, 3, 3, **kw)
    _, b, _, _ = _run(n, 3, 3, profile=1, **kw)
    assert max((a.u - b.u).abs().max(), (a.v - b.v).abs().max()) < 1e-9
    assert (a.pt - b.pt).abs().max() < 1e-8 * b.pt.abs().max()
