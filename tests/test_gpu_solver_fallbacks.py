"""What stands in for a solve that cannot run: no memory for the direct or the
resident solve, and a direct solve that does not reach the tolerance."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402
from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402


def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def _flow(n, limit=None, **kw):
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 3)
    ctx = R.Context(28, 7, 3)
    if limit is not None:
        R.debug_set_solver_bytes(ctx, limit)
    tol = 1e-11 if kw.get("precision") else 1e-12
    flow = R.flow_from_nodes(ctx, nd, **{**dict(Re=100.0, dt=0.08 / (n - 1), tol=tol), **kw})
    gu, gv = (_d(g) for g in O.lid_bc(nd))
    return R, ctx, flow, gu, gv


# 20: a dense inverse of 1.28 MB, resident copies of at most 94 KB; 65: no
# direct solve; a limit of 0 refuses every solver's memory, 500,000 the inverse
@pytest.mark.parametrize("n,limit", [(20, 0), (20, 500000), (65, 0)])
@pytest.mark.parametrize("precision", [0, 1])
def test_out_of_memory_leaves_the_launched_solve(n, limit, precision):
    """Three steps with the solvers' memory refused and without: velocities
    within 1e-9 (MIXED 1e-6) and p~ within 1e-8 (1e-5), the bars between the
    forms of the solve elsewhere."""
    got = []
    for lim in (limit, None):
        R, ctx, flow, gu, gv = _flow(n, lim, precision=precision)
        st = R.State.zeros(flow)
        assert R.step(ctx, flow, st, gu, gv, 3)["steps"] == 3
        got.append(st)
    a, b = got
    tu, tp = (1e-6, 1e-5) if precision else (1e-9, 1e-8)
    assert max((a.u - b.u).abs().max(), (a.v - b.v).abs().max()) < tu
    assert (a.pt - b.pt).abs().max() < tp * b.pt.abs().max()


@pytest.mark.parametrize("limit", [None, 0])
@pytest.mark.parametrize("group", [1, 6])
def test_krylov_takes_over_from_a_stalled_direct_solve(limit, group):
    """A tolerance of 1e-15 is below what the refinement's residual reaches;
    the Krylov recurrence goes on from its iterate through all six steps, with
    the hierarchy built then, whether or not there is memory for the resident
    form.  Within 1e-9 and 1e-8 of the launched form alone: both solve to the
    rounding level."""
    got = []
    for profile in (0, 1):
        R, ctx, flow, gu, gv = _flow(20, profile=profile)
        st = R.State.zeros(flow)
        R.step(ctx, flow, st, gu, gv, 1)  # builds the plan, with its direct solve
        if limit is not None:
            R.debug_set_solver_bytes(ctx, limit)
        flow.tol = 1e-15
        for _ in range(6 // group):
            assert R.step(ctx, flow, st, gu, gv, group)["steps"] == group
        assert st.j == 7
        got.append(st)
    a, b = got
    assert max((a.u - b.u).abs().max(), (a.v - b.v).abs().max()) < 1e-9
    assert (a.pt - b.pt).abs().max() < 1e-8 * b.pt.abs().max()


@pytest.mark.parametrize("profile", [0, 1])
def test_iteration_cap_holds_for_the_viscous_solve(profile):
    """A stiff viscous system that takes more than 84 iterations fails with 0.6
    times as many (50 at least, so that the direct solve stays in place), in
    the resident form and as separate launches, and leaves the state."""
    its = None
    for cap in (20000, None):
        R, ctx, flow, gu, gv = _flow(33, Re=0.5, dt=0.05, profile=profile)
        st = R.State.zeros(flow)
        flow.max_iter = cap or int(0.6 * its)
        if cap:
            its = R.step(ctx, flow, st, gu, gv, 1)["helm_iters"]
            assert its > 84
            continue
        with pytest.raises(R.RbffdError) as e:
            R.step(ctx, flow, st, gu, gv, 1)
        assert e.value.code == R.ERR_NOT_CONVERGED and "viscous" in str(e.value)
        assert e.value.stats["steps"] == 0 and st.j == 0 and not st.u.any()
        assert flow.max_iter <= e.value.stats["helm_iters"] <= flow.max_iter + 1


@pytest.mark.parametrize("precision", [0, 1])
def test_a_stalled_direct_solve_is_not_tried_at_every_step(precision):
    """32 steps in one call launch no more than 1.5 times what 32 calls do (a
    batch of 32 steps enqueued again after each stall launches three times as
    much), give their bits, and a loosened tolerance has the direct solve back
    at once (at most 8 products a step).  MIXED flows stall at the rounding level of
    the FP64 residual, where the Krylov solve stalls, too: the call reports it."""
    runs = []
    for group in (32, 1):
        R, ctx, flow, gu, gv = _flow(20, precision=precision)
        st = R.State.zeros(flow)
        R.step(ctx, flow, st, gu, gv, 1)
        flow.tol = 1e-16
        if precision:
            with pytest.raises(R.RbffdError) as e:
                R.step(ctx, flow, st, gu, gv, group)
            assert e.value.code == R.ERR_NOT_CONVERGED and st.j == 1
        launches = 0
        if not precision:
            flow.tol = 1e-15
            for _ in range(32 // group):
                launches += R.step(ctx, flow, st, gu, gv, group)["launches"]
            assert st.j == 33
        runs.append((launches, st))
        flow.tol = 1e-11
        other = R.State.zeros(flow)
        assert R.step(ctx, flow, other, gu, gv, 4)["poisson_iters"] <= 4 * 8
    (a, x), (b, y) = runs
    assert a <= 1.5 * b
    assert torch.equal(x.u, y.u) and torch.equal(x.pt, y.pt)


@pytest.mark.parametrize("profile", [0, 1])
def test_pressure_graphs_are_refused_alike(profile):
    """A graph whose coarsest matrix is not positive (two P-nodes of an edge
    1e-14 apart, whose weight of 1e28 leaves nothing of the others) is refused
    when the plan is built, by the hierarchy and by a flow solved directly."""
    R, ctx, flow, gu, gv = _flow(20, profile=profile)
    e, bc = flow.tensors["p_edges"], flow.tensors["p_bc"].bool()
    a, b = (int(v) for v in e[~bc[e[:, 0].long()] & ~bc[e[:, 1].long()]][50])
    for k in ("px", "py"):
        flow.tensors[k] = flow.tensors[k].clone()
        flow.tensors[k][b] = flow.tensors[k][a]
    flow.tensors["px"][b] += 1e-14
    st = R.State.zeros(flow)
    with pytest.raises(R.RbffdError) as err:
        R.step(ctx, flow, st, gu, gv, 1)
    assert err.value.code == R.ERR_INVALID_ARG and "not positive" in str(err.value)
    assert st.j == 0


# 1.10M and 1.21M rows: either side of the limit for rows of 28 entries; another
# width stays resident
@pytest.mark.parametrize("n,stencil,resident", [(1050, (28, 7, 3), True),
                                                (1100, (28, 7, 3), False),
                                                (1100, (21, 5, 2), True)])
def test_large_systems_take_the_faster_form(n, stencil, resident):
    """A resident solve is one launch, a launched one some 25 an iteration."""
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 3)
    ctx = R.Context(*stencil)
    flow = R.flow_from_nodes(ctx, nd, Re=1000.0, dt=0.08 / (n - 1), tol=1e-6)
    gu, gv = (_d(g) for g in O.lid_bc(nd))
    st = R.State.zeros(flow)
    stats = R.step(ctx, flow, st, gu, gv, 1)
    assert stats["poisson_iters"] >= 10
    assert (stats["launches"] < 10 * stats["poisson_iters"]) == resident, stats
