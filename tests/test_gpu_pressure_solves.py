"""The three forms of the preconditioned pressure solve at the sizes where they
meet: the direct solve of small systems (at most 4,096 P-nodes), the resident
Krylov kernel above it, and the launch-by-launch solve (taken when it is
profiled), each against the oracle's sparse LU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402
from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402


def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


# 81 rows: fewer than the SMs; 1,089 and 1,681: odd and uneven shares of rows;
# 4,096: the largest direct system; 4,225: the smallest resident one (two levels)
@pytest.mark.parametrize("n", [9, 33, 41, 64, 65])
@pytest.mark.parametrize("precision,profile", [(0, 0), (1, 0), (0, 1)])
def test_forms_match_the_oracle(n, precision, profile):
    """Five steps from rest to 1e-12 (MIXED 1e-11).  FP64: velocities within
    1e-9 and p~ within 1e-8 relative, the bars of the 20 x 20 cavity; MIXED:
    1e-6 and 1e-5, the bars of the MIXED path."""
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 3)
    ctx = R.Context(28, 7, 3)
    Re, dt = 100.0, 0.08 / (n - 1)
    flow = R.flow_from_nodes(ctx, nd, Re=Re, dt=dt, tol=1e-11 if precision else 1e-12,
                             precision=precision, profile=profile)
    st = R.State.zeros(flow)
    gu, gv = O.lid_bc(nd)
    stats = R.step(ctx, flow, st, _d(gu), _d(gv), 5)
    fs = O.FractionalStep(nd, Re=Re, dt=dt, viscous_solver="krylov" if n > 40 else "lu")
    s = fs.initial_state()
    for _ in range(5):
        s = fs.step(s, gu, gv)
    tu, tp = (1e-6, 1e-5) if precision else (1e-9, 1e-8)
    assert np.abs(st.u.cpu().numpy() - s.u).max() < tu
    assert np.abs(st.v.cpu().numpy() - s.v).max() < tu
    assert np.abs(st.pt.cpu().numpy() - s.pt).max() < tp * np.abs(s.pt).max()
    # the direct solve needs at most a few products a step, the Krylov one many
    direct = n <= 64 and not profile
    assert (stats["poisson_iters"] <= 20) == direct, stats["poisson_iters"]


# either side of 300,000 rows, where the resident kernel's block grows
@pytest.mark.parametrize("n", [547, 548])
def test_resident_and_launched_solves_agree(n):
    """A step from the lid's start by the resident kernel and, in a profiled
    flow, by separate launches, both to 1e-12: velocities within 1e-9 and p~
    within 1e-8 relative, the bars above."""
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 3)
    gu, gv = (_d(g) for g in O.lid_bc(nd))
    got = []
    for profile in (0, 1):
        ctx = R.Context(28, 7, 3)
        flow = R.flow_from_nodes(ctx, nd, Re=100.0, dt=0.08 / (n - 1), tol=1e-12, profile=profile)
        st = R.State.zeros(flow)
        R.step(ctx, flow, st, gu, gv, 1)
        got.append(st)
    a, b = got
    assert max((a.u - b.u).abs().max(), (a.v - b.v).abs().max()) < 1e-9
    assert (a.pt - b.pt).abs().max() < 1e-8 * b.pt.abs().max()
