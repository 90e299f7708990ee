"""The ensemble's kernels at every number of columns per thread and shape of
the coarse product: one or two members (one column per thread in the pressure
solve), 4 to 64 (four), on node sets without (12 x 12) and with (50 x 50)
levels below the dense coarsest one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402
from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402

_ref = {}


def _oracle(n, Re, lid, steps, dt):
    key = (n, Re, lid)
    if key not in _ref:
        nd = ns.jittered_cavity(n, 4)
        fs = O.FractionalStep(nd, Re=Re, dt=dt, viscous_solver="krylov")
        gu, gv = O.lid_bc(nd, lid)
        s = fs.initial_state()
        for _ in range(steps):
            s = fs.step(s, gu, gv)
        _ref[key] = s
    return _ref[key]


@pytest.mark.parametrize("n", [12, 50])
@pytest.mark.parametrize("E", [1, 2, 4, 8, 16, 32, 64])
def test_members_match_the_oracle(n, E):
    """Three steps from rest; the first and last members against the oracle
    with the MIXED bars (velocities 1e-6 of the lid speed, p~ 1e-5)."""
    from paper_2206_06495_gb300 import rbffd as R
    nd = ns.jittered_cavity(n, 4)
    ctx = R.Context(28, 7, 3)
    dt = 0.1 / (n - 1)
    Re = np.linspace(300.0, 900.0, 64)[:E]
    lid = np.linspace(0.8, 1.2, 64)[:E]
    flow = R.flow_from_nodes(ctx, nd, Re=1.0, dt=dt, precision=R.PREC_MIXED, tol=1e-11)
    g = np.zeros((nd.N, E))
    g[nd.v_wall == ns.WALL_TOP] = lid
    gu = torch.as_tensor(g.ravel(), device="cuda")
    st = R.ensemble_zeros(flow, E)
    R.ensemble_step(ctx, flow, Re, st, gu, torch.zeros_like(gu), 3)
    u = st.u.cpu().numpy().reshape(nd.N, E)
    v = st.v.cpu().numpy().reshape(nd.N, E)
    pt = st.pt.cpu().numpy().reshape(nd.M, E)
    for e in {0, E - 1}:
        s = _oracle(n, float(Re[e]), float(lid[e]), 3, dt)
        assert np.abs(u[:, e] - s.u).max() < 1e-6 * lid[e]
        assert np.abs(v[:, e] - s.v).max() < 1e-6 * lid[e]
        assert np.abs(pt[:, e] - s.pt).max() < 1e-5 * np.abs(s.pt).max()
