"""rbffd_stats of a small open flow: its two viscous systems' iterations add up
in the resident solve as in the launched one."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2206_06495_gb300 import nodesets as ns  # noqa: E402


def test_viscous_iterations_of_both_components_are_counted():
    """Three steps of the small wake in the resident form and, profiled, as
    separate launches: the same method from the same guesses, so the counts
    differ by the rounding of single solves only, at most a quarter."""
    from paper_2206_06495_gb300 import rbffd as R
    from paper_2206_06495_gb300 import wake
    nd = ns.cylinder_wake(h_wall=0.06, h_wake=0.08, h_far=0.5, x0=-3.0, x1=6.0, y0=-3.0, y1=3.0)
    its = []
    for profile in (0, 1):
        ctx = R.Context(28, 7, 3)
        flow = wake.wake_flow(ctx, nd, Re=100.0, dt=0.005, tol=1e-12, profile=profile)
        gu, gv = wake.wake_data(nd)
        st = R.State.zeros(flow)
        st.u.fill_(1.0)
        its.append(R.step(ctx, flow, st, gu, gv, 3)["helm_iters"])
    assert abs(its[0] - its[1]) <= 0.25 * its[1], its
