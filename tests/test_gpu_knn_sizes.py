"""The stencil search's two forms (a warp per query up to 32 neighbours, a
thread per query above) against the oracle's brute force, on sets where the
bucket grid is uneven: clustered, nearly collinear, tied, and so small that the
first block of cells covers everything."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import rbffd_oracle as O  # noqa: E402


def _sets(kind, rng):
    if kind == "uniform":
        return rng.random((700, 2)), rng.random((333, 2))
    if kind == "clustered":  # most nodes in one cell of the global grid
        b = np.concatenate([0.5 + 1e-3 * rng.random((900, 2)), rng.random((60, 2))])
        return b, np.concatenate([b[::7], rng.random((40, 2))])
    if kind == "strip":
        b = rng.random((500, 2)) * [1.0, 1e-4]
        return b, b[::3]
    if kind == "lattice":  # four-way ties
        g = np.stack(np.meshgrid(np.arange(21.0), np.arange(21.0)), -1).reshape(-1, 2)
        return g, g
    return rng.random((70, 2)), rng.random((5, 2)) * 3.0 - 1.0  # few nodes, queries outside


# k = 1: one neighbour; 28: the paper's; 31, 32: the last of the warp form;
# 33, 64: the thread form
@pytest.mark.parametrize("kind", ["uniform", "clustered", "strip", "lattice", "few"])
@pytest.mark.parametrize("k", [1, 28, 31, 32, 33, 64])
def test_search_equals_brute_force(kind, k):
    from paper_2206_06495_gb300 import rbffd as R
    rng = np.random.default_rng(3)
    b, a = _sets(kind, rng)
    d = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    ctx = R.Context(k, 3, -1)  # plain RBF: any stencil size; only the stencils are compared
    idx, _, _ = R.build_weights(ctx, d(a[:, 0]), d(a[:, 1]), d(b[:, 0]), d(b[:, 1]), R.OP_DX)
    got = idx.cpu().numpy()[:, : len(a)].T
    assert np.array_equal(got, O.knn(a[:, 0], a[:, 1], b[:, 0], b[:, 1], k))


@pytest.mark.parametrize("k", [1, 2, 32, 33])
def test_masked_search_with_a_forced_first_node(k):
    """Slot 0 forced, k - 1 searched among the unmasked (k = 33: 32 searched,
    33 slots)."""
    from paper_2206_06495_gb300 import rbffd as R
    rng = np.random.default_rng(5)
    b = rng.random((400, 2))
    rows = np.arange(0, 400, 9).astype(np.int32)
    mask = np.ones(400, bool)
    mask[rows] = False
    d = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    ctx = R.Context(k, 3, -1)
    idx, _, _ = R.build_weights_masked(ctx, d(b[rows, 0]), d(b[rows, 1]), d(b[:, 0]), d(b[:, 1]),
                                       R.OP_DX, beta_mask=d(mask.astype(np.uint8)),
                                       alpha_self=d(rows))
    got = idx.cpu().numpy()[:, : rows.size].T
    ref = O.knn(b[rows, 0], b[rows, 1], b[:, 0], b[:, 1], k, beta_mask=mask, alpha_self=rows)
    assert np.array_equal(got, ref)
