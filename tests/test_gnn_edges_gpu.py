"""The warm-start network's kernels at graph sizes around a warp, a block and
a block of 1,024 threads, with a hub of n/2 neighbours and isolated nodes,
against the FP64 oracle.

Tolerances: a neighbourhood mean adds at most n/64 terms per lane in a chain
and a five-level tree, at n = 2,050 about 40 2^-24 = 2.4e-6 relative, then a
sum of 6 and one of 64 terms: 1e-5 on the prediction (of order 1) and on the
loss, 2e-5 of the largest entry on the gradient, as in the parity tests.  The
fitted scale comes from sums carried in about 48 bits and is rounded once:
2^-23."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fastalign_ref as R  # noqa: E402
from oracle import gnn_ref as G  # noqa: E402
from paper_2607_11952_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n", [1, 2, 31, 33, 257, 1025, 2050])
def test_forward_and_gradient(n):
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api, gnn
    rng = np.random.default_rng(n)
    live = max(1, n - n // 8)
    e = np.concatenate([rng.integers(0, live, (2 * live, 2)),
                        np.stack([np.zeros(n // 2, np.int64), np.arange(n // 2)], axis=1)])
    e = synth.canonical_edges(n, e[:, 0], e[:, 1])
    F = rng.standard_normal((n, G.FIN)).astype(np.float32)
    y = rng.standard_normal(n).astype(np.float32)
    theta = gnn.init_params(n)
    graph, m = api.Graph(n, e), gnn.WarmStartModel(theta)
    a = m.predict(graph, torch.from_numpy(F).cuda())
    L.fa_gnn_backward(m.h, graph.handle, m.ws(n), a, torch.from_numpy(y).cuda(), m.grad, m.loss)
    A = R.row_normalized(n, e)
    a_ref, _ = G.forward(A, F.astype(np.float64), theta.astype(np.float64))
    loss_ref, g_ref = G.backward(A, F.astype(np.float64), theta.astype(np.float64), y)
    np.testing.assert_allclose(a.cpu().numpy(), a_ref, rtol=1e-5, atol=1e-5)
    assert abs(m.loss.item() - loss_ref) <= 1e-5 * loss_ref
    g = m.grad.cpu().numpy().astype(np.float64)
    np.testing.assert_allclose(g[:-1], g_ref[:-1], rtol=0, atol=2e-5 * np.abs(g_ref[:-1]).max())
    assert abs(g[-1]) < 1e-4


@pytest.mark.parametrize("n", [2, 33, 1025, 5000])
@pytest.mark.parametrize("shrink", [0, 1, 2])
def test_fit_scale(n, shrink):
    from paper_2607_11952_gb300 import _lib as L
    rng = np.random.default_rng(n)
    y = (3.0 + rng.standard_normal(n)).astype(np.float32)
    p = (0.5 * y + 0.7 * rng.standard_normal(n) + 40.0).astype(np.float32)   # far from centred
    if n > 10:
        p[3], p[5], p[7] = np.inf, np.nan, 1e9
    out = torch.empty(1, device="cuda")
    for pred in (p, np.full(n, 7.25, np.float32)):
        L.fa_gnn_fit_scale(n, torch.from_numpy(pred).cuda(), torch.from_numpy(y).cuda(), 45.0, out,
                           shrink=shrink)
        want = G.fit_scale(pred, y, 45.0, shrink)
        assert abs(out.item() - want) <= 2.0 ** -23 * max(1.0, want)


@pytest.mark.parametrize("n", [33, 1025])
def test_mean_of_an_infinite_potential_is_infinite(n):
    """A sum that leaves the finite numbers keeps its sign: the centred finite
    potentials are then -inf, as with a float64 sum."""
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api, gnn
    graph, m = api.Graph(n, np.zeros((0, 2), np.int64)), gnn.WarmStartModel(gnn.init_params(n))
    lv, zero = torch.randn(n, device="cuda"), torch.zeros(n, device="cuda")
    lv[n // 2] = float("inf")
    F = torch.empty(n, G.FIN, device="cuda")
    L.fa_gnn_features(graph.handle, lv, zero, zero, zero, 1, F, m.ws(n))
    want = torch.full((n,), -float("inf"), device="cuda")
    want[n // 2] = float("nan")
    torch.testing.assert_close(F[:, 0], want, rtol=0, atol=0, equal_nan=True)
    assert torch.isfinite(F[:, 1:]).all()
