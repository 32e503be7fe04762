"""Sums that float64 holds and float32 does not: the plan change of plans
whose entries sum to more than 3.4e38, and the warm-start network's sums of
values whose sum, or whose products, leave float32's range on either side.

Tolerances: plan entries are exp(log_u) in float32 (2 ulps), so 2^-22 of the
sum; a fitted scale, a loss and a mean are float64 results rounded once, of
inputs whose differences are formed to 2^-24: 1e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import gnn_ref as G  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


NONE = np.zeros((0, 2), np.int64)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2", [(1, 2), (5, 40), (9000, 300)])
def test_plan_change_beyond_float32(n1, n2, dtype):
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    al = api.Aligner(api.Graph(n1, NONE), api.Graph(n2, NONE), api.Params(dtype=dtype))
    al.K.zero_()
    al.K[:, :n2] = 1.0
    al.log_u.fill_(88.0)                                   # exp = 1.65e38
    al.log_v.zero_()
    other = torch.zeros_like(al.K)
    got = L.fa_plan_change(al.ctx, al.K, al.log_u, al.log_v, other, al.log_u, al.log_v)
    want = n1 * n2 * np.exp(88.0)
    assert abs(got - want) <= 2.0 ** -22 * want
    al.log_u[n1 - 1] = 89.0                                # exp = inf
    with pytest.raises(L.FastAlignError) as e:
        L.fa_plan_change(al.ctx, al.K, al.log_u, al.log_v, other, al.log_u, al.log_v)
    assert e.value.status == L.FA_ERR_NUMERIC
    al.close()


@pytest.mark.parametrize("scale", [1e-25, 1e-12, 1e25])
@pytest.mark.parametrize("n", [33, 5000, 16384, 20000])
def test_fit_scale_of_tiny_and_huge_values(n, scale):
    from paper_2607_11952_gb300 import _lib as L
    rng = np.random.default_rng(n)
    y = (scale * rng.standard_normal(n)).astype(np.float32)
    p = (1.7 * y.astype(np.float64) + 0.2 * scale * rng.standard_normal(n)).astype(np.float32)
    out = torch.empty(1, device="cuda")
    for shrink in (0, 1):
        L.fa_gnn_fit_scale(n, torch.from_numpy(p).cuda(), torch.from_numpy(y).cuda(), 1e30, out,
                           shrink=shrink)
        want = G.fit_scale(p.astype(np.float64), y.astype(np.float64), 1e30, shrink)
        assert 0.1 < want < 0.9
        assert abs(out.item() - want) <= 1e-6


@pytest.mark.parametrize("n", [1025, 17000])
def test_loss_and_means_of_huge_values(n):
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api, gnn
    graph, m = api.Graph(n, NONE), gnn.WarmStartModel(gnn.init_params(n))
    rng = np.random.default_rng(n)
    y = (1e19 * rng.uniform(-1, 1, n)).astype(np.float32)   # squares sum to more than 3.4e38
    a = m.predict(graph, torch.zeros(n, G.FIN, device="cuda"))
    L.fa_gnn_backward(m.h, graph.handle, m.ws(n), a, torch.from_numpy(y).cuda(), m.grad, m.loss)
    r = y.astype(np.float64) - y.astype(np.float64).mean()
    want = (r * r).mean()
    assert abs(m.loss.item() - want) <= 1e-6 * want
    lv = torch.full((n,), 3e38, device="cuda")
    F = torch.empty(n, G.FIN, device="cuda")
    L.fa_gnn_features(graph.handle, lv, lv, lv, None, 1, F, m.ws(n))
    for c in (0, 1, 3):
        assert torch.equal(F[:, c], torch.zeros(n, device="cuda"))
