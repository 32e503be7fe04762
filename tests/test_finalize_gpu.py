"""Column finalisation at the edges of its blocks: column counts around one
32-column block, around the switch to 128-column blocks (16,384 columns) and
one past them, with numbers of partial rows that leave every remainder of the
block's row groups and of the four rows in flight.

One static Sinkhorn step against float64.  Tolerance: a row sum adds at most
84 rounded terms in a chain (64 vectors per thread, then trees) and a column
sum at most n1 = 200, so u and then a column sum are off by at most about
284 2^-24 = 1.7e-5 relative; logf and the stored logarithm add 1e-6 each."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n2", [1, 31, 33, 129, 5000, 16383, 16384, 16513])
@pytest.mark.parametrize("n1,G", [(1, 0), (37, 0), (200, 1), (200, 33), (200, 100), (200, 0)])
def test_one_step_matches_float64(n2, n1, G, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    if G:
        monkeypatch.setenv("FA_SWEEP_G", str(G))
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params())
    gen = torch.Generator(device="cuda").manual_seed(n1 * 100003 + n2)
    al.K.zero_()
    al.K[:, :n2] = torch.rand(n1, n2, generator=gen, device="cuda") + 0.05
    lv = 0.5 * torch.randn(n2, generator=gen, device="cuda")
    _, err, _ = al.sinkhorn(2, warm_log_v=lv)
    K = al.K[:, :n2].double()
    v = torch.exp(lv.double())
    u = 1.0 / (n1 * (K @ v))
    v2 = 1.0 / (n2 * (K.T @ u))
    u2 = 1.0 / (n1 * (K @ v2))
    want_err = (v2 * (K.T @ u2) - 1.0 / n2).abs().sum().item()
    assert (al.log_v.double() - torch.log(v2)).abs().max().item() < 2e-5
    assert (al.log_u.double() - torch.log(u2)).abs().max().item() < 4e-5
    # the plan's mass is 1: the error sums differences of that relative size
    assert abs(err - want_err) < 6e-5
    assert math.isfinite(err)
