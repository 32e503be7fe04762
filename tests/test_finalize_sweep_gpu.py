"""The column finalisation at narrow widths, where a solve without further
switches runs in one launch and does not reach it: the sweep is asked for, and
the launch count shows that sweep and finalisation ran.  One row, rows that
leave every thread group but some without a partial row, and the largest
number of partial rows.  Tolerances as in test_finalize_gpu."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n2", [1, 31, 33, 129, 4096])
@pytest.mark.parametrize("n1", [1, 37, 200, 1500])
def test_sweep_and_finalisation_match_float64(n2, n1, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    monkeypatch.setenv("FA_SWEEP_KIND", "0")
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params())
    gen = torch.Generator(device="cuda").manual_seed(n1 * 100003 + n2)
    al.K.zero_()
    al.K[:, :n2] = torch.rand(n1, n2, generator=gen, device="cuda") + 0.05
    lv = 0.5 * torch.randn(n2, generator=gen, device="cuda")
    launches = L.fa_kernel_launch_count()
    _, err, _ = al.sinkhorn(2, warm_log_v=lv)
    assert L.fa_kernel_launch_count() - launches == 4
    K = al.K[:, :n2].double()
    v = torch.exp(lv.double())
    u = 1.0 / (n1 * (K @ v))
    v2 = 1.0 / (n2 * (K.T @ u))
    u2 = 1.0 / (n1 * (K @ v2))
    want_err = (v2 * (K.T @ u2) - 1.0 / n2).abs().sum().item()
    # a column sum adds n1 rounded terms, a row sum at most 84 in a chain
    rel = (n1 + 84) * 2.0 ** -24
    assert (al.log_v.double() - torch.log(v2)).abs().max().item() < max(2e-5, 1.2 * rel)
    assert (al.log_u.double() - torch.log(u2)).abs().max().item() < max(4e-5, 2.4 * rel)
    assert abs(err - want_err) < max(6e-5, 4 * rel)
