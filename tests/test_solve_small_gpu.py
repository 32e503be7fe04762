"""The one-launch solve against the oracle's float64 scaling iteration and
against the sweeps, at sizes where it can go wrong: fewer rows than CTAs of a
cluster, one row more than a cluster's, one column, a last eighth of padding,
row counts that leave CTAs without a row, the largest kernel that fits and
one past it; tolerance tests that end it early.

Tolerance: a row or column sum of n terms in trees and chains of at most 100
is off by 100 2^-24 = 6e-6 relative at the very most; the scalings carry
that through an iteration, contract all but their common factor, and that
factor by at most as much per iteration again (10 here): 1e-4 absolute on the
logarithms, as the sweep tests use."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fastalign_ref as R  # noqa: E402
from paper_2607_11952_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _make(n1, n2, dtype, seed=0):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import api
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params(dtype=dtype))
    rng = synth.rng_for(seed + 7 * n1 + n2)
    K = synth.random_kernel_rows(n1, n2, rng)
    lv = synth.random_log_scalings(n2, rng)
    al.K.zero_()
    al.K[:, :n2].copy_(torch.from_numpy(K).cuda())
    return al, K.astype(np.float64), lv


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2", [(1, 1), (3, 130), (8, 1), (9, 127), (130, 897), (153, 129),
                                   (1000, 1000), (1217, 400), (300, 3000), (2600, 2600),
                                   (2900, 2900)])
def test_matches_oracle_and_sweeps(n1, n2, dtype, monkeypatch):
    from paper_2607_11952_gb300 import _lib as L
    al, K, lv = _make(n1, n2, dtype)
    w = torch.from_numpy(lv).cuda()
    launches = L.fa_kernel_launch_count()
    it, err, _ = al.sinkhorn(10, warm_log_v=w)
    one = L.fa_kernel_launch_count() - launches == 1
    # which path ran: at 2,600 FP32 it depends on how many clusters the device holds
    assert one == (n1 <= 2600 or dtype == "bf16") or (n1 == 2600 and dtype == "f32")
    u, v, errs = R.sinkhorn_scaling(K, np.full(n1, 1 / n1), np.full(n2, 1 / n2), 10,
                                    v0=np.exp(lv.astype(np.float64)))
    lu, lvo = al.log_u.cpu().double().numpy(), al.log_v.cpu().double().numpy()
    assert it == 10
    assert np.abs(lu - np.log(u)).max() < 1e-4
    assert np.abs(lvo - np.log(v)).max() < 1e-4
    assert abs(err - errs[-1]) < 1e-5 + 1e-4 * errs[-1]
    # the rows of the returned plan are exact to FP32 rounding
    T = np.exp(lu)[:, None] * K * np.exp(lvo)[None, :]
    assert np.abs(T.sum(axis=1) * n1 - 1).max() < 1e-5
    monkeypatch.setenv("FA_SWEEP_KIND", "0")           # the sweeps on the same kernel
    it2, err2, _ = al.sinkhorn(10, warm_log_v=w)
    assert it2 == 10 and abs(err - err2) < 1e-5 + 1e-4 * err
    assert np.abs(al.log_u.cpu().double().numpy() - lu).max() < 1e-4
    assert np.abs(al.log_v.cpu().double().numpy() - lvo).max() < 1e-4


@pytest.mark.parametrize("check", [1, 3])
def test_stops_where_the_sweeps_stop(check, monkeypatch):
    from paper_2607_11952_gb300 import _lib as L
    al, _, lv = _make(700, 650, "f32")
    w = torch.from_numpy(lv).cuda()
    for tol in (1e-2, 1e-4):
        it, err, st = al.sinkhorn(200, tol, check, w)
        assert st == L.FA_OK and err <= tol
        monkeypatch.setenv("FA_SWEEP_KIND", "0")
        it2, err2, _ = al.sinkhorn(200, tol, check, w)
        monkeypatch.delenv("FA_SWEEP_KIND")
        assert it == it2 and abs(err - err2) <= 1e-3 * err + 1e-6
    it, err, st = al.sinkhorn(4, 1e-12, check, w)
    assert it == 4 and st == L.FA_ERR_NOT_CONVERGED
    it, _, _ = al.sinkhorn(1, warm_log_v=w)            # one iteration returns its own start
    assert it == 1 and torch.equal(al.log_v, w)


def test_reports_an_empty_row_and_recovers():
    from paper_2607_11952_gb300 import _lib as L
    al, _, lv = _make(200, 300, "f32")
    w = torch.from_numpy(lv).cuda()
    keep = al.K[5].clone()
    al.K[5] = 0.0
    with pytest.raises(L.FastAlignError) as e:
        al.sinkhorn(3, warm_log_v=w)
    assert e.value.status == L.FA_ERR_NUMERIC
    al.K[5] = keep
    it, _, st = al.sinkhorn(3, warm_log_v=w)
    assert it == 3 and st == L.FA_OK and bool(torch.isfinite(al.log_u).all())
