"""The shapes that the BF16 sweep's cluster rule plans between 12,000 and
57,000 columns (two rows per step in clusters of 2 to 7, uneven slabs), and
the sweep that carries K in registers in clusters of 2, 4 and 8, against the
float64 scaling iteration of the oracle.

Row counts: 701 (odd, so the last step has one row; most clusters take
several steps) and 37 (one step for some clusters, none for the rest).  The
column counts leave padding and a ragged last vector round.  Ten iterations:
both sweep directions, from a general start.

Tolerance: as for the workload's own shape, relative errors of a few 1e-6 per
FP32 sum that the iteration does not amplify past 1e-4 on log u and log v."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fastalign_ref as R  # noqa: E402
from paper_2607_11952_gb300 import synth  # noqa: E402

ITERS = 10
# columns, forced cluster size (0: the planner's), expected (Q, S, R)
SHAPES = [(12_000, 0, (2, 3, 2)), (21_000, 4, (4, 3, 2)), (43_000, 8, (8, 3, 2)),
          (24_000, 0, (3, 4, 2)), (27_000, 0, (3, 5, 2)), (40_000, 0, (5, 4, 2)),
          (44_000, 0, (5, 5, 2)), (48_000, 0, (6, 4, 2)), (52_000, 0, (6, 5, 2)),
          (56_500, 0, (7, 4, 2))]


@pytest.fixture(autouse=True)
def own_rule(monkeypatch):
    import __graft_entry__
    __graft_entry__.build()
    for k in ("KIND", "Q", "R", "NS", "NT", "G", "SMAX", "ANYQ", "L", "MB"):
        monkeypatch.delenv("FA_SWEEP_" + k, raising=False)


def test_planned_shapes():
    from paper_2607_11952_gb300 import _lib as L

    def shape(ld):
        p = L.fa_sweep_plan(50_000, ld, L.FA_BF16)
        assert p["kind"] == 0 and p["NT"] == 256
        return p["Q"], p["S"], p["R"]

    for n2, forced, expect in SHAPES:
        if not forced:
            assert shape((n2 + 127) // 128 * 128) == expect, n2
    # where clusters of three rounds or of seven CTAs measured slower than these
    assert shape(17_536) == (2, 5, 2)
    assert shape(51_200) == (5, 5, 1)
    assert shape(61_696) == shape(65_152) == (8, 4, 2)


@pytest.mark.gpu
@pytest.mark.parametrize("n1", [701, 37])
@pytest.mark.parametrize("n2,forced,expect", SHAPES)
def test_shapes_match_oracle(n1, n2, forced, expect, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    if forced:
        monkeypatch.setenv("FA_SWEEP_Q", str(forced))
    rng = synth.rng_for(n1 + n2)
    K = synth.random_kernel_rows(n1, n2, rng)
    lv0 = synth.random_log_scalings(n2, rng)
    u, v, errs = R.sinkhorn_scaling(K.astype(np.float64), np.full(n1, 1 / n1),
                                    np.full(n2, 1 / n2), ITERS,
                                    v0=np.exp(lv0.astype(np.float64)))
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params(dtype="bf16"))
    try:
        p = L.fa_sweep_plan(n1, al.ld, L.FA_BF16)
        assert (p["Q"], p["S"], p["R"]) == expect, p
        al.K.zero_()
        al.K[:, :n2].copy_(torch.from_numpy(K).cuda())
        it, err, st = al.sinkhorn(ITERS, warm_log_v=torch.from_numpy(lv0).cuda())
        lu, lv = al.log_u.double().cpu().numpy(), al.log_v.double().cpu().numpy()
    finally:
        al.close()
    assert it == ITERS and st == L.FA_OK
    assert np.abs(lu - np.log(u)).max() <= 1e-4
    assert np.abs(lv - np.log(v)).max() <= 1e-4
    assert abs(err - errs[-1]) < 1e-5 + 1e-4 * errs[-1]
