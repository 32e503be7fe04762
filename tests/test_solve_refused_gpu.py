"""A one-launch solve whose cooperative launch the device refuses (more CTAs
than it holds at once) must run as sweeps: the same bits as the sweeps give
when they are asked for, the state untouched before, and the one launch again
in the next call."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_11952_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm", [True, False])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_refused_launch_runs_the_sweeps(dtype, warm, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    n1, n2 = 500, 430
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params(dtype=dtype))
    rng = synth.rng_for(n1)
    al.K.zero_()
    al.K[:, :n2].copy_(torch.from_numpy(synth.random_kernel_rows(n1, n2, rng)).cuda())
    v0 = torch.from_numpy(synth.random_log_scalings(n2, rng)).cuda()

    def solve():
        al.log_v.copy_(v0)
        n = L.fa_kernel_launch_count()
        out = al.sinkhorn(40, 1e-4, 3, v0 if warm else None)
        return out, al.log_u.clone(), al.log_v.clone(), L.fa_kernel_launch_count() - n

    one, _, _, launches = solve()
    assert launches == 1
    L.fa_ctx_selftest_solve(al.ctx, -2, 50)
    got = solve()
    monkeypatch.setenv("FA_SWEEP_KIND", "0")
    want = solve()
    monkeypatch.delenv("FA_SWEEP_KIND")
    assert got[0] == want[0] and got[3] == want[3] > 1
    assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
    assert solve()[3] == 1
    al.close()
