"""The one-launch solve when one of its waits runs out, without a GPU fault:
one CTA withholds its partial sums, so that every CTA's wait for them (or for
a column sum formed from them) ends at its limit.  fa_sinkhorn must report
FA_ERR_TIMEOUT soon after that limit however many iterations were asked for
(a CTA that gave up leaves instead of running on), and the same context must
solve as before in its next call.
"""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_11952_gb300 import synth  # noqa: E402


def test_arguments_are_checked_on_the_host():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import _lib as L
    assert L.lib().fa_ctx_selftest_solve(None, 0, 50) == L.FA_ERR_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2", [(200, 300), (1000, 1000), (3, 4000)])
def test_a_silent_cta_is_reported_and_the_context_recovers(n1, n2, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params(dtype=dtype))
    rng = synth.rng_for(n1 + n2)
    al.K.zero_()
    al.K[:, :n2].copy_(torch.from_numpy(synth.random_kernel_rows(n1, n2, rng)).cuda())
    w = torch.from_numpy(synth.random_log_scalings(n2, rng)).cuda()
    it, err, _ = al.sinkhorn(20, warm_log_v=w)
    want_u, want_v = al.log_u.clone(), al.log_v.clone()
    ctas = min(n1, torch.cuda.get_device_properties(0).multi_processor_count // 2)
    for silent in (0, ctas - 1):
        L.fa_ctx_selftest_solve(al.ctx, silent, 50)
        t0 = time.perf_counter()
        with pytest.raises(L.FastAlignError) as ei:
            al.sinkhorn(20000, 1e-12, 1, w)
        waited = time.perf_counter() - t0
        assert ei.value.status == L.FA_ERR_TIMEOUT
        assert 0.04 <= waited <= 1.5      # two waits in turn at most, not one per iteration
        it2, err2, st = al.sinkhorn(20, warm_log_v=w)
        assert (it2, err2, st) == (it, err, L.FA_OK)
        assert torch.equal(al.log_u, want_u) and torch.equal(al.log_v, want_v)
    with pytest.raises(L.FastAlignError) as ei:
        L.fa_ctx_selftest_solve(al.ctx, 1 << 20, 50)
    assert ei.value.status == L.FA_ERR_ARG
    al.close()
