"""fa_plan_init writes ones, zero padding and uniform log-scalings at widths
around its 16-byte vectors and blocks, also into a K that is not 16-byte
aligned, and nothing outside it."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2,offset", [(1, 1, 0), (3, 130, 1), (5000, 127, 0), (7, 2049, 0),
                                          (40, 9000, 3)])
def test_plan_init(dtype, n1, n2, offset):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import _lib as L
    from paper_2607_11952_gb300 import api
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params(dtype=dtype))
    buf = torch.full((al.K.numel() + 16,), 7.0, dtype=al.K.dtype, device="cuda")
    K = buf[offset:offset + al.K.numel()].view(al.K.shape)
    L.fa_plan_init(al.ctx, K, al.log_u, al.log_v)
    assert bool((K[:, :n2] == 1).all()) and bool((K[:, n2:] == 0).all())
    assert bool((buf[:offset] == 7).all()) and bool((buf[offset + K.numel():] == 7).all())
    assert torch.allclose(al.log_u, torch.full_like(al.log_u, -math.log(n1)), rtol=2e-7, atol=0)
    assert torch.allclose(al.log_v, torch.full_like(al.log_v, -math.log(n2)), rtol=2e-7, atol=0)
