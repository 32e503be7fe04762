"""Read-out kernels (fa_topk, fa_rank, fa_plan_change) at the sizes where they
can go wrong: rows shorter than one vector, one warp's pass and its
remainder, more columns than one pass; k from 1 to the largest; many equal
scores; scores that are -inf or NaN; a kernel that is not 16-byte aligned.
The order is checked exactly: with log_v = 0 a score is the stored kernel
value itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _make(n1, n2, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import api
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e), api.Params(dtype=dtype))
    al.log_v.zero_()
    al.log_u.zero_()
    al.K.zero_()
    return al


def _values(n1, n2, seed):
    """Scores with many ties, some -inf and some NaN (exact in BF16)."""
    rng = np.random.default_rng(seed)
    K = rng.integers(0, 40, (n1, n2)).astype(np.float32) / 64.0
    K[rng.random((n1, n2)) < 0.05] = -np.inf
    K[rng.random((n1, n2)) < 0.05] = np.nan
    K[0] = -np.inf                       # a row without any valid score
    return K


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2,k", [(1, 1, 1), (3, 7, 10), (9, 128, 32), (17, 255, 8),
                                     (5, 257, 32), (33, 1029, 10), (8, 5000, 17)])
@pytest.mark.parametrize("offset", [0, 1])
def test_topk_and_rank_orders(dtype, n1, n2, k, offset):
    from paper_2607_11952_gb300 import _lib as L
    al = _make(n1, n2, dtype)
    K = _values(n1, n2, 7 * n2 + k)
    al.K[:, :n2].copy_(torch.from_numpy(K))
    buf = torch.zeros(al.K.numel() + 8, dtype=al.K.dtype, device="cuda")
    Kd = buf[offset:offset + al.K.numel()].view(al.K.shape)    # offset 1: not 16-byte aligned
    Kd.copy_(al.K)
    idx = torch.empty((n1, k), dtype=torch.int32, device="cuda")
    score = torch.empty((n1, k), dtype=torch.float32, device="cuda")
    L.fa_topk(al.ctx, Kd, al.log_v, k, idx, score)
    want_i = np.full((n1, k), -1, np.int64)
    want_s = np.full((n1, k), -np.inf, np.float32)
    for i in range(n1):
        ok = np.flatnonzero(K[i] > -np.inf)
        top = ok[np.lexsort((ok, -K[i, ok]))][:k]
        want_i[i, :len(top)] = top
        want_s[i, :len(top)] = K[i, top]
    np.testing.assert_array_equal(idx.cpu().numpy(), want_i)
    np.testing.assert_array_equal(score.cpu().numpy(), want_s)

    rng = np.random.default_rng(n2)
    rows, cols = rng.integers(0, n1, 40), rng.integers(0, n2, 40)
    out = torch.empty(40, dtype=torch.int32, device="cuda")
    r = torch.as_tensor(rows, dtype=torch.int32).cuda()
    c = torch.as_tensor(cols, dtype=torch.int32).cuda()
    L.fa_rank(al.ctx, Kd, al.log_v, r, c, out)
    ref = K[rows, cols][:, None]
    x, j = K[rows], np.arange(n2)[None, :]
    want = 1 + ((x > ref) | ((x == ref) & (j < cols[:, None]))).sum(axis=1)
    np.testing.assert_array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2,offset", [(1, 1, 0), (3, 1030, 1), (1300, 2051, 0)])
def test_plan_change_sums(dtype, n1, n2, offset):
    """Against float64 sums.  Every plan value carries three float32 roundings
    (expf, two products), so a difference is off by at most about 4 ulp of the
    larger value: 4 2^-23 of the two plans' mass in all."""
    from paper_2607_11952_gb300 import _lib as L
    al = _make(n1, n2, dtype)
    gen = torch.Generator(device="cuda").manual_seed(n2)
    al.K[:, :n2] = torch.rand(n1, n2, generator=gen, device="cuda").to(al.K.dtype)
    buf = torch.zeros(al.K.numel() + 8, dtype=al.K.dtype, device="cuda")
    Kb = buf[offset:offset + al.K.numel()].view(al.K.shape)
    Kb[:, :n2] = torch.rand(n1, n2, generator=gen, device="cuda").to(al.K.dtype)
    lu, lv = torch.randn(n1, device="cuda"), torch.randn(n2, device="cuda")
    al.log_u.copy_(0.5 * lu)
    al.log_v.copy_(0.5 * lv)
    got = L.fa_plan_change(al.ctx, al.K, al.log_u, al.log_v, Kb, lu, lv)
    same = L.fa_plan_change(al.ctx, al.K, al.log_u, al.log_v, al.K, al.log_u, al.log_v)

    def plan(K, u, v):
        return torch.exp(u.double())[:, None] * K[:, :n2].double() * torch.exp(v.double())[None]
    A, B = plan(al.K, al.log_u, al.log_v), plan(Kb, lu, lv)
    assert abs(got - (A - B).abs().sum().item()) <= 4 * 2.0 ** -23 * (A.sum() + B.sum()).item()
    assert same == 0.0
    al.log_u[n1 - 1] = float("nan")
    with pytest.raises(L.FastAlignError):
        L.fa_plan_change(al.ctx, al.K, al.log_u, al.log_v, Kb, lu, lv)
