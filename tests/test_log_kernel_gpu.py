"""The logarithm of the previous plan's kernel in the outer step.  With zero
costs, zero scalings and a large proximal weight p = lam_p / eps, the step's
kernel is K^p over its row's maximum, and an error of the logarithm appears p
times as large.

Tolerance, relative: p times one ulp of the largest logarithm in the row
(logf's documented bound) and again for the row's maximum, one rounding of
the exponent x and of x minus its maximum (2^-24 |x|), two ulps of expf."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("lo,hi,p", [(0.99, 1.0, 100.0), (0.74, 0.76, 20.0), (1.49, 1.51, 20.0),
                                     (0.3, 3.0, 4.0), (1e-12, 1.0, 1.0), (2e-40, 1e-39, 1.0)])
def test_kernel_power(lo, hi, p, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import api
    n1, n2 = 70, 333
    e = np.zeros((0, 2), np.int64)
    al = api.Aligner(api.Graph(n1, e), api.Graph(n2, e),
                     api.Params(dtype=dtype, eps=1.0, lam_p=p, lam_e=0.0, lam_n=0.0, lam_a=0.0))
    rng = np.random.default_rng(int(p))
    K0 = torch.from_numpy(np.exp(rng.uniform(np.log(lo), np.log(hi), (n1, n2))).astype(np.float32))
    al.K.zero_()
    al.K[:, :n2].copy_(K0.cuda())
    K0 = al.K[:, :n2].double().cpu().numpy()
    al.C_node.zero_()
    al.log_u.zero_()
    al.log_v.zero_()
    al.align_iter()
    L = np.log(K0)
    x = p * (L - L.max(axis=1, keepdims=True))
    want = np.exp(x)
    got = al.K[:, :n2].double().cpu().numpy()
    al.close()
    big = np.abs(L).max()
    ulp = 2.0 ** (np.floor(np.log2(big)) - 23)
    tol = 2 * p * ulp + 2 * 2.0 ** -24 * p * big + np.abs(x).max() * 2.0 ** -24 + 2 * 2.0 ** -23
    if dtype == "bf16":
        tol += 2.0 ** -8                    # the result's storage
    # a result below the smallest normal number is not resolved to that
    ok = want > 1e-37
    assert np.abs(got / np.where(ok, want, 1) - 1)[ok].max() <= tol
