"""Sparse x dense products at the sizes where the gather engine can go wrong:
graphs smaller than a row tile or a column panel, one past them, a hub row
split over every warp and over several batches of edge records, isolated
nodes, no edges at all, a kernel that is only 8-byte aligned.

Node cost against the oracle: within 5e-6 of its largest entry, as in the
parity tests (FP32 GEMM and FP32 sums of convex combinations).  One outer
iteration from T0: the exponent of K is formed in FP32 with |x| up to about
150 from a few operations, about 1e-5, so K within 2e-5 in norm; BF16
storage adds its rounding, 2^-9 of each entry at most."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fastalign_ref as R  # noqa: E402
from paper_2607_11952_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _graph(n, seed, deg=6):
    """Random edges, node 0 tied to most others, the last tenth isolated."""
    rng = np.random.default_rng(seed)
    live = max(1, n - n // 10)
    e = rng.integers(0, live, (deg * live // 2, 2))
    hub = np.stack([np.zeros(live, np.int64), np.arange(live)], axis=1)[rng.random(live) < 0.8]
    return synth.canonical_edges(n, *np.concatenate([e, hub]).T)


def _setup(n1, n2, dtype, edges=True):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2607_11952_gb300 import api
    none = np.zeros((0, 2), np.int64)
    e1, e2 = (_graph(n1, n1), _graph(n2, n2 + 1)) if edges else (none, none)
    rng = np.random.default_rng(n1 + n2)
    X1 = rng.standard_normal((n1, 7)).astype(np.float32)
    X2 = rng.standard_normal((n2, 7)).astype(np.float32)
    m = max(1, min(n1, n2) // 9)
    anchors = np.stack([rng.permutation(n1)[:m], rng.permutation(n2)[:m]], axis=1)
    # FP32 node cost in both forms; an edge weight that makes lam_e Z_e, with
    # T0 = 1 / (n1 n2), of order 1 (larger ones would leave |x| in the thousands)
    p = api.Params(dtype=dtype, gemm="simt", lam_e=0.5 * n1 * n2 if edges else 1.0, lam_n=0.1)
    al = api.Aligner(api.Graph(n1, e1), api.Graph(n2, e2), p)
    al.node_cost(X1, X2, anchors)
    al.plan_init()
    op = R.Params(lam_e=p.lam_e, lam_n=p.lam_n)
    return al, op, R.phase1(n1, n2, e1, e2, X1, X2, anchors, op)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n1,n2", [(1, 1), (2, 3), (16, 17), (33, 31), (40, 257), (129, 300),
                                   (700, 513), (2100, 130), (260, 2300)])
def test_products_match_oracle(n1, n2, dtype):
    al, op, ph = _setup(n1, n2, dtype)
    C = al.C_node.cpu().numpy()
    assert np.all(C[:, n2:] == 0.0)
    assert np.abs(C[:, :n2] - ph.C_node).max() <= 5e-6 * max(1.0, np.abs(ph.C_node).max())
    al.align_iter()
    C_eff = R.outer_step(ph, np.full((n1, n2), -math.log(n1 * n2)), op)
    logK = -C_eff / op.eps
    assert np.abs(logK).max() < 160      # what the bound on K rests on
    want = np.exp(logK - logK.max(axis=1, keepdims=True))
    K = al.K.float().cpu().numpy()
    assert np.all(K[:, n2:] == 0.0)
    rel = np.linalg.norm(K[:, :n2] - want) / np.linalg.norm(want)
    assert rel <= 2e-5 + (2.0 ** -9 if dtype == "bf16" else 0.0), rel


def test_no_edges():
    al, op, ph = _setup(50, 70, "f32", edges=False)
    assert np.all(al.C_node.cpu().numpy() == 0.0)
    al.align_iter()
    K = al.K[:, :70].cpu().numpy()
    C_eff = R.outer_step(ph, np.full((50, 70), -math.log(3500)), op)
    logK = -C_eff / op.eps
    want = np.exp(logK - logK.max(axis=1, keepdims=True))
    assert np.linalg.norm(K - want) <= 2e-5 * np.linalg.norm(want)


def test_kernel_of_eight_byte_alignment():
    """The same outer step on a copy of K that starts 8 bytes past a 16-byte
    boundary gives the same bits."""
    from paper_2607_11952_gb300 import _lib as L
    al, _, _ = _setup(300, 411, "bf16")
    buf = torch.zeros(al.K.numel() + 8, dtype=al.K.dtype, device="cuda")
    Kd = buf[4:4 + al.K.numel()].view(al.K.shape)
    Kd.copy_(al.K)
    lu, lv = al.log_u.clone(), al.log_v.clone()
    L.fa_align_iter(al.ctx, Kd, lu, lv, al.C_node)
    al.align_iter()
    assert torch.equal(Kd, al.K) and torch.equal(lv, al.log_v)
