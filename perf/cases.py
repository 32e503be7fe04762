"""Performance cases of the alignment framework: what a user's program has it do.

A case is a dict with a ``kind`` (which public entry point it goes through),
sizes, the storage type of the plan's kernel and the options of the call.

  align    one whole ``Aligner.align`` call, cold start (Algorithm 1)
  learned  one whole ``Aligner.align`` call with the trained warm start and
           the outer loop's convergence test (BF16 storage)
  solve    ``Aligner.sinkhorn``: one Sinkhorn solve on a fixed kernel
  outer    ``Aligner.align_iter``: one outer step (costs, Gibbs kernel) from
           a saved plan, as a resumed run does
  phase1   ``Aligner.node_cost``: Phase 1 (RWR, node similarity, propagation)
  readout  ``Aligner.topk`` and ``Aligner.rank`` on a finished plan
  train    ``WarmStartModel.train_step``: forward, backward and Adam of the
           warm-start network

Sizes are those of the repository's own workloads (``synth.CONFIGS``, the
training pairs of ``gnn``) or lie between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_11952_gb300 import api, gnn, synth

L2_BYTES = 126e6        # a kernel smaller than this need not be re-read from HBM


def listed():
    return [
        # the Barabasi-Albert 1k workload in full: every kernel at its
        # smallest, 10 outer x 50 Sinkhorn iterations
        dict(name="align_1k_f32", kind="align", n=1000, outer=10, sink=50, dtype="f32"),
        # the flagship form (learned warm start, BF16) on a pair of the size
        # the network is trained on, with the plan-change test of the outer loop
        dict(name="learned_5k_bf16", kind="learned", n=5000, outer=2, sink=30, d=128, deg=10.0,
             gamma=2.1, noise=0.15),
        # one solve of the 1k workload: 50 iterations of a 4 MB kernel
        dict(name="solve_1k_f32", kind="solve", n1=1000, n2=1000, iters=50, check=0, dtype="f32"),
        # one solve of the 10k workload: 100 FP32 iterations, fixed count
        dict(name="solve_10k_f32", kind="solve", n1=10000, n2=10000, iters=100, check=0,
             dtype="f32"),
        # an uneven pair with odd sizes, as real graph pairs are, solved to a
        # tolerance that is tested every 5 iterations, under an iteration cap
        dict(name="solve_uneven_bf16", kind="solve", n1=30011, n2=23993, iters=40, check=5,
             dtype="bf16"),
        # the 50k workload's Sinkhorn phase, 20 iterations, tested every 5
        dict(name="solve_50k_bf16", kind="solve", n1=50000, n2=50000, iters=20, check=5,
             dtype="bf16"),
        # one outer step of the 10k workload in plain FP32
        dict(name="outer_10k_f32", kind="outer", n1=10000, n2=10000, d=64, deg=8.0, gamma=2.5,
             noise=0.10, anchors=0.05, dtype="f32"),
        # one outer step of the 50k workload (heavy-tailed degrees, BF16)
        dict(name="outer_50k_bf16", kind="outer", n1=50000, n2=50000, d=128, deg=10.0, gamma=2.1,
             noise=0.15, anchors=0.05, dtype="bf16"),
        # Phase 1 of the 10k workload (FP32 operands: three-product TF32)
        dict(name="phase1_10k_f32", kind="phase1", n1=10000, n2=10000, d=64, deg=8.0, gamma=2.5,
             noise=0.10, anchors=0.05, dtype="f32"),
        # Phase 1 of the 50k workload (BF16 operands, 2500 anchors)
        dict(name="phase1_50k_bf16", kind="phase1", n1=50000, n2=50000, d=128, deg=10.0,
             gamma=2.1, noise=0.15, anchors=0.05, dtype="bf16"),
        # top-10 of every row and the rank of every true pair on the 20k
        # evaluation pair
        dict(name="readout_20k_bf16", kind="readout", n1=20000, n2=20000, k=10, dtype="bf16"),
        # one optimiser step on a training pair (n in 2000..5000)
        dict(name="train_4k", kind="train", n=4000, deg=10.0, gamma=2.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["align", "learned", "solve", "solve", "solve", "outer", "outer", "phase1",
                       "phase1", "readout", "train"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "align":
        return dict(kind=kind, n=_log_int(rng, 300, 3000), outer=rng.randint(2, 10),
                    sink=rng.randint(20, 50), dtype=dtype)
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 2000, 30000), deg=round(rng.uniform(6, 16), 2),
                    gamma=round(rng.uniform(2.1, 2.8), 2))
    graph = dict(d=rng.choice([32, 64, 100, 128, 256]), deg=round(rng.uniform(6, 16), 2),
                 gamma=round(rng.uniform(2.1, 2.8), 2), noise=round(rng.uniform(0.05, 0.2), 3))
    if kind == "learned":
        return dict(kind=kind, n=_log_int(rng, 1500, 10000), outer=2, sink=rng.randint(20, 40),
                    **graph)
    if kind == "solve":
        n1 = _log_int(rng, 500, 45000)
        n2 = min(50000, max(300, int(n1 * rng.uniform(0.6, 1.3))))
        most = 10 if max(n1, n2) > 20000 else 50
        return dict(kind=kind, n1=n1, n2=n2, iters=rng.randint(10, 2 * most),
                    check=rng.choice([0, 5, 10]), dtype=dtype)
    if kind == "readout":
        n1 = _log_int(rng, 1000, 35000)
        return dict(kind=kind, n1=n1, n2=max(500, int(n1 * rng.uniform(0.6, 1.1))),
                    k=rng.choice([1, 5, 10, 20]), dtype=dtype)
    top = 30000 if kind == "outer" else 24000
    n1 = _log_int(rng, 900, top)
    n2 = max(600, int(n1 * rng.uniform(0.6, 1.0)))
    return dict(kind=kind, n1=n1, n2=n2, anchors=rng.choice([0.02, 0.05, 0.1]), dtype=dtype,
                **graph)


# ------------------------------------------------------------ inputs
def _chung_lu(n, gamma, deg, rng):
    """About n deg / 2 edges whose endpoints are drawn in proportion to
    power-law weights (exponent gamma) capped at the square root of their sum."""
    w = np.arange(1, n + 1, dtype=np.float64) ** (-1.0 / (gamma - 1.0))
    w *= deg / w.mean()
    w = np.minimum(w, math.sqrt(deg * n))
    cum = np.cumsum(w)
    m = int(n * deg / 2)
    ends = np.searchsorted(cum, rng.random(2 * m) * cum[-1]).astype(np.int64)
    return synth.canonical_edges(n, np.minimum(ends[:m], n - 1), np.minimum(ends[m:], n - 1))


def _pair(case, seed):
    """(edges1, edges2, X1, X2, anchors, truth): G2 is G1 (or the subgraph
    induced by n2 of its nodes) relabelled, with edge noise; X2 is X1
    relabelled with noise.  Attributes are made on the GPU."""
    n1 = case.get("n1", case.get("n"))
    n2 = min(case.get("n2", n1), n1)
    rng = np.random.default_rng([seed, n1, n2])
    e1 = _chung_lu(n1, case["gamma"], case["deg"], rng)
    e1 = rng.permutation(n1)[e1]
    kept = np.sort(rng.permutation(n1)[:n2])
    perm = rng.permutation(n2)
    truth = np.full(n1, -1, np.int64)
    truth[kept] = perm
    e2 = truth[e1]
    e2 = e2[(e2 >= 0).all(axis=1)]
    e2 = e2[rng.random(len(e2)) >= case["noise"]]
    add = rng.integers(0, n2, (int(case["noise"] * len(e2)), 2))
    e2 = synth.canonical_edges(n2, np.concatenate([e2[:, 0], add[:, 0]]),
                               np.concatenate([e2[:, 1], add[:, 1]]))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    d = case["d"]
    X1 = torch.randn(n1, d, device="cuda", generator=gen)
    X2 = torch.empty(n2, d, device="cuda")
    X2[torch.from_numpy(perm).cuda()] = X1[torch.from_numpy(kept).cuda()] + 0.1 * torch.randn(
        n2, d, device="cuda", generator=gen)
    pick = np.sort(rng.permutation(n2)[: int(round(case.get("anchors", 0.05) * n2))])
    anchors = np.stack([kept[pick], perm[pick]], axis=1)
    return e1, e2, X1, X2, anchors, truth


def _ld(n2):
    return (n2 + 127) // 128 * 128


def _gibbs(n1, n2, dtype, seed):
    """A row-stabilised Gibbs kernel (n1 x ld, padding 0) as the method makes
    them: entries exp(x) with x spread over tens of log units, every row's
    maximum 1 at one column -- for 70% of the rows a partner of its own, for
    the others any column, so that columns compete and the solve converges as
    slowly as the method's own do.  Also log-scalings of a previous plan."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    K = torch.zeros(n1, _ld(n2), device="cuda",
                    dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
    step = max(1, (1 << 28) // n2)
    for i in range(0, n1, step):
        x = torch.randn(min(step, n1 - i), n2, device="cuda", generator=gen)
        K[i:i + step, :n2] = x.mul_(6.0).sub_(45.0).clamp_(max=0.0).exp_()
    m = min(n1, n2)
    rows = torch.randperm(n1, device="cuda", generator=gen)[:m]
    cols = torch.randperm(n2, device="cuda", generator=gen)[:m]
    peak = torch.randint(0, n2, (n1,), device="cuda", generator=gen)
    own = int(0.7 * m)
    peak[rows[:own]] = cols[:own]
    K[torch.arange(n1, device="cuda"), peak] = 1.0
    log_u = 0.5 * torch.randn(n1, device="cuda", generator=gen) - 0.5 * math.log(n1)
    log_v = 0.5 * torch.randn(n2, device="cuda", generator=gen) - 0.5 * math.log(n2)
    return K, log_u, log_v, rows, cols


def _train_inputs(case, seed):
    rng = np.random.default_rng([seed, case["n"]])
    n = case["n"]
    e = rng.permutation(n)[_chung_lu(n, case["gamma"], case["deg"], rng)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    F = torch.randn(n, gnn.FIN, device="cuda", generator=gen)
    y = 0.3 * torch.randn(n, device="cuda", generator=gen) + 0.2 * F[:, 0] * F[:, 3]
    return e, F, y


def _aligner(n1, n2, e1, e2, dtype):
    return api.Aligner(api.Graph(n1, e1), api.Graph(n2, e2), api.Params(dtype=dtype))


def _no_edges():
    return np.zeros((0, 2), np.int64)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    if kind == "align":
        g = synth.config_pair("ba1k", n=case["n"], seed=seed)
        st["al"] = _aligner(g.n1, g.n2, g.edges1, g.edges2, case["dtype"])
        st["X1"], st["X2"] = torch.from_numpy(g.X1).cuda(), torch.from_numpy(g.X2).cuda()
        st["anchors"] = g.anchors
    elif kind == "learned":
        n = case["n"]
        e1, e2, st["X1"], st["X2"], st["anchors"], _ = _pair(case, seed)
        st["al"] = _aligner(n, n, e1, e2, "bf16")
        st["model"] = gnn.WarmStartModel.load()
    elif kind == "solve":
        K, _, st["log_v"], _, _ = _gibbs(case["n1"], case["n2"], case["dtype"], seed)
        # the solve reads the kernel alone: the pair's edges play no part in it
        st["al"] = _aligner(case["n1"], case["n2"], _no_edges(), _no_edges(), case["dtype"])
        st["al"].K = K
    elif kind == "outer":
        e1, e2, X1, X2, anchors, _ = _pair(case, seed)
        al = st["al"] = _aligner(case["n1"], case["n2"], e1, e2, case["dtype"])
        al.node_cost(X1, X2, anchors)
        st["K"], st["log_u"], st["log_v"], _, _ = _gibbs(case["n1"], case["n2"], case["dtype"],
                                                         seed)
    elif kind == "phase1":
        e1, e2, st["X1"], st["X2"], st["anchors"], _ = _pair(case, seed)
        st["al"] = _aligner(case["n1"], case["n2"], e1, e2, case["dtype"])
    elif kind == "readout":
        K, _, log_v, rows, cols = _gibbs(case["n1"], case["n2"], case["dtype"], seed)
        al = st["al"] = _aligner(case["n1"], case["n2"], _no_edges(), _no_edges(), case["dtype"])
        al.K = K
        al.log_v.copy_(log_v)
        st["rows"], st["cols"] = rows.cpu().numpy(), cols.cpu().numpy()
    elif kind == "train":
        e, st["F"], st["y"] = _train_inputs(case, seed)
        st["graph"] = api.Graph(case["n"], e)
        st["model"] = gnn.WarmStartModel(seed=1)
    return st


# ------------------------------------------------------------ one pass
def run(st):
    case, kind = st["case"], st["kind"]
    if kind == "train":
        loss = st["model"].train_step(st["graph"], st["F"], st["y"], 3e-3)
        return {"loss": loss, "grad": st["model"].grad}
    al = st["al"]
    if kind == "align":
        al.align(st["X1"], st["X2"], st["anchors"], case["outer"], case["sink"])
        return {"K": al.K, "scalings": torch.cat([al.log_u, al.log_v])}
    if kind == "learned":
        warm = gnn.WarmStarter(al, "learned", st["model"])
        al.align(st["X1"], st["X2"], st["anchors"], case["outer"], case["sink"], check_every=5,
                 warm=warm, plan_tol=0.0)
        return {"K": al.K, "scalings": torch.cat([al.log_u, al.log_v])}
    if kind == "solve":
        # tol 1e-8 is below what FP32 scalings reach: the cap ends the solve
        tol = 1e-8 if case["check"] else -1.0
        it, err, _ = al.sinkhorn(case["iters"], tol, max(1, case["check"]), st["log_v"])
        # the L1 marginal error is absolute (the plan's mass is 1): mass + error
        return {"log_u": al.log_u, "log_v": al.log_v, "mass_err": 1.0 + err, "iters": it}
    if kind == "outer":
        al.K.copy_(st["K"])
        al.log_u.copy_(st["log_u"])
        al.log_v.copy_(st["log_v"])
        al.align_iter()
        return {"K": al.K, "log_u": al.log_u, "log_v": al.log_v}
    if kind == "phase1":
        al.node_cost(st["X1"], st["X2"], st["anchors"])
        return {"C_node": al.C_node}
    idx, score = al.topk(case["k"])
    return {"idx": idx, "score": score, "rank": al.rank(st["rows"], st["cols"])}


# ------------------------------------------------------------ work of a pass
def work(case):
    kind = case["kind"]
    n1 = case.get("n1", case.get("n"))
    n2 = case.get("n2", n1)
    b = 2 if case.get("dtype", "bf16") == "bf16" else 4
    N = float(n1) * n2
    nnz = case.get("deg", 6.0) * (n1 + n2) / 2    # stored entries per graph, on average
    gather = 2.0 * nnz * (n1 + n2)                # FLOPs of one P1 D P2^T
    L = case.get("anchors", 0.05) * n2
    d = case.get("d", 32)

    def solve(iters):
        reads = iters if b * N > L2_BYTES else 1
        return b * N * reads + 4.0 * (n1 + n2) * 2, 4.0 * N * iters

    phase1 = (4.0 * N + 4.0 * d * (n1 + n2), 2.0 * N * (d + L) + gather)
    outer = ((2 * b + 4.0) * N, 2 * gather + 10.0 * N)
    if kind == "solve":
        by, fl = solve(case["iters"])
    elif kind == "outer":
        by, fl = outer
    elif kind == "phase1":
        by, fl = phase1
    elif kind == "readout":
        by, fl = b * N + 8.0 * n1 * case["k"] + 12.0 * n1, 2.0 * N
    elif kind == "train":
        n = case["n"]
        e = case["deg"] * n
        by = 4.0 * n * (gnn.FIN + 1) + 8.0 * e + 8.0 * gnn.NP
        fl = 6.0 * n * gnn.FIN * gnn.HID + 2.0 * e * (gnn.FIN + 2)
    else:
        s = solve(case["sink"])
        by = phase1[0] + case["outer"] * (outer[0] + s[0])
        fl = phase1[1] + case["outer"] * (outer[1] + s[1])
    return {"bytes": float(by), "flops": float(fl)}


# ------------------------------------------------------------ the same in 64 bits
def _adjacency(n, edges):
    """Edges in both directions (rows, cols) without duplicates or loops, and degrees."""
    e = np.asarray(edges, np.int64)
    u, v = np.minimum(e[:, 0], e[:, 1]), np.maximum(e[:, 0], e[:, 1])
    key = np.unique((u * n + v)[u != v])
    u, v = key // n, key % n
    r, c = np.concatenate([u, v]), np.concatenate([v, u])
    deg = np.bincount(r, minlength=n).astype(np.float64)
    order = np.lexsort((c, r))
    r, c = torch.from_numpy(r[order]).cuda(), torch.from_numpy(c[order]).cuda()
    return r, c, torch.from_numpy(deg).cuda()


def _csr(n, r, c, vals):
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
    return torch.sparse_csr_tensor(ptr, c, vals, (n, n))


def _rwr64(n, g, seeds, p):
    r, c, deg = g
    A = _csr(n, r, c, 1.0 / deg[r])
    R0 = torch.zeros(n, max(1, len(seeds)), dtype=torch.float64, device="cuda")
    if len(seeds):
        R0[torch.from_numpy(np.asarray(seeds)).cuda(), torch.arange(len(seeds)).cuda()] = 1.0
    R = R0.clone()
    for _ in range(p.k_rwr):
        R = (1 - p.beta) * (A @ R) + p.beta * R0
    return R


def _unit(X):
    X = X.double()
    s = X.norm(dim=1, keepdim=True)
    return torch.where(s > 0, X / s, torch.zeros_like(X))


def _pad(C, n2):
    out = torch.zeros(C.shape[0], _ld(n2), dtype=torch.float64, device="cuda")
    out[:, :n2] = C
    return out


class _Exact:
    """Algorithm 1 in 64 bits (dense torch and CSR products)."""

    def __init__(self, n1, n2, e1, e2, X1, X2, anchors):
        p = self.p = api.Params()
        self.n1, self.n2 = n1, n2
        g1, g2 = _adjacency(n1, e1), _adjacency(n2, e2)
        R1, R2 = _rwr64(n1, g1, anchors[:, 0], p), _rwr64(n2, g2, anchors[:, 1], p)

        def intra(n, g, R, by):
            r, c, deg = g
            dots = torch.cat([(R[a] * R[b]).sum(1) for a, b in
                              zip(r.split(20000), c.split(20000))])
            return _csr(n, r, c, dots / deg[r if by == 0 else c])

        self.P1 = [intra(n1, g1, R1, 0), _csr(n1, g1[0], g1[1], 1.0 / g1[2][g1[1]])]
        self.P2 = [intra(n2, g2, R2, 1), _csr(n2, g2[0], g2[1], 1.0 / g2[2][g2[1]])]
        C = p.alpha * torch.exp(-(R1 @ R2.T)) + (1 - p.alpha) * torch.exp(
            -(_unit(X1) @ _unit(X2).T))
        A1 = _csr(n1, g1[0], g1[1], 1.0 / g1[2][g1[0]])
        A2 = _csr(n2, g2[0], g2[1], 1.0 / g2[2][g2[0]])
        for _ in range(p.k_prop):
            C = (A2 @ (A1 @ C).T.contiguous()).T.contiguous()
        self.C_node = C
        self.C_anc = torch.full((n1, n2), -math.log(p.eps_anc), dtype=torch.float64,
                                device="cuda")
        a = torch.from_numpy(np.asarray(anchors)).cuda()
        self.C_anc[a[:, 0], a[:, 1]] = -math.log(p.eps_anc + 1.0)

    def outer(self, log_T):
        """The next row-stabilised kernel and the first column update."""
        p, T = self.p, torch.exp(log_T)
        Ze, Zn = ((P2 @ (P1 @ T).T.contiguous()).T for P1, P2 in zip(self.P1, self.P2))
        C = (self.C_node + p.lam_e * Ze - p.lam_n * torch.log(Zn.clamp(min=p.delta))
             + p.lam_a * self.C_anc)
        x = -C / p.eps + (p.lam_p / p.eps) * log_T
        K = torch.exp(x - x.max(dim=1, keepdim=True).values)
        return K, -math.log(self.n2) - torch.log(K.sum(0))


def _solve64(K, log_v, iters):
    n1, n2 = K.shape
    log_v = log_v.double()
    for t in range(iters):
        v = torch.exp(log_v)
        u = 1.0 / (n1 * (K @ v))
        c = K.T @ u
        if t + 1 < iters:
            log_v = -math.log(n2) - torch.log(c)
    return torch.log(u), log_v, (v * c - 1.0 / n2).abs().sum()


def exact(case, seed):
    kind = case["kind"]
    if kind == "learned":
        return None         # a whole engine in 16-bit storage
    if kind == "solve":
        K, _, log_v, _, _ = _gibbs(case["n1"], case["n2"], case["dtype"], seed)
        log_u, log_v, err = _solve64(K[:, : case["n2"]].double(), log_v, case["iters"])
        return {"log_u": log_u, "log_v": log_v, "mass_err": 1.0 + err, "iters": None}
    if kind == "readout":
        K, _, log_v, _, _ = _gibbs(case["n1"], case["n2"], case["dtype"], seed)
        v = torch.exp(log_v.double())
        score = torch.cat([torch.topk(k[:, : case["n2"]].double() * v, case["k"], dim=1).values
                           for k in K.split(2000)])
        return {"idx": None, "score": score, "rank": None}
    if kind == "train":
        e, F, y = _train_inputs(case, seed)
        r, c, deg = _adjacency(case["n"], e)
        A = _csr(case["n"], r, c, 1.0 / deg[r]).to_sparse_coo()
        H, fin = gnn.HID, gnn.FIN
        th = torch.from_numpy(gnn.init_params(1)).cuda().double().requires_grad_(True)
        W1, b1, w2, b2 = th.split([fin * H, H, H, 1])
        hid = torch.relu(torch.sparse.mm(A, F.double()) @ W1.view(fin, H) + b1)
        a = torch.sparse.mm(A, (hid @ w2).view(-1, 1)).view(-1) + b2
        res = (a - a.mean()) - (y.double() - y.double().mean())
        loss = (res * res).mean()
        loss.backward()
        return {"loss": loss.detach().view(1), "grad": th.grad}
    if kind == "align":
        g = synth.config_pair("ba1k", n=case["n"], seed=seed)
        ex = _Exact(g.n1, g.n2, g.edges1, g.edges2, torch.from_numpy(g.X1).cuda(),
                    torch.from_numpy(g.X2).cuda(), g.anchors)
        log_T = torch.full((g.n1, g.n2), -math.log(g.n1) - math.log(g.n2), dtype=torch.float64,
                           device="cuda")
        for _ in range(case["outer"]):
            K, log_v = ex.outer(log_T)
            log_u, log_v, _ = _solve64(K, log_v, case["sink"])
            log_T = log_u[:, None] + torch.log(K) + log_v[None, :]
        return {"K": _pad(K, g.n2), "scalings": torch.cat([log_u, log_v])}
    if max(case["n1"], case["n2"]) > 16000:
        return None         # the dense 64-bit products take too long
    e1, e2, X1, X2, anchors, _ = _pair(case, seed)
    ex = _Exact(case["n1"], case["n2"], e1, e2, X1, X2, anchors)
    if kind == "phase1":
        return {"C_node": _pad(ex.C_node, case["n2"])}
    K, log_u, log_v, _, _ = _gibbs(case["n1"], case["n2"], case["dtype"], seed)
    log_T = (log_u.double()[:, None] + torch.log(K[:, : case["n2"]].double())
             + log_v.double()[None, :])
    K, log_v = ex.outer(log_T)
    return {"K": _pad(K, case["n2"]), "log_u": torch.zeros_like(log_u, dtype=torch.float64),
            "log_v": log_v}
