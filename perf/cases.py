"""The work a user of the solver has it do, as cases that can be timed and
whose outputs can be compared.

A case is one call sequence of a program that fits a sparse matrix: factors
in (device tensors), one sweep (or a few block steps, the losses, the
embedding with its nearest-neighbour search), results out.  Problem sizes are
those of the repository's workloads (paper_2608_21607_gb300/workloads.py) and
benchmark: the connectome-shaped power-law graph (139,255 nodes, mean
out-degree 20, r = 16 / 64 / 256), the planted 20,000 x 20,000 matrix
(r = 32, 5% dense), the identity of 4,096, the planted 600 x 400 matrix, the
community graph for the Delta form with range search.
"""
import math
import types

import numpy as np
import torch

from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

PREC = {"bf16": N.NMD_BF16, "fp32": N.NMD_FP32}
SKIP = {"none": N.NMD_SKIP_NONE, "range": N.NMD_SKIP_RANGE}


def _sweep(name, S, m, n, r, block, *, schedule="stoch", precision="bf16", form="z", skip="none", eta=0.5,
           gamma=0.9):
    return {"name": name, "kind": "sweep", "S": S, "m": m, "n": n, "r": r, "block": block, "schedule": schedule,
            "precision": precision, "form": form, "skip": skip, "eta": eta, "gamma": gamma}


def listed():
    return [
        # the smallest fit: a few-hundred-row matrix, exact alternating least
        # squares over ragged blocks; launches and latency only
        _sweep("tiny-exact", "planted4", 600, 400, 4, 128, schedule="exact", eta=1.0, gamma=0.0),
        # a small stochastic fit (identity, rank-3 completion): 16 short steps
        _sweep("identity-r3", "identity", 4096, 4096, 3, 512, eta=1.0, gamma=0.9),
        # thresholded similarity matrix, 5% dense: the support term weighs as
        # much as the dense contraction
        _sweep("planted-r32", "planted32", 20000, 20000, 32, 2048, eta=1.0, gamma=0.0),
        # connectome shape at the paper's end-to-end setting: r = 16, about 100
        # mini-batches per epoch (odd block size, ragged chunks; a smaller step
        # for the many small mini-batches)
        _sweep("connectome-r16", "powerlaw", 139255, 139255, 16, 1393, eta=0.1),
        # the headline: connectome shape, r = 64, blocks of 4096
        _sweep("connectome-r64", "powerlaw", 139255, 139255, 64, 4096),
        # the same in the fp32-accurate mode
        _sweep("connectome-r64-fp32", "powerlaw", 139255, 139255, 64, 4096, precision="fp32"),
        # the largest rank, blocks of 8192
        _sweep("connectome-r256", "powerlaw", 69627, 69627, 256, 8192),
        # parallel least squares: each block of rows against the whole other factor
        _sweep("exact-r64", "powerlaw", 40011, 40011, 64, 4096, schedule="exact", eta=1.0, gamma=0.0),
        # Delta form with range search on clustered factors (most of max(0, L) is zero)
        _sweep("communities-range-r64", "communities", 24576, 24576, 64, 8192, form="delta", skip="range",
               gamma=0.0),
        # a user's own schedule: steps on (row block, column block) pairs
        {"name": "combined-r64", "kind": "combined", "S": "powerlaw", "m": 40011, "n": 40011, "r": 64,
         "block": 4096, "schedule": "stoch", "precision": "bf16", "form": "z", "skip": "none", "eta": 0.5,
         "gamma": 0.9, "pairs": 8},
        # the losses of a fit, as evaluated between sweeps
        {"name": "loss-r64", "kind": "loss", "S": "powerlaw", "m": 139255, "n": 139255, "r": 64, "block": 4096,
         "schedule": "stoch", "precision": "bf16", "form": "z", "skip": "none", "eta": 0.5, "gamma": 0.9},
        # downstream: cell embedding and held-out 1-NN search over all cells
        {"name": "embed-nn-r64", "kind": "embed", "S": "powerlaw", "m": 139255, "n": 139255, "r": 64,
         "block": 4096, "schedule": "stoch", "precision": "bf16", "form": "z", "skip": "none", "eta": 0.5,
         "gamma": 0.9},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep"] * 7 + ["combined", "loss", "embed"])
    S = rng.choice(["powerlaw"] * 4 + ["planted32", "planted32", "planted4", "identity", "communities"])
    if S == "communities":
        kind = "sweep"
    if kind == "embed":
        S = "powerlaw"
    c = {"kind": kind, "S": S, "schedule": "stoch", "precision": rng.choice(["bf16", "bf16", "fp32"]),
         "form": rng.choice(["z", "z", "delta"]), "skip": "none", "eta": 0.5, "gamma": 0.9}
    if S == "communities":
        # every block of 8192 holds all 64 communities of 128-row runs
        n = 8192 * rng.randint(1, 4) - rng.randint(0, 60)
        c.update(m=n, n=n, r=64, block=8192, form="delta", skip="range", gamma=0.0)
        return c
    top = {"powerlaw": 139255, "planted32": 20000, "planted4": 5000, "identity": 20000}[S]
    r = {"planted32": lambda: rng.randint(20, 40), "planted4": lambda: rng.randint(3, 6),
         "identity": lambda: rng.randint(3, 8)}.get(S, lambda: _logint(rng, 4, 256))()
    if kind == "embed":
        r = min(r, 128)
    for _ in range(1000):
        n = _logint(rng, max(600, 30 * r), top)
        m = n if S in ("powerlaw", "identity") else _logint(rng, max(600, 30 * r), top)
        # blocks of 10 r rows or more, at most about 100 per side
        big = max(m, n)
        block = _logint(rng, max(128, 10 * r, big // 100), max(256, 20 * r, big // 100 + 1, min(8192, big // 2)))
        rp = next(p for p in (16, 32, 64, 128, 256) if r <= p)
        cost = m * n * max(rp, 32) * (3 if c["precision"] == "fp32" else 1) * (3 if kind == "embed" else 1)
        ragged = [x % block for x in (m, n)]
        if cost <= 139255 ** 2 * 64 * 3 and all(q == 0 or q >= 5 * r for q in ragged) and \
                not (c["precision"] == "fp32" and rp == 256 and n > 40000):
            break
    c.update(m=m, n=n, r=r, block=block)
    # the step shrinks with the number of mini-batches (with momentum 0.9, eta
    # near 1 diverges within a sweep of many steps)
    blocks = -(-max(m, n) // block)
    if S.startswith("planted"):
        c.update(eta=1.0, gamma=0.0)
    else:
        c.update(eta=round(min(0.5, 10.0 / blocks), 3))
    if kind == "sweep" and rng.random() < 0.2:
        c.update(schedule="exact", eta=1.0, gamma=0.0)
    if kind == "combined":
        c["pairs"] = rng.randint(2, 8)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed, salt):
    g = torch.Generator(device=_dev())
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _csr(m, n, rows, cols, vals):
    ptr = torch.zeros(m + 1, dtype=torch.int64, device=rows.device)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return WL.CSR(m, n, ptr.cpu().numpy(), cols.to(torch.int32).cpu().numpy(), vals.float().cpu().numpy())


def _powerlaw(n, seed, mean_degree=20.0, exponent=2.2):
    """Directed graph: power-law out-degree, uniform targets, no self loops,
    values ceil(exp(1 + N(0, 1))) (repeated targets are merged)."""
    g = _gen(seed, 1)
    u = 1.0 - torch.rand(n, generator=g, device=_dev(), dtype=torch.float64)
    base = u ** (-1.0 / (exponent - 1.0))
    lo, hi = 0.0, 2.0 * mean_degree
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        if float(torch.clamp(torch.floor(mid * base), max=n - 1).mean()) >= mean_degree:
            hi = mid
        else:
            lo = mid
    deg = torch.clamp(torch.floor(hi * base), max=n - 1).long()
    rows = torch.repeat_interleave(torch.arange(n, device=_dev()), deg)
    cols = torch.randint(0, n - 1, (rows.numel(),), generator=g, device=_dev())
    cols += (cols >= rows).long()
    keys = torch.unique(rows * n + cols)
    vals = torch.ceil(torch.exp(1.0 + torch.randn(keys.numel(), generator=g, device=_dev())))
    return _csr(n, n, keys // n, keys % n, vals)


def _planted(m, n, d, seed):
    """max(0, U V^T - tau): tau = 0.5 at d = 4, else the 95th percentile of
    sampled entries; 1% multiplicative noise."""
    g = _gen(seed, 2)
    U = torch.randn(m, d, generator=g, device=_dev())
    V = torch.randn(n, d, generator=g, device=_dev())
    tau = 0.5
    if d > 4:
        k = 1_000_000
        i = torch.randint(0, m, (k,), generator=g, device=_dev())
        j = torch.randint(0, n, (k,), generator=g, device=_dev())
        tau = float(torch.sort((U[i] * V[j]).sum(1)).values[int(0.95 * k)])
    rows, cols, vals = [], [], []
    for r0 in range(0, m, 4096):
        L = U[r0:r0 + 4096] @ V.T - tau
        at = (L > 0).nonzero()
        rows.append(at[:, 0] + r0)
        cols.append(at[:, 1])
        vals.append(L[at[:, 0], at[:, 1]])
    v = torch.cat(vals)
    v = torch.clamp(v * (1.0 + 0.01 * torch.randn(v.numel(), generator=g, device=_dev())), min=1e-30)
    return _csr(m, n, torch.cat(rows), torch.cat(cols), v)


def _community_factors(n, r, seed, noise, clusters=64, run=128, neg=0.6):
    """Factor rows in tight groups of directions, communities in runs of 128."""
    g = _gen(seed, 3)
    cl = (torch.arange(n, device=_dev()) // run) % min(clusters, r)
    W = torch.zeros(n, r, device=_dev())
    W[torch.arange(n, device=_dev()), cl] = 1.0
    H = torch.zeros(n, r, device=_dev())
    H[:, :min(clusters, r)] = -neg
    H[torch.arange(n, device=_dev()), cl] += 2.0
    W += noise * torch.randn(n, r, generator=g, device=_dev())
    H += noise * torch.randn(n, r, generator=g, device=_dev())
    W *= 0.5 + 1.5 * torch.rand(n, 1, generator=g, device=_dev())
    H *= 0.5 + 1.5 * torch.rand(n, 1, generator=g, device=_dev())
    return W, H.T.contiguous(), cl


def _communities(n, W, H):
    """S = max(0, W H): a zero-loss point of the clustered factors."""
    rows, cols, vals = [], [], []
    for r0 in range(0, n, 4096):
        L = W[r0:r0 + 4096].double() @ H.double()
        at = (L > 0).nonzero()
        rows.append(at[:, 0] + r0)
        cols.append(at[:, 1])
        vals.append(L[at[:, 0], at[:, 1]].float())
    v = torch.cat(vals)
    rows, cols = torch.cat(rows), torch.cat(cols)
    keep = v > 0
    return _csr(n, n, rows[keep], cols[keep], v[keep])


def _inputs(case, seed):
    """(S, W, H, labels): S as host CSR, the factors as device tensors."""
    m, n, r = case["m"], case["n"], case["r"]
    labels = None
    if case["S"] == "communities":
        W, H, _ = _community_factors(n, r, seed, 0.002)
        return _communities(n, W, H), W, H, None
    if case["kind"] == "embed":
        W, H, labels = _community_factors(n, r, seed, 0.1)
        labels = labels.int().contiguous()
    else:   # iid N(0, 0.1^2), the usual start
        g = _gen(seed, 4)
        W = 0.1 * torch.randn(m, r, generator=g, device=_dev())
        H = 0.1 * torch.randn(r, n, generator=g, device=_dev())
    if case["S"] == "powerlaw":
        S = _powerlaw(n, seed)
    elif case["S"] == "identity":
        S = WL.identity(n)
    else:
        S = _planted(m, n, 4 if case["S"] == "planted4" else 32, seed)
    return S, W, H, labels


def _pairs(case, seed):
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 5])
    kr, kc = -(-case["m"] // case["block"]), -(-case["n"] // case["block"])
    return [(int(rng.integers(kr)), int(rng.integers(kc))) for _ in range(case["pairs"])]


def prepare(case, seed):
    S, W, H, labels = _inputs(case, seed)
    sol = N.Solver(S, case["r"], block_rows=case["block"], block_cols=case["block"],
                   schedule=N.NMD_EXACT if case["schedule"] == "exact" else N.NMD_STOCH, eta=case["eta"],
                   gamma=case["gamma"], precision=PREC[case["precision"]],
                   epilogue=N.NMD_EPI_DELTA if case["form"] == "delta" else N.NMD_EPI_Z,
                   seed=int(seed) & 0x7FFFFFFF, skip_zero_chunks=SKIP[case["skip"]])
    st = types.SimpleNamespace(kind=case["kind"], sol=sol, W=W, H=H, labels=labels)
    if st.kind in ("sweep", "combined"):
        st.Wo, st.Ho = torch.empty_like(W), torch.empty_like(H)
    if st.kind == "combined":
        st.pairs = _pairs(case, seed)
    if st.kind in ("loss", "embed"):
        sol.set_factors(W, H)
    return st


def run(st):
    sol = st.sol
    if st.kind == "loss":
        return sol.loss()
    if st.kind == "embed":
        xi, sigma = sol.embed()
        nn, best, errors = N.nearest_neighbors(xi, st.labels)
        return {"xi": xi, "sigma": sigma, "nn": nn, "best": best, "errors": errors}
    sol.set_factors(st.W, st.H)
    if st.kind == "sweep":
        sol.sweep()
    else:
        for i, j in st.pairs:
            sol.block_update_combined(N.NMD_ROW, i, j)
            sol.block_update_combined(N.NMD_COL, i, j)
    sol.get_factors_device(st.Wo, st.Ho)
    return {"W": st.Wo, "H": st.Ho}


def _nnz(case):
    m, n = case["m"], case["n"]
    return {"powerlaw": 20 * n, "identity": n, "planted32": 0.05 * m * n, "planted4": 0.37 * m * n,
            "communities": m * n / 64}[case["S"]]


def work(case):
    m, n, r, b = case["m"], case["n"], case["r"], case["block"]
    nnz = _nnz(case)
    if case["kind"] == "loss":
        return {"bytes": 4 * r * (m + n) + 8 * nnz, "flops": 2 * m * n * r}
    if case["kind"] == "embed":
        return {"bytes": 4 * r * (m + n) + 8 * r * n + 8 * n, "flops": 2 * n * n * 2 * r + 8 * n * r * r}
    # factors in and out, S once
    base = 8 * r * (m + n) + 8 * nnz
    if case["kind"] == "combined":
        steps = 2 * case["pairs"]
        bm, bn = min(b, m), min(b, n)
        return {"bytes": base, "flops": steps * (4 * bm * bn * r + (bm + bn) * 2 * r * r)}
    kr, kc = -(-m // b), -(-n // b)
    if case["schedule"] == "exact":
        return {"bytes": base, "flops": 8 * m * n * r + 4 * (m + n) * r * r}
    return {"bytes": base, "flops": 8 * m * n * r + 2 * r * r * (m * kc + n * kr + m + n)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the definitions
# ---------------------------------------------------------------------------

_M64 = (1 << 64) - 1


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _order(seed, sweep, side, K):
    """SplitMix64-driven Fisher-Yates order of the blocks of one side."""
    s = _mix(seed & _M64) ^ _mix(((sweep << 1) | side) & _M64)
    p = list(range(K))
    for i in range(K - 1, 0, -1):
        s = (s + 0x9E3779B97F4A7C15) & _M64
        j = _mix(s) % (i + 1)
        p[i], p[j] = p[j], p[i]
    return p


class _Exact:
    def __init__(self, case, S, W, H):
        self.case = case
        self.F = [W.double(), H.double().T.contiguous()]           # W (m x r), B = H^T (n x r)
        self.E = [torch.zeros_like(f) for f in self.F]
        rp = torch.from_numpy(np.asarray(S.row_ptr)).to(_dev())
        self.rows = torch.repeat_interleave(torch.arange(S.m, device=_dev()), rp[1:] - rp[:-1])
        self.cols = torch.from_numpy(np.asarray(S.col_idx)).to(_dev()).long()
        self.vals = torch.from_numpy(np.asarray(S.vals)).to(_dev()).double()

    def step(self, f, m0, m1, q0, q1, momentum):
        """Rows [m0, m1) of factor f from rows [q0, q1) of the other one."""
        M, Q = self.F[f], self.F[1 - f][q0:q1]
        mi, qi = (self.rows, self.cols) if f == 0 else (self.cols, self.rows)
        keep = (mi >= m0) & (mi < m1) & (qi >= q0) & (qi < q1)
        mi, qi, v = mi[keep], qi[keep] - q0, self.vals[keep]
        if f == 1:
            mi, o = torch.sort(mi, stable=True)
            qi, v = qi[o], v[o]
        c = torch.linalg.cholesky(Q.T @ Q)
        eta, gamma = self.case["eta"], self.case["gamma"]
        per = max(1, min(m1 - m0, (1 << 28) // max(1, q1 - q0)))
        for a in range(m0, m1, per):
            z = min(m1, a + per)
            Z = torch.clamp(M[a:z] @ Q.T, max=0.0)
            lo, hi = (int(x) for x in torch.searchsorted(mi, torch.tensor([a, z], device=_dev())))
            Z[mi[lo:hi] - a, qi[lo:hi]] = v[lo:hi]
            X = torch.cholesky_solve((Z @ Q).T, c).T
            U = eta * (X - M[a:z])
            if momentum:
                U = U + gamma * self.E[f][a:z]
                self.E[f][a:z] = U
            M[a:z] += U


def _exact_cost(case):
    return case["m"] * case["n"] * case["r"] * (2 if case["kind"] in ("loss", "combined") else 8)


def exact(case, seed):
    if _exact_cost(case) > 1.2e13:
        return None
    S, W, H, _ = _inputs(case, seed)
    m, n, b = case["m"], case["n"], case["block"]
    kr, kc = -(-m // b), -(-n // b)
    if case["kind"] == "embed":
        A, B = W.double(), H.double().T.contiguous()
        qa, ra = torch.linalg.qr(A)
        qb, rb = torch.linalg.qr(B)
        u, s, vt = torch.linalg.svd(ra @ rb.T)
        xi = torch.cat([qa @ u * s.sqrt(), qb @ vt.T * s.sqrt()], 1)
        xi /= xi.norm(dim=1, keepdim=True)
        best = torch.empty(n, dtype=torch.float64, device=_dev())
        for a in range(0, n, 2048):
            G = xi[a:a + 2048] @ xi.T
            k = torch.arange(G.shape[0], device=_dev())
            G[k, k + a] = -math.inf
            best[a:a + 2048] = G.max(1).values
        return {"xi": None, "sigma": s, "nn": None, "best": best, "errors": None}
    x = _Exact(case, S, W, H)
    if case["kind"] == "loss":
        A, B = x.F
        r2 = r1 = sa = sb = smin = smax = 0.0
        for a in range(0, m, 2048):
            L = torch.clamp(A[a:a + 2048] @ B.T, min=0.0)
            lo, hi = (int(q) for q in torch.searchsorted(x.rows, torch.tensor([a, min(m, a + 2048)], device=_dev())))
            i, j, v = x.rows[lo:hi], x.cols[lo:hi], x.vals[lo:hi]
            l = (A[i] * B[j]).sum(1)
            sh = torch.clamp(l, min=0.0)
            L[i - a, j] = 0.0
            r2 += float((L * L).sum())
            r1 += float(L.sum())
            sa += float(((v - l) ** 2).sum())
            sb += float(((v - sh) ** 2).sum())
            smin += float(torch.minimum(v, sh).sum())
            smax += float(torch.maximum(v, sh).sum())
        fro = float(x.vals.square().sum().sqrt())
        return {"obj": math.sqrt(r2 + sa) / fro, "rmse": math.sqrt(r2 + sb) / fro, "wjd": 1.0 - smin / (r1 + smax),
                "s_fro": fro, "sum_relu2": r2, "sum_relu": r1}
    rng_ = lambda k, size: (k * b, min(size, (k + 1) * b))   # noqa: E731
    if case["kind"] == "combined":
        for i, j in _pairs(case, seed):
            x.step(0, *rng_(i, m), *rng_(j, n), True)
            x.step(1, *rng_(j, n), *rng_(i, m), True)
    else:
        s = int(seed) & 0x7FFFFFFF
        pr, pc = _order(s, 0, 0, kr), _order(s, 0, 1, kc)
        if case["schedule"] == "exact":
            for i in pr:
                x.step(0, *rng_(i, m), 0, n, False)
            for j in pc:
                x.step(1, *rng_(j, n), 0, m, False)
        else:
            for t in range(max(kr, kc)):
                if t < kc:
                    x.step(0, 0, m, *rng_(pc[t], n), True)
                if t < kr:
                    x.step(1, 0, n, *rng_(pr[t], m), True)
    return {"W": x.F[0], "H": x.F[1].T.contiguous()}
