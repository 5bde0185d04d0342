"""The work that a user of this package has it do, as measurable cases.

Each case is one call through the public entry points of
``paper_1312_6838_gb300.css`` on seeded synthetic inputs, or one forward and
backward pass for the differentiable residual.  Sizes are those of the
package's configurations (``css_inputs.CONFIGS``), its tests and its benchmark,
with ragged ones between them.  ``exact`` restates every computed result in
FP64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1312_6838_gb300 import css

_DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_SIZE = {"f64": 8, "f32": 4, "bf16": 2}
_DEV = "cuda"


def listed():
    return [
        # One small problem, the smallest instance of a batched workload called
        # on its own: launches and latency are all of it.
        dict(name="select_f32_64x128", kind="select", dtype="f32", m=64, n=128, k=8, rank=8, noise=1e-2),
        # The paper's medium data sets in plain FP64.
        dict(name="select_f64_500x1000", kind="select", dtype="f64", m=500, n=1000, k=50, rank=50, noise=1e-2),
        # The memory-efficient centralized selection at scale, streamed in BF16.
        dict(name="select_bf16_4096x65536", kind="select", dtype="bf16", m=4096, n=65536, k=256, rank=256, noise=1e-3,
             decay=True),
        # The same method in FP32 on a matrix as it comes: odd sizes, columns
        # that start on no 16-byte boundary.
        dict(name="select_f32_1999x30011", kind="select", dtype="f32", m=1999, n=30011, k=100, rank=128, noise=1e-3,
             decay=True),
        # Many independent instances of uneven sizes in one call.
        dict(name="batched_bf16_1024", kind="batched", dtype="bf16", count=1024),
        # Algorithm 4 on 64 uneven column blocks with the concise representation
        # of the data (B = A Omega) already at hand.
        dict(name="distributed_bf16_2048x262144", kind="distributed", dtype="bf16", m=2048, n=262144, r=400, blocks=64,
             l=100, k=100, rank=400, noise=1e-3),
        # Columns of A chosen to reconstruct another matrix (Algorithm 3).
        dict(name="gcss_f32_1500x24001", kind="gcss", dtype="f32", m=1500, n=24001, r=200, k=64, rank=100, noise=1e-3),
        # The random projection of the distributed variant: BF16 at scale, and
        # FP32 with odd sizes.
        dict(name="project_bf16_2048x262144", kind="project", dtype="bf16", m=2048, n=262144, r=400, rank=400,
             noise=1e-3),
        dict(name="project_f32_1500x50001", kind="project", dtype="f32", m=1500, n=50001, r=200, rank=100, noise=1e-3),
        # Reconstruction error at a fixed selection, forward and backward.
        dict(name="residual_f32_4096x16384", kind="residual", dtype="f32", m=4096, n=16384, k=128, rank=128,
             noise=1e-3),
        # The embedding of every column into the span of a selection (Sec. 3.2).
        dict(name="embed_bf16_4096x65536", kind="embed", dtype="bf16", m=4096, n=65536, l=256, rank=256, noise=1e-3,
             decay=True),
        # The approximate SVD from such an embedding.
        dict(name="lowrank_256x65536", kind="lowrank", dtype="f64", m=4096, n=65536, l=256, k=128, rank=256, noise=1e-3),
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]; rarely a round one."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    v = min(hi, max(lo, v))
    return max(lo, v // 8 * 8) if rng.random() < 0.4 else v


def draw(rng):
    kind = rng.choice(["select", "select", "select", "batched", "distributed", "gcss", "project", "residual",
                       "residual", "embed", "lowrank"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "select":
        dtype = rng.choice(["f64", "f32", "bf16"])
        m = _log(rng, 64, 1024 if dtype == "f64" else 4096)
        n = _log(rng, 128, 8192 if dtype == "f64" else 32768)
        k = min(_log(rng, 8, 256), m // 2, n // 2)
        return dict(kind=kind, dtype=dtype, m=m, n=n, k=k, rank=max(8, k), noise=1e-2, decay=rng.random() < 0.3)
    if kind == "batched":
        return dict(kind=kind, dtype=dtype, count=_log(rng, 8, 512))
    if kind == "distributed":
        blocks = _log(rng, 8, 64)
        return dict(kind=kind, dtype=dtype, m=_log(rng, 256, 2048), n=_log(rng, 16384, 131072), r=_log(rng, 32, 400),
                    blocks=blocks, l=_log(rng, 16, 64), k=_log(rng, 16, 100), rank=100, noise=1e-3)
    if kind == "gcss":
        dtype = rng.choice(["f64", "f32", "bf16"])
        m = _log(rng, 64, 512 if dtype == "f64" else 2048)
        n = _log(rng, 256, 4096 if dtype == "f64" else 32768)
        return dict(kind=kind, dtype=dtype, m=m, n=n, r=_log(rng, 8, 400), k=min(_log(rng, 8, 128), m // 2, n // 2),
                    rank=max(16, m // 8), noise=1e-3)
    if kind == "project":
        return dict(kind=kind, dtype=dtype, m=_log(rng, 128, 4096), n=_log(rng, 1024, 131072), r=_log(rng, 16, 400),
                    rank=64, noise=1e-3)
    if kind == "residual":
        dtype = rng.choice(["f64", "f32", "bf16"])
        m = _log(rng, 256, 1024 if dtype == "f64" else 4096)
        n = _log(rng, 512, 4096 if dtype == "f64" else 16384)
        k = min(_log(rng, 8, 128), m // 4)
        return dict(kind=kind, dtype=dtype, m=m, n=n, k=k, rank=k, noise=1e-3)
    if kind == "embed":
        m = _log(rng, 256, 4096)
        return dict(kind=kind, dtype=dtype, m=m, n=_log(rng, 1024, 65536), l=min(_log(rng, 8, 256), m // 4), rank=128,
                    noise=1e-3, decay=True)
    l = _log(rng, 16, 256)
    return dict(kind=kind, dtype="f64", m=_log(rng, 512, 4096), n=_log(rng, 1024, 65536), l=l, k=max(8, l // 2),
                rank=l, noise=1e-3)


# ------------------------------------------------------------------ inputs --
def _gen(seed):
    return torch.Generator(device=_DEV).manual_seed(int(seed) % (1 << 62))


def _normal(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device=_DEV, dtype=dtype)


def _matrix(g, m, n, rank, noise, dtype, decay=False):
    """A column-major m x n matrix U V + noise N; with `decay`, U and V have
    orthonormal columns and the singular values are 1 / i."""
    work = torch.float64 if dtype == torch.float64 else torch.float32
    rank = min(rank, m, n)
    U = _normal(g, m, rank, dtype=work)
    V = _normal(g, n, rank, dtype=work)
    if decay:
        U = torch.linalg.qr(U)[0] / torch.arange(1, rank + 1, device=_DEV, dtype=work)
        V = torch.linalg.qr(V)[0]
    A = torch.empty((n, m), dtype=dtype, device=_DEV)   # its rows are the columns
    step = max(1, (1 << 26) // m)
    for c in range(0, n, step):
        X = V[c:c + step] @ U.t()
        X += noise * _normal(g, X.shape[0], m, dtype=work)
        A[c:c + step] = X
    return A.t()


def _columns(g, n, k):
    return torch.randperm(n, generator=g, device=_DEV)[:k].to(torch.int32)


def _offsets(n, blocks, seed):
    """Offsets of log-normal block widths (sigma 0.8) that sum to n."""
    w = np.random.RandomState(int(seed) % (1 << 32)).lognormal(0.0, 0.8, blocks)
    least = min(100, n // (2 * blocks))
    at = least * np.arange(blocks + 1) + np.concatenate([[0], np.cumsum(w)]) / w.sum() * (n - least * blocks)
    at = [int(v) for v in at]
    at[-1] = n
    return at


def prepare(case, seed):
    g = _gen(seed)
    kind, dtype = case["kind"], _DTYPES[case["dtype"]]
    state = {"case": case}
    if kind == "batched":
        sizes = np.random.RandomState(4)   # a workload has its sizes; the seed draws the values
        As, ks = [], []
        for _ in range(case["count"]):
            m, n, k = int(sizes.randint(64, 1025)), int(sizes.randint(128, 4097)), int(sizes.randint(8, 65))
            As.append(_matrix(g, m, n, k, 1e-2, dtype))
            ks.append(min(k, m, n))
        return {**state, "A": As, "k": ks}
    m, n = case["m"], case["n"]
    A = _matrix(g, m, n, case["rank"], case["noise"], dtype, case.get("decay", False))
    if kind in ("gcss", "distributed"):
        # the target: random combinations of the columns, as B = A Omega gives
        r = case["r"]
        acc = torch.float64 if dtype == torch.float64 else torch.float32
        B = torch.zeros((r, m), dtype=acc, device=_DEV)
        step = 16384
        for c in range(0, n, step):
            X = A[:, c:c + step].to(acc)
            B += (_normal(g, r, X.shape[1], dtype=acc) / math.sqrt(r)) @ X.t()
        state["B"] = B.t()
        if kind == "distributed":
            state["offsets"] = _offsets(n, case["blocks"], seed)
    elif kind == "project":
        state["Omega"] = (_normal(g, case["r"], n) / math.sqrt(case["r"])).to(dtype).t()
    elif kind == "residual":
        state["S"] = _columns(g, n, case["k"])
        A = A.detach().requires_grad_()
    elif kind == "embed":
        state["S"] = _columns(g, n, case["l"])
    elif kind == "lowrank":
        # an embedding as css.embed returns it: Q = orth(A_S), W = Q^T A
        S = _columns(g, n, case["l"]).long()
        Q = torch.linalg.qr(A[:, S])[0]
        state["Q"] = Q.t().contiguous().t()
        state["W"] = (Q.t() @ A).contiguous()
        return state
    state["A"] = A
    return state


# --------------------------------------------------------------------- run --
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "select":
        r = css.select(state["A"], case["k"])
        return {"sel": r.sel, "trace": r.trace, "n_sel": r.n_sel}
    if kind == "batched":
        rs = css.select_batched(state["A"], state["k"])
        return {"sel": torch.cat([r.sel for r in rs]), "trace": torch.cat([r.trace for r in rs])}
    if kind == "distributed":
        r = css.distributed(state["A"], state["B"], state["offsets"], case["l"], case["k"])
        return {"sel": r.sel, "trace": r.trace, "n_sel": r.n_sel, "block_sel": r.block_sel}
    if kind == "gcss":
        r = css.gcss_select(state["A"], state["B"], case["k"])
        return {"sel": r.sel, "trace": r.trace, "n_sel": r.n_sel}
    if kind == "project":
        return {"B": css.project(state["A"], state["Omega"])}
    if kind == "residual":
        loss = css.residual(state["A"], state["S"])
        (grad,) = torch.autograd.grad(loss, state["A"])
        return {"loss": loss.detach(), "grad": grad}
    if kind == "embed":
        r = css.embed(state["A"], state["S"])
        return {"Q": r.Q, "W": r.W}
    r = css.lowrank(state["W"], case["k"], state["Q"])
    return {"sigma": r.sigma, "Uw": r.Uw, "U": r.U, "V": r.V, "tail": r.tail}


def work(case):
    kind, e = case["kind"], _SIZE[case["dtype"]]
    if kind == "batched":
        sizes = np.random.RandomState(4)
        total = {"bytes": 0.0, "flops": 0.0}
        for _ in range(case["count"]):
            m, n, k = int(sizes.randint(64, 1025)), int(sizes.randint(128, 4097)), int(sizes.randint(8, 65))
            one = work(dict(kind="select", dtype=case["dtype"], m=m, n=n, k=min(k, m, n)))
            total = {q: total[q] + one[q] for q in total}
        return total
    m, n = float(case["m"]), float(case["n"])
    k = float(case.get("k", 0))
    if kind == "select":
        # the scores' contraction with A A^T (its symmetric halves), then per
        # pick two products with every column and one with A A^T
        return {"bytes": e * m * n + 12 * k, "flops": 2 * m * m * n + k * (4 * m * n + 2 * m * m)}
    if kind in ("gcss", "distributed"):
        acc = 8.0 if case["dtype"] == "f64" else 4.0
        r = float(case["r"])
        nb = case.get("blocks", 1)
        l = float(case.get("l", k))
        flops = 2 * m * r * n + l * (4 * m * n + 4 * m * r * nb)
        if kind == "distributed":
            flops += k * (4 * m * nb * l + 4 * m * r)
        return {"bytes": e * m * n + acc * m * r + 12 * k + (4 * nb * l if kind == "distributed" else 0), "flops": flops}
    if kind == "project":
        r = float(case["r"])
        return {"bytes": e * (m * n + n * r) + 4 * m * r, "flops": 2 * m * n * r}
    if kind == "residual":
        # W = Q^T A, R = A - Q W, R W^T
        return {"bytes": 2 * e * m * n, "flops": 6 * m * n * k}
    if kind == "embed":
        l = float(case["l"])
        return {"bytes": e * m * n + 8 * (m * l + l * n), "flops": 2 * m * n * l + 8 * m * l * l}
    l = float(case["l"])
    return {"bytes": 8 * (l * n + m * l + k * (n + m + l + 1)), "flops": l * l * n + 2 * k * l * (n + m) + 10 * l ** 3}


# ------------------------------------------------------------------- exact --
def _greedy(A, k, f, target, tau):
    """The greedy selection in FP64: picks and error trace.  `f` are the
    initial numerators; `target(q)` the vector whose products with the columns
    update them and the squared norm that goes with it."""
    g = A.square().sum(0)
    least = tau * g
    Q = torch.empty((k, A.shape[0]), dtype=torch.float64, device=A.device)
    f = f.clone()
    free = g > 0
    picks, drops = [], []
    for t in range(k):
        score = torch.where(free & (g > least), f.clamp_min(0) / g, torch.full_like(f, -1.0))
        p = torch.argmax(score)
        drops.append(f[p] / g[p])
        picks.append(p)
        a = A.index_select(1, p.view(1)).view(-1)
        q = a
        for _ in range(2):
            q = q - Q[:t].t() @ (Q[:t] @ q)
        q = q / torch.linalg.vector_norm(q)
        y, s = target(q)
        y = y - Q[:t].t() @ (Q[:t] @ y)
        P = torch.stack([q, y]) @ A
        w, h = P[0], P[1]
        f = f - 2 * w * h + s * w * w
        g = g - w * w
        Q[t] = q
        free = free.index_fill(0, p.view(1), False)
    return torch.stack(picks), torch.stack(drops)


def _trace(total, drops):
    return torch.cat([total.view(1), total - torch.cumsum(drops, 0)])


def _tau(dtype):
    return 1e-12 if dtype == "f64" else 1e-6


def _select_exact(A, k, dtype):
    A = A.double()
    C = A @ A.t()

    def target(q):
        y = C @ q
        return y, q @ y

    f = torch.cat([(A[:, c:c + 8192] * (C @ A[:, c:c + 8192])).sum(0) for c in range(0, A.shape[1], 8192)])
    picks, drops = _greedy(A, k, f, target, _tau(dtype))
    return picks, _trace(A.square().sum(), drops)


def _gcss_exact(A, B, k, dtype):
    A, B = A.double(), B.double()

    def target(q):
        u = B.t() @ q
        return B @ u, u @ u

    f = torch.cat([(B.t() @ A[:, c:c + 8192]).square().sum(0) for c in range(0, A.shape[1], 8192)])
    picks, drops = _greedy(A, k, f, target, _tau(dtype))
    return picks, _trace(B.square().sum(), drops)


def exact(case, seed):
    kind = case["kind"]
    state = prepare(case, seed)
    with torch.no_grad():
        if kind == "select":
            _, trace = _select_exact(state["A"], case["k"], case["dtype"])
            return {"sel": None, "trace": trace, "n_sel": None}
        if kind == "batched":
            if case["count"] > 300:
                # every instance would take too long: nothing is said here, and
                # the drawn batches are checked instead
                return None
            traces = [_select_exact(A, k, case["dtype"])[1] for A, k in zip(state["A"], state["k"])]
            return {"sel": None, "trace": torch.cat(traces)}
        if kind == "distributed":
            A, B, at = state["A"], state["B"], state["offsets"]
            union = []
            for lo, hi in zip(at[:-1], at[1:]):
                picks, _ = _gcss_exact(A[:, lo:hi], B, min(case["l"], hi - lo), case["dtype"])
                union.append(picks + lo)
            _, trace = _gcss_exact(A[:, torch.cat(union)], B, case["k"], case["dtype"])
            return {"sel": None, "trace": trace, "n_sel": None, "block_sel": None}
        if kind == "gcss":
            _, trace = _gcss_exact(state["A"], state["B"], case["k"], case["dtype"])
            return {"sel": None, "trace": trace, "n_sel": None}
        if kind == "project":
            A, Om = state["A"], state["Omega"]
            B = torch.zeros((case["m"], case["r"]), dtype=torch.float64, device=_DEV)
            for c in range(0, case["n"], 16384):
                B += A[:, c:c + 16384].double() @ Om[c:c + 16384].double()
            return {"B": B}
        if kind in ("residual", "embed"):
            A = state["A"].detach().double()
            AS = A[:, state["S"].long()]
            Q, R = torch.linalg.qr(AS)
            sign = torch.sign(torch.diagonal(R))
            Q, R = Q * sign, R * sign[:, None]
            W = Q.t() @ A
            if kind == "embed":
                return {"Q": Q, "W": W}
            E = A - Q @ W
            E -= Q @ (Q.t() @ E)
            E[:, state["S"].long()] = 0
            grad = 2 * E
            # T = R^-1 W;  dL/dA_S = -2 E T^T
            T = torch.linalg.solve_triangular(R, W, upper=True)
            grad[:, state["S"].long()] = -2 * (E @ T.t())
            return {"loss": E.square().sum(), "grad": grad}
        W, Q, k = state["W"], state["Q"], case["k"]
        U, s, Vt = torch.linalg.svd(W.cpu(), full_matrices=False)
        U, s, Vt = U.to(_DEV), s.to(_DEV), Vt.to(_DEV)
        # the largest entry of each left vector is positive
        sign = torch.sign(U.gather(0, U.abs().argmax(0, keepdim=True)))
        U, Vt = U * sign, Vt * sign.t()
        return {"sigma": s[:k], "Uw": U[:, :k], "U": Q @ U[:, :k], "V": Vt[:k].t(), "tail": s[k:].square().sum()}
