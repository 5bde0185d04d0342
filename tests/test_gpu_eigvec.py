"""The eigenvector estimate (eigvec.cu) before the Jacobi rounds of css_lowrank:
sizes around its blocks, and spectra that FP32 separates, resolves in part or
not at all."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _spectrum(kind, l):
    i = np.arange(1, l + 1)
    return {"flat": 1.0 + 0.5 * np.cos(i), "graded": 1.0 / i, "steep": 10.0 ** (-12.0 * i / l),
            "clusters": 1.0 + (i % 3) + 1e-9 * i, "equal": np.ones(l), "rank": (i <= l // 2) * 1.0 / i,
            "tiny": 1e-140 / i, "huge": 1e140 / i}[kind]


@pytest.mark.parametrize("l,kind", [(31, "flat"), (32, "flat"), (33, "graded"), (63, "clusters"), (64, "rank"),
                                    (65, "steep"), (96, "equal"), (127, "flat"), (128, "clusters"), (129, "graded"),
                                    (64, "tiny"), (64, "huge"), (200, "steep"), (257, "clusters")])
def test_lowrank_spectra(l, kind):
    from paper_1312_6838_gb300 import css
    rng = np.random.default_rng(l)
    n = 4 * l + 5
    s = np.sort(_spectrum(kind, l))[::-1]
    U = np.linalg.qr(rng.standard_normal((l, l)))[0]
    V = np.linalg.qr(rng.standard_normal((n, l)))[0]
    W = (U * s) @ V.T
    r = css.lowrank(torch.from_numpy(W).cuda(), l)
    sig, Uw = r.sigma.cpu().numpy(), r.Uw.cpu().numpy()
    top = s[0]
    ref = np.linalg.svd(W / top, compute_uv=False)
    w2 = float(np.sum(ref ** 2))
    tol = 4 * (n + l) * 2.0 ** -52 * w2   # the Gram route's resolution
    assert np.all(np.diff(sig) <= 0)
    assert np.all(np.abs((sig / top) ** 2 - ref ** 2) <= tol)
    np.testing.assert_allclose(Uw.T @ Uw, np.eye(l), atol=1e-12)
    G = (W / top) @ (W / top).T
    assert np.abs(G @ Uw - Uw * (sig / top) ** 2).max() <= tol
    again = css.lowrank(torch.from_numpy(W).cuda(), l)
    assert torch.equal(again.sigma, r.sigma) and torch.equal(again.Uw, r.Uw)
