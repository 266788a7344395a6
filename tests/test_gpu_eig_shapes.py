"""Facet eigen-solves at the edges of the channel counts (one pair, odd counts with the
dummy index, the two-pass task split above 62 channels) and of the chunk counts (partials
added by the solve itself, or first by the chunk sums): nuclear dual
P = Z V diag(min(1, alpha / s)) V^T and weights mu_bar / (s + mu_bar) against numpy's SVD
in float64, an all-zero facet included."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (channels, image side): 64^2 is 4 chunks of 1024 pixels, 272^2 is 73 (past the 64 that the
# solve adds itself), 512^2 is 256
CASES = [(1, 64), (2, 64), (3, 64), (9, 64), (17, 64), (32, 64), (33, 64), (47, 64), (62, 64), (63, 64), (64, 64),
         (5, 512), (12, 512), (33, 512)]


def _context(n, L, mu_bar):
    from paper_2003_07358_gb300.fhs import Context, CubeParams
    rng = np.random.default_rng(1)
    uv = rng.uniform(-1.0, 1.0, (16 * L, 2)).astype(np.float32)
    return Context([CubeParams(n1=n, n2=n, L=L, Qy=1, Qx=1, overlap=0.1, window="triangular",
                               M_lb=np.full((L, 1), 16, dtype=np.int64), uv=uv, eta=np.ones(L), mu=0.1,
                               mu_bar=np.array([mu_bar]), eps=np.ones((L, 1)))])


@pytest.mark.parametrize("L,n", CASES)
def test_dual_and_weights(L, n):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    rng = np.random.default_rng(100 * L + n)
    N = n * n
    V, _ = np.linalg.qr(rng.standard_normal((L, L)))
    s = np.logspace(1, -1, L)                            # 10 .. 0.1 (times about sqrt N)
    Z = (rng.standard_normal((N, L)) * s) @ V.T
    Z = Z.astype(np.float32).astype(np.float64)
    U, sv, Vt = np.linalg.svd(Z, full_matrices=False)
    mu_bar = float(sv[L // 2] * 1.5)
    tb = np.linspace(0.2, 1.0, L).astype(np.float32)
    m = np.minimum(1.0, mu_bar * tb.astype(np.float64) / sv)
    M = (Vt.T * m) @ Vt
    ref = Z @ M
    ctx = _context(n, L, mu_bar)
    X = torch.as_tensor(np.ascontiguousarray(Z.T.reshape(L, n, n), dtype=np.float32), device="cuda")
    P = torch.zeros(L * N, device="cuda")
    A = torch.zeros((L, n, n), device="cuda")
    ctx.fhs_prox_nuclear_facets(0, X, P, torch.as_tensor(tb[None, :], device="cuda"), A)
    got = P.double().cpu().numpy().reshape(L, N).T
    # FP32 rows times an FP32 matrix: (L + 2) roundings of 2^-24 on |z| |M|
    tol = 2.0 * (L + 2) * 2.0 ** -24 * np.linalg.norm(Z) * np.linalg.norm(M)
    assert np.linalg.norm(got - ref) <= tol
    theta = torch.empty(ctx.sizes(0)["n_coef"], device="cuda")
    theta_bar = torch.empty(L, device="cuda")
    ctx.fhs_reweight(0, X, theta, theta_bar)
    want = mu_bar / (sv + mu_bar)
    assert np.max(np.abs(theta_bar.double().cpu().numpy() - want) / want) <= 2.0 ** -23
    # all-zero facet: duals stay zero, weights are one
    P.zero_()
    X.zero_()
    ctx.fhs_prox_nuclear_facets(0, X, P, torch.as_tensor(tb[None, :], device="cuda"), A)
    ctx.fhs_reweight(0, X, theta, theta_bar)
    assert not P.any()
    assert bool((theta_bar == 1.0).all())
    ctx.close()
