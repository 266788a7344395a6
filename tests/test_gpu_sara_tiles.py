"""Fused SARA passes (analysis, l2,1 dual, synthesis, weights) against the per-pass kernels at
the edges of their tiles: images smaller than a tile, sides that leave ragged tiles at every
level, and enough channels that the 64 x 64 synthesis tiles and the per-basis launches run."""
from __future__ import annotations

import numpy as np
import pytest

from _fixtures import REL_TOL

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n1,n2,L", [(16, 16, 1), (32, 48, 3), (96, 64, 5), (144, 192, 2), (256, 96, 33), (512, 512, 15),
                                     (768, 384, 17), (1024, 512, 64)])
def test_fast_and_plain_paths_agree(n1, n2, L):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2003_07358_gb300.fhs import Context, CubeParams
    rng = np.random.default_rng(n1 + n2 + L)
    uv = rng.uniform(-1.0, 1.0, (16 * L, 2)).astype(np.float32)
    ctx = Context([CubeParams(n1=n1, n2=n2, L=L, Qy=1, Qx=1, overlap=0.1, window="sine",
                              M_lb=np.full((L, 1), 16, dtype=np.int64), uv=uv, eta=np.ones(L), mu=2.0,
                              mu_bar=np.ones(1), eps=np.ones((L, 1)))])
    g = torch.Generator(device="cuda").manual_seed(n1 * L)
    I = ctx.sizes(0)["n_coef"]
    x = torch.randn((L, n1, n2), generator=g, device="cuda")
    W0 = torch.randn(L * I, generator=g, device="cuda")
    theta = torch.rand(I, generator=g, device="cuda")
    A0 = torch.randn((L, n1, n2), generator=g, device="cuda")
    got = {}
    for path in ("fast", "plain"):
        ctx.fhs_set_path(path)
        W, A, th, tb = W0.clone(), A0.clone(), torch.empty(I, device="cuda"), torch.empty(L, device="cuda")
        ctx.fhs_prox_l21_sara_facets(0, x, W, theta, A)
        ctx.fhs_reweight(0, x, th, tb)
        got[path] = (W, A - A0, th, tb)
    for a, b in zip(got["fast"], got["plain"]):
        assert float(torch.linalg.vector_norm((a - b).double())) <= REL_TOL * float(torch.linalg.vector_norm(b.double()))
    ctx.close()
