"""Phi and Re Phi^dagger on image sides whose grids take the two-for-one mid-size transforms
(every transform length from 96 to 3072, rows and columns of different kinds) against the
FP64 oracle; sides of 16 and 32, sides 9 * 16 and plain-path contexts keep the others."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import nufft as nu

from _fixtures import REL_TOL, rel_err, to_dev_c64, to_dev_f32, vis_to_user

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIDES = [(16, 16), (32, 48), (48, 64), (96, 128), (128, 96), (192, 256), (256, 192), (384, 512), (512, 384),
         (768, 192), (48, 768), (1024, 96), (192, 1024), (1536, 48), (48, 1536), (144, 64)]


@pytest.mark.parametrize("n1,n2", SIDES)
@pytest.mark.parametrize("path", ["fast", "plain"])
def test_measure_and_adjoint(n1, n2, path):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2003_07358_gb300.fhs import Context, CubeParams
    rng = np.random.default_rng(n1 * 10000 + n2)
    L, M = 2, 700
    uv = rng.uniform(-3.1, 3.1, (L * M, 2)).astype(np.float32)
    ctx = Context([CubeParams(n1=n1, n2=n2, L=L, Qy=1, Qx=1, overlap=0.1, window="sine",
                              M_lb=np.full((L, 1), M, dtype=np.int64), uv=uv, eta=np.ones(L), mu=0.1,
                              mu_bar=np.ones(1), eps=np.ones((L, 1)))])
    ctx.fhs_set_path(path)
    x = rng.standard_normal((L, n1, n2)).astype(np.float32)
    y = torch.empty(L * M, dtype=torch.complex64, device="cuda")
    ctx.fhs_measure(0, to_dev_f32(torch, x), y)
    assert rel_err(vis_to_user(ctx, torch, y), nu.measure_cube(x.astype(np.float64), uv, [M] * L)) < REL_TOL
    v = (rng.standard_normal(L * M) + 1j * rng.standard_normal(L * M)).astype(np.complex64)
    vi = torch.empty_like(y)
    ctx.fhs_vis_to_internal(0, to_dev_c64(torch, v), vi)
    out = torch.empty((L, n1, n2), device="cuda")
    ctx.fhs_adjoint(0, vi, out)
    ref = nu.adjoint_cube_real(v.astype(np.complex128), uv, [M] * L, n1, n2)
    assert rel_err(out.cpu().numpy(), ref) < REL_TOL
    ctx.close()
