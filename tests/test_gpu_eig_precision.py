"""What the facet Grams and their eigen-solves keep of FP64: singular vectors of channels many
decades fainter than the others, on both Gram kernels of the fast path (up to 8 channels, and
tensor cores) and on the CUDA-core one; duals and
weights of images far from 1 in scale, and weights of nearly
dependent channels, whose singular values lie below 2^-24 of the largest."""
from __future__ import annotations

import numpy as np
import pytest

from oracle.prox import jacobi_svd

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _context(n, L, mu_bar):
    from paper_2003_07358_gb300.fhs import Context, CubeParams
    rng = np.random.default_rng(1)
    uv = rng.uniform(-1.0, 1.0, (16 * L, 2)).astype(np.float32)
    return Context([CubeParams(n1=n, n2=n, L=L, Qy=1, Qx=1, overlap=0.1, window="triangular",
                               M_lb=np.full((L, 1), 16, dtype=np.int64), uv=uv, eta=np.ones(L), mu=0.1,
                               mu_bar=np.array([mu_bar]), eps=np.ones((L, 1)))])


def _sky(n, L, seed):
    """Non-negative sources with power-law spectra, [L][n][n] in float64: their channels are nearly
    dependent, the singular values fall to the rounding of FP32."""
    rng = np.random.default_rng(seed)
    nu, r = np.linspace(1.0, 2.0, L), np.arange(n)
    x = np.zeros((L, n, n))
    for _ in range(60):
        y0, x0, w, a, index = (rng.uniform(*b) for b in ((0, n), (0, n), (1, 4), (0.1, 1), (-1, 1)))
        blob = np.exp(-(r - y0) ** 2 / (2 * w * w))[:, None] * np.exp(-(r - x0) ** 2 / (2 * w * w))
        x += (a * nu ** index)[:, None, None] * blob
    return x


def _dual(x, mu_bar, tb):
    L, n = x.shape[:2]
    ctx = _context(n, L, mu_bar)
    P, A = torch.zeros(L * n * n, device="cuda"), torch.zeros((L, n, n), device="cuda")
    ctx.fhs_prox_nuclear_facets(0, torch.as_tensor(x, device="cuda"), P, torch.as_tensor(tb[None, :], device="cuda"), A)
    ctx.close()
    return P.double().cpu().numpy().reshape(L, n * n).T


@pytest.mark.parametrize("L", [2, 4, 7, 8, 12, 20, 37])
@pytest.mark.parametrize("amps", [(1e-9,), (1e-11,), (1e-13,), (1e-11, 3e-12)])
def test_faint_channels(L, amps):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    if len(amps) >= L:
        pytest.skip("a bright channel is needed")
    n = 64
    rng = np.random.default_rng(L)
    x = _sky(n, L, L)
    faint = [L // 2, L - 1][:len(amps)] if L > 2 else [1]
    for l, a in zip(faint, amps):
        x[l] *= a
    x = (x * (1.0 + 0.2 * rng.standard_normal(x.shape))).astype(np.float32)
    Z = x.reshape(L, -1).T.astype(np.float64)
    U, s, V = jacobi_svd(Z)                          # one-sided: small singular values to full relative accuracy
    tb = np.linspace(0.3, 1.0, L).astype(np.float32)
    mu_bar = 0.1 * s[0]
    m = np.minimum(1.0, mu_bar * tb.astype(np.float64) / s)
    M = (V * m) @ V.T
    got, ref = _dual(x, mu_bar, tb), Z @ M
    # FP32 rows times an FP32 matrix: (L + 2) roundings of 2^-24 on the terms of each channel
    terms = np.linalg.norm(np.abs(Z) @ np.abs(M), axis=0)
    err = np.linalg.norm(got - ref, axis=0)
    assert np.all(err <= 2.0 * (L + 2) * 2.0 ** -24 * terms), (err / terms)[faint]


def _weights(x, mu_bar):
    L, n = x.shape[:2]
    ctx = _context(n, L, mu_bar)
    theta, theta_bar = torch.empty(ctx.sizes(0)["n_coef"], device="cuda"), torch.empty(L, device="cuda")
    ctx.fhs_reweight(0, torch.as_tensor(x, device="cuda"), theta, theta_bar)
    ctx.close()
    return theta_bar.double().cpu().numpy()


def _weights_tol(s, mu_bar):
    """Relative error of mu_bar / (s + mu_bar): an eigenvalue of an FP64 Gram is off by a few
    2^-53 of the largest (4 here), so s by at most 2^-25.5 s_max; theta_bar and mu_bar are FP32."""
    return 2.0 ** -25.5 * s[0] / (s + mu_bar) + 2.0 ** -23


@pytest.mark.parametrize("L", [3, 8, 20, 38, 64])
@pytest.mark.parametrize("scale", [1e-25, 1e-20, 1e-12, 1e12, 1e18, 1e25])
def test_weights_at_any_scale(L, scale):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    n = 64
    rng = np.random.default_rng(L)
    V, _ = np.linalg.qr(rng.standard_normal((L, L)))
    Z = (rng.standard_normal((n * n, L)) * np.logspace(0, -3, L)) @ V.T
    x = np.ascontiguousarray((Z.T * scale).reshape(L, n, n)).astype(np.float32)
    s = np.linalg.svd(x.reshape(L, -1).T.astype(np.float64), compute_uv=False)
    mu_bar = 0.01 * s[0]
    want = mu_bar / (s + mu_bar)
    assert np.all(np.abs(_weights(x, mu_bar) - want) <= _weights_tol(s, mu_bar) * want)


@pytest.mark.parametrize("L,n", [(8, 64), (20, 64), (33, 256), (38, 96), (38, 288), (45, 96), (64, 96), (64, 288)])
@pytest.mark.parametrize("faint", [False, True])
def test_weights_of_dependent_channels(L, n, faint):
    """Both sides of 64 chunks of 1024 pixels (256^2 and 288^2); `faint`: with a channel 1e-9 of the
    others, whose singular value FP64 rotations keep although it lies below 2^-26 of the largest."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    x = _sky(n, L, L)
    if faint:
        x[L // 2] *= 1e-9
    x = x.astype(np.float32)
    s = torch.linalg.svdvals(torch.as_tensor(x.reshape(L, -1).T.astype(np.float64), device="cuda")).cpu().numpy()
    for f in (1e-2, 1e-3, 1e-4):
        mu_bar = f * s[0]
        want = mu_bar / (s + mu_bar)
        got = _weights(x, mu_bar)
        assert np.all(np.abs(got - want) <= _weights_tol(s, mu_bar) * want), (f, np.max(np.abs(got - want) / want))


@pytest.mark.parametrize("L", [1, 3, 4, 5, 8, 12])
@pytest.mark.parametrize("scale", [1e-32, 1e-23, 1e-19, 1e-14, 1e14, 1e18, 1e25])
def test_dual_at_any_scale(L, scale):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    n = 64
    rng = np.random.default_rng(L)
    V, _ = np.linalg.qr(rng.standard_normal((L, L)))
    Z = (rng.standard_normal((n * n, L)) * np.logspace(0, -3, L)) @ V.T * scale
    x = np.ascontiguousarray(Z.T.reshape(L, n, n)).astype(np.float32)
    x[:, : n // 2] *= np.float32(1e-3)               # CTAs on either side of the limits
    Z = x.reshape(L, -1).T.astype(np.float64)
    U, s, Vt = np.linalg.svd(Z / scale, full_matrices=False)
    tb = np.linspace(0.3, 1.0, L).astype(np.float32)
    m = np.minimum(1.0, 0.05 * s[0] * tb.astype(np.float64) / s)
    M = (Vt.T * m) @ Vt
    got = _dual(x, 0.05 * s[0] * scale, tb)
    # FP32 rows times an FP32 matrix, in units of the scale; below 1e-31 FP32's own spacing too
    tol = 2.0 * (L + 2) * 2.0 ** -24 * np.linalg.norm(Z / scale) * np.linalg.norm(M) + n * np.sqrt(L) * 2.0 ** -149 / scale
    assert np.linalg.norm(got / scale - (Z / scale) @ M) <= tol


@pytest.mark.parametrize("L", [2, 4, 7, 8, 10, 16, 24, 32, 36, 64])
def test_dual_beside_a_bright_pixel(L):
    """A bright pixel whose values have 7 bits (every Gram kernel forms their products exactly) and
    independent faint noise elsewhere: s_1 is about 6e4 times the others, whose thresholds and vectors
    show in the faint pixels (their own products with M are accurate to FP32)."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    n = 64
    rng = np.random.default_rng(2000 + L)
    x = rng.standard_normal((L, n, n))
    x[:, :16] = 0.0                                  # the source has a Gram chunk of its own
    x[:, 0, 0] = rng.integers(96, 128, L) * 2.0 ** np.floor(np.log2(6e4 * np.sqrt(48.0 * n / L) / 112))
    x = x.astype(np.float32)
    Z = x.reshape(L, -1).T.astype(np.float64)
    U, s, Vt = np.linalg.svd(Z, full_matrices=False)
    tb = np.linspace(0.3, 1.0, L).astype(np.float32)
    mu_bar = float(s[L // 2])
    m = np.minimum(1.0, mu_bar * tb.astype(np.float64) / s)
    M = (Vt.T * m) @ Vt
    got, ref, faint = _dual(x, mu_bar, tb), Z @ M, slice(16 * n, None)
    # FP32 rows times an FP32 matrix, and an FP64 solve: about 8 sweeps of L rotations of a row, two
    # roundings each, 2^-53 of the largest eigenvalue and adding up at random
    tol = 2.0 * (L + 2) * 2.0 ** -24 * np.linalg.norm(np.abs(Z[faint]) @ np.abs(M))
    tol += 4.0 * np.sqrt(L) * 2.0 ** -53 * (s[0] / s[-1]) ** 2 * np.linalg.norm(ref[faint])
    assert np.linalg.norm(got[faint] - ref[faint]) <= tol


@pytest.mark.parametrize("L", [2, 4, 8])
def test_dual_of_one_large_facet(L):
    """A facet of 4096^2 pixels, where a thread of the Gram kernel adds thousands of products:
    channels that differ by 1e-6, whose dual is that much of them, scaled by alpha / s_j."""
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    n = 4096
    g = torch.Generator(device="cuda").manual_seed(L)
    b = torch.rand((1, n * n), generator=g, device="cuda", dtype=torch.float64) ** 4
    c = torch.linspace(0.6, 1.4, L, device="cuda", dtype=torch.float64)[:, None]
    x = (b * c + 1e-6 * b.square().mean().sqrt() * torch.randn((L, n * n), generator=g, device="cuda")).float()
    # the singular values through a basis whose first vector is the spectrum c: its Gram is graded, and so
    # are its Cholesky factor's entries, which one-sided rotations keep
    basis = torch.linalg.qr(torch.cat([c, torch.eye(L, device="cuda", dtype=torch.float64)[:, 1:]], 1))[0]
    Y = basis.T @ x.double()
    R = np.linalg.cholesky((Y @ Y.T).cpu().numpy()).T
    U, s, V = jacobi_svd(R)
    V = basis.cpu().numpy() @ V
    alpha = 0.5 * float(s[-1])
    ctx = _context(n, L, alpha)
    P, A = torch.zeros(L * n * n, device="cuda"), torch.zeros((L, n, n), device="cuda")
    ctx.fhs_prox_nuclear_facets(0, x.view(L, n, n), P, torch.ones((1, L), device="cuda"), A)
    ctx.close()
    for j in range(1, L):
        v = torch.as_tensor(np.ascontiguousarray(V[:, j]), device="cuda")
        z, p = v @ x.double(), v @ P.view(L, -1).double()
        m = float((p @ z) / (z @ z)) / (alpha / s[j])
        # s_j^2 from a Gram to 2^-47 of s_1^2 (float pairs), and 2^-10 for the solve and FP32
        assert abs(m - 1.0) <= 0.5 * 2.0 ** -47 * (s[0] / s[j]) ** 2 + 2.0 ** -10, (j, m - 1.0, s[0] / s[j])
