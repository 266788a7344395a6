"""Sub-iterations of the preconditioned data duals at the edges of their launch (one and two
steps, sixteen blocks, fewer visibilities than a CTA and several CTAs per
channel) with a caller's U spread over four decades, against the FP64 oracle."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import pdfb as pd

from _fixtures import REL_TOL, make_context, make_problem, rel_err, vis_to_internal, vis_to_user

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,M,B,n_sub", [(32, 90, 1, 1), (32, 700, 16, 2), (64, 6100, 3, 5), (64, 6100, 16, 40)])
def test_one_iteration_matches_oracle(n, M, B, n_sub):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    spec, inp, prob = make_problem("tiny", n=n, L=2, m_abs=M, B=B, power_iters=5)
    rng = np.random.default_rng(n_sub)
    U = (10.0 ** rng.uniform(-4.0, 0.0, prob.uv.shape[0])).astype(np.float32)
    prob.U, prob.n_sub = U.astype(np.float64), n_sub
    st = pd.initial_state(prob, inp.x_true)
    st.v[:] = (0.1 * prob.U * (rng.standard_normal(U.size) + 1j * rng.standard_normal(U.size))).astype(np.complex64)
    ctx = make_context(prob, torch)
    ctx.fhs_set_preconditioning(0, n_sub, U)
    X = torch.as_tensor(inp.x_true.astype(np.float32), device="cuda")
    state = ctx.new_state(0)
    state["v"] = vis_to_internal(ctx, torch, st.v)
    state["u_prev"] = vis_to_internal(ctx, torch, st.u_prev)
    it = [{"X": X, "Xcheck": X.clone(), "y": vis_to_internal(ctx, torch, prob.y), "state": state}]
    ctx.fhs_pdfb_iter(it, 1)
    # v = U (d - w) is a difference of d = v / U + 2 u - u_prev - y and its projection: the
    # per-operator bar applies to the terms it is formed from
    u = pd.measure_all(prob, st.X)
    terms = np.abs(st.v) + prob.U * (2 * np.abs(u) + np.abs(st.u_prev) + np.abs(prob.y))
    pd.pdfb_iteration(prob, st)
    assert np.linalg.norm(vis_to_user(ctx, torch, state["v"]) - st.v) < REL_TOL * np.linalg.norm(terms)
    assert rel_err(X.double().cpu().numpy(), st.X) < REL_TOL
    ctx.close()
