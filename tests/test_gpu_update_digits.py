"""FP64 block updates from exact integer digits inside bdg_solve (blocks of
8192 rows and more): block sizes whose updates take one to five stages and
every width of the output tile, against the same solve with every contraction
in double-float (BDG_GRAM_TC=0) and against the oracle's operator.  Bounds:
the solver's own 1e-10 on residuals (10 % for another FFT's rounding) and on
eigenvalues, 1e-8 on the bi-orthogonality, as for every other solve."""
import numpy as np
import pytest

import synth
from gpu_util import make_plan, need_torch_cuda, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,m", [(6, 14), (14, 25), (30, 46), (36, 52)])
def test_update_digits_in_a_solve(k, m, monkeypatch):
    torch = need_torch_cuda()
    from oracle import lrep
    from paper_2506_08308_gb300 import bdg
    w = synth.Workload("s2d_64", (64, 64), (-8.0, -8.0), (8.0, 8.0), (1.0, 1.3), 30.0, -1.0, 0.0, 0.1, k=k, m=m,
                       gs_seed=3, block_seed=4)
    V, phi, mu, op = oracle_problem(w)
    X0 = torch.from_numpy(synth.random_block(w, w.m, complex_=True)).cuda()
    plan = make_plan(w, V, phi, prec=bdg.FP64, tol=1e-10, maxit=600)
    om, UV, resid, nconv = plan.solve(k, m, X0=X0)
    monkeypatch.setenv("BDG_GRAM_TC", "0")
    om_df, _, _, nconv_df = plan.solve(k, m, X0=X0)
    plan.close()
    assert nconv == nconv_df == k and np.all(resid[:k] <= 1e-10)
    np.testing.assert_allclose(om[:k], om_df[:k], rtol=1e-10, atol=0)
    uv = UV[:k].cpu().numpy().real
    assert lrep.residual_uv(op, uv, om[:k]).max() <= 1.1e-10
    U, Vv = uv[:, :3].reshape(k, -1), uv[:, 3:].reshape(k, -1)
    assert np.abs(lrep.weight(w) * (U @ U.T - Vv @ Vv.T) - np.eye(k)).max() < 1e-8
