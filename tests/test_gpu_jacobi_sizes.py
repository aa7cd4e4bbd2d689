"""The small eigensolver's cluster and one-CTA Jacobi kernels around their
switch (64 columns), at odd and even counts of pair positions per CTA and at
the largest size, through bdg_biortho (whose real embedding is four times the
block's columns): F^H G = I on the kept columns and zeros in the others, to the
FP64 bound of the other bi-orthogonalisation tests.  (The kept rank itself is
the choice of one vector per complex direction, not of these kernels.)"""
import numpy as np
import pytest

import synth
from gpu_util import make_plan, need_torch_cuda, oracle_problem

pytestmark = pytest.mark.gpu

W = synth.Workload("s2d_16", (16, 16), (-6.0, -6.0), (6.0, 6.0), (1.0, 1.4), 12.0, -1.0, 0.05, 0.3, gs_seed=8)


@pytest.mark.parametrize("ncol,copies", [(15, 0), (16, 0), (17, 0), (23, 0), (24, 5), (33, 0), (40, 0), (40, 3)])
def test_jacobi_sizes(ncol, copies):
    torch = need_torch_cuda()
    V, phi, mu, op = oracle_problem(W)
    plan = make_plan(W, V, phi)
    rng = np.random.default_rng(ncol + copies)
    z = lambda: rng.standard_normal((3 * W.npts, ncol)) + 1j * rng.standard_normal((3 * W.npts, ncol))  # noqa: E731
    F0 = z()
    G0 = F0 + 0.5 * z()
    F0[:, :copies] = F0[:, copies : 2 * copies]      # a block that loses rank
    dev = lambda M: torch.from_numpy(np.ascontiguousarray(M.T.reshape(ncol, 3, -1))).cuda()  # noqa: E731
    F, G = dev(F0), dev(G0)
    r = plan.biortho(F, G)
    plan.close()
    assert 0 < r <= ncol - copies
    Fg, Gg = (t.cpu().numpy().reshape(ncol, -1).T for t in (F, G))
    assert np.abs(Fg[:, :r].conj().T @ Gg[:, :r] - np.eye(r)).max() < 1e-10
    assert not Fg[:, r:].any() and not Gg[:, r:].any()
