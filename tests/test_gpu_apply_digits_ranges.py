"""FP64 products in integer digits (axes of 128 and 256 points, more than 2048
lines) at the ends of their ranges."""
import numpy as np
import pytest

import synth
from gpu_util import make_plan, need_torch_cuda

pytestmark = pytest.mark.gpu


def _setup(n):
    from oracle import apply as ap
    d = len(n)
    w = synth.Workload("digits", n, (-6.0,) * d, (6.0,) * d, (1.0, 1.3, 0.8)[:d], 30.0, -1.5, 0.05, 0.1, gs_seed=4)
    V, phi, mu = synth.potential(w), synth.initial_spinor(w) * 0.3, np.array([1.1, 0.9, 1.3])
    return w, ap.Operator(w, phi, V, mu), make_plan(w, V, phi, mu=mu)


def test_more_than_a_million_vectors():
    """More groups of 16 vectors than gridDim.y holds: the same bits as the
    same vectors in parts."""
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    w, op, plan = _setup((128,))
    part = 1 << 16
    nvec = 16 * part + 400
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of device memory")
    x = torch.empty((nvec, 6, 128), dtype=torch.complex128, device="cuda")
    torch.view_as_real(x).normal_(generator=torch.Generator(device="cuda").manual_seed(1))
    y = plan.apply(x, bdg.UV)
    for i in range(0, nvec, part):
        assert torch.equal(y[i:i + part], plan.apply(x[i:i + part], bdg.UV)), i
    plan.close()
