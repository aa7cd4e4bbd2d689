"""FP32 products on grids that put every line length on the contiguous and on
a strided axis, with odd numbers of rows and vectors (the two-lines-per-thread
kernels' last pair is then half empty), the narrow strided tile (stride 8),
and blocks that are aligned to one complex64 element only."""
import numpy as np
import pytest

import synth
from gpu_util import make_plan, need_torch_cuda

pytestmark = pytest.mark.gpu

GRIDS = [(32,), (64,), (512,), (1024,), (32, 8), (64, 8), (1024, 8), (8, 32), (16, 128), (32, 512), (512, 32),
         (128, 16), (256, 64), (8, 1024), (8, 8, 64), (64, 32, 8), (16, 64, 32)]


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_apply_f32_lines(n):
    torch = need_torch_cuda()
    from oracle import apply as ap
    from paper_2506_08308_gb300 import bdg
    d = len(n)
    w = synth.Workload("lines", n, (-4.0,) * d, (4.0,) * d, (1.0, 1.3, 0.8)[:d], 20.0, -1.0, 0.05, 0.1, gs_seed=3)
    V, phi, mu = synth.potential(w), synth.initial_spinor(w) * 0.3, np.array([1.1, 0.9, 1.3])
    op = ap.Operator(w, phi, V, mu)
    plan = make_plan(w, V, phi, mu=mu)
    kin = 0.5 * sum((np.pi * k / 8.0) ** 2 for k in n)
    norm = kin + np.max(np.abs(op.Apt).sum(axis=2) + np.abs(op.Bpt).sum(axis=2))
    for nvec in (1, 3):
        x = synth.random_block(w, nvec, seed=21 + nvec).astype(np.complex64)
        buf = torch.zeros(2 * x.size + 2, dtype=torch.complex64, device="cuda")
        xt = buf[1:1 + x.size].view(x.shape)                  # 8 bytes past a 16-byte boundary
        yt = buf[1 + x.size:1 + 2 * x.size].view(x.shape)
        xt.copy_(torch.from_numpy(x))
        for mode in (bdg.UV, bdg.FG):
            yt.fill_(float("nan"))
            plan.apply(xt, mode, out=yt)
            ref = op.apply_fft(x.astype(np.complex128), mode)
            err = np.linalg.norm((yt.cpu().numpy() - ref).ravel()) / (norm * np.linalg.norm(x.ravel()))
            # forward and inverse transforms and the coupling: about 30 roundings of 2^-24 in a row
            assert err < 30 * 2.0 ** -24, (mode, nvec, err)
            assert buf[0] == 0 and buf[-1] == 0
    plan.close()
