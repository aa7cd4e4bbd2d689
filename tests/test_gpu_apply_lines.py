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


@pytest.mark.parametrize("n", GRIDS, ids=lambda n: "x".join(map(str, n)))
def test_apply_f64_few_lines(n):
    """FP64 products of one and three vectors (few lines: four points per
    thread) against the oracle, and those of a block of more than 5000 lines
    (the other kernels) against its vectors taken one by one."""
    torch = need_torch_cuda()
    from oracle import apply as ap
    from paper_2506_08308_gb300 import bdg
    d = len(n)
    w = synth.Workload("lines", n, (-4.0,) * d, (4.0,) * d, (1.0, 1.3, 0.8)[:d], 20.0, -1.0, 0.05, 0.1, gs_seed=3)
    V, phi, mu = synth.potential(w), synth.initial_spinor(w) * 0.3, np.array([1.1, 0.9, 1.3])
    op = ap.Operator(w, phi, V, mu)
    plan = make_plan(w, V, phi, mu=mu)
    for nvec in (1, 3):
        x = synth.random_block(w, nvec, seed=31 + nvec)
        for mode in (bdg.UV, bdg.FG):
            y = plan.apply(torch.from_numpy(x).cuda(), mode).cpu().numpy()
            ref = op.apply_fft(x, mode)
            # about 40 roundings of 2^-53 in a row, relative to the largest symbol times x (y is of its size)
            assert np.linalg.norm((y - ref).ravel()) < 1e-13 * np.linalg.norm(ref.ravel()), (mode, nvec)
    many = 5000 * max(n) // (6 * plan.npts) + 1
    xt = torch.randn((many, 6, plan.npts), dtype=torch.complex128, device="cuda",
                     generator=torch.Generator(device="cuda").manual_seed(5))
    for mode in (bdg.UV, bdg.FG):
        y = plan.apply(xt, mode)
        one = torch.cat([plan.apply(xt[i:i + 1], mode) for i in (0, many // 2, many - 1)])
        two = y[[0, many // 2, many - 1]]
        assert float((one - two).norm() / two.norm()) < 1e-13
    plan.close()
