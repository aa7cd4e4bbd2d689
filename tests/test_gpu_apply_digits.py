"""FP64 products whose axes of 128 and 256 points run in integer digits on the
tensor cores (more than 2048 lines): each axis alone and together, a last
tile that is not full, lines of very different size side by side, zero lines,
and lines that hold a NaN or an infinity."""
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


@pytest.mark.parametrize("n,nvec", [((256,), 343), ((128,), 350), ((128, 128), 3), ((256, 128), 2), ((8, 256), 43),
                                    ((256, 8), 43), ((128, 32), 11), ((64, 128), 6), ((16, 8, 128), 3),
                                    ((128, 8, 16), 3), ((8, 256, 16), 3)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_apply_digits_against_oracle(n, nvec):
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    w, op, plan = _setup(n)
    x = synth.random_block(w, nvec, seed=5)
    x[::3] *= 1e-40
    x[1, 4] = 0.0
    xt = torch.from_numpy(x).cuda()
    for mode in (bdg.UV, bdg.FG):
        y = plan.apply(xt, mode).cpu().numpy()
        for i in sorted({0, 1, nvec // 2, nvec - 1}):
            ref = op.apply_fft(x[i:i + 1], mode)[0]
            # per component; the reference's own FFT roundings included
            for c in range(6):
                assert np.linalg.norm(y[i, c] - ref[c]) < 3e-15 * np.linalg.norm(ref), (mode, i, c)
    plan.close()


def test_apply_digits_non_finite_lines():
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    w, op, plan = _setup((128, 128))
    x = synth.random_block(w, 3, seed=9)
    clean = plan.apply(torch.from_numpy(x).cuda(), bdg.FG).cpu().numpy().reshape(3, 6, 128, 128)
    x = x.reshape(3, 6, 128, 128)
    x[1, 4, 17, 90] = np.nan
    x[2, 0, 5, 6] = complex(np.inf, 0.0)
    y = plan.apply(torch.from_numpy(x.reshape(3, 6, -1)).cuda(), bdg.FG).cpu().numpy().reshape(3, 6, 128, 128)
    assert np.array_equal(y[0], clean[0])
    for v, c, i, j in ((1, 4, 17, 90), (2, 0, 5, 6)):
        assert np.all(~np.isfinite(y[v, c, i, :].real)) and np.all(~np.isfinite(y[v, c, :, j].real))
        far = np.ones((128, 128), dtype=bool)
        far[i, :] = far[:, j] = False
        assert np.array_equal(y[v, c][far], clean[v, c][far])
    plan.close()
