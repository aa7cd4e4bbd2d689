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


@pytest.mark.parametrize("n,nvec", [((256, 256), 2), ((128, 8, 128), 2), ((256,), 350)])
def test_small_coupling_beside_a_large_one(n, nvec):
    """UV form with v = 0: the last three components are -B u alone, with a
    relative accuracy of the sum of |B u|'s three terms: 8 units of 2^-53 for
    B's entries (six roundings at most) and the products."""
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    w, op, plan = _setup(n)
    x = synth.random_block(w, nvec, seed=5)
    x[:, 3:] = 0.0
    y = plan.apply(torch.from_numpy(x).cuda(), bdg.UV).cpu().numpy()[:, 3:]
    a, b, c = (synth.initial_spinor(w) * 0.3).reshape(3, -1).astype(np.longdouble)
    bn, bs = np.longdouble(w.beta_n), np.longdouble(w.beta_s)
    B = [[(bn + bs) * a * a, (bn + bs) * a * b, bn * a * c + bs * (b * b - a * c)],
         [(bn + bs) * a * b, bn * b * b + 2 * bs * a * c, (bn + bs) * b * c],
         [bn * a * c + bs * (b * b - a * c), (bn + bs) * b * c, (bn + bs) * c * c]]
    # (terms of an entry before they cancel)
    S = [[abs(e) for e in r] for r in B]
    S[0][2] = S[2][0] = abs(bn * a * c) + abs(bs) * (b * b + abs(a * c))
    S[1][1] = abs(bn) * b * b + 2 * abs(bs * a * c)
    for j in range(3):
        for part in ("real", "imag"):
            u = getattr(x[:, :3], part).astype(np.longdouble)
            ref = -sum(B[j][k] * u[:, k] for k in range(3))
            size = sum(S[j][k] * abs(u[:, k]) for k in range(3))
            err = abs(getattr(y[:, j], part) - ref) / size
            assert err.max() < 8 * 2.0 ** -53, (j, part, err.max())
    plan.close()


@pytest.mark.parametrize("n,nvec", [((128,), 350), ((256,), 350), ((128, 64), 6), ((256, 32), 9)])
@pytest.mark.parametrize("k", [-960, -1000, -1030])
def test_lines_of_very_small_values(n, nvec, k):
    """Lines down to subnormal values, with zeros between them: x 2^k gives the
    result 2^k times that of x, to 2^-54 of a line's largest value and to
    2^-1074 (the spacing of subnormal numbers, at which the passes that stay
    FFTs and the coupling round) times the l1 norm N^2 / 4 of an axis' kernel
    (kappa < 1); four times that for the roundings one after another."""
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    w, op, plan = _setup(n)
    x = synth.random_block(w, nvec, seed=6)
    x[:, :, ::3] = 0.0
    x[::4] *= 1e-12                  # lines of other sizes in the same tile
    x[1] = 0.0
    x = np.ldexp(np.ldexp(x.view(np.float64), k), -k).view(np.complex128)   # (what survives as a subnormal)
    xk = np.ldexp(x.view(np.float64), k).view(np.complex128)
    for mode in (bdg.UV, bdg.FG):
        y = plan.apply(torch.from_numpy(x).cuda(), mode).cpu().numpy()
        yk = plan.apply(torch.from_numpy(xk).cuda(), mode).cpu().numpy()
        yk = np.ldexp(yk.view(np.float64), -k).view(np.complex128)
        tol = sum(m * m for m in n) * (2.0 ** -56 * np.abs(x).max(axis=(1, 2)) + 2.0 ** (-1074 - k))
        assert np.all(np.abs(yk - y).max(axis=(1, 2)) <= tol), np.abs(yk - y).max(axis=(1, 2)) / tol
    plan.close()
