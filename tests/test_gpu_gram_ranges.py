"""FP64 Grams from integer digits (bdg_gram on C128 blocks of 8192 rows and
more) at the ends of their ranges."""
import ctypes

import numpy as np
import pytest

from gpu_util import need_torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,Q,n", [(2, 3, 8192), (9, 33, 8447), (24, 24, 12288)])
def test_columns_of_very_small_values(P, Q, n):
    """Powers of two on a block go to the result unchanged, also where they
    take its columns near the smallest normal number, with zeros in them."""
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    g = torch.Generator(device="cuda").manual_seed(P + Q)
    A = torch.randn((P, n), dtype=torch.complex128, device="cuda", generator=g)
    B = torch.randn((Q, n), dtype=torch.complex128, device="cuda", generator=g)
    A[:, ::3] = 0.0
    B[:, 1::5] = 0.0
    G = bdg.gram(A, B, engine=bdg.GRAM_SIMT).cpu().numpy()
    for ka, kb in ((-1000, 900), (900, -1005), (-990, 0)):
        Gk = bdg.gram(A * 2.0 ** (ka // 2) * 2.0 ** (ka - ka // 2), B * 2.0 ** (kb // 2) * 2.0 ** (kb - kb // 2),
                      engine=bdg.GRAM_SIMT).cpu().numpy()
        assert np.array_equal(np.ldexp(Gk, -(ka + kb)), G), (ka, kb)


def _apart(rng, n, kind):
    """(A, B) whose products of columns have sums |a b| from |a| |b| down to 0."""
    x = np.linspace(-12.0, 12.0, 256, endpoint=False)
    line = np.arange(n) % 256
    if kind == "gaussians":      # unit Gaussians at distances of 0 to 8 on every line
        g = np.stack([np.exp(-0.5 * (x - c) ** 2)[line] for c in (-4.0, -3.0, 0.0, 3.0, 4.0)])
        a = np.concatenate([g, g[::-1]])
        b = np.concatenate([g[1:], g[:2]])
    elif kind == "rows":         # large values on even rows, on odd rows, on all
        s = np.stack([np.where(np.arange(n) % 2 == k, 1.0, f) for k in (0, 1) for f in (0.0, 1e-9, 1e-3)])
        a, b = np.concatenate([s, s[:2] * 0 + 1]), s
    else:                        # one large value per 256 rows, elsewhere in A than in B
        a, b = np.full((8, n), 1e-6), np.full((10, n), 1e-5)
        for c in range(8):
            a[c, c::256] = 1.0
        for c in range(10):
            b[c, 40 + 5 * c::256] = 1.0
        b[8:, 1::256] = 1.0
    a = a * rng.standard_normal(a.shape) * 10.0 ** rng.integers(-3, 4, size=(a.shape[0], 1))
    b = b * rng.standard_normal(b.shape)
    return a[::2] + 1j * a[1::2], b[::2] + 1j * b[1::2]


@pytest.mark.parametrize("kind", ["gaussians", "rows", "peaks"])
@pytest.mark.parametrize("n", [8192, 16384 + 37])
def test_columns_whose_large_parts_lie_apart(kind, n):
    """The error stays relative to sum |a b| where that is far below |a| |b|,
    down to exact zeros: 2^-46, of double-float products (2^-48 for the operands'
    rounding and for the product of the low parts left out, 2^-47 for the sum of
    the cross terms; sums of these columns have few terms or even out)."""
    torch = need_torch_cuda()
    from oracle import lrep
    from paper_2506_08308_gb300 import bdg
    A, B = _apart(np.random.default_rng(n), n, kind)
    if kind == "gaussians":      # (tiles with nothing to form again as well)
        A = np.concatenate([A, np.random.default_rng(1).standard_normal((70, n)) + 0j])
    S, Sabs = lrep.pair_gram(A, B)

    def public(A, B):
        return bdg.gram(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), engine=bdg.GRAM_SIMT).cpu().numpy()

    def checked(A, B):   # by digits whatever the public call's rule says
        A, B = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
        G = torch.empty((2 * A.shape[0], 2 * B.shape[0]), dtype=torch.float64, device="cuda")
        f = bdg.load().bdg_kernel_gram
        i, p, q = ctypes.c_int, ctypes.c_void_p, ctypes.c_longlong
        f.argtypes = [i, i, p, q, i, p, q, i, q, p, p]
        assert f(1, -7, A.data_ptr(), n, A.shape[0], B.data_ptr(), n, B.shape[0], n, G.data_ptr(),
                 torch.cuda.current_stream().cuda_stream) == 0
        return G.cpu().numpy()

    bad = A.copy()
    bad[0, 5] = complex(np.nan, 0.0)
    for gram in (public, checked):
        G = gram(A, B)
        assert np.all(G[Sabs == 0] == 0.0)
        err = np.abs(G - S)[Sabs > 0] / Sabs[Sabs > 0]
        assert err.max() < 2.0 ** -46, (gram.__name__, err.max())
        G2 = gram(bad, B)
        assert not np.isfinite(G2[0]).any() and np.array_equal(G2[2:], G[2:])
