"""The solver's digit contractions on their own (csrc/kernel_entries.cu): Grams
of four and seven digits and block updates.  The operands are integers (times
powers of two) whose results double precision holds, and whose digits below
the leading ones all count, so that every kept digit product shows.  (A
negative value is cut one unit too low; the integers are positive where the
results are compared closer than that.)"""
import ctypes

import numpy as np
import pytest

from gpu_util import need_torch_cuda

pytestmark = pytest.mark.gpu


def _lib():
    from paper_2506_08308_gb300 import bdg
    lib = bdg.load()
    vp, ll, i, d = ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int, ctypes.c_double
    lib.bdg_kernel_gram.argtypes = [i, i, vp, ll, i, vp, ll, i, ll, vp, vp]
    lib.bdg_kernel_update.argtypes = [vp, ll, i, vp, d, d, vp, ll, i, ll, vp]
    return lib


def _gram(torch, A, B, digits):
    G = torch.full((2 * A.shape[0], 2 * B.shape[0]), float("nan"), dtype=torch.float64, device="cuda")
    e = _lib().bdg_kernel_gram(int(A.dtype == torch.complex128), digits, A.data_ptr(), A.stride(0), A.shape[0],
                               B.data_ptr(), B.stride(0), B.shape[0], A.shape[1], G.data_ptr(),
                               torch.cuda.current_stream().cuda_stream)
    assert e == 0
    return G.cpu().numpy()


def _real_columns(X):
    """(2P, n) real columns of complex columns (P, n)."""
    return np.stack([X.real, X.imag], 1).reshape(2 * X.shape[0], -1)


def _complex_columns(R):
    return R[::2] + 1j * R[1::2]


SHAPES = [(1, 2, 8192), (2, 1, 8193), (9, 5, 8447), (20, 20, 8449), (65, 24, 8704), (24, 33, 9001), (40, 40, 12288),
          (64, 65, 8193)]


@pytest.mark.parametrize("digits,fp64", [(7, True), (4, True), (4, False)])
@pytest.mark.parametrize("P,Q,n", SHAPES)
def test_gram_keeps_every_digit(P, Q, n, digits, fp64):
    """In every 256 rows A has one value 2^54 (four digits: 2^29), where B is
    zero, and integers below 2^43 (2^18) against powers of two in B: they lie in
    the lower digits, down to the last bit of the last.  Seven digits: the eight
    weight sums of 256 rows are put together in units of four, at most two off,
    and added in FP64, exactly below 2^53 (four chunks hold values).  Four: all
    sums are integers that two floats hold."""
    torch = need_torch_cuda()
    rng = np.random.default_rng(P + 10 * Q + n)
    top, low, rows = (54, 43, 4 * 256) if digits == 7 else (29, 18, n)
    a = np.zeros((2 * P, n))
    a[:, :rows] = rng.integers(0, 1 << low, size=(2 * P, rows))
    big = np.arange(0, n, 256) + rng.integers(0, min(256, n % 256 or 256), size=(n + 255) // 256)
    a[:, big] = 2.0 ** top
    scale = 2.0 ** rng.integers(-8, 9, size=2 * Q)
    b = np.repeat(scale[:, None], n, 1)
    b[:, big] = 0.0
    dt = torch.complex128 if fp64 else torch.complex64
    A, B = (torch.from_numpy(_complex_columns(r)).to(dt).cuda() for r in (a, b))
    a[:, big] = 0.0
    want = a.sum(1)[:, None] * scale[None, :]
    tol = scale[None, :] * (8.0 if digits == 7 else 0.0)
    G, GT = _gram(torch, A, B, digits), _gram(torch, B, A, digits).T
    for g in (G, GT):
        assert np.all(np.abs(g - want) <= tol), np.max(np.abs(g - want) / scale)
    # powers of two that take the columns near the smallest normal number
    ka, kb = (-1000, 900) if fp64 else (-130, 100)
    Gk = _gram(torch, A * 2.0 ** (ka // 2) * 2.0 ** (ka - ka // 2), B * 2.0 ** kb, digits)
    assert np.array_equal(Gk, np.ldexp(G, ka + kb))


@pytest.mark.parametrize("digits,fp64", [(7, True), (4, True), (4, False)])
def test_gram_non_finite_columns(digits, fp64):
    torch = need_torch_cuda()
    dt = torch.complex128 if fp64 else torch.complex64
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn((70, 8500), dtype=dt, device="cuda", generator=g)
    B = torch.randn((30, 8500), dtype=dt, device="cuda", generator=g)
    ref = _gram(torch, A, B, digits)
    A[68, 8499] = complex(float("inf"), A[68, 8499].imag.item())
    B[7, 4000] = complex(B[7, 4000].real.item(), float("nan"))
    G = _gram(torch, A, B, digits)
    bad = np.zeros_like(G, dtype=bool)
    bad[136], bad[:, 15] = True, True
    assert np.array_equal(~np.isfinite(G), bad) and np.array_equal(G[~bad], ref[~bad])


@pytest.mark.parametrize("beta,alpha,signed", [(0.0, 1.0, False), (1.0, -1.0, False), (-2.0, 1.0, True)])
@pytest.mark.parametrize("P,Q,n", [(8, 4, 8192), (8, 8, 8193), (16, 9, 8319), (17, 16, 8320), (33, 20, 9000), (48, 24, 8193),
                                   (73, 25, 8319), (74, 32, 8447), (80, 26, 8192), (80, 32, 20001)])
def test_update_keeps_every_digit(P, Q, n, beta, alpha, signed):
    """Integers of up to 37 bits beside a column of 2^45 that meets coefficients
    of zero: rows are cut against the large column in units of 2^-9, the results
    (below 2^53) come from the lower digits, and nothing is rounded.  Negative
    values are one unit too low, in A (signed) 2^-9 at most, in C (alpha < 0)
    2^-47."""
    torch = need_torch_cuda()
    rng = np.random.default_rng(P + 10 * Q + n)
    top = (1 << 37) // (2 * P)
    a = rng.integers(-top if signed else 0, top, size=(2 * P, n)).astype(np.float64)
    big = int(rng.integers(0, 2 * P))
    a[big] = 2.0 ** 45
    a[big, ::3] = 0.0
    C = rng.integers(0, 256, size=(2 * P, 2 * Q)).astype(np.float64)
    C[big] = 0.0
    C[:, 2 * Q - 1] = 0.0
    y = rng.integers(-1000, 1001, size=(2 * Q, n)).astype(np.float64)
    want = alpha * (C.T @ a) + beta * y    # (every product and sum an integer below 2^53)
    tol = 0.0
    if signed:
        tol = np.where(C.any(0), 1.0 + 2.0 ** -9 * C.sum(0), 0.0)[:, None]
    if alpha < 0:   # (2^37 bounds the sum of a row; and a rounding of as much again)
        tol = 2.0 * 2.0 ** (37 - 47)
    for tiny in (False, True):   # powers of two on rows (down to 1e-301) and on all of C
        s, c = np.ones(n), 1.0
        if tiny:
            s[::7], s[1::7], c = 2.0 ** -1000, 2.0 ** -520, 2.0 ** 520
        A = torch.from_numpy(_complex_columns(a * s)).cuda()
        Ck, Y0, w = C * c, y * (s * c), want * (s * c)
        Y = torch.from_numpy(_complex_columns(Y0)).cuda()
        Y = torch.cat([Y, torch.full((1, n), 7.0, dtype=Y.dtype, device="cuda")])
        Cd = torch.from_numpy(Ck).cuda()
        e = _lib().bdg_kernel_update(A.data_ptr(), A.stride(0), P, Cd.data_ptr(), beta, alpha, Y.data_ptr(), n, Q, n,
                                     torch.cuda.current_stream().cuda_stream)
        assert e == 0
        Yh = Y.cpu().numpy()
        assert np.all(np.abs(_real_columns(Yh[:Q]) - w) <= tol * (s * c)), tiny
        assert np.all(Yh[Q] == 7.0)


def test_update_non_finite_rows_and_columns():
    torch = need_torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(2)
    A = torch.randn((24, 8200), dtype=torch.complex128, device="cuda", generator=g)
    C = torch.randn((48, 50), dtype=torch.float64, device="cuda", generator=g)

    def run():
        Y = torch.zeros((25, 8200), dtype=torch.complex128, device="cuda")
        assert _lib().bdg_kernel_update(A.data_ptr(), 8200, 24, C.data_ptr(), 0.0, 1.0, Y.data_ptr(), 8200, 25, 8200,
                                        torch.cuda.current_stream().cuda_stream) == 0
        return _real_columns(Y.cpu().numpy())

    ref = run()
    A[3, 17] = complex(float("nan"), 0.0)
    A[23, 8199] = complex(0.0, float("inf"))
    C[5, 31] = float("inf")
    got = run()
    bad = np.zeros_like(ref, dtype=bool)
    bad[:, [17, 8199]] = True
    bad[31] = True
    assert np.array_equal(~np.isfinite(got), bad) and np.array_equal(got[~bad], ref[~bad])
