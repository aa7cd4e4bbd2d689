"""FP64 Grams from exact integer digits (bdg_gram on C128 blocks of 8192 rows
and more) against the oracle's pair_gram: one and several column tiles, part
tiles, a last chunk of one row, columns whose size changes by many orders
within and between chunks, zero columns, and columns with a NaN or an
infinity."""
import numpy as np
import pytest

from gpu_util import need_torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,Q,n", [(1, 2, 8192), (2, 1, 8193), (9, 33, 8447), (24, 24, 9000), (65, 8, 8449),
                                   (40, 41, 10000), (73, 24, 8704), (72, 72, 12288)])
def test_gram_digits_against_oracle(P, Q, n):
    torch = need_torch_cuda()
    from oracle import lrep
    from paper_2506_08308_gb300 import bdg
    g = torch.Generator(device="cuda").manual_seed(P + 3 * Q + n)
    A = torch.randn((P, n), dtype=torch.complex128, device="cuda", generator=g)
    B = torch.randn((Q, n), dtype=torch.complex128, device="cuda", generator=g)
    r = torch.linspace(-20, 20, n, device="cuda", dtype=torch.float64)
    A *= torch.exp(-0.5 * r * r)          # 87 orders of magnitude, chunk after chunk
    A[::3] *= 1e-30
    B[::4] *= 1e20
    B[Q // 2] *= 1e-12 ** (torch.arange(n, device="cuda") % 2)   # alternating rows
    B[-1].imag.zero_()
    G = bdg.gram(A, B, engine=bdg.GRAM_SIMT).cpu().numpy()
    S, Sabs = lrep.pair_gram(A.cpu().numpy(), B.cpu().numpy())
    # an operand is off by at most 2^-47 of its chunk's largest value: about
    # 2 x 6 x 2^-47 of sum |a b| row by row, averaged over more than 8000 rows
    err = np.abs(G - S) / np.maximum(Sabs, 1e-300)
    assert err.max() < 1e-14, (err.max(), np.unravel_index(err.argmax(), err.shape))
    assert np.all(G[:, 2 * Q - 1] == 0)
    assert np.array_equal(G, bdg.gram(A, B, engine=bdg.GRAM_SIMT).cpu().numpy())


def test_gram_digits_non_finite_columns():
    torch = need_torch_cuda()
    from paper_2506_08308_gb300 import bdg
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn((5, 9001), dtype=torch.complex128, device="cuda", generator=g)
    B = torch.randn((30, 9001), dtype=torch.complex128, device="cuda", generator=g)
    ref = bdg.gram(A, B, engine=bdg.GRAM_SIMT)
    A[1, 9000] = complex(float("nan"), 1.0)
    B[7, 4000] = complex(1.0, float("inf"))
    G = bdg.gram(A, B, engine=bdg.GRAM_SIMT)
    bad = torch.zeros_like(G, dtype=torch.bool)
    bad[2], bad[:, 15] = True, True
    assert bool((~torch.isfinite(G) == bad).all())
    keep = ~bad
    keep[3] = keep[:, 14] = False          # the other parts of the changed elements
    assert torch.equal(G[keep], ref[keep])
