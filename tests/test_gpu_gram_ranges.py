"""FP64 Grams from integer digits (bdg_gram on C128 blocks of 8192 rows and
more) at the ends of their ranges."""
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
