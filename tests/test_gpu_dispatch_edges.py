"""Both sides of the sizes where a kernel variant is chosen."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_06805_gb300 as P
    P.lib()
    return P


@pytest.mark.parametrize("M,N,K", [(4, 4625, 8), (43, 431, 8), (37, 500, 8), (100, 185, 9), (36, 1029, 16),
                                   (370, 100, 16), (371, 100, 16), (740, 100, 31), (741, 100, 31)])
def test_fp64_products_of_8_to_31_terms(M, N, K):
    """A warp per output or 64 x 64 tiles. Both sides are FP64 sums of 2 K
    products: within 2 K 2^-53 of the sum of their magnitudes."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    cn = lambda *s: torch.view_as_complex(torch.randn(*s, 2, generator=g, device="cuda", dtype=torch.float64))
    A, B = cn(M, K), cn(N, K)
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    tol = 8 * K * 2.0 ** -53 * (A.abs() @ B.abs().T)
    assert bool(((C - A @ B.T).abs() <= tol).all())
