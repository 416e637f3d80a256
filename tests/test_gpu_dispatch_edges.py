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


@pytest.mark.parametrize("N,r,n", [(304, 70, 50), (305, 70, 50), (1000, 2100, 60), (2432, 33, 20), (2433, 33, 20)])
def test_pivoted_cholesky_threads_per_row(N, r, n):
    """A block, a warp or eight threads per row of the generator, against the
    oracle; its condition is that of a random matrix with 3/4 of its rank taken
    (remainders above 1e-2 of the diagonal), so FP64 sums of r terms agree to
    far below 1e-11."""
    from oracle import cholesky
    P = _gpu()
    rng = np.random.default_rng(N + r)
    B = rng.standard_normal((N, r)) + 1j * rng.standard_normal((N, r))
    n = min(n, 3 * r // 4)
    ref, piv_ref = cholesky.pivoted_cholesky(B, 0.0, max_vec=n)
    L, piv = P.cholesky_dev(torch.from_numpy(B).cuda(), 0.0, n)
    assert np.array_equal(piv, piv_ref)
    assert np.abs(L.cpu().numpy() - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("M,N,K,tier", [(20000, 41, 33, "fp16x3"), (40000, 100, 32, "fp16x3"), (9000, 9, 40, "fp16x3"),
                                        (60000, 9, 16, "fp16x3"), (2100, 1000, 40, "fp16x3"),
                                        (40000, 4, 8, "fp64"), (20000, 4, 16, "fp64"), (5000, 250, 2, "fp64")])
def test_short_k_products_whole_or_cut(M, N, K, tier):
    """The short side whole or cut over blocks: sums of 2 K products in FP32
    (2 K 2^-24) or FP64 (2 K 2^-53), against the sum of their magnitudes."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    cn = lambda *s: torch.view_as_complex(torch.randn(*s, 2, generator=g, device="cuda", dtype=torch.float64))
    A, B = cn(M, K), cn(N, K)
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, tier)
    tol = 8 * K * 2.0 ** (-53 if tier == "fp64" else -24) * (A.abs() @ B.abs().T)
    assert bool(((C - A @ B.T).abs() <= tol).all())
