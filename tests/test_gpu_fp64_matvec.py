"""FP64 matrix-vector products: a lane's sums run over few terms."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", ["row", "column"])
@pytest.mark.parametrize("n,K", [(64, 300), (320, 12000), (1823, 4559), (1824, 4560), (3000, 4000), (9728, 20000), (12001, 4097), (20000, 513)])
def test_fp64_matrix_vector_sums_are_short(n, K, side):
    """One term of 2^53 before K - 1 terms of 1: a sum that holds the large one
    loses every 1 that follows it (a tie, to even). A lane keeps four sums, so
    at most K / 128 are lost, and each of the ten additions that join the four
    sums, the lanes and the warps rounds off at most 1."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_06805_gb300 as P
    P.lib()
    V = torch.ones((n, K), dtype=torch.complex128, device="cuda")
    V[:, 0] = 2.0 ** 53
    x = torch.ones((1, K), dtype=torch.complex128, device="cuda")
    A, B = (x, V) if side == "row" else (V, x)
    C = torch.empty((A.shape[0], B.shape[0]), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    lost = (K - 1) - (C.real - 2.0 ** 53)
    assert bool((lost.abs() <= K / 128 + 10).all())
    assert bool((C.imag == 0).all())
