"""FP64 products whose rows' largest elements do not meet: every element to
FP64's accuracy against the sum of its own terms' magnitudes,
S = sum_k |a_k| |b_k| (real and imaginary part apart), not only against the
rows' norms. On both sides of the sizes that take the tensor cores."""
import numpy as np
import pytest

from oracle import ccsd, integrals
from paper_2506_06805_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_06805_gb300 as P
    P.lib()
    return P


def _cn(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float64))


def _check(P, A, B):
    """An FP64 sum of 2 K products is within 2 K 2^-53 S of the exact one,
    whatever its order; here and in the reference."""
    C = torch.empty((A.shape[0], B.shape[0]), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    ref = torch.complex(A.real @ B.real.T - A.imag @ B.imag.T, A.real @ B.imag.T + A.imag @ B.real.T)
    ar, ai, br, bi = (x.abs() for x in (A.real, A.imag, B.real, B.imag))
    tol = 4.0 * A.shape[1] * 2.0 ** -53
    assert bool(((C - ref).real.abs() <= tol * (ar @ br.T + ai @ bi.T)).all())
    assert bool(((C - ref).imag.abs() <= tol * (ar @ bi.T + ai @ br.T)).all())
    return C


SIZES = [(300, 260, 500), (700, 650, 64), (64, 640, 1025), (129, 2000, 40), (5, 40000, 160),
         (130, 97, 20000), (40, 30, 50)]


@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("d", [0, 2, 3, 4, 8, 12, 20])
def test_columns_scaled_oppositely(M, N, K, d):
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    s = 10.0 ** (-d * torch.arange(K, device="cuda", dtype=torch.float64) / K)
    _check(P, _cn(g, M, K) * s, _cn(g, N, K) / s)


@pytest.mark.parametrize("M,N,K", SIZES)
@pytest.mark.parametrize("kind", ["sparse", "small imaginary", "spikes", "one pair", "log-normal"])
def test_structured_operands(M, N, K, kind):
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M * N + K)
    A, B = _cn(g, M, K), _cn(g, N, K)
    if kind == "sparse":
        A *= torch.rand(M, K, generator=g, device="cuda") < 0.05
        B *= torch.rand(N, K, generator=g, device="cuda") < 0.05
    elif kind == "small imaginary":
        A, B = torch.complex(A.real, 1e-11 * A.imag), torch.complex(B.real, 1e-13 * B.imag)
    elif kind == "spikes":  # single large elements in some rows and some columns
        A[::7, K // 3] *= 1e12
        A[:, K // 2] *= 1e7
        B[::5, K // 4] *= 1e9
    elif kind == "one pair":  # 1 beside 1e20, met by 1 beside 0: S is 1e-20 of the rows' product
        A[2, :], B[3, :] = 0, 0
        A[2, 0], A[2, 1], B[3, 1] = 1e20, 1.0, 1.0
        B[4, 1] = 1e-20
    else:
        A *= torch.exp(3 * torch.randn(M, K, generator=g, device="cuda", dtype=torch.float64))
        B *= torch.exp(3 * torch.randn(N, K, generator=g, device="cuda", dtype=torch.float64))
    C = _check(P, A, B)
    if kind == "one pair":
        assert C[2, 3].item() == 1.0


def test_long_even_rows():
    """Rows of one magnitude and 20000 terms (part of the sums in FP32), whose
    halves are then scaled oppositely, unsplit in K."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(7)
    M, N, K = 1600, 1300, 20000
    for f in (1.0, 1e-2, 1e-5):
        A, B = _cn(g, M, K), _cn(g, N, K)
        A /= A.abs()
        B /= B.abs()
        A[:, K // 2:] *= f
        B[:, :K // 2] *= f
        _check(P, A, B)


@pytest.mark.parametrize("o,v,X", [(6, 41, 163), (17, 19, 60)])
def test_residual_with_graded_virtuals(o, v, X):
    """Strided, conjugated, transposed and accumulating products: vectors that
    fall by 10^8 along the virtuals and amplitudes that rise by as much. Each
    (a, b) block of the residual against its own size, for a context that may
    use the tensor cores and for one that may not (a memory limit); the oracle
    sums up to 1e4 terms in FP64, 1e-12, of which the blocks keep 1e-2."""
    P = _gpu()
    eps, L = synth.make_system(o, v, X, seed=5)
    s = np.concatenate([np.ones(o), 10.0 ** (-8.0 * np.arange(v) / v)])
    L = 4 * L * s[:, None] * s[None, :]
    rng = np.random.default_rng(2)
    t1 = 0.02 * (rng.standard_normal((o, v)) + 1j * rng.standard_normal((o, v))) / s[o:]
    t2 = 0.01 * (rng.standard_normal((o, o, v, v)) + 1j * rng.standard_normal((o, o, v, v)))
    t2 = t2 - t2.transpose(1, 0, 2, 3)
    t2 = (t2 - t2.transpose(0, 1, 3, 2)) / s[o:][:, None] / s[o:]
    R1, R2 = ccsd.residuals(integrals.blocks_from_cholesky(L, o), eps, t1, t2)
    d1, d2 = torch.from_numpy(t1).cuda(), torch.from_numpy(t2).cuda()
    for limit in (0, 1 << 36):
        r1, r2 = torch.empty_like(d1), torch.empty_like(d2)
        with P.System(eps, L, n_occ=o, tier="fp64") as c:
            if limit:
                c.set_memory_limit(limit)
            c.residual_dev(d1, d2, r1, r2)
        assert (np.abs(r1.cpu().numpy() - R1) <= 1e-10 * np.abs(R1).max(0)).all()
        diag = np.eye(v, dtype=bool)  # a = b: zero
        err = np.abs(r2.cpu().numpy() - R2).max((0, 1))
        assert (err <= 1e-10 * np.abs(R2).max((0, 1)))[~diag].all()
