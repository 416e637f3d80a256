"""Kernel variants chosen by size, at the sizes where the choice or the edges
of a tile can go wrong, against the oracle or numpy."""
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


def _amps(rng, o, v, s=1e-2):
    t = s * (rng.standard_normal((o, o, v, v)) + 1j * rng.standard_normal((o, o, v, v)))
    t = t - t.transpose(1, 0, 2, 3)
    return t - t.transpose(0, 1, 3, 2)


# FP16 rounds both operands to 2^-11; FP16x3 and FP32 accumulation 2^-22 and up
LADDER_TOL = {"fp16": 4e-3, "fp16x3": 2e-6, "fp64": 1e-12}


@pytest.mark.parametrize("tier", ["fp16", "fp16x3", "fp64"])
@pytest.mark.parametrize("o,v,slab", [(2, 2, 0), (3, 3, 0), (4, 17, 0), (3, 33, 0),
                                      (3, 33, 8 * 33 ** 3), (4, 26, 5 * 8 * 26 ** 3)])
def test_ladder_row_ranges(tier, o, v, slab):
    """Slabs of every a, of one a and of a few, split into row ranges."""
    P = _gpu()
    X = 2 * v + 1
    eps, L = synth.make_system(o, v, X, seed=11)
    tau = _amps(np.random.default_rng(o * v), o, v)
    ref = ccsd.ladder_term(integrals.blocks_from_cholesky(L, o).vvvv, tau)
    out = torch.zeros((o, o, v, v), dtype=torch.complex128, device="cuda")
    with P.System(eps, L, n_occ=o, tier=tier) as s:
        if slab:
            s.set_slab_budget(slab)
        s.ladder_dev(torch.from_numpy(tau).cuda(), out)
    err = np.abs(out.cpu().numpy() - ref).max() / np.abs(ref).max()
    assert err <= LADDER_TOL[tier]


def _cn(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda", dtype=torch.float64))


def _rownorm(x):
    """Row 2-norms without under- or overflow."""
    top = x.abs().amax(1)
    scaled = torch.view_as_real(x).flatten(1) / torch.where(top == 0, 1.0, top)[:, None]
    return torch.linalg.vector_norm(scaled, dim=1) * top


def _check_product(A, B, C):
    """Both sides are FP64 sums of K terms: sqrt(K) 2^-52 of |a_m| |b_n|."""
    ref = A @ B.T
    tol = A.shape[1] ** 0.5 * 2.0 ** -52 * _rownorm(A)[:, None] * _rownorm(B)[None, :]
    assert bool(((C - ref).abs() <= tol).all())


@pytest.mark.parametrize("M,N,K", [(257, 129, 300), (129, 2000, 33), (64, 640, 1025), (5, 40000, 160),
                                   (700, 700, 64), (300, 130, 40000), (130, 130, 65537),
                                   (1200, 64, 65600), (64, 2500, 65600)])
def test_fp64_product_on_tensor_cores(M, N, K):
    """Ragged tiles, few rows, a split K, K in two blocks, and operands whose
    digit planes exceed the plane budget (the last two, blocked in M and N)."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, B = _cn(g, M, K), _cn(g, N, K)
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    _check_product(A, B, C)


def test_fp64_product_extreme_rows():
    """Rows of any scale (to the smallest denormals), zero rows, rows with one
    large element, and Inf / NaN, which the tensor-core form leaves to the
    FP64 kernel."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(3)
    M, N, K = 300, 260, 500
    A, B = _cn(g, M, K), _cn(g, N, K)
    A[1] = 0
    A[2] *= 1e-310
    A[3] *= 1e280
    B[3] *= 1e-280
    A[4] *= 1e150
    B[4] *= 1e150
    A[5, 7] *= 1e12
    B[6] = 0.5 + 0.5j
    A[6] = 1.0
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    ref = A @ B.T
    tol = K ** 0.5 * 2.0 ** -52 * _rownorm(A)[:, None] * _rownorm(B)[None, :]
    ok = (C - ref).abs() <= tol + 1e-321  # the products of row 2 are themselves denormal
    ok[3, 4] = not bool(torch.isfinite(C[3, 4]))  # 1e430
    assert bool(ok.all())
    assert bool((C[1] == 0).all())
    for bad in (float("inf"), float("nan")):
        A2 = A.clone()
        A2[10, 20] = bad
        P.zgemm_dev(A2, B, C, "fp64")
        keep = torch.arange(M, device="cuda") != 10
        ok = (C - ref).abs() <= tol + 1e-321
        ok[3, 4] = True
        assert bool(ok[keep].all())
        assert not bool(torch.isfinite(torch.view_as_real(C[10])).any(-1).any())


@pytest.mark.parametrize("o,v,X", [(6, 41, 163), (9, 30, 121), (17, 19, 60)])
def test_fp64_residual_and_sigma_on_tensor_cores(o, v, X):
    """Strided, conjugated, transposed and accumulating products of the FP64
    residual and sigma at sizes that take the tensor-core form."""
    from oracle import ipeom
    P = _gpu()
    eps, L = synth.make_system(o, v, X, seed=5)
    L = 4 * L
    rng = np.random.default_rng(2)
    t1 = 0.02 * (rng.standard_normal((o, v)) + 1j * rng.standard_normal((o, v)))
    t2 = _amps(rng, o, v)
    g = integrals.blocks_from_cholesky(L, o)
    R1, R2 = ccsd.residuals(g, eps, t1, t2)
    io, jo = np.triu_indices(o, 1)
    av, bv = np.triu_indices(v, 1)
    d1, d2 = torch.from_numpy(t1).cuda(), torch.from_numpy(t2).cuda()
    r1, r2 = torch.empty_like(d1), torch.empty_like(d2)
    with P.System(eps, L, n_occ=o, tier="fp64") as s:
        s.residual_dev(d1, d2, r1, r2)
        s.set_amplitudes(t1, t2[io, jo][:, av, bv])
        H = ipeom.hbar(g, eps, t1, t2)
        n = ipeom.dim(o, v)
        x = rng.standard_normal((7, n)) + 1j * rng.standard_normal((7, n))
        xd = torch.from_numpy(x).cuda()
        sd, ld = torch.empty_like(xd), torch.empty_like(xd)
        s.sigma_dev(xd, sd)
        s.left_sigma_dev(xd, ld)
    for got, ref in ((r1, R1), (r2, R2),
                     (sd, np.array([ipeom.sigma(H, x[k], o, v) for k in range(7)])),
                     (ld, np.array([ipeom.left_sigma(H, x[k], o, v) for k in range(7)]))):
        assert np.abs(got.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("M,N,K", [(1, 3000, 2), (100, 3200, 1), (250, 1025, 17), (200, 5000, 32),
                                   (1024, 7, 3), (90000, 9, 2)])
def test_fp64_short_k_products_cut_on_both_sides(M, N, K):
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, B = _cn(g, M, K), _cn(g, N, K)
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    _check_product(A, B, C)


@pytest.mark.parametrize("M,N,K", [(2048, 200, 16), (300, 2500, 20), (1000, 40000, 48), (8, 2048, 33)])
def test_fp32_short_k_products_cut_on_both_sides(M, N, K):
    """FP32 products and sums of 2 K terms: 2 K 2^-24 of |a_m| |b_n|."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A, B = _cn(g, M, K), _cn(g, N, K)
    C = torch.empty((M, N), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp16x3")
    tol = 2 * K * 2.0 ** -24 * _rownorm(A)[:, None] * _rownorm(B)[None, :]
    assert bool(((C - A @ B.T).abs() <= tol).all())


@pytest.mark.parametrize("N,r,n", [(1, 1, 1), (5, 3, 3), (33, 40, 33), (257, 2100, 40), (300000, 9, 9)])
def test_pivoted_cholesky_sizes(N, r, n):
    """Fewer rows than a block, more coefficients than shared memory holds,
    several passes per block."""
    from oracle import cholesky
    P = _gpu()
    rng = np.random.default_rng(N + r)
    B = rng.standard_normal((N, r)) + 1j * rng.standard_normal((N, r))
    ref, piv_ref = cholesky.pivoted_cholesky(B, 0.0, max_vec=n)
    L, piv = P.cholesky_dev(torch.from_numpy(B).cuda(), 0.0, n)
    # the last vectors of a full-rank run stand on small remainders
    m = min(n, max(1, 3 * min(N, r) // 4))
    assert np.array_equal(piv[:m], piv_ref[:m])
    assert np.abs(L.cpu().numpy()[:m] - ref[:m]).max() <= 1e-11 * np.abs(ref).max()
    if n > m:
        Lh = L.cpu().numpy()
        if len(Lh) == min(N, r):
            M = B @ B.conj().T if N <= 1000 else None
            if M is not None:
                assert np.abs(M - Lh.T @ Lh.conj()).max() <= 1e-10 * np.abs(M).max()


def test_pivoted_cholesky_beyond_the_rank_and_non_finite():
    P = _gpu()
    rng = np.random.default_rng(4)
    B = rng.standard_normal((500, 12)) + 1j * rng.standard_normal((500, 12))
    L, piv = P.cholesky_dev(torch.from_numpy(B).cuda(), 0.0, 80)  # tau 0: rounding remainders only
    Lh = L.cpu().numpy()
    assert len(piv) >= 12 and np.abs(Lh[12:]).max(initial=0.0) <= 1e-5 * np.abs(Lh).max()
    M = B @ B.conj().T
    assert np.abs(M - Lh.T @ Lh.conj()).max() <= 1e-11 * np.abs(M).max()
    B[7, 3] = np.inf
    with pytest.raises(P.CCError) as e:
        P.cholesky_dev(torch.from_numpy(B).cuda(), 0.0, 8)
    assert e.value.code == -6  # CC_ERR_NUMERIC


@pytest.mark.parametrize("n,K", [(1, 5000), (1, 129), (320, 12001), (2432, 1024), (2431, 1023),
                                 (9729, 131), (12000, 300)])
@pytest.mark.parametrize("side", ["row", "column"])
def test_fp64_matrix_vector(n, K, side):
    """A block, a warp or a quarter of a warp per output, with remainders."""
    P = _gpu()
    g = torch.Generator(device="cuda").manual_seed(n + K)
    V, x = _cn(g, n, K), _cn(g, 1, K)
    A, B = (x, V) if side == "row" else (V, x)
    C = torch.empty((A.shape[0], B.shape[0]), dtype=torch.complex128, device="cuda")
    P.zgemm_dev(A, B, C, "fp64")
    _check_product(A, B, C)


def test_fp64_solve_on_tensor_cores_with_and_without_graphs():
    """The captured sigma replays the digit-plane products (their planes are
    part of the graph's key); FP64 to the last steps of the Davidson."""
    P = _gpu()
    eps, L = synth.make_system(9, 41, 163, seed=8)
    roots = []
    for graphs in (True, False):
        with P.System(eps, 3 * L, n_occ=9, tier="fp64", eom_tier="fp64") as s:
            s.set_graphs(graphs)
            s.ccsd(tol=1e-10)
            roots.append(s.ipeom(4, tol=1e-9)[0])
    assert np.abs(np.sort_complex(roots[0]) - np.sort_complex(roots[1])).max() <= 1e-10
