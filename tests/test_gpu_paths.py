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
