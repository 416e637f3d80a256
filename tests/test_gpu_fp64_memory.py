"""FP64 work in as much memory as it takes without digit planes: the planes are
given up when an allocation fails, and when a cap is set."""
import numpy as np
import pytest

from paper_2506_06805_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_06805_gb300 as P
    P.lib()
    return P


class Pool:
    """Allocator callbacks over torch that refuse to hold more than a budget."""

    def __init__(self):
        self.held, self.used, self.peak, self.budget, self.refused = {}, 0, 0, None, 0

    def alloc(self, n, _user):
        if self.budget is not None and self.used + n > self.budget:
            self.refused += 1
            return None
        p = torch.cuda.caching_allocator_alloc(int(n), 0)
        self.held[p] = n
        self.used += n
        self.peak = max(self.peak, self.used)
        return p

    def free(self, p, _user):
        self.used -= self.held.pop(p)
        torch.cuda.caching_allocator_delete(p)


def _inputs(o, v):
    X = 4 * v
    eps, L = synth.make_system(o, v, X, seed=3)
    rng = np.random.default_rng(1)
    t2 = 0.01 * (rng.standard_normal((o, o, v, v)) + 1j * rng.standard_normal((o, o, v, v)))
    t2 = t2 - t2.transpose(1, 0, 2, 3)
    t2 = t2 - t2.transpose(0, 1, 3, 2)
    t1 = 0.01 * (rng.standard_normal((o, v)) + 1j * rng.standard_normal((o, v)))
    return eps, L, torch.from_numpy(t1).cuda(), torch.from_numpy(t2).cuda()


@pytest.mark.parametrize("call", ["ladder", "residual"])
@pytest.mark.parametrize("slab", [0, 8 << 20])
def test_fp64_work_fits_where_the_pipe_form_fits(call, slab):
    """A capped context (FP64 pipe, no planes) sets the budget; a context
    without a cap then has to do with as much, to the same result (FP64 sums of
    up to 5184 terms: 1e-12)."""
    P = _gpu()
    o, v = 10, 72
    eps, L, t1, t2 = _inputs(o, v)
    out = []
    budget = None
    for capped in (True, False):
        pool = Pool()
        with P.System(eps, L, n_occ=o, tier="fp64") as s:
            s.set_allocator(pool.alloc, pool.free)
            if slab:
                s.set_slab_budget(slab)
            s.dump_integrals(0)  # the stored integrals, before the budget counts
            if capped:
                s.set_memory_limit(1 << 36)
            base = pool.used
            pool.peak = base
            pool.budget = None if capped else base + budget
            r1, r2 = torch.zeros_like(t1), torch.zeros_like(t2)
            if call == "ladder":
                s.ladder_dev(t2, r2)
            else:
                s.residual_dev(t1, t2, r1, r2)
            torch.cuda.synchronize()
            if capped:
                budget = pool.peak - base
            else:
                assert pool.refused > 0 and pool.peak <= pool.budget
            out.append((r1, r2))
    for a, b in zip(*out):
        assert float((a - b).abs().max()) <= 1e-12 * float(a.abs().max() if a.abs().max() > 0 else 1.0)


def test_a_cap_gives_the_planes_back():
    """The planes do not count against a cap set after FP64 work: one byte
    above what the context held before it is accepted."""
    P = _gpu()
    o, v = 10, 72
    eps, L, t1, t2 = _inputs(o, v)
    with P.System(eps, L, n_occ=o, tier="fp64") as s:
        s.set_memory_limit(1 << 36)  # the work's other lasting buffers, first
        r1, r2 = torch.zeros_like(t1), torch.zeros_like(t2)
        s.residual_dev(t1, t2, r1, r2)
        s.set_memory_limit(0)
        held = int(s.stats()["device_bytes_held"])
        s.residual_dev(t1, t2, r1, r2)
        assert int(s.stats()["device_bytes_held"]) > held
        s.set_memory_limit(held + 1)
        assert int(s.stats()["device_bytes_held"]) <= held
