"""Performance cases: the calls a user of this framework makes, over the sizes
they are made at.

The sizes are those of ``synth.CONFIGS`` (tiny, mid, small, medium), of the
uneven batch (n_occ 20-50, n_virt 150-400, n_aux = 4 n_virt) and of the
natural-spinor and Cholesky benchmarks of ``kernel_bench``, with ragged ones
between them. ``listed`` holds the named cases, ``draw`` more of the same
ranges, ``prepare`` what a user's program has in hand before the call (on the
GPU), ``run`` the call, ``work`` its minimal traffic and operations and
``exact`` its value in 64 bits from plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_06805_gb300 as cd
from paper_2506_06805_gb300 import synth


def listed():
    return [
        # One CCSD iteration's residual in the default tier (FP64) at the
        # smallest configuration: launches and latency.
        {"name": "residual-tiny-fp64", "kind": "residual", "tier": "fp64", "o": 10, "v": 30, "X": 120},
        # The same in an ordinary system whose amplitudes are wanted in FP64.
        {"name": "residual-mid-fp64", "kind": "residual", "tier": "fp64", "o": 12, "v": 72, "X": 288},
        # The particle-particle ladder alone in FP64, ragged in every extent.
        {"name": "ladder-ragged-fp64", "kind": "ladder", "tier": "fp64", "o": 15, "v": 131, "X": 517},
        # A CCSD iteration in the tier the benchmark runs CCSD in: small and
        # medium configurations (the latter is the time-to-roots workload).
        {"name": "residual-small-fp16", "kind": "residual", "tier": "fp16", "o": 20, "v": 160, "X": 640},
        {"name": "residual-medium-fp16", "kind": "residual", "tier": "fp16", "o": 40, "v": 300, "X": 1200},
        # The ladder in the split tier (a CCSD that escalated, or one asked
        # for FP32-like accuracy), a member of the uneven batch.
        {"name": "ladder-ragged-fp16x3", "kind": "ladder", "tier": "fp16x3", "o": 23, "v": 187, "X": 748},
        # The Davidson's sigma build of the time-to-roots workload: 8 roots.
        {"name": "sigma-medium-fp16x3", "kind": "sigma", "tier": "fp16x3", "o": 40, "v": 300, "X": 1200, "k": 8},
        # Left vectors of a small system, an odd number of them (some roots
        # have converged).
        {"name": "left-sigma-small-fp16x3", "kind": "left_sigma", "tier": "fp16x3", "o": 20, "v": 160, "X": 640, "k": 5},
        # The complex product by itself, default tier.
        {"name": "zgemm-fp64", "kind": "zgemm", "tier": "fp64", "M": 1536, "N": 1000, "K": 1200},
        # Setting a system up from device-resident Cholesky vectors and
        # truncating it to frozen natural spinors (default tier).
        {"name": "fns-fp64", "kind": "fns", "tier": "fp64", "o": 18, "v": 150, "X": 450, "keep": 60},
        # Pivoted Cholesky decomposition of a pair matrix.
        {"name": "cholesky", "kind": "cholesky", "N": 43681, "r": 320, "n": 240},
        # A whole calculation on resident vectors: CCSD from the MP2 start,
        # H-bar and the Davidson for 8 roots, in the benchmark's tiers.
        {"name": "solve-small", "kind": "solve", "tier": "fp16", "o": 20, "v": 160, "X": 640, "roots": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual64", "residual16", "ladder64", "ladder16", "sigma", "left_sigma",
                       "zgemm", "fns", "cholesky", "solve"])
    if kind == "residual64":
        v = _log(rng, 30, 120)
        return {"kind": "residual", "tier": "fp64", "o": rng.randint(8, 16), "v": v, "X": 4 * v + rng.randint(0, 7)}
    if kind == "residual16":
        v = _log(rng, 100, 260)
        return {"kind": "residual", "tier": rng.choice(["fp16", "fp16", "fp16x3", "tf32"]),
                "o": rng.randint(14, 36), "v": v, "X": 4 * v}
    if kind == "ladder64":
        v = _log(rng, 40, 131)
        return {"kind": "ladder", "tier": "fp64", "o": rng.randint(8, 20), "v": v, "X": 4 * v + rng.randint(0, 9)}
    if kind == "ladder16":
        v = _log(rng, 120, 280)
        return {"kind": "ladder", "tier": rng.choice(["fp16", "fp16x3"]), "o": rng.randint(14, 36), "v": v, "X": 4 * v}
    if kind in ("sigma", "left_sigma"):
        v = _log(rng, 90, 260)
        return {"kind": kind, "tier": "fp16x3", "o": rng.randint(12, 36), "v": v, "X": 4 * v, "k": rng.randint(1, 12)}
    if kind == "zgemm":
        return {"kind": "zgemm", "tier": rng.choice(["fp64", "fp64", "fp16x3", "fp16"]),
                "M": _log(rng, 100, 4000), "N": _log(rng, 100, 2000), "K": _log(rng, 100, 2500)}
    if kind == "fns":
        v = _log(rng, 60, 180)
        return {"kind": "fns", "tier": "fp64", "o": rng.randint(8, 20), "v": v, "X": 3 * v, "keep": max(2, int(0.4 * v))}
    if kind == "cholesky":
        r = rng.randint(100, 320)
        return {"kind": "cholesky", "N": _log(rng, 5000, 60000), "r": r, "n": int(0.75 * r)}
    v = _log(rng, 60, 160)
    return {"kind": "solve", "tier": "fp16", "o": rng.randint(10, 22), "v": v, "X": 4 * v, "roots": rng.randint(2, 8)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
DEV = "cuda"


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(7919 * int(seed) + stream)
    return g


def _cnormal(shape, g):
    x = torch.randn(*shape, 2, generator=g, device=DEV, dtype=torch.float64)
    return torch.view_as_complex(x)


def _vectors(case, seed):
    """Orbital energies (host) and Cholesky vectors (device)."""
    o, v, X = case["o"], case["v"], case["X"]
    eps = synth.make_eps(np.random.default_rng(seed), o, v)
    return eps, synth.cholesky_chunks_device(seed + 1, o + v, X, 0, X, device=DEV)


def _system(case, eps, L):
    s = cd.System(eps, None, n_occ=case["o"], n_aux=case["X"], tier=case["tier"],
                  eom_tier="fp16x3" if case["tier"] == "fp16" else None)
    s.add_cholesky(0, case["X"], L)
    return s


def _packed_t2(case, eps, seed):
    """Amplitudes of first-order size over unique pairs: random integrals of
    the magnitude the vectors give, over the orbital-energy denominators."""
    o, v, X = case["o"], case["v"], case["X"]
    e = torch.from_numpy(eps).to(DEV)
    io, jo = torch.triu_indices(o, o, 1, device=DEV)
    av, bv = torch.triu_indices(v, v, 1, device=DEV)
    d = (e[io] + e[jo])[:, None] - (e[o + av] + e[o + bv])[None, :]
    g = _cnormal((len(io), len(av)), _gen(seed, 3)) * (synth.L_SCALE ** 2 / math.sqrt(4.0 * X))
    return g / d, io, jo, av, bv


def _amplitudes(case, eps, seed):
    """t1 [o][v] and the full antisymmetric t2 [o][o][v][v]."""
    o, v = case["o"], case["v"]
    u, io, jo, av, bv = _packed_t2(case, eps, seed)
    t2 = torch.zeros((o, o, v, v), dtype=torch.complex128, device=DEV)
    half = torch.zeros((len(io), v, v), dtype=torch.complex128, device=DEV)
    half[:, av, bv] = u
    half -= half.transpose(1, 2).clone()
    t2[io, jo] = half
    t2[jo, io] = -half
    t1 = _cnormal((o, v), _gen(seed, 4)) * 1e-4
    return t1, t2


def _ip_vectors(case, seed):
    """Davidson vectors: a leading 1h part and a small 2h1p part, unit norm."""
    o, v, k = case["o"], case["v"], case["k"]
    dim = o + o * (o - 1) // 2 * v
    r = _cnormal((k, dim), _gen(seed, 5))
    r[:, o:] *= 0.3 * math.sqrt(o / (dim - o))
    return r / torch.linalg.vector_norm(r, dim=1, keepdim=True)


def _generator(case, seed):
    """Generator of a pair matrix whose spectrum decays over five decades."""
    B = _cnormal((case["N"], case["r"]), _gen(seed, 6))
    return (B * torch.logspace(0, -2.5, case["r"], device=DEV, dtype=torch.float64)).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind == "zgemm":
        st["A"] = _cnormal((case["M"], case["K"]), _gen(seed, 1))
        st["B"] = _cnormal((case["N"], case["K"]), _gen(seed, 2))
        st["C"] = torch.empty((case["M"], case["N"]), dtype=torch.complex128, device=DEV)
        return st
    if kind == "cholesky":
        st["B"] = _generator(case, seed)
        return st
    eps, L = _vectors(case, seed)
    st["eps"] = eps
    if kind == "fns":
        st["L"] = L
        return st
    st["sys"] = s = _system(case, eps, L)
    del L
    if kind == "solve":
        return st
    t1, t2 = _amplitudes(case, eps, seed)
    if kind == "ladder":
        st["tau"], st["out"] = t2, torch.empty_like(t2)
    elif kind == "residual":
        st["t1"], st["t2"] = t1, t2
        st["r1"], st["r2"] = torch.empty_like(t1), torch.empty_like(t2)
    else:  # sigma, left_sigma: amplitudes and H-bar in hand, as in the Davidson
        u = _packed_t2(case, eps, seed)[0]
        del t2
        s.set_amplitudes(t1.cpu().numpy(), u.cpu().numpy())
        st["r"] = _ip_vectors(case, seed)
        st["s"] = torch.empty_like(st["r"])
        (s.sigma_dev if kind == "sigma" else s.left_sigma_dev)(st["r"], st["s"])
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "zgemm":
        cd.zgemm_dev(st["A"], st["B"], st["C"], c["tier"])
        return st["C"]
    if kind == "cholesky":
        L, piv = cd.cholesky_dev(st["B"], 0.0, c["n"])
        return {"L": L, "piv": piv}
    if kind == "fns":
        s = _system(c, st["eps"], st["L"])
        kept = s.fns_truncate(n_keep=c["keep"])
        out = {"kept": kept, "occ": s.fns_occupations(c["v"])}
        s.close()
        return out
    s = st["sys"]
    if kind == "ladder":
        s.ladder_dev(st["tau"], st["out"])
        return st["out"]
    if kind == "residual":
        s.residual_dev(st["t1"], st["t2"], st["r1"], st["r2"])
        return {"r1": st["r1"], "r2": st["r2"]}
    if kind == "sigma":
        s.sigma_dev(st["r"], st["s"])
        return st["s"]
    if kind == "left_sigma":
        s.left_sigma_dev(st["r"], st["s"])
        return st["s"]
    s.reset_amplitudes()
    e = s.ccsd(tol=1e-8)
    w, r1w = s.ipeom(c["roots"], tol=1e-7)
    return {"e": np.array([e]), "w": w, "r1w": r1w}


def work(case):
    """Operations: 8 per complex multiply-add, with the permutational
    symmetry of the pair indices used in the ladder; bytes: each input read
    once, each output written once."""
    kind = case["kind"]
    z = 16.0
    if kind == "zgemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": z * (M * K + N * K + M * N), "flops": 8.0 * M * N * K}
    if kind == "cholesky":
        # each vector is a new combination of the generator's r columns
        N, r, n = case["N"], case["r"], case["n"]
        return {"bytes": z * N * (r + n), "flops": 8.0 * N * r * n}
    o, v, X = case["o"], case["v"], case["X"]
    nab, nij, n2 = v * (v - 1) / 2, o * (o - 1) / 2, float(o) * o * v * v
    ladder = 8.0 * (X * v ** 3 * (v - 1) / 2 + nab * nab * nij)
    if kind == "ladder":
        return {"bytes": z * (X * v * v + 2 * n2), "flops": ladder}
    rest = 8.0 * (2.0 * o ** 3 * v ** 3           # ring and its intermediate
                  + 2.0 * o ** 4 * v * v          # hole ladder
                  + 4.0 * X * o * o * v * v)      # integrals times t1 through L
    lvec = z * X * (o + v) ** 2
    if kind == "residual":
        return {"bytes": lvec + z * 2 * n2, "flops": ladder + rest}
    if kind in ("sigma", "left_sigma"):
        k = case["k"]
        dim = o + nij * v
        return {"bytes": z * (3 * n2 + 2 * o ** 3 * v + 2 * k * dim),
                "flops": 8.0 * k * (o ** 3 * v * v + o ** 4 * v + o * o * v * v + o ** 3 * v)}
    if kind == "fns":
        nk = case["keep"]
        return {"bytes": 2 * lvec, "flops": 8.0 * (X * n2 / 2 + n2 * v / 2 + X * v * v * nk + X * v * nk * nk)}
    it = 5  # CCSD iterations such a system takes; four sigma builds of the block
    sig = 8.0 * case["roots"] * (o ** 3 * v * v + o ** 4 * v)
    return {"bytes": it * (lvec + z * 4 * n2), "flops": it * (ladder + rest) + 4 * sig}


# ---------------------------------------------------------------------------
# the same values in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _blocks(L, o):
    d = {"oo": L[:, :o, :o], "ov": L[:, :o, o:], "vo": L[:, o:, :o], "vv": L[:, o:, o:]}
    g = {}
    g["oooo"] = torch.einsum("pmi,pnj->mnij", d["oo"], d["oo"])
    g["oooo"] = g["oooo"] - g["oooo"].transpose(2, 3)
    g["ooov"] = torch.einsum("pmi,pne->mnie", d["oo"], d["ov"]) - torch.einsum("pme,pni->mnie", d["ov"], d["oo"])
    x = torch.einsum("pia,pjb->ijab", d["ov"], d["ov"])
    g["oovv"] = x - x.transpose(2, 3)
    g["ovvo"] = torch.einsum("pme,pbj->mbej", d["ov"], d["vo"]) - torch.einsum("pmj,pbe->mbej", d["oo"], d["vv"])
    return d, g


def _ladder64(lvv, tau):
    """1/2 sum_cd <ab||cd> tau_ij^cd, a row block at a time; tau is
    antisymmetric, so the direct part alone counts twice."""
    X, v, _ = lvv.shape
    o = tau.shape[0]
    out = torch.empty_like(tau)
    lt = lvv.permute(0, 2, 1).reshape(X, v * v)  # [P][(d, b)]
    for a in range(v):
        w = (lvv[:, a, :].T @ lt).reshape(v * v, v)  # [(c, d)][b] = sum_P L_ac L_bd
        out[:, :, a, :] = (tau.reshape(o * o, v * v) @ w).reshape(o, o, v)
    return out


def _pij(x):
    return x - x.transpose(0, 1)


def _pab(x):
    return x - x.transpose(2, 3)


def _asym(t1):
    x = torch.einsum("ia,jb->ijab", t1, t1)
    return x - x.transpose(2, 3)


def _f_terms(d, g, t1, half_tau):
    c = torch.einsum("mf,pmf->p", t1, d["ov"])
    y = torch.einsum("paf,mf->pam", d["vv"], t1)
    fae = torch.einsum("p,pae->ae", c, d["vv"]) - torch.einsum("pme,pam->ae", d["ov"], y) \
        - 0.5 * torch.einsum("mnaf,mnef->ae", half_tau, g["oovv"])
    fmi = torch.einsum("ne,mnie->mi", t1, g["ooov"]) + 0.5 * torch.einsum("inef,mnef->mi", half_tau, g["oovv"])
    fme = torch.einsum("nf,mnef->me", t1, g["oovv"])
    return fae, fmi, fme, y


def _residual64(case, eps, L, t1, t2):
    """Right-hand sides of the CCSD singles and doubles equations."""
    o = case["o"]
    d, g = _blocks(L, o)
    x = _asym(t1)
    tau, half = t2 + x, t2 + 0.5 * x
    fae, fmi, fme, y = _f_terms(d, g, t1, half)
    r1 = t1 @ fae.T - (fmi.T @ t1) + torch.einsum("imae,me->ia", t2, fme) \
        + torch.einsum("nf,nafi->ia", t1, g["ovvo"]) + 0.5 * torch.einsum("mnae,nmie->ia", t2, g["ooov"])
    q = torch.einsum("imef,pme->pif", t2, d["ov"])
    r1 = r1 - torch.einsum("paf,pif->ia", d["vv"], q)
    r2 = g["oovv"].conj().clone()
    fbe = fae - 0.5 * torch.einsum("mb,me->be", t1, fme)
    fmj = fmi + 0.5 * torch.einsum("je,me->mj", t1, fme)
    r2 += _pab(torch.einsum("ijae,be->ijab", t2, fbe))
    r2 -= _pij(torch.einsum("imab,mj->ijab", t2, fmj))
    u = torch.einsum("je,mnie->mnij", t1, g["ooov"])
    w4 = g["oooo"] + u - u.transpose(2, 3) + 0.5 * torch.einsum("ijef,mnef->mnij", tau, g["oovv"])
    # 1/4 tau <mn||ef> tau is counted once here and left out of the ladder
    r2 += 0.5 * torch.einsum("mnab,mnij->ijab", tau, w4)
    # particle ladder over <ab||cd> - P(ab) t_m^b <am||ef>
    bare = _ladder64(d["vv"], tau)
    amij = torch.empty((o, o, case["v"], o), dtype=t2.dtype, device=t2.device)
    for i in range(o):
        z = torch.einsum("jef,pme->jpmf", tau[i], d["ov"])
        amij[i] = torch.einsum("jpmf,paf->jam", z, d["vv"])
    # sum_ef (ae|mf) tau_ij^ef = -sum_ef (af|me) tau_ij^ef
    r2 += bare + _pab(torch.einsum("ijam,mb->ijab", amij, t1))
    zz = 0.5 * t2 + torch.einsum("jf,nb->jnfb", t1, t1)
    wm = g["ovvo"] + torch.einsum("pme,pbj->mbej", d["ov"], y) \
        - torch.einsum("pmj,pbe->mbej", torch.einsum("pmf,jf->pmj", d["ov"], t1), d["vv"]) \
        + torch.einsum("nb,mnje->mbej", t1, g["ooov"]) - torch.einsum("jnfb,mnef->mbej", zz, g["oovv"])
    ring = torch.einsum("imae,mbej->ijab", t2, wm) \
        - torch.einsum("ma,mbij->ijab", t1, torch.einsum("ie,mbej->mbij", t1, g["ovvo"]))
    r2 += _pij(_pab(ring))
    v_o = torch.einsum("pai,pbj->ijab", y, d["vo"])
    r2 += _pij(_pab(v_o))
    r2 -= _pab(torch.einsum("ma,ijmb->ijab", t1, g["ooov"].conj()))
    return r1, r2


def _hbar64(case, eps, L, t1, t2):
    o = case["o"]
    d, g = _blocks(L, o)
    e = torch.from_numpy(eps).to(DEV).to(torch.complex128)
    tau = t2 + _asym(t1)
    hvv, hoo, hov, y = _f_terms(d, g, t1, tau)
    hoo, hvv = hoo + torch.diag(e[:o]), hvv + torch.diag(e[o:])
    u = torch.einsum("je,mnie->mnij", t1, g["ooov"])
    h4 = g["oooo"] + u - u.transpose(2, 3) + 0.5 * torch.einsum("ijef,mnef->mnij", tau, g["oovv"])
    h3 = g["ooov"] + torch.einsum("if,mnfe->mnie", t1, g["oovv"])
    q = torch.einsum("jnfb,mnef->mbej", t2, g["oovv"])
    hr = g["ovvo"] + torch.einsum("pme,pbj->mbej", d["ov"], y) \
        - torch.einsum("pmj,pbe->mbej", torch.einsum("pmf,jf->pmj", d["ov"], t1), d["vv"]) \
        + torch.einsum("nb,mnje->mbej", t1, g["ooov"]) - q \
        - torch.einsum("nb,mnej->mbej", t1, torch.einsum("mnef,jf->mnej", g["oovv"], t1))
    yy = torch.einsum("mnie,jnbe->mbij", g["ooov"], t2) + torch.einsum("ie,mbej->mbij", t1, g["ovvo"] - q)
    hb = g["ooov"].conj().permute(2, 3, 0, 1) - torch.einsum("me,ijbe->mbij", hov, t2) \
        - torch.einsum("nb,mnij->mbij", t1, h4) + yy - yy.transpose(2, 3)
    for i in range(o):
        z = torch.einsum("jef,pme->jpmf", tau[i], d["ov"])
        hb[:, :, i, :] += torch.einsum("jpmf,pbf->mbj", z, d["vv"])
    return {"oo": hoo, "vv": hvv, "ov": hov, "oooo": h4, "ooov": h3, "ovvo": hr, "ovoo": hb,
            "oovv": g["oovv"], "t2": t2}


def _sigma64(case, h, r, left):
    o, v, k = case["o"], case["v"], case["k"]
    io, jo = torch.triu_indices(o, o, 1, device=DEV)
    r1 = r[:, :o]
    r2 = torch.zeros((k, o, o, v), dtype=r.dtype, device=DEV)
    u = r[:, o:].reshape(k, len(io), v)
    r2[:, io, jo] = u
    r2[:, jo, io] = -u
    if left:
        s1 = -r1 @ h["oo"].T - 0.5 * torch.einsum("mbij,Kijb->Km", h["ovoo"], r2)
        s2 = torch.einsum("Ki,me->Kime", r1, h["ov"]) - 0.5 * torch.einsum("Ki,mnie->Kmne", r1, h["ooov"]) \
            + 0.5 * r2 @ h["vv"] - torch.einsum("mi,Kijb->Kmjb", h["oo"], r2) \
            + 0.25 * torch.einsum("Kijb,mnij->Kmnb", r2, h["oooo"]) \
            + torch.einsum("Kijb,mbej->Kime", r2, h["ovvo"])
        x = 0.5 * torch.einsum("Kijb,ijeb->Ke", r2, h["t2"])
        s2 = s2 - 0.5 * torch.einsum("Ke,mnef->Kmnf", x, h["oovv"])
        s2 = s2 - s2.transpose(1, 2)
    else:
        s1 = -r1 @ h["oo"] + torch.einsum("me,Kime->Ki", h["ov"], r2) \
            - 0.5 * torch.einsum("mnie,Kmne->Ki", h["ooov"], r2)
        x = torch.einsum("mi,Kmjb->Kijb", h["oo"], r2)
        y = torch.einsum("mbej,Kime->Kijb", h["ovvo"], r2)
        s2 = -torch.einsum("mbij,Km->Kijb", h["ovoo"], r1) + r2 @ h["vv"].T - x + x.transpose(1, 2) \
            + 0.5 * torch.einsum("mnij,Kmnb->Kijb", h["oooo"], r2) + y - y.transpose(1, 2)
        xe = 0.5 * torch.einsum("mnef,Kmnf->Ke", h["oovv"], r2)
        s2 = s2 - torch.einsum("Ke,ijeb->Kijb", xe, h["t2"])
    return torch.cat([s1, s2[:, io, jo].reshape(k, -1)], dim=1)


def _cholesky64(B, n):
    N = B.shape[0]
    d = (B.real.square() + B.imag.square()).sum(1)
    L = torch.zeros((n, N), dtype=B.dtype, device=B.device)
    piv = np.zeros(n, dtype=np.int64)
    for k in range(n):
        p = int(torch.argmax(d))
        col = B @ B[p].conj()
        if k:
            col = col - L[:k].T @ L[:k, p].conj()
        L[k] = col / torch.sqrt(d[p])
        d = d - (L[k].real.square() + L[k].imag.square())
        piv[k] = p
    return {"L": L, "piv": piv}


def exact(case, seed):
    kind = case["kind"]
    if kind == "zgemm":
        return _cnormal((case["M"], case["K"]), _gen(seed, 1)) @ _cnormal((case["N"], case["K"]), _gen(seed, 2)).T
    if kind == "cholesky":
        return _cholesky64(_generator(case, seed), case["n"])
    if kind == "solve":  # iterates to its tolerances
        return None
    o, v = case["o"], case["v"]
    # plain FP64 runs at about 1 TF/s on this card: leave out what takes long
    X, vv = case["X"], float(v) * v
    flops = 0.0 if kind == "fns" else 8.0 * (X + o * o) * vv * vv
    if kind not in ("fns", "ladder"):
        flops += 8.0 * (5.0 * (o * v) ** 3 + 2.0 * X * o * vv * (o + v))
    if flops > 14e12:
        return None
    eps, L = _vectors(case, seed)
    if kind == "fns":
        Lov = L[:, :o, o:]
        x = torch.einsum("pia,pjb->ijab", Lov, Lov)
        e = torch.from_numpy(eps).to(DEV)
        d = e[:o, None, None, None] + e[None, :o, None, None] - e[None, None, o:, None] - e[None, None, None, o:]
        t = (x - x.transpose(2, 3)).conj() / d
        t = t.permute(2, 0, 1, 3).reshape(v, -1)
        occ = torch.linalg.eigvalsh(0.5 * (t @ t.conj().T))
        return {"kept": None, "occ": occ.flip(0).cpu().numpy()}
    t1, t2 = _amplitudes(case, eps, seed)
    if kind == "ladder":
        return _ladder64(L[:, o:, o:].contiguous(), t2)
    if kind == "residual":
        r1, r2 = _residual64(case, eps, L, t1, t2)
        return {"r1": r1, "r2": r2}
    h = _hbar64(case, eps, L, t1, t2)
    return _sigma64(case, h, _ip_vectors(case, seed), kind == "left_sigma")
