"""What the performance work on this library measures.

Each case is one piece of work that a user of the library has it do, through
the calls of ``paper_0912_1459_gb300.cdsigma``: the Cholesky decomposition of
the integral supermatrix, the AO->MO transform of its vectors, the self-energy
on an energy grid, the Newton quasiparticle solve, the MP2 energy, the
gradient of the quasiparticle energies, a batch of small molecules and the
whole pipeline.  FP64 is what the calls do unless they are told otherwise; the
split-precision forms are what the throughput runs use.

Sizes are those of the workloads of this repository (24 functions in a cube,
240 functions, clusters of 4 to 40 centres, the 840-function cage), ``draw``
takes everything between them.  Inputs are seeded:

* geometries: centres uniform in a ball (clusters) or the vertices of a
  truncated icosahedron displaced by 0.02 bohr (thermal motion), the same
  geometric exponent ladder on every centre;
* C = S^(-1/2) Q with Q random orthogonal, so C^T S C = 1;
* energies: occupied uniform in [-1.5, -0.3] Ha, virtual in [0.05, 3] Ha;
* factors for the calls that start from them: normal deviates whose spread
  falls off along J as the Cholesky vectors' does, scaled so that the
  self-energy is of the order of a tenth of a Hartree and the quasiparticle
  picture holds for the orbitals around the gap.

``exact`` states the method in 64 bits with torch alone.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_0912_1459_gb300 import cdsigma as G

TIE = 1e-12


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a small molecule's decomposition, the default precision: launches
        # and the steps' serial chain are everything
        {"name": "cd_small_fp64", "kind": "cd", "precision": "fp64", "atoms": 6, "ladder": 4,
         "delta": 1e-6, "cage": False},
        # a middle-sized molecule in the default precision
        {"name": "cd_mid_fp64", "kind": "cd", "precision": "fp64", "atoms": 20, "ladder": 12,
         "delta": 1e-5, "cage": False},
        # the cage in the form the throughput runs use (exact slices on the
        # tensor cores)
        {"name": "cd_cage_ozaki", "kind": "cd", "precision": "ozaki", "atoms": 60, "ladder": 14,
         "delta": 1e-4, "cage": True},
        # transform of a middle-sized molecule's vectors, default precision
        {"name": "mo_mid_fp64", "kind": "mo", "precision": "fp64", "nbf": 240, "nocc": 40,
         "M": 720, "np": 10},
        # transform of the cage's vectors on the tensor cores
        {"name": "mo_cage_ozaki", "kind": "mo", "precision": "ozaki", "nbf": 840, "nocc": 180,
         "M": 896, "np": 20},
        # spectrum around the gap of a middle-sized molecule, default
        # precision: Sigma on a grid, then the Newton solve that recomputes it
        {"name": "spectrum_mid_fp64", "kind": "spectrum", "precision": "fp64", "cached": False,
         "nbf": 240, "nocc": 40, "M": 720, "np": 10, "nE": 16},
        # HOMO and LUMO of the cage in FP64, the numerators kept for Newton:
        # the check that a split-precision run is held against
        {"name": "spectrum_cage_fp64", "kind": "spectrum", "precision": "fp64", "cached": True,
         "nbf": 840, "nocc": 180, "M": 896, "np": 2, "nE": 64},
        # the cage's 20 gap orbitals on the tensor cores, as the throughput
        # runs do it: grid with the numerators kept, Newton from them
        {"name": "spectrum_cage_bf16x3", "kind": "spectrum", "precision": "bf16x3",
         "cached": True, "nbf": 840, "nocc": 180, "M": 896, "np": 20, "nE": 64},
        # MP2 energy from the factors on the tensor cores
        {"name": "mp2_bf16x3", "kind": "mp2", "precision": "bf16x3", "nbf": 480, "nocc": 100,
         "M": 600},
        # backward pass of the quasiparticle energies of 8 gap orbitals
        {"name": "gradient_cage_bf16x3", "kind": "gradient", "precision": "bf16x3", "nbf": 840,
         "nocc": 180, "M": 896, "np": 8},
        # twelve clusters of uneven size in one batch: decomposition,
        # transform, self-energy grids
        {"name": "batch_clusters", "kind": "batch", "clusters": 12, "lo": 4, "hi": 40,
         "ladder": 10, "delta": 1e-5},
        # the cage from the basis to its self-energy grid, decomposition and
        # transform overlapped
        {"name": "pipeline_cage", "kind": "pipeline", "atoms": 60, "ladder": 14, "delta": 1e-4,
         "cage": True, "nocc": 180, "np": 20, "nE": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cd", "cd", "mo", "mo", "spectrum", "spectrum", "spectrum", "mp2",
                       "gradient", "batch", "pipeline"])
    if kind == "cd":
        prec = rng.choice(["fp64", "ozaki"])
        ladder = rng.randint(4, 14)
        atoms = _log(rng, 4, 24) if prec == "fp64" else _log(rng, 10, 60)
        return {"kind": kind, "precision": prec, "atoms": atoms, "ladder": ladder,
                "delta": rng.choice([1e-4, 1e-5]), "cage": False}
    if kind == "batch":
        lo = rng.randint(4, 12)
        return {"kind": kind, "clusters": rng.randint(2, 12), "lo": lo,
                "hi": rng.randint(lo + 4, 36), "ladder": rng.randint(6, 10), "delta": 1e-5}
    if kind == "pipeline":
        atoms, ladder = _log(rng, 12, 52), rng.randint(6, 14)
        nbf = atoms * ladder
        return {"kind": kind, "atoms": atoms, "ladder": ladder, "delta": 1e-4, "cage": False,
                "nocc": max(4, nbf // 5), "np": 2 * rng.randint(1, 8), "nE": _log(rng, 8, 64)}
    nbf = _log(rng, 24, 840)
    nocc = max(4, int(nbf * rng.uniform(0.12, 0.25)))
    M = max(20, int(nbf * rng.uniform(1.05, 3.0) if nbf < 500 else nbf * rng.uniform(0.7, 1.05)))
    np_ = 2 * rng.randint(1, min(8, nocc // 2))
    if kind == "mo":
        prec = rng.choice(["fp64", "ozaki"])
        if prec == "fp64" and nbf > 480:   # stays below the largest listed case
            M = min(M, 240)
        return {"kind": kind, "precision": prec, "nbf": nbf, "nocc": nocc, "M": M, "np": np_}
    if kind == "spectrum":
        prec = rng.choice(["fp64", "bf16x3"])
        cached = rng.choice([True, False])
        nE = _log(rng, 1, 64)
        if prec == "fp64" and nbf > 200:   # stays below the largest listed case
            np_ = min(np_, 4)
        if prec == "fp64" and nbf > 420:
            np_, cached, nE = 2, True, min(nE, 32)
            nocc = min(nocc, 180)
        return {"kind": kind, "precision": prec, "cached": cached, "nbf": nbf, "nocc": nocc,
                "M": min(M, 896), "np": np_, "nE": nE}
    if kind == "mp2":
        prec = rng.choice(["fp64", "bf16x3"])
        nbf = _log(rng, 24, 200 if prec == "fp64" else 640)
        return {"kind": kind, "precision": prec, "nbf": nbf,
                "nocc": max(4, int(nbf * rng.uniform(0.12, 0.25))),
                "M": max(20, int(nbf * rng.uniform(0.8, 1.5)))}
    prec = rng.choice(["fp64", "bf16x3"])
    nbf = _log(rng, 24, 240 if prec == "fp64" else 840)
    nocc = max(4, int(nbf * rng.uniform(0.12, 0.215)))
    return {"kind": kind, "precision": prec, "nbf": nbf, "nocc": nocc,
            "M": max(20, min(896, int(nbf * rng.uniform(0.9, 1.6)))),
            "np": 2 * rng.randint(1, 4)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _put(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(_dev())


def _ball(rng, n):
    radius, pts = 3.0 * n ** (1.0 / 3.0), []
    while len(pts) < n:
        p = rng.uniform(-radius, radius, 3)
        if p @ p <= radius * radius and all(((p - q) ** 2).sum() >= 1.0 for q in pts):
            pts.append(p)
    return np.array(pts)


def _cage(rng):
    phi = (1.0 + math.sqrt(5.0)) / 2.0
    pts = set()
    for b in ((0.0, 1.0, 3 * phi), (1.0, 2 + phi, 2 * phi), (phi, 2.0, 2 * phi + 1)):
        for c in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
            for s in itertools.product((1.0, -1.0), repeat=3):
                pts.add(tuple(round(s[k] * b[c[k]], 12) + 0.0 for k in range(3)))
    return np.array(sorted(pts)) * 1.35 + 0.02 * rng.standard_normal((60, 3))


def _basis(rng, atoms, ladder, cage):
    centres = _cage(rng) if cage else _ball(rng, atoms)
    lo, hi = (0.08, 30.0) if cage else (0.1, 10.0)
    ex = lo * (hi / lo) ** (np.arange(ladder) / (ladder - 1))
    return (np.repeat(centres, ladder, axis=0), np.tile(ex, len(centres)),
            np.repeat(np.arange(len(centres), dtype=np.int32), ladder))


def _overlap(xyz, al):
    p = al[:, None] + al[None, :]
    r2 = ((xyz[:, None, :] - xyz[None, :, :]) ** 2).sum(-1)
    return (2.0 * np.sqrt(al[:, None] * al[None, :]) / p) ** 1.5 * np.exp(
        -al[:, None] * al[None, :] / p * r2)


def _orbitals(rng, S):
    w, U = np.linalg.eigh(S)
    Q, R = np.linalg.qr(rng.standard_normal(S.shape))
    return ((U / np.sqrt(w)) @ U.T) @ (Q * np.sign(np.diag(R)))


def _energies(rng, nocc, nvir):
    return np.concatenate([np.sort(rng.uniform(-1.5, -0.3, nocc)),
                           np.sort(rng.uniform(0.05, 3.0, nvir))])


def _gap(nocc, n):
    return np.arange(nocc - n // 2, nocc + n - n // 2, dtype=np.int32)


def _grid(eq, nE):
    if nE == 1:
        return eq[:, None].copy()
    return eq[:, None] + (-0.25 + 0.5 * np.arange(nE) / (nE - 1))[None, :]


def _factors(seed, nocc, nvir, M, orbitals):
    """Lov [o, v, M] and, for the orbitals given, Lp [np, nmo, M]."""
    g = torch.Generator(device=_dev())
    g.manual_seed(seed * 7919 + 17)
    fall = torch.exp(-torch.arange(M, dtype=torch.float64, device=_dev()) / (0.2 * M))
    x2 = 0.3 / (nocc * nvir * max(nocc, nvir))      # mean square of an MO integral
    scale = (x2 / float((fall ** 4).sum())) ** 0.25
    Lov = torch.randn((nocc, nvir, M), dtype=torch.float64, device=_dev(), generator=g)
    Lov *= fall * scale
    Lp = None
    if orbitals is not None:
        Lp = torch.randn((len(orbitals), nocc + nvir, M), dtype=torch.float64, device=_dev(),
                         generator=g)
        Lp *= fall * scale
    return Lov, Lp


def _clusters(case):
    """(centres, orbitals, energies) of each cluster: uneven sizes over the whole range."""
    n, span = case["clusters"], case["hi"] - case["lo"]
    return [(case["lo"] + (span * ((5 * i + 2) % n) + n // 2) // max(n - 1, 1) % (span + 1),
             2 + 2 * (i % 2), 8 + (19 * i + 11) % 57) for i in range(n)]


def _rank_cap(nbf, cage):
    """Room for the vectors that a user of these bases keeps."""
    return 1280 if cage else min(G.npair(nbf), max(6 * nbf, 512) if nbf <= 240 else 1536)


def prepare(case, seed):
    rng = np.random.default_rng([seed, 20091214])
    kind = case["kind"]
    if kind in ("cd", "pipeline"):
        xyz, al, at = _basis(rng, case["atoms"], case["ladder"], case["cage"])
        nbf, cap = len(al), _rank_cap(len(al), case["cage"])
        st = {"xyz": _put(xyz), "alpha": _put(al), "atom": _put(at), "delta": case["delta"],
              "cap": cap}
        lib = G.load()
        st["L"] = torch.zeros((cap, G.npair(nbf)), dtype=torch.float64, device=_dev())
        if kind == "cd":
            st["precision"] = case["precision"]
            st["ws"] = torch.empty(lib.cds_cd_workspace_bytes_prec(
                nbf, cap, G.PRECISIONS[case["precision"]]), dtype=torch.uint8, device=_dev())
        else:
            o, n = case["nocc"], case["np"]
            eps = _energies(rng, o, nbf - o)
            orbs = _gap(o, n)
            st.update(C=_put(_orbitals(rng, _overlap(xyz, al))), eps=_put(eps), nocc=o,
                      orbs=_put(orbs), E=_put(_grid(eps[orbs], case["nE"])))
            st["Lov"] = torch.empty(o * (nbf - o) * cap, dtype=torch.float64, device=_dev())
            st["Lp"] = torch.empty(n * nbf * cap, dtype=torch.float64, device=_dev())
            st["ws"] = torch.empty(lib.cds_cd_decompose_to_mo_workspace_bytes(
                nbf, nbf, o, cap, n, G.PRECISIONS["ozaki"]), dtype=torch.uint8, device=_dev())
            st["cache"] = torch.empty(lib.cds_sigma2_cache_bytes(
                nbf, o, n, G.PRECISIONS["bf16x3"]), dtype=torch.uint8, device=_dev())
    elif kind == "mo":
        n, o, M = case["nbf"], case["nocc"], case["M"]
        ladder = 12 if n % 12 == 0 else 8
        atoms = -(-n // ladder)
        xyz, al, _ = _basis(rng, atoms, ladder, False)
        xyz, al = xyz[:n], al[:n]
        S = _overlap(xyz, al)
        g = torch.Generator(device=_dev())
        g.manual_seed(seed * 7919 + 31)
        mu, nu = np.tril_indices(n)[1], np.tril_indices(n)[0]
        fall = torch.exp(-torch.arange(M, dtype=torch.float64, device=_dev()) / (0.2 * M))
        L = torch.randn((M, G.npair(n)), dtype=torch.float64, device=_dev(), generator=g)
        L *= _put(S[nu, mu])[None, :]       # a pair's vector is as large as its overlap
        L *= fall[:, None]
        orbs = _gap(o, case["np"])
        st = {"L": L, "C": _put(_orbitals(rng, S)), "nocc": o, "orbs": _put(orbs),
              "precision": case["precision"]}
        st["ws"] = torch.empty(G.load().cds_cd_to_mo_workspace_bytes(n, n, o, M, len(orbs)),
                               dtype=torch.uint8, device=_dev())
    elif kind == "batch":
        mols, parts = [], {k: [] for k in ("xyz", "alpha", "atom", "C", "orb", "eps", "E")}
        for nat, np_, nE in _clusters(case):
            xyz, al, at = _basis(rng, nat, case["ladder"], False)
            nbf = len(al)
            o = max(4, nbf // 5)
            orbs = _gap(o, np_)
            eps = _energies(rng, o, nbf - o)
            mols.append((nbf, o, len(orbs), nE, min(G.npair(nbf), 4 * nbf + 64)))
            for k, a in (("xyz", xyz), ("alpha", al), ("atom", at), ("orb", orbs), ("eps", eps),
                         ("C", _orbitals(rng, _overlap(xyz, al))), ("E", _grid(eps[orbs], nE))):
                parts[k].append(np.ascontiguousarray(a).ravel())
        st = {k: _put(np.concatenate(v)) for k, v in parts.items()}
        st.update(mols=mols, delta=case["delta"],
                  batch=G.Batch(mols, _dev(), "bf16x3", cd_precision="ozaki"))
        st["batch"].L.zero_()
        st["batch"].piv.zero_()
    else:
        n, o, M = case["nbf"], case["nocc"], case["M"]
        eps = _energies(rng, o, n - o)
        orbs = _gap(o, case["np"]) if kind != "mp2" else None
        Lov, Lp = _factors(seed, o, n - o, M, orbs)
        st = {"Lov": Lov, "eps": _put(eps), "nocc": o, "precision": case["precision"]}
        lib, prec = G.load(), G.PRECISIONS[case["precision"]]
        if kind == "mp2":
            st["ws"] = torch.empty(max(1, lib.cds_mp2_workspace_bytes(n, o, M, prec)),
                                   dtype=torch.uint8, device=_dev())
        else:
            st.update(Lp=Lp, orbs=_put(orbs))
        if kind == "spectrum":
            k = case["np"]
            st.update(E=_put(_grid(eps[orbs], case["nE"])), cached=case["cached"])
            st["ws"] = torch.empty(max(1, lib.cds_sigma2_workspace_bytes(
                n, o, M, k, case["nE"], prec)), dtype=torch.uint8, device=_dev())
            if case["cached"]:
                st["cache"] = torch.empty(max(1, lib.cds_sigma2_cache_bytes(n, o, k, prec)),
                                          dtype=torch.uint8, device=_dev())
        if kind == "gradient":
            # converged roots and upstream gradients, as a backward pass has them
            st["omega"] = _put(eps[orbs] + rng.uniform(-0.05, 0.05, len(orbs)))
            st["g"] = _put(rng.standard_normal(len(orbs)))
    st["kind"] = kind
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _vectors(s, L, piv, D, de):
    """The caller's buffers: the vectors in front, the rows that are left zero."""
    M = L.shape[0]
    s["L"][M:] = 0.0
    return {"rank": M, "L": s["L"], "D": D, "delta_eff": de,
            "piv": torch.nn.functional.pad(piv, (0, s["cap"] - M))}


def run(s):
    kind = s["kind"]
    if kind == "cd":
        L, piv, D, de = G.cds_cd_decompose(s["xyz"], s["alpha"], s["atom"], s["delta"],
                                           max_rank=s["cap"], L_out=s["L"], workspace=s["ws"],
                                           precision=s["precision"])
        return _vectors(s, L, piv, D, de)
    if kind == "mo":
        Lov, Lp = G.cds_cd_to_mo(s["L"], s["C"], s["nocc"], s["orbs"], workspace=s["ws"],
                                 precision=s["precision"])
        return {"Lov": Lov, "Lp": Lp}
    if kind == "spectrum":
        if s["cached"]:
            sig, ds, cache = G.cds_sigma2_diag_cache(s["Lov"], s["Lp"], s["eps"], s["nocc"],
                                                     s["E"], s["precision"], cache=s["cache"],
                                                     workspace=s["ws"])
            w, P, it, status = G.cds_qp_solve_cached(cache, s["orbs"], s["eps"],
                                                     s["Lp"].shape[1], s["nocc"],
                                                     precision=s["precision"])
        else:
            sig, ds = G.cds_sigma2_diag(s["Lov"], s["Lp"], s["eps"], s["nocc"], s["E"],
                                        s["precision"], workspace=s["ws"])
            w, P, it, status = G.cds_qp_solve(s["Lov"], s["Lp"], s["orbs"], s["eps"], s["nocc"],
                                              precision=s["precision"])
        return {"sigma": sig, "dsigma": ds, "omega": w, "pole": P, "iters": it, "status": status}
    if kind == "mp2":
        e, pair = G.cds_mp2_energy(s["Lov"], s["eps"], s["nocc"], s["precision"],
                                   workspace=s["ws"])
        return {"e": e, "pair": pair}
    if kind == "gradient":
        de, dov, dp = G.cds_qp_gradient(s["Lov"], s["Lp"], s["orbs"], s["eps"], s["nocc"],
                                        s["omega"], s["g"], s["precision"])
        return {"d_eps": de, "d_Lov": dov, "d_Lp": dp}
    if kind == "batch":
        b = s["batch"]
        ranks = b.cd_decompose(s["xyz"], s["alpha"], s["atom"], s["delta"], precision="ozaki")
        b.cd_to_mo(s["C"], s["orb"], precision="ozaki")
        b.sigma2(s["eps"], s["E"])
        for c, m in enumerate(s["mols"]):
            b.view("L", c, (m[4], G.npair(m[0])))[ranks[c]:] = 0.0
            b.view("piv", c, (m[4],))[ranks[c]:] = 0
        return {"ranks": np.array(ranks), "L": b.L, "piv": b.piv, "D": b.D, "Lov": b.Lov,
                "Lp": b.Lp, "sigma": b.sigma, "dsigma": b.dsigma}
    L, piv, D, de, Lov, Lp = G.cds_cd_decompose_to_mo(
        s["xyz"], s["alpha"], s["atom"], s["delta"], s["C"], s["nocc"], s["orbs"],
        max_rank=s["cap"], L_out=s["L"], Lov_out=s["Lov"], Lp_out=s["Lp"], workspace=s["ws"],
        transform="ozaki", cd_precision="ozaki")
    sig, ds, _ = G.cds_sigma2_diag_cache(Lov, Lp, s["eps"], s["nocc"], s["E"], "bf16x3",
                                         cache=s["cache"])
    s["Lov"][Lov.numel():] = 0.0
    s["Lp"][Lp.numel():] = 0.0
    return dict(_vectors(s, L, piv, D, de), Lov=s["Lov"], Lp=s["Lp"], sigma=sig, dsigma=ds)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _typical_rank(nbf, delta):
    """Vectors that s-Gaussian bases of these shapes take (used for the work only)."""
    return int(min(nbf * (nbf + 1) // 2, nbf * {1e-4: 1.1, 1e-5: 3.0, 1e-6: 5.0}[delta]))


def _work_cd(nbf, M):
    """Every vector written once, every projection sum taken once."""
    npr = nbf * (nbf + 1) // 2
    return 8.0 * npr * (M + 1), 1.0 * npr * M * (M + 60)


def _work_mo(nbf, nocc, M, k):
    npr, v = nbf * (nbf + 1) // 2, nbf - nocc
    out = nocc * v * M + k * nbf * M
    return 8.0 * (npr * M + nbf * nbf + out), 2.0 * M * (
        (nocc + k) * nbf * nbf + nocc * v * nbf + k * nbf * nbf)


def _work_sigma(nbf, nocc, M, k, evals):
    """One contraction per orbital, a division and two sums per element and energy."""
    v = nbf - nocc
    el = nocc * v * nbf
    return 8.0 * (nocc * v * M + k * nbf * M + 2 * k * evals), k * el * (2.0 * M + 3.0 * evals)


def work(case):
    kind = case["kind"]
    if kind == "cd":
        nbf = case["atoms"] * case["ladder"]
        by, fl = _work_cd(nbf, _typical_rank(nbf, case["delta"]))
    elif kind == "mo":
        by, fl = _work_mo(case["nbf"], case["nocc"], case["M"], case["np"])
    elif kind == "spectrum":
        by, fl = _work_sigma(case["nbf"], case["nocc"], case["M"], case["np"], case["nE"] + 4)
    elif kind == "mp2":
        o, v = case["nocc"], case["nbf"] - case["nocc"]
        by, fl = 8.0 * o * v * case["M"], 1.0 * (o * v) ** 2 * (case["M"] + 2)
    elif kind == "gradient":
        o, n, M, k = case["nocc"], case["nbf"], case["M"], case["np"]
        by = 16.0 * (o * (n - o) * M + k * n * M)
        fl = 6.0 * k * o * (n - o) * n * M
    elif kind == "batch":
        by = fl = 0.0
        for nat, np_, nE in _clusters(case):
            nbf = nat * case["ladder"]
            M, o = _typical_rank(nbf, case["delta"]), max(4, nbf // 5)
            for b, f in (_work_cd(nbf, M), _work_mo(nbf, o, M, np_),
                         _work_sigma(nbf, o, M, np_, nE)):
                by, fl = by + b, fl + f
    else:
        nbf = case["atoms"] * case["ladder"]
        M = _typical_rank(nbf, case["delta"])
        by = fl = 0.0
        for b, f in (_work_cd(nbf, M), _work_mo(nbf, case["nocc"], M, case["np"]),
                     _work_sigma(nbf, case["nocc"], M, case["np"], case["nE"])):
            by, fl = by + b, fl + f
    return {"bytes": float(by), "flops": float(fl)}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
def _exact_cd(xyz, al, delta, cap):
    n = al.shape[0]
    nu, mu = torch.tril_indices(n, n, device=al.device)
    a, b = al[mu], al[nu]
    p = a + b
    P = (a[:, None] * xyz[mu] + b[:, None] * xyz[nu]) / p[:, None]
    r2 = ((xyz[mu] - xyz[nu]) ** 2).sum(1)
    K = (2 * a / math.pi) ** 0.75 * (2 * b / math.pi) ** 0.75 * torch.exp(-a * b / p * r2) / p

    def integral(q, Q, Kq):
        T = p * q / (p + q) * ((P - Q) ** 2).sum(1)
        x = torch.sqrt(torch.clamp(T, min=1e-10))
        f0 = torch.where(T < 1e-10, 1.0 - T / 3.0, 0.5 * math.sqrt(math.pi) * torch.erf(x) / x)
        return 2.0 * math.pi ** 2.5 * K * Kq / torch.sqrt(p + q) * f0

    D = integral(p, P, K)
    scale = D.max()
    top = float(scale)
    deff = max(float(delta), D.numel() * 2.0 ** -52 * top)
    L = torch.zeros((cap, D.numel()), dtype=torch.float64, device=al.device)
    piv = []
    for k in range(cap):
        g = D.max()
        if k % 8 == 0 and float(g) <= deff:
            break
        i = ((D >= g - TIE * scale) & (D > deff)).int().argmax().view(1)
        col = integral(p[i], P[i], K[i]) - (L[:k, i].T @ L[:k]).view(-1)
        row = col / torch.sqrt(D[i])
        L[k] = row
        D = D - row * row
        D[i] = 0.0
        piv.append(torch.cat([i.double(), g.view(1)]))
    else:
        g = D.max()
    # the stop test is read every 8 steps: drop what came after it
    tops = torch.stack(piv)[:, 1] if piv else torch.zeros(0)
    M = int((tops > deff).sum())
    for k in range(M, len(piv)):
        D = D + L[k] * L[k]
    return L[:M], torch.stack(piv)[:M, 0].to(torch.int32), D, deff


def _exact_mo(L, C, nocc, orbs):
    n = C.shape[0]
    nu, mu = torch.tril_indices(n, n, device=C.device)
    M = L.shape[0]
    ov = torch.empty((nocc, n - nocc, M), dtype=torch.float64, device=C.device)
    pp = torch.empty((len(orbs), n, M), dtype=torch.float64, device=C.device)
    Co, Cv, Cp = C[:, :nocc], C[:, nocc:], C[:, orbs.long()]
    step = max(1, min(M, (1 << 27) // (n * n)))
    for k in range(0, M, step):
        A = torch.zeros((min(step, M - k), n, n), dtype=torch.float64, device=C.device)
        A[:, nu, mu] = L[k:k + step]
        A[:, mu, nu] = L[k:k + step]
        ov[:, :, k:k + step] = ((Co.T @ A) @ Cv).permute(1, 2, 0)
        pp[:, :, k:k + step] = ((Cp.T @ A) @ C).permute(1, 2, 0)
    return ov, pp


class _Sigma:
    """Sigma of one orbital: numerators of both sums, evaluated at any energies."""

    def __init__(self, ov, lq, eps, o):
        flat, v = ov.reshape(-1, ov.shape[2]), ov.shape[1]
        Y = (lq[:o] @ flat.T).view(o, o, v)
        U = (lq[o:] @ flat.T).view(v, o, v)
        eo, ev = eps[:o], eps[o:]
        self.parts = [((2 * Y - Y.transpose(0, 1)) * Y,
                       ev[None, None, :] - eo[:, None, None] - eo[None, :, None]),
                      ((2 * U - U.transpose(0, 2)) * U,
                       eo[None, :, None] - ev[:, None, None] - ev[None, None, :])]
        self.ints = (Y, U)

    def at(self, w):
        s = d = 0.0
        for num, base in self.parts:
            r = 1.0 / (base + w)
            t = num * r
            s, d = s + t.sum(), d - (t * r).sum()
        return s, d


def _exact_grid(ov, lp, eps, o, E):
    out = torch.empty((2,) + tuple(E.shape), dtype=torch.float64, device=E.device)
    for t in range(E.shape[0]):
        f = _Sigma(ov, lp[t], eps, o)
        for e in range(E.shape[1]):
            out[0, t, e], out[1, t, e] = f.at(E[t, e])
    return out[0], out[1]


def _into(s, cd):
    """The decomposition with its vectors in the state's buffer."""
    s["L"][:len(cd[1])] = cd[0]
    return (s["L"][:len(cd[1])],) + cd[1:]


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    if kind == "cd":
        return _vectors(s, *_into(s, _exact_cd(s["xyz"], s["alpha"], s["delta"], s["cap"])))
    if kind == "mo":
        ov, pp = _exact_mo(s["L"], s["C"], s["nocc"], s["orbs"])
        return {"Lov": ov, "Lp": pp}
    if kind == "spectrum":
        eps, o = s["eps"], s["nocc"]
        sig, ds = _exact_grid(s["Lov"], s["Lp"], eps, o, s["E"])
        w = torch.empty(len(s["orbs"]), dtype=torch.float64)
        pole = torch.empty_like(w)
        it = torch.empty(len(w), dtype=torch.int32)
        for t, q in enumerate(s["orbs"].tolist()):
            f = _Sigma(s["Lov"], s["Lp"][t], eps, o)
            x = eq = float(eps[q])
            for n in range(50):
                a, b = (float(y) for y in f.at(x))
                P = 1.0 / (1.0 - b)
                new = x + (eq + a - x) * P
                done, x = abs(new - x) <= 1e-5, new
                if done:
                    break
            w[t], pole[t], it[t] = x, P, n + 1
        return {"sigma": sig, "dsigma": ds, "omega": w, "pole": pole, "iters": it,
                "status": None}
    if kind == "mp2":
        ov, eps, o = s["Lov"], s["eps"], s["nocc"]
        ev, pair = eps[o:], torch.empty(o, dtype=torch.float64, device=eps.device)
        for i in range(o):
            X = (ov.reshape(-1, ov.shape[2]) @ ov[i].T).view(o, -1, ov.shape[1])   # j, b, a
            den = eps[i] + eps[:o, None, None] - ev[None, :, None] - ev[None, None, :]
            pair[i] = ((2 * X - X.transpose(1, 2)) * X / den).sum()
        return {"e": pair.sum().view(1), "pair": pair}
    if kind == "gradient":
        ov, eps, o = s["Lov"], s["eps"], s["nocc"]
        flat = ov.reshape(-1, ov.shape[2])
        de, dov, dp = torch.zeros_like(eps), torch.zeros_like(flat), torch.zeros_like(s["Lp"])
        for t, q in enumerate(s["orbs"].tolist()):
            f = _Sigma(ov, s["Lp"][t], eps, o)
            (n1, b1), (n2, b2) = f.parts
            Y, U = f.ints
            d1, d2 = b1 + s["omega"][t], b2 + s["omega"][t]
            r1, r2 = n1 / d1 ** 2, n2 / d2 ** 2
            W = s["g"][t] / (1.0 + r1.sum() + r2.sum())
            de[o:] += W * (r2.sum((1, 2)) + r2.sum((0, 1)) - r1.sum((0, 1)))
            de[:o] += W * (r1.sum((1, 2)) + r1.sum((0, 2)) - r2.sum((0, 2)))
            de[q] += W
            G1 = (W * (4 * Y - 2 * Y.transpose(0, 1)) / d1).view(o, -1)
            G2 = (W * (4 * U - 2 * U.transpose(0, 2)) / d2).view(U.shape[0], -1)
            dp[t, :o], dp[t, o:] = G1 @ flat, G2 @ flat
            dov += G1.T @ s["Lp"][t, :o] + G2.T @ s["Lp"][t, o:]
        return {"d_eps": de, "d_Lov": dov.view_as(ov), "d_Lp": dp}
    if kind == "pipeline":
        L, piv, D, de = _into(s, _exact_cd(s["xyz"], s["alpha"], s["delta"], s["cap"]))
        ov, pp = _exact_mo(L, s["C"], s["nocc"], s["orbs"])
        sig, ds = _exact_grid(ov, pp, s["eps"], s["nocc"], s["E"])
        for key, val in (("Lov", ov), ("Lp", pp)):
            s[key].zero_()
            s[key][:val.numel()] = val.view(-1)
        return dict(_vectors(s, L, piv, D, de), Lov=s["Lov"], Lp=s["Lp"], sigma=sig, dsigma=ds)
    b, at = s["batch"], {"x": 0, "C": 0, "k": 0, "E": 0}
    out = {"ranks": [], "D": [], "sigma": [], "dsigma": [], "L": b.L, "piv": b.piv, "Lov": b.Lov,
           "Lp": b.Lp}
    for c, (nbf, o, k, nE, cap) in enumerate(s["mols"]):
        xyz = s["xyz"][3 * at["x"]:3 * (at["x"] + nbf)].view(nbf, 3)
        al, eps = s["alpha"][at["x"]:at["x"] + nbf], s["eps"][at["x"]:at["x"] + nbf]
        C = s["C"][at["C"]:at["C"] + nbf * nbf].view(nbf, nbf)
        L, piv, D, _ = _exact_cd(xyz, al, s["delta"], cap)
        ov, pp = _exact_mo(L, C, o, s["orb"][at["k"]:at["k"] + k])
        sig, ds = _exact_grid(ov, pp, eps, o, s["E"][at["E"]:at["E"] + k * nE].view(k, nE))
        for key, val in (("L", L), ("piv", piv), ("ov", ov), ("p", pp)):
            b.view(key, c, tuple(val.shape)).copy_(val)
        out["ranks"].append(len(piv))
        for key, val in (("D", D), ("sigma", sig), ("dsigma", ds)):
            out[key].append(val.reshape(-1))
        at = {"x": at["x"] + nbf, "C": at["C"] + nbf * nbf, "k": at["k"] + k,
              "E": at["E"] + k * nE}
    for key in ("D", "sigma", "dsigma"):
        out[key] = torch.cat(out[key])
    out["ranks"] = np.array(out["ranks"])
    return out
