"""FP64 self-energy, Newton and MP2 from exact-slice tensor-core integrals
(bases of 64 orbitals and more), against the oracle, where the tiles and the
energy groups end: 32-blocks of occupied and virtual orbitals, 64-row operand
tiles, 16-column k-steps and 256-column chunks of M, one / eight / more
energies, 64-energy zones, a grid that runs through poles.

Tolerances, set from the arithmetic: integrals carry at most (M + 4) roundings
of 2^-53 against sum |a||b| (the slices' own truncation is 2^-60 of the row
scales), every numerator three times that of X^2, every denominator and sum a
few units; with M <= 300 and no pole nearer than 1e-3 Ha that is below 1e-11
of the sum of the terms' magnitudes, which is what the tests allow.
"""
import numpy as np
import pytest
import torch

from oracle import sigma2

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def factors(o, v, M, n, seed=0):
    rng = np.random.default_rng(seed)
    fall = 0.05 * np.exp(-np.arange(M) / (0.3 * M))
    eps = np.concatenate([np.sort(rng.uniform(-1.5, -0.3, o)), np.sort(rng.uniform(0.05, 3.0, v))])
    Lov = rng.standard_normal((o, v, M)) * fall
    Lp = rng.standard_normal((n, o + v, M)) * fall
    return Lov, Lp, eps


def magnitude(lq, ov, eps, o, E):
    """sum of |term| over both sums of Eq. SE at each energy."""
    v, M = ov.shape[1:]
    Y = (lq[:o] @ ov.reshape(-1, M).T).reshape(o, o, v)
    U = (lq[o:] @ ov.reshape(-1, M).T).reshape(v, o, v)
    eo, ev = eps[:o], eps[o:]
    n1 = (2 * np.abs(Y) + np.abs(Y.transpose(1, 0, 2))) * np.abs(Y)
    n2 = (2 * np.abs(U) + np.abs(U.transpose(2, 1, 0))) * np.abs(U)
    out = []
    for e in E:
        d1 = np.abs(e + ev[None, None, :] - eo[:, None, None] - eo[None, :, None])
        d2 = np.abs(e + eo[None, :, None] - ev[:, None, None] - ev[None, None, :])
        out.append(((n1 / d1).sum() + (n2 / d2).sum(), (n1 / d1 ** 2).sum() + (n2 / d2 ** 2).sum()))
    return np.array(out).T


@pytest.mark.parametrize("o,v,M,n,nE,span", [
    (4, 60, 1, 1, 1, 0.25),       # 64 orbitals, one vector, one energy
    (32, 33, 16, 2, 8, 0.25),     # 65 orbitals: blocks of 32 and 33, all energies direct
    (33, 64, 17, 3, 9, 0.25),     # moments from 9 energies on
    (12, 85, 255, 2, 64, 0.25),
    (40, 96, 257, 1, 65, 0.1),    # second 256-column chunk, second energy zone
    (20, 50, 40, 2, 24, 1.5),     # the grid runs through both sums' poles
    (63, 1, 30, 2, 12, 0.25),     # one virtual orbital
    (1, 70, 30, 2, 12, 0.25),     # one occupied orbital
])
def test_sigma_against_oracle(o, v, M, n, nE, span):
    Lov, Lp, eps = factors(o, v, M, n)
    q = np.clip(np.arange(o - n // 2 - 1, o - n // 2 - 1 + n), 0, o + v - 1)
    E = eps[q][:, None] + (np.linspace(-span, span, nE)[None, :] if nE > 1 else 0.01)
    poles = np.concatenate([(eps[:o, None, None] + eps[None, :o, None] - eps[None, None, o:]).ravel(),
                            (eps[o:, None, None] + eps[None, o:, None] - eps[None, None, :o]).ravel()])
    for t in range(n):            # keep every energy 1e-3 Ha away from every pole
        for k in range(nE):
            while np.abs(poles - E[t, k]).min() < 1e-3:
                E[t, k] += 7e-4
    s, ds = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), o, dev(E), "fp64")
    sc, dsc, cache = G.cds_sigma2_diag_cache(dev(Lov), dev(Lp), dev(eps), o, dev(E), "fp64")
    assert torch.equal(s, sc) and torch.equal(ds, dsc)
    for t in range(n):
        rs, rd = sigma2.sigma2_from_factors(Lp[t], Lov, eps, o, E[t])
        ms, md = magnitude(Lp[t], Lov, eps, o, E[t])
        assert np.all(np.abs(s[t].cpu().numpy() - rs) <= 1e-11 * ms)
        assert np.all(np.abs(ds[t].cpu().numpy() - rd) <= 1e-11 * md)
    # Newton that recomputes and Newton from the kept numerators: the same bits
    orbs = dev(q.astype(np.int32))
    a = G.cds_qp_solve(dev(Lov), dev(Lp), orbs, dev(eps), o, precision="fp64")
    b = G.cds_qp_solve_cached(cache, orbs, dev(eps), o + v, o, precision="fp64")
    for x, y in zip(a, b):
        assert torch.equal(x, y)


def test_repeated_and_nan_energies():
    """One energy repeated (no interval to expand on) and a NaN among the energies."""
    Lov, Lp, eps = factors(20, 50, 40, 1)
    E = np.full((1, 12), eps[19] + 0.01)
    s, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), 20, dev(E), "fp64")
    one, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), 20, dev(E[:, :1]), "fp64")
    np.testing.assert_allclose(s.cpu().numpy(), np.repeat(one.cpu().numpy(), 12, 1), rtol=1e-12)
    E = eps[19] + np.linspace(-0.1, 0.1, 12)[None, :]
    ok, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), 20, dev(E), "fp64")
    E[0, 5] = np.nan
    s, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), 20, dev(E), "fp64")
    s, ok = s.cpu().numpy()[0], ok.cpu().numpy()[0]
    assert np.isnan(s[5])
    np.testing.assert_allclose(np.delete(s, 5), np.delete(ok, 5), rtol=1e-11)


def test_non_finite_factor_touches_only_its_orbital():
    """An infinite factor entry: the plain FP64 products take the call, the
    other orbitals' values stay."""
    Lov, Lp, eps = factors(20, 50, 40, 3)
    E = eps[18:21][:, None] + np.linspace(-0.1, 0.1, 4)[None, :]
    ok, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), 20, dev(E), "fp64")
    Lp[1, 3, 7] = np.inf
    s, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), 20, dev(E), "fp64")
    assert not torch.isfinite(s[1]).any()
    torch.testing.assert_close(s[[0, 2]], ok[[0, 2]], rtol=1e-12, atol=0)


def test_a_small_workspace_is_still_served():
    """The workspace of the fused FP64 kernel (32 x 32 items, two doubles per
    item and energy) is accepted and gives the same values."""
    o, v, M, nE = 20, 50, 40, 4
    Lov, Lp, eps = factors(o, v, M, 2)
    E = eps[19:21][:, None] + np.linspace(-0.1, 0.1, nE)[None, :]
    big, _ = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), o, dev(E), "fp64")
    lib = G.load()
    items = 2 * (v * 1 + o * 3)
    ws = torch.empty(items * nE * 16 + 256, dtype=torch.uint8, device=DEV)
    s, ds = torch.empty((2, 2, nE), dtype=torch.float64, device=DEV)
    t = [dev(x) for x in (Lov, Lp, eps, E)]
    st = lib.cds_sigma2_diag(o + v, o, M, t[0].data_ptr(), t[1].data_ptr(), 2, t[2].data_ptr(),
                             t[3].data_ptr(), nE, 0, s.data_ptr(), ds.data_ptr(), ws.data_ptr(),
                             ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.testing.assert_close(s, big, rtol=1e-11, atol=0)


@pytest.mark.parametrize("o,v,M", [(4, 60, 20), (33, 65, 33)])
def test_mp2_against_oracle(o, v, M):
    Lov, _, eps = factors(o, v, M, 1)
    e, pair = G.cds_mp2_energy(dev(Lov), dev(eps), o, "fp64")
    X = np.einsum("iaK,jbK->ijab", Lov, Lov)
    den = (eps[:o, None, None, None] + eps[None, :o, None, None]
           - eps[None, None, o:, None] - eps[None, None, None, o:])
    ref = ((2 * X - X.transpose(0, 1, 3, 2)) * X / den).sum((1, 2, 3))
    np.testing.assert_allclose(pair.cpu().numpy(), ref, rtol=1e-11)
    np.testing.assert_allclose(float(e[0]), ref.sum(), rtol=1e-11)
