"""FP64 products of rows of wide dynamic range (localised orbitals, factors graded in
opposite senses): every result is good to its own sum of magnitudes S = sum |a||b|, as a
sum of FP64 products is, however small S is beside the rows' largest entries.

Tolerances: one product is off by at most (K + 4) 2^-53 S, the reference's FP64 sums by
as much again.  Two products in a row (the transform) take 4 (N + 4) 2^-53 of |C|'|A||C|.
Self-energy: the numerators are six times as far off as X^2, denominators (no pole nearer
than 0.1 Ha) and sums a few units more: 8 x 2 (M + 16) 2^-53 of the terms' magnitudes
with S in the place of |X|."""
import numpy as np
import pytest
import torch

from oracle import sigma2

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")
U = 2.0 ** -53


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def magnitudes(lq, ov, eps, o, E):
    v, M = ov.shape[1:]
    Y = (np.abs(lq[:o]) @ np.abs(ov).reshape(-1, M).T).reshape(o, o, v)
    X = (np.abs(lq[o:]) @ np.abs(ov).reshape(-1, M).T).reshape(v, o, v)
    eo, ev = eps[:o], eps[o:]
    n1, n2 = (2 * Y + Y.transpose(1, 0, 2)) * Y, (2 * X + X.transpose(2, 1, 0)) * X
    out = []
    for e in E:
        d1 = np.abs(e + ev[None, None, :] - eo[:, None, None] - eo[None, :, None])
        d2 = np.abs(e + eo[None, :, None] - ev[:, None, None] - ev[None, None, :])
        out.append(((n1 / d1).sum() + (n2 / d2).sum(), (n1 / d1 ** 2).sum() + (n2 / d2 ** 2).sum()))
    return np.array(out).T


@pytest.mark.parametrize("o,v,M,nE,t", [(4, 60, 2, 1, 1e-6), (20, 50, 17, 12, 1e-14), (33, 64, 260, 2, 1e-30),
                                        (12, 85, 40, 64, 1.0)])
def test_self_energy(o, v, M, nE, t):
    rng = np.random.default_rng(M)
    ramp = t ** (np.arange(M) / (M - 1))
    Lov = rng.standard_normal((o, v, M)) * ramp
    Lp = rng.standard_normal((2, o + v, M)) * ramp[::-1]
    Lp[1, 5] = 0.0
    eps = np.concatenate([np.sort(rng.uniform(-1.5, -0.3, o)), np.sort(rng.uniform(0.05, 3.0, v))])
    E = np.array([-0.25, 0.0])[:, None] + np.linspace(0.0, 0.02, nE)    # between the two sums' poles
    s, ds = G.cds_sigma2_diag(dev(Lov), dev(Lp), dev(eps), o, dev(E), "fp64")
    for q in range(2):
        rs, rd = sigma2.sigma2_from_factors(Lp[q], Lov, eps, o, E[q])
        ms, md = magnitudes(Lp[q], Lov, eps, o, E[q])
        tol = 16 * (M + 16) * U
        assert np.all(np.abs(s[q].cpu().numpy() - rs) <= tol * ms)
        assert np.all(np.abs(ds[q].cpu().numpy() - rd) <= tol * md)


def unpacked(L, N):
    il = np.tril_indices(N)
    A = np.zeros((L.shape[0], N, N))
    A[:, il[0], il[1]] = L
    A[:, il[1], il[0]] = L
    return A


@pytest.mark.parametrize("N,M,o,np_,fall", [(33, 3, 8, 1, 2.0), (70, 9, 21, 2, 0.7), (130, 3, 30, 0, 0.4),
                                            (260, 5, 40, 3, 0.2), (300, 2, 70, 2, 0.0)])
def test_transform(N, M, o, np_, fall):
    """Orbitals and vectors that fall off from a function of their own; one vector zero,
    one tiny, one large (beyond the slices' range in one case)."""
    rng = np.random.default_rng(N)
    x = np.arange(N)
    C = rng.standard_normal((N, N)) * np.exp(-fall * np.abs(x[:, None] - x[None, :]))
    il = np.tril_indices(N)
    at = rng.integers(0, N, M)[:, None]
    L = rng.standard_normal((M, il[0].size)) * np.exp(
        -fall * (np.abs(il[0][None, :] - at) + np.abs(il[1][None, :] - at)))
    L[1] *= 1e180 if N == 130 else 1e80
    if M > 2:
        L[2] *= 1e-60
    if M > 3:
        L[3] = 0.0
    orbs = np.linspace(0, N - 1, np_).astype(np.int32)
    Lov, Lp = G.cds_cd_to_mo(dev(L), dev(C), o, dev(orbs))
    A = unpacked(L, N)

    def both(c, a):
        return (np.einsum("mi,Kmn,na->iaK", c[:, :o], a, c[:, o:], optimize=True),
                np.einsum("mt,Kmn,nq->tqK", c[:, orbs], a, c, optimize=True))

    for got, ref, mag in zip((Lov, Lp), both(C, A), both(np.abs(C), np.abs(A))):
        err = np.abs(got.cpu().numpy() - ref)
        assert np.all(err <= 4 * (N + 4) * U * mag + 1e-300)
