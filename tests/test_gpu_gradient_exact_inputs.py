"""The tensor-core gradient where the split products are exact: factors that are small
integers times a power of two have no low parts and their sums are whole in FP32, so what
is left is the pass over the integrals (denominators, reciprocals, G, the sums over its
elements), and the splits of G.

Tolerances.  d_eps: FP64 sums of r, each element a few units of 2^-53 off, in any order:
1e-12 of the sum of magnitudes.  d_Lov, d_Lp: G in two bf16 parts is good to 2^-16, the
sums to 2^-24 of the magnitudes per term: (2^-16 + K 2^-24) sum |G||L|, 2e-5 + 6e-8 K as
used, K = o v for d_Lp and 2 (o + v) for d_Lov."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("o,v,M", [(5, 9, 8), (33, 70, 24), (7, 130, 33), (40, 33, 16)])
def test_against_64_bits(o, v, M):
    rng = np.random.default_rng(o)
    unit = 2.0 ** -6
    ov = dev(rng.integers(-4, 5, (o, v, M)) * unit)
    lp = dev(rng.integers(-4, 5, (2, o + v, M)) * unit)
    eps = dev(np.concatenate([np.sort(rng.uniform(-1.5, -0.3, o)), np.sort(rng.uniform(0.05, 3.0, v))]))
    orbs = dev(np.array([o - 1, o], dtype=np.int32))
    w = eps[orbs.long()] + dev(np.array([0.0625, -0.03125]))
    g = dev(np.array([1.0, -0.5]))
    de, dov, dp = G.cdsigma.cds_qp_gradient(ov, lp, orbs, eps, o, w, g, "bf16x3")
    flat = ov.reshape(-1, M)
    re, me = torch.zeros_like(eps), torch.zeros_like(eps)
    rov, mov = torch.zeros_like(flat), torch.zeros_like(flat)
    eo, ev = eps[:o], eps[o:]
    for t in range(2):
        Y = (lp[t, :o] @ flat.T).view(o, o, v)                 # x, j, a
        U = (lp[t, o:] @ flat.T).view(v, o, v)                 # x, j, b
        d1 = w[t] + ev[None, None, :] - eo[:, None, None] - eo[None, :, None]
        d2 = w[t] + eo[None, :, None] - ev[:, None, None] - ev[None, None, :]
        n1, n2 = 2 * Y - Y.transpose(0, 1), 2 * U - U.transpose(0, 2)
        r1, r2 = n1 * Y / d1 ** 2, n2 * U / d2 ** 2
        W = g[t] / (1.0 + r1.sum() + r2.sum())
        a1, a2 = r1.abs(), r2.abs()
        wide = W.abs() * (1 + (a1.sum() + a2.sum()) * W.abs() / g[t].abs())   # W's own sums
        re[o:] += W * (r2.sum((1, 2)) + r2.sum((0, 1)) - r1.sum((0, 1)))
        re[:o] += W * (r1.sum((1, 2)) + r1.sum((0, 2)) - r2.sum((0, 2)))
        re[orbs[t].long()] += W
        me[o:] += wide * (a2.sum((1, 2)) + a2.sum((0, 1)) + a1.sum((0, 1)))
        me[:o] += wide * (a1.sum((1, 2)) + a1.sum((0, 2)) + a2.sum((0, 2)))
        me[orbs[t].long()] += wide
        G1, G2 = (W * 2 * n1 / d1).view(o, -1), (W * 2 * n2 / d2).view(v, -1)
        rov += G1.T @ lp[t, :o] + G2.T @ lp[t, o:]
        mov += G1.abs().T @ lp[t, :o].abs() + G2.abs().T @ lp[t, o:].abs()
        rp = torch.cat([G1 @ flat, G2 @ flat])
        mp = torch.cat([G1.abs() @ flat.abs(), G2.abs() @ flat.abs()])
        assert ((dp[t] - rp).abs() <= (2e-5 + 6e-8 * o * v) * mp + 1e-300).all()
    assert ((de - re).abs() <= 1e-12 * me).all()
    assert ((dov.reshape(-1, M) - rov).abs() <= (2e-5 + 6e-8 * 2 * (o + v)) * mov + 1e-300).all()
