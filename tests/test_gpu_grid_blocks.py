"""The self-energy on the tensor cores where its last column block changes form: blocks of
up to 96 valid columns take one MMA per product, wider ones one for two of them, and the
grid from the kept numerators ends at the next 16 columns.

BF16X3 against FP64: factors carry 2^-17 each and the lo.lo product is dropped, so an
integral is off by at most 3 x 2^-17 of the product p of its factors' norms, and a numerator
(2 X - X') X, |X| <= p, by 6 p times that, below 2^-12 p^2.  The energies are kept 0.5 Ha
from every pole, so Sigma is off by at most 2^-12 / 0.5 of the sum of p^2, its derivative by
2^-12 / 0.25.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("o,v", [(15, 16), (17, 95), (20, 97), (8, 112), (33, 127), (16, 129), (97, 225)])
def test_bf16x3_grid_against_fp64(o, v):
    rng = np.random.default_rng(o + v)
    M, nmo = 48, o + v
    Lov = rng.standard_normal((o, v, M)) / np.sqrt(M)
    Lp = rng.standard_normal((2, nmo, M)) / np.sqrt(M)
    eps = np.concatenate([np.sort(rng.uniform(-1.5, -1.0, o)), np.sort(rng.uniform(1.0, 1.5, v))])
    # poles e_a + e_b - e_i >= 3 and e_i + e_j - e_a <= -3: these energies are 0.5 away
    E = np.linspace(-2.5, 2.5, 7) + np.zeros((2, 1))
    d = [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (Lov, Lp, eps, E)]
    s, ds, _ = G.cds_sigma2_diag_cache(d[0], d[1], d[2], o, d[3], "bf16x3")
    r, dr = G.cds_sigma2_diag(d[0], d[1], d[2], o, d[3], "fp64")
    mag = ((d[1] ** 2).sum((1, 2)) * (d[0] ** 2).sum())[:, None]
    assert ((s - r).abs() <= 2.0 ** -12 * mag / 0.5).all()
    assert ((ds - dr).abs() <= 2.0 ** -12 * mag / 0.25).all()
