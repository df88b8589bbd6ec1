"""The tensor-core gradient's G pass at the edges of its tiles: 32 x 32 tiles of
(x, c2), four c1 in turn, orbitals in chunks of eight; against the FP64 gradient
(its own kernels), 1e-3 of the largest entry, the bound the split precision is
held to elsewhere.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402
from paper_0912_1459_gb300 import cdsigma as C  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("o,v,M,n", [(1, 1, 3, 1), (3, 31, 8, 2), (4, 32, 20, 1), (5, 33, 17, 9), (33, 65, 40, 3)])
def test_gradient_against_fp64(prec, o, v, M, n):
    rng = np.random.default_rng(o * 100 + v)
    eps = np.concatenate([np.sort(rng.uniform(-1.5, -0.3, o)), np.sort(rng.uniform(0.05, 3.0, v))])
    orbs = (np.arange(n) % (o + v)).astype(np.int32)
    x = [rng.standard_normal((o, v, M)) * 0.1, rng.standard_normal((n, o + v, M)) * 0.1, orbs, eps]
    x = [torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in x]
    w = torch.from_numpy(rng.uniform(-0.2, 0.0, n)).to(DEV)
    g = torch.from_numpy(rng.standard_normal(n)).to(DEV)
    ref = C.cds_qp_gradient(x[0], x[1], x[2], x[3], o, w, g, "fp64")
    got = C.cds_qp_gradient(x[0], x[1], x[2], x[3], o, w, g, prec)
    for a, b in zip(got, ref):
        assert (a - b).abs().max().item() <= 1e-3 * b.abs().max().item()
