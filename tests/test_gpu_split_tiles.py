"""The split products' GEMM where its tiles change: one tile and many, last tiles that are
nearly empty, widths that are rounded up to 16 columns, several tiles of columns.

Each operand is hi + lo to 2^-17 (BF16X3) or 2^-22 (TF32X3) of itself, the lo.lo product
is dropped and sums are FP32: with u twice that a product is off by at most 4 u |a||b|
and a sum of N by N 2^-24 more; the bound below adds both transforms' terms.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("precision,u", [("bf16x3", 2.0 ** -16), ("tf32x3", 2.0 ** -21)])
@pytest.mark.parametrize("N,M,o,np_", [
    (5, 3, 2, 1),        # one tile, 16 columns
    (60, 40, 17, 3),     # 2,400 rows: fewer tiles than SMs
    (96, 203, 17, 16),   # 19,488 rows: 32 rows in the last tile; 33 columns
    (96, 204, 30, 3),
    (130, 160, 64, 66),  # 130 columns: two tiles of 80
    (200, 128, 60, 1),
])
def test_against_fp64(precision, u, N, M, o, np_):
    rng = np.random.default_rng(N + M)
    L = rng.standard_normal((M, N * (N + 1) // 2))
    C = np.linalg.qr(rng.standard_normal((N, N)))[0]
    orbs = np.linspace(0, N - 1, np_).astype(np.int32)
    d = [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (L, C, orbs)]
    Lov, Lp = G.cds_cd_to_mo(d[0], d[1], o, d[2], precision=precision)
    il = torch.tril_indices(N, N, device=DEV)
    A = torch.zeros((M, N, N), dtype=torch.float64, device=DEV)
    A[:, il[0], il[1]] = d[0]
    A[:, il[1], il[0]] = d[0]
    Cj = torch.cat([d[1][:, :o], d[1][:, d[2].long()]], 1)
    w = 4 * u + N * 2.0 ** -24
    T = A @ Cj
    ref = torch.einsum("knr,nq->rqk", T, d[1])
    bound = torch.einsum("knr,nq->rqk", w * (A.abs() @ Cj.abs()) + w * T.abs(), d[1].abs())
    assert ((Lov - ref[:o, o:]).abs() <= bound[:o, o:]).all()
    assert ((Lp - ref[o:]).abs() <= bound[o:]).all()
