"""The exact-slice transform's operand slicing, eight neighbouring rows per block,
where a band ends inside the matrix and where a vector's magnitude leaves the
range of the integer form (tiny, zero and huge rows go through float pairs).

Tolerance: operands carry 42 bits below each row's largest entry, so with C
orthogonal an element is off by at most N (2^-42 + 2^-45) of the product of the
two rows' scales (twice their largest entries) per product, two products; the
tests allow 8 N^2 2^-42 of the vector's largest entry.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("N,o", [(3, 1), (8, 3), (9, 4), (31, 6), (100, 20), (257, 30)])
def test_transform_of_mixed_magnitudes(N, o):
    rng = np.random.default_rng(N)
    scales = np.array([1.0, 0.0, 1e-30, 1e20, 3e-7, 1.0, 1e-120])
    L = rng.standard_normal((len(scales), N * (N + 1) // 2)) * scales[:, None]
    L[5] *= np.exp(-rng.uniform(0, 60, L.shape[1]))      # a wide range inside one vector
    C = np.linalg.qr(rng.standard_normal((N, N)))[0]
    orbs = np.array([0, N - 1], dtype=np.int32)
    d = [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (L, C, orbs)]
    Lov, Lp = G.cds_cd_to_mo(d[0], d[1], o, d[2], precision="ozaki")
    il = np.tril_indices(N)
    for k in range(len(scales)):
        A = np.zeros((N, N))
        A[il] = L[k]
        A[il[1], il[0]] = L[k]
        tol = 8 * N * N * 2.0 ** -42 * np.abs(L[k]).max()
        if scales[k] == 1e-120:      # below the float range: no more than its own size
            tol = N * N * np.abs(L[k]).max()
        np.testing.assert_allclose(Lov[:, :, k].cpu().numpy(), C[:, :o].T @ A @ C[:, o:], rtol=0, atol=tol)
        np.testing.assert_allclose(Lp[:, :, k].cpu().numpy(), C[:, orbs].T @ A @ C, rtol=0, atol=tol)
