"""The exact-slice transform's products at the edges of their tiles: 320 summands is the
most that the accumulator of three pairs holds before it is emptied (one more, two, three
chunks, and the largest basis), tiles of 16 to 96 columns, and rows whose digits are all
at their largest, equal signs, so that every sum is as large as it can be.

Tolerance: operands carry 42 bits below each row's largest entry, so with |C| <= 1 an
element is off by at most N (2^-42 + 2^-45) of the product of the two rows' scales (twice
their largest entries) per product, two products, the first one's entries up to N times
larger: 8 N^2 2^-42 of the vector's largest entry, times the largest column sum of |C|
over its largest entry squared for the columns that are not orthogonal.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


def transform(L, C, o, orbs):
    d = [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in (L, C, orbs)]
    Lov, Lp = G.cds_cd_to_mo(d[0], d[1], o, d[2], precision="ozaki")
    N = C.shape[0]
    il = torch.tril_indices(N, N, device=DEV)
    ref = []
    for k in range(L.shape[0]):
        A = torch.zeros((N, N), dtype=torch.float64, device=DEV)
        A[il[0], il[1]] = d[0][k]
        A[il[1], il[0]] = d[0][k]
        ref.append(((Lov[:, :, k] - d[1][:, :o].T @ A @ d[1][:, o:]).abs().max().item(),
                    (Lp[:, :, k] - d[1][:, torch.from_numpy(orbs).long().to(DEV)].T @ A @ d[1]).abs().max().item()))
    return ref


@pytest.mark.parametrize("N,o,np_", [
    (319, 13, 3),      # one chunk; 16 rows of Cj, 306 columns in 4 tiles
    (320, 80, 16),     # one chunk, full; 96 rows of Cj: the widest tile
    (321, 81, 16),     # a second chunk of one; 97: two tiles
    (352, 30, 2),
    (641, 70, 4),      # three chunks
    (1040, 100, 1),    # the largest basis, four chunks
])
def test_tiles_against_fp64(N, o, np_):
    rng = np.random.default_rng(N)
    L = rng.standard_normal((3, N * (N + 1) // 2))
    L *= np.array([1.0, 1e-5, 1e4])[:, None]
    C = np.linalg.qr(rng.standard_normal((N, N)))[0]
    orbs = np.linspace(0, N - 1, np_).astype(np.int32)
    for k, (a, b) in enumerate(transform(L, C, o, orbs)):
        tol = 8 * N * N * 2.0 ** -42 * np.abs(L[k]).max()
        assert a <= tol and b <= tol


@pytest.mark.parametrize("N", [320, 337, 1040])
def test_largest_digits(N):
    """Every entry just below its row's scale: digits of 127, sums of one sign."""
    L = np.full((2, N * (N + 1) // 2), 1.0 - 2.0 ** -42)
    L[1] *= -1.0
    C = np.full((N, N), 1.0 - 2.0 ** -42)
    for a, b in transform(L, C, 8, np.array([0, N - 1], dtype=np.int32)):
        tol = 8 * N * N * 2.0 ** -42 * N
        assert a <= tol and b <= tol
