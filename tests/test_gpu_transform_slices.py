"""The FP64 transform where its forms change hands: FP64 units below 32
functions, FP64 first product and tensor-core second product up to 256,
tensor cores throughout above; ragged vectors, orbitals and tiles; no
requested orbitals, one occupied one; operands that are not finite.

Tolerance: with C orthogonal (no cancellation) two products of N terms carry
at most 2 (N + 4) roundings of 2^-53 relative to sum |C||A||C|, which is at most
N max|A| here; the tests allow 4 N 2^-53 N max|A|.
"""
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


def case(N, M, seed=0):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((M, N * (N + 1) // 2)), np.linalg.qr(rng.standard_normal((N, N)))[0]


def reference(L, C, o, orbs):
    N = C.shape[0]
    il = np.tril_indices(N)
    A = np.zeros((L.shape[0], N, N))
    A[:, il[0], il[1]] = L
    A[:, il[1], il[0]] = L
    return (np.einsum("mi,Kmn,na->iaK", C[:, :o], A, C[:, o:], optimize=True),
            np.einsum("mt,Kmn,nq->tqK", C[:, orbs], A, C, optimize=True))


@pytest.mark.parametrize("N,M,o,np_", [
    (31, 5, 7, 2), (32, 33, 8, 1), (33, 40, 1, 3), (65, 70, 64, 2), (130, 37, 21, 5),
    (256, 11, 40, 9), (257, 11, 40, 9), (300, 7, 129, 0), (300, 7, 30, 1), (272, 300, 5, 2),
])
def test_transform_against_reference(N, M, o, np_):
    L, C = case(N, M)
    orbs = np.linspace(0, N - 1, np_).astype(np.int32)
    Lov, Lp = G.cds_cd_to_mo(dev(L), dev(C), o, dev(orbs))
    rov, rp = reference(L, C, o, orbs)
    tol = 4 * N * 2.0 ** -53 * N * np.abs(L).max()
    np.testing.assert_allclose(Lov.cpu().numpy(), rov, rtol=0, atol=tol)
    np.testing.assert_allclose(Lp.cpu().numpy(), rp, rtol=0, atol=tol)


@pytest.mark.parametrize("N", [70, 260])
def test_non_finite_vector_touches_only_itself(N):
    L, C = case(N, 9)
    orbs = dev(np.array([1, 40], dtype=np.int32))
    a, b = G.cds_cd_to_mo(dev(L), dev(C), 20, orbs)
    L[3, 17] = np.inf
    c, d = G.cds_cd_to_mo(dev(L), dev(C), 20, orbs)
    keep = [k for k in range(9) if k != 3]
    assert not torch.isfinite(c[..., 3]).all() and not torch.isfinite(d[..., 3]).all()
    tol = 4 * N * 2.0 ** -53 * N * 6.0
    torch.testing.assert_close(c[..., keep], a[..., keep], rtol=0, atol=tol)
    torch.testing.assert_close(d[..., keep], b[..., keep], rtol=0, atol=tol)
