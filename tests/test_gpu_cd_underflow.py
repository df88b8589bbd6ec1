"""FP64 decomposition of pairs whose diagonal (rho_I|rho_I) underflows: two tight
functions on centres far apart.  Their vectors (1e-150 and less) are still FP64
numbers, and every form projects them like any other pair's.

Against the launch-per-step form.  Both are sums of K <= 150 products bounded by
sqrt(D0_I) sqrt(D0_P), sqrt(D0_P) <= 3, divided by sqrt(D_P) >= 3e-3: each good to K
2^-53 10^3 sqrt(D0_I), 2e-11 of it; the errors of the rows they are made from add up
over K steps, so 1e-8 sqrt(D0_I) is allowed.
"""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def diagonal_roots(b):
    """sqrt((rho_I|rho_I)) without forming the square."""
    nu, mu = np.tril_indices(b.nbf)
    a, c = b.alpha[mu], b.alpha[nu]
    p = a + c
    r2 = ((b.xyz[mu] - b.xyz[nu]) ** 2).sum(1)
    k = (2 * a / np.pi) ** 0.75 * (2 * c / np.pi) ** 0.75 * np.exp(-a * c / p * r2) / p
    return k * np.sqrt(2 * np.pi ** 2.5 / np.sqrt(2 * p))


@pytest.mark.parametrize("atoms,ladder,gap,cap", [(10, 6, 5.0, 150), (4, 4, 12.0, 60)])
def test_underflowing_pairs_are_projected(atoms, ladder, gap, cap):
    c = np.zeros((atoms, 3))
    c[:, 0] = gap * np.arange(atoms)
    b = W.make_basis(c, W.geometric_exponents(0.1, 10.0, ladder))
    args = [dev(b.xyz), dev(b.alpha), dev(b.atom.astype(np.int32))]
    lib, n = G.load(), b.nbf
    prec = G.cdsigma.PRECISIONS["fp64"]
    out = []
    for rank in (cap, 0):            # with room for the one-launch form, and without
        ws = torch.empty(lib.cds_cd_workspace_bytes_prec(n, rank, prec), dtype=torch.uint8, device=DEV)
        L = torch.zeros((cap, G.npair(n)), dtype=torch.float64, device=DEV)
        piv = torch.zeros(cap, dtype=torch.int32, device=DEV)
        D = torch.empty(G.npair(n), dtype=torch.float64, device=DEV)
        M, de = ctypes.c_int32(0), ctypes.c_double(0.0)
        p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        st = lib.cds_cd_decompose(n, p(args[0]), p(args[1]), p(args[2]), 1e-5, G.cdsigma.SCHEMES["full"],
                                  cap, prec, p(L), p(piv), p(D), ctypes.byref(M), ctypes.byref(de), p(ws),
                                  ws.numel(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        torch.cuda.synchronize()
        assert st == 0
        out.append((M.value, piv.cpu().numpy(), L.cpu().numpy()))
    (M, piv, L), (M0, piv0, L0) = out
    assert M == M0 and np.array_equal(piv, piv0)
    root = diagonal_roots(b)
    under = (root < 1e-155) & (root > 1e-290)
    assert under.sum() > 5 and np.abs(L0[:, under]).max() > 0
    assert np.all(np.abs(L - L0) <= 1e-8 * root[None, :] + 1e-300)
