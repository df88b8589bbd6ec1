"""The one-launch FP64 decomposition at the sizes where its layout changes: one
pair, one group of pairs, a last group that is nearly empty, one and several pairs
per thread, the largest that it serves and the first beyond; with and without exact
ties between residuals.

Against the launch-per-step form, which the same call takes when its workspace has no
room for the rows: equal pivots, vectors and residuals to 1e-11.  Both forms are FP64:
a sum of K products of vectors (|L| <= 2) is good to K 2^-53 x 4 in either, K <= 200,
divided by sqrt(D_P) >= 1e-2, i.e. 1e-11 at most.
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


def basis(kind, nbf, ladder):
    atoms = -(-nbf // ladder)
    if kind == "ring":      # equivalent centres: every residual has exact partners
        c = W.ring_centres(atoms, 0.4 * atoms)
    else:
        c = W.ball_centres(atoms, 1.5 * atoms ** (1.0 / 3.0) + 1.0, 0.7, np.random.default_rng(5))
    b = W.make_basis(c, W.geometric_exponents(0.15, 6.0, ladder))
    return dev(b.xyz[:nbf]), dev(b.alpha[:nbf]), dev(b.atom[:nbf].astype(np.int32))


def run(args, delta, cap, scheme, ws_bytes):
    n = args[1].shape[0]
    npr = G.npair(n)
    L = torch.full((max(cap, 1), npr), float("nan"), dtype=torch.float64, device=DEV)
    piv = torch.full((max(cap, 1),), -1, dtype=torch.int32, device=DEV)
    D = torch.empty(npr, dtype=torch.float64, device=DEV)
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device=DEV)
    M, de = ctypes.c_int32(0), ctypes.c_double(0.0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = G.load().cds_cd_decompose(n, p(args[0]), p(args[1]), p(args[2]), delta,
                                   G.cdsigma.SCHEMES[scheme], cap, G.cdsigma.PRECISIONS["fp64"], p(L),
                                   p(piv), p(D), ctypes.byref(M), ctypes.byref(de), p(ws), ws_bytes,
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    return st, M.value, de.value, L[:M.value], piv[:M.value], D


@pytest.mark.parametrize("kind,nbf,ladder,delta,cap,scheme", [
    ("ball", 1, 2, 1e-4, 4, "full"),          # one pair
    ("ball", 7, 4, 1e-4, 28, "full"),         # 28 pairs: one CTA
    ("ball", 8, 4, 1e-4, 36, "full"),         # 36: a second CTA of four pairs
    ("ring", 24, 4, 1e-4, 200, "full"),
    ("ball", 24, 4, 1e-4, 11, "full"),        # the rank cap stops it
    ("ball", 99, 9, 1e-3, 200, "atomic"),     # 4,950: two warps per CTA
    ("ring", 240, 12, 1e-2, 200, "full"),     # 28,920: 192 pairs per CTA
    ("ball", 278, 14, 1e-2, 200, "full"),     # 38,781: 256 pairs, one per thread
    ("ball", 279, 14, 1e-2, 200, "full"),     # 39,060: two per thread
    ("ball", 395, 14, 5e-2, 200, "full"),     # 78,210: three per thread
    ("ball", 482, 14, 5e-2, 60, "full"),      # 116,403: the largest
    ("ball", 484, 14, 5e-2, 60, "full"),      # beyond: a launch per step in both calls
])
def test_against_a_launch_per_step(kind, nbf, ladder, delta, cap, scheme):
    args = basis(kind, nbf, ladder)
    lib = G.load()
    need = lib.cds_cd_workspace_bytes_prec(nbf, cap, G.cdsigma.PRECISIONS["fp64"])
    st0, M0, de0, L0, p0, D0 = run(args, delta, cap, scheme,
                                   min(need, lib.cds_cd_workspace_bytes_prec(nbf, 0, G.cdsigma.PRECISIONS["fp64"])))
    st, M, de, L, p, D = run(args, delta, cap, scheme, need)
    assert (st, M, de) == (st0, M0, de0)
    assert torch.equal(p, p0)
    assert (L - L0).abs().max().item() <= 1e-11
    assert (D - D0).abs().max().item() <= 1e-11
