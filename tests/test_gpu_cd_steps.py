"""The tensor-core decomposition's in-kernel steps at the sizes where their
layout changes: one block of 512 pairs, two, one per SM, two side by side, more
than the SMs hold at once; with and without exact ties between residuals.

Against the FP64 decomposition: the pivots are equal (ties included: the lowest
index in the 1e-12 band on both sides) and the vectors agree to 1e-9, the
bound the projections' 56-bit slices and the float-pair sums are held to
elsewhere (2^-44 per operation, a few thousand of them, vectors up to 2).
"""
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


def basis(kind, atoms, ladder):
    if kind == "ring":      # equivalent centres: every residual has exact partners
        c = W.ring_centres(atoms, 0.4 * atoms)
    else:
        c = W.ball_centres(atoms, 1.5 * atoms ** (1.0 / 3.0) + 1.0, 0.7, np.random.default_rng(3))
    b = W.make_basis(c, W.geometric_exponents(0.15, 6.0, ladder))
    return dev(b.xyz), dev(b.alpha), dev(b.atom.astype(np.int32))


@pytest.mark.parametrize("kind,atoms,ladder,delta", [
    ("ball", 6, 4, 1e-6),       # 300 pairs: one block
    ("ring", 6, 4, 1e-6),
    ("ball", 8, 4, 1e-6),       # 528 pairs: two blocks
    ("ring", 20, 6, 1e-4),      # 15 blocks
    ("ball", 40, 10, 1e-2),     # 157 blocks: two side by side
    ("ring", 48, 10, 1e-2),     # 226 blocks
    ("ball", 70, 10, 3e-2),     # 480 blocks: more than 3 x 152
])
def test_pivots_and_vectors_against_fp64(kind, atoms, ladder, delta):
    args = basis(kind, atoms, ladder)
    L, piv, D, _ = G.cds_cd_decompose(*args, delta, "full", max_rank=min(1024, G.npair(atoms * ladder)),
                                      precision="ozaki")
    Lr, pr, Dr, _ = G.cds_cd_decompose(*args, delta, "full", max_rank=min(1024, G.npair(atoms * ladder)),
                                       precision="fp64")
    assert torch.equal(piv, pr)
    assert (L - Lr).abs().max().item() <= 1e-9
    assert (D - Dr).abs().max().item() <= 1e-9


def test_rank_cap_inside_a_pass():
    args = basis("ball", 20, 6)
    Lr, pr, _, _ = G.cds_cd_decompose(*args, 1e-6, "full", precision="fp64")
    L = torch.empty((11, Lr.shape[1]), dtype=torch.float64, device=DEV)
    with pytest.raises(G.CdsError) as ei:
        G.cds_cd_decompose(*args, 1e-6, "full", max_rank=11, L_out=L, precision="ozaki")
    assert ei.value.status == 4
    assert (L - Lr[:11]).abs().max().item() <= 1e-9
