"""The batched FP64 decomposition in several waves: molecules of uneven size side by
side, larger ones alone with one, two and three pairs per thread, one pair only; and a
batch that holds a molecule too large for the one-launch form.

Against a launch per step for the whole batch (a workspace without the region of the
one-launch form): equal ranks and pivots, vectors and residuals to 1e-11, as two FP64
forms of sums of K <= 200 products of vectors (|L| <= 2) divided by sqrt(D_P) >= 1e-1;
and the single-molecule call bit for bit."""
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


def basis(nbf, seed):
    ladder = 14 if nbf > 99 else 4
    atoms = -(-nbf // ladder)
    c = W.ball_centres(atoms, 1.5 * atoms ** (1.0 / 3.0) + 1.0, 0.7, np.random.default_rng(seed))
    b = W.make_basis(c, W.geometric_exponents(0.15, 6.0, ladder))
    return b.xyz[:nbf], b.alpha[:nbf], b.atom[:nbf].astype(np.int32)


@pytest.mark.parametrize("sizes", [
    (24, 240, 1, 300, 99, 240, 7, 395),      # four waves: three, two, one pair per thread, uneven sharing
    (7, 7, 7),
    (24, 484, 99),                           # 117,370 pairs: a launch per step for all
])
@pytest.mark.parametrize("scheme", ["full", "atomic"])
def test_waves(sizes, scheme):
    mols = [(n, max(1, n // 5), 1, 1, min(G.npair(n), 200)) for n in sizes]
    parts = [basis(n, i) for i, n in enumerate(sizes)]
    flat = [dev(np.concatenate([x[k].ravel() for x in parts])) for k in range(3)]
    lib = G.load()
    out = []
    for region in (True, False):
        b = G.cdsigma.Batch(mols, DEV, "bf16x3")
        if not region:
            small = lib.cds_batch_workspace_bytes(len(mols), b.mols, G.cdsigma.PRECISIONS["bf16x3"])
            assert small < b.ws.numel() or 484 in sizes
            b.ws = b.ws[:small]
        b.L.zero_()
        b.piv.zero_()
        ranks = b.cd_decompose(*flat, 5e-2, scheme)
        out.append((list(ranks), b))
    (r, b), (r0, b0) = out
    assert r == r0 and torch.equal(b.piv, b0.piv)
    assert (b.L - b0.L).abs().max().item() <= 1e-11
    assert (b.D - b0.D).abs().max().item() <= 1e-11
    if 484 in sizes:
        return
    for i, (x, m) in enumerate(zip(parts, mols)):
        L, piv, D, _ = G.cds_cd_decompose(dev(x[0]), dev(x[1]), dev(x[2]), 5e-2, scheme, max_rank=m[4])
        assert r[i] == L.shape[0]
        assert torch.equal(b.view("L", i, (m[4], G.npair(m[0])))[:r[i]], L)
        assert torch.equal(b.view("piv", i, (m[4],))[:r[i]], piv)
