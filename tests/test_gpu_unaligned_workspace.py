"""Workspaces that start on an 8-byte boundary: nothing asks the caller for more than
the alignment of a double.  The results are those of an aligned workspace, bit for bit."""
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
FP64 = 0


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def p(t):
    return ctypes.c_void_p(t.data_ptr())


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def shifted(need, shift):
    return torch.empty(need + 64, dtype=torch.uint8, device=DEV)[shift:shift + need]


def ball(atoms, ladder):
    c = W.ball_centres(atoms, 1.5 * atoms ** (1.0 / 3.0) + 1.0, 0.7, np.random.default_rng(5))
    return W.make_basis(c, W.geometric_exponents(0.15, 6.0, ladder))


@pytest.mark.parametrize("shift", [8, 24])
def test_decomposition(shift):
    b, lib, cap = ball(6, 10), G.load(), 200
    n = b.nbf
    a = [dev(b.xyz), dev(b.alpha), dev(b.atom.astype(np.int32))]
    out = []
    for s in (0, shift):
        ws = shifted(lib.cds_cd_workspace_bytes_prec(n, cap, FP64), s)
        L = torch.zeros((cap, G.npair(n)), dtype=torch.float64, device=DEV)
        piv = torch.zeros(cap, dtype=torch.int32, device=DEV)
        D = torch.empty(G.npair(n), dtype=torch.float64, device=DEV)
        M = ctypes.c_int32(0)
        assert lib.cds_cd_decompose(n, p(a[0]), p(a[1]), p(a[2]), 1e-4, 0, cap, FP64, p(L), p(piv), p(D),
                                    ctypes.byref(M), None, p(ws), ws.numel(), stream()) == 0
        out.append((M.value, L, piv, D))
    assert out[0][0] == out[1][0] and all(torch.equal(x, y) for x, y in zip(out[0][1:], out[1][1:]))


def test_batch_decomposition():
    bs = [ball(k, 6) for k in (3, 5, 9)]
    mols = [(b.nbf, 4, 2, 4, min(G.npair(b.nbf), 400)) for b in bs]
    xyz = dev(np.concatenate([b.xyz.ravel() for b in bs]))
    al = dev(np.concatenate([b.alpha for b in bs]))
    at = dev(np.concatenate([b.atom for b in bs]).astype(np.int32))
    out = []
    for s in (0, 8):
        batch = G.cdsigma.Batch(mols, DEV, "bf16x3", cd_precision="fp64")
        batch.ws = shifted(batch.ws.numel(), s)
        batch.L.zero_()
        batch.piv.zero_()
        ranks = batch.cd_decompose(xyz, al, at, 1e-4)
        out.append((list(ranks), batch.L.clone(), batch.piv.clone(), batch.D.clone()))
    assert out[0][0] == out[1][0] and all(torch.equal(x, y) for x, y in zip(out[0][1:], out[1][1:]))


@pytest.mark.parametrize("N", [70, 260])
def test_transform(N):
    rng, lib, M, o = np.random.default_rng(1), G.load(), 5, 13
    L, C = dev(rng.standard_normal((M, G.npair(N)))), dev(np.linalg.qr(rng.standard_normal((N, N)))[0])
    orb = dev(np.array([2, 40], dtype=np.int32))
    out = []
    for s in (0, 8):
        ws = shifted(lib.cds_cd_to_mo_workspace_bytes(N, N, o, M, 2), s)
        Lov = torch.empty((o, N - o, M), dtype=torch.float64, device=DEV)
        Lp = torch.empty((2, N, M), dtype=torch.float64, device=DEV)
        assert lib.cds_cd_to_mo(N, N, o, M, p(L), p(C), p(orb), 2, FP64, p(Lov), p(Lp), p(ws), ws.numel(),
                                stream()) == 0
        out.append((Lov, Lp))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_self_energy_and_mp2():
    rng, lib = np.random.default_rng(2), G.load()
    o, v, M, n, nE = 20, 50, 40, 2, 12
    Lov = dev(0.05 * rng.standard_normal((o, v, M)))
    Lp = dev(0.05 * rng.standard_normal((n, o + v, M)))
    eps = dev(np.concatenate([np.sort(rng.uniform(-1.5, -0.3, o)), np.sort(rng.uniform(0.05, 3.0, v))]))
    E = dev(np.array([-0.3, 0.05])[:, None] + np.linspace(-0.1, 0.1, nE))
    out = []
    for s in (0, 8):
        ws = shifted(lib.cds_sigma2_workspace_bytes(o + v, o, M, n, nE, FP64), s)
        sig, ds = torch.empty((2, n, nE), dtype=torch.float64, device=DEV)
        assert lib.cds_sigma2_diag(o + v, o, M, p(Lov), p(Lp), n, p(eps), p(E), nE, FP64, p(sig), p(ds), p(ws),
                                   ws.numel(), stream()) == 0
        ws = shifted(lib.cds_mp2_workspace_bytes(o + v, o, M, FP64), s)
        e, pair = torch.empty(1, dtype=torch.float64, device=DEV), torch.empty(o, dtype=torch.float64, device=DEV)
        assert lib.cds_mp2_energy(o + v, o, M, p(Lov), p(eps), FP64, p(pair), p(e), p(ws), ws.numel(),
                                  stream()) == 0
        out.append((sig, ds, e, pair))
    assert all(torch.equal(x, y) for x, y in zip(*out))
