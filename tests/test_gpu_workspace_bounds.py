"""Scratch of the FP64 self-energy, Newton, MP2 and transform: what the calls ask for is
bounded whatever the size of the molecule, and a smaller workspace takes the spectators
in panels (any number of them, the last one narrower), with the results of everything at once.

Tolerance: the integrals are the same numbers; the partial sums of a panel are added in
another order, 2^-53 of the magnitudes for each of at most 40 panels: 1e-13 of the largest
value of a smooth grid."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_0912_1459_gb300 as G  # noqa: E402

DEV = torch.device("cuda:0")
FP64, GB = 0, 1 << 30


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def p(t):
    return ctypes.c_void_p(t.data_ptr())


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("nmo,nocc,M", [(2000, 400, 2000), (4000, 800, 4000), (5000, 1000, 12000)])
def test_requests_are_bounded(nmo, nocc, M):
    lib = G.load()
    assert lib.cds_sigma2_workspace_bytes(nmo, nocc, M, 20, 64, FP64) <= 5 * GB
    assert lib.cds_qp_workspace_bytes(nmo, nocc, M, 20, FP64) <= 5 * GB
    assert lib.cds_mp2_workspace_bytes(nmo, nocc, M, FP64) <= 5 * GB
    # the transform: one size for all precisions, whose other forms hold batches of 32 vectors
    # of up to 16 bytes per element
    assert lib.cds_cd_to_mo_workspace_bytes(nmo, nmo, nocc, M, 20) <= max(5 * GB, 32 * 16 * nmo * (nmo + nocc + 20))


def factors(o, v, M, n):
    rng = np.random.default_rng(o)
    fall = 0.05 * np.exp(-np.arange(M) / (0.3 * M))
    eps = np.concatenate([np.sort(rng.uniform(-1.5, -0.3, o)), np.sort(rng.uniform(0.05, 3.0, v))])
    return (dev(rng.standard_normal((o, v, M)) * fall), dev(rng.standard_normal((n, o + v, M)) * fall), dev(eps))


# spectators per panel follow from the workspace: shares of what lies between the fixed
# part and everything at once
def test_a_workspace_without_room_is_refused():
    lib = G.load()
    Lov, Lp, eps = factors(20, 50, 8, 2)
    orb = dev(np.array([18, 19], dtype=np.int32))
    w, it = torch.empty((2, 2), dtype=torch.float64, device=DEV), torch.empty((2, 2), dtype=torch.int32, device=DEV)
    e = torch.empty(21, dtype=torch.float64, device=DEV)
    ws = torch.empty(4096, dtype=torch.uint8, device=DEV)
    for have in (0, 1, 256, 1024):
        assert lib.cds_qp_solve(70, 20, 8, p(Lov), p(Lp), p(orb), 2, p(eps), 1e-5, 50, FP64, p(w[0]), p(w[1]),
                                p(it[0]), p(it[1]), p(ws), have, stream()) == 6
        assert lib.cds_mp2_energy(70, 20, 8, p(Lov), p(eps), FP64, p(e[1:]), p(e), p(ws), have, stream()) == 6
    E = eps[18:20].view(2, 1).contiguous()
    assert lib.cds_sigma2_diag(70, 20, 8, p(Lov), p(Lp), 2, p(eps), p(E), 1, FP64, p(w[0]), p(w[1]), p(ws), 1024,
                               stream()) == 6
    # no occupied orbital: no sums, but Newton's own arrays all the same
    assert lib.cds_qp_solve(70, 0, 8, None, p(Lp), p(orb), 2, p(eps), 1e-5, 50, FP64, p(w[0]), p(w[1]), p(it[0]),
                            p(it[1]), p(ws), 512, stream()) == 6


@pytest.mark.parametrize("o,v,M,n,nE", [(40, 200, 50, 3, 12), (33, 130, 17, 2, 1), (65, 140, 33, 2, 5),
                                        (70, 330, 20, 2, 70)])
def test_self_energy_in_panels(o, v, M, n, nE):
    lib, nmo = G.load(), o + v
    Lov, Lp, eps = factors(o, v, M, n)
    q = np.arange(o - 1, o - 1 + n)
    E = eps[dev(q)][:, None] + dev(np.linspace(-0.05, 0.05, nE))[None, :]
    full = lib.cds_sigma2_workspace_bytes(nmo, o, M, n, nE, FP64)
    nc = lib.cds_sigma2_cache_bytes(nmo, o, n, FP64)
    out = []
    for share in (1.0, 0.8, 0.3, 0.2):
        ws = torch.empty(int(full * share), dtype=torch.uint8, device=DEV)
        cache = torch.zeros(nc // 8, dtype=torch.float64, device=DEV)
        s, ds = torch.empty((2, n, nE), dtype=torch.float64, device=DEV)
        assert lib.cds_sigma2_diag_cache(nmo, o, M, p(Lov), p(Lp), n, p(eps), p(E), nE, FP64, p(s), p(ds),
                                         p(cache), nc, p(ws), ws.numel(), stream()) == 0
        need = lib.cds_qp_workspace_bytes(nmo, o, M, n, FP64)
        wq = torch.empty(int(need * share), dtype=torch.uint8, device=DEV)
        w = torch.empty((2, n), dtype=torch.float64, device=DEV)
        it = torch.empty((2, n), dtype=torch.int32, device=DEV)
        assert lib.cds_qp_solve(nmo, o, M, p(Lov), p(Lp), p(dev(q.astype(np.int32))), n, p(eps), 1e-8, 50, FP64,
                                p(w[0]), p(w[1]), p(it[0]), p(it[1]), p(wq), wq.numel(), stream()) == 0
        out.append((s, ds, cache, w))
    s0, ds0, cache0, w0 = out[0]
    for s, ds, cache, w in out[1:]:
        assert (s - s0).abs().max() <= 1e-13 * s0.abs().max()
        assert (ds - ds0).abs().max() <= 1e-13 * ds0.abs().max()
        assert torch.equal(cache, cache0)
        assert (w - w0).abs().max() <= 1e-12


@pytest.mark.parametrize("o,v,M,shares", [(40, 100, 30, (0.7, 0.06, 0.04, 0.015)), (33, 65, 17, (0.5, 0.06, 0.04))])
def test_mp2_in_panels(o, v, M, shares):
    lib = G.load()
    Lov, _, eps = factors(o, v, M, 1)
    full = lib.cds_mp2_workspace_bytes(o + v, o, M, FP64)
    ref = None
    for share in (1.0,) + shares:
        ws = torch.empty(int(full * share), dtype=torch.uint8, device=DEV)
        e, pair = torch.empty(1, dtype=torch.float64, device=DEV), torch.empty(o, dtype=torch.float64, device=DEV)
        assert lib.cds_mp2_energy(o + v, o, M, p(Lov), p(eps), FP64, p(pair), p(e), p(ws), ws.numel(),
                                  stream()) == 0
        ref = pair if ref is None else ref
        assert (pair - ref).abs().max() <= 1e-13 * ref.abs().max()


def test_the_most_pairs_of_orbitals():
    """o v = 1023 x 4100, just below 2^22: against the fused kernel (the least workspace)."""
    o, v, M = 1023, 4100, 1
    lib, nmo = G.load(), o + v
    Lov, Lp, eps = factors(o, v, M, 1)
    E = eps[o - 1:o].view(1, 1) + 0.2
    items = v * 33 * 32 // 2 + o * 130 * 129 // 2
    out = []
    for size in (lib.cds_sigma2_workspace_bytes(nmo, o, M, 1, 1, FP64), items * 16 + 1024):
        ws = torch.empty(size, dtype=torch.uint8, device=DEV)
        s, ds = torch.empty((2, 1, 1), dtype=torch.float64, device=DEV)
        assert lib.cds_sigma2_diag(nmo, o, M, p(Lov), p(Lp), 1, p(eps), p(E), 1, FP64, p(s), p(ds), p(ws),
                                   ws.numel(), stream()) == 0
        out.append((s, ds))
    assert abs((out[0][0] / out[1][0]).item() - 1) <= 1e-10
    assert abs((out[0][1] / out[1][1]).item() - 1) <= 1e-10
