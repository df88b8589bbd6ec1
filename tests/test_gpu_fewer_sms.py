"""Decompositions on a stream with fewer SMs than the device (a green context): the
cooperative launches have to fit those, or leave the call to the launch-per-step form.

FP64: against the whole device's results as two FP64 forms, 1e-11 (|L| <= 2, K <= 200
vectors, sqrt(D_P) >= 1e-2).  Tensor-core form: the same bits, its sums do not depend on
which CTA forms them."""
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
SM = 1                                    # CU_DEV_RESOURCE_TYPE_SM


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.fixture
def few():
    """A stream on 16 or so SMs."""
    torch.zeros(1, device=DEV)            # the primary context
    cu = ctypes.CDLL("libcuda.so.1")
    device, n = ctypes.c_int(0), ctypes.c_uint(1)
    res, part, rest = (ctypes.create_string_buffer(512) for _ in range(3))
    desc, ctx, stream = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    try:
        steps = [lambda: cu.cuDeviceGet(ctypes.byref(device), torch.cuda.current_device()),
                 lambda: cu.cuDeviceGetDevResource(device, res, SM),
                 lambda: cu.cuDevSmResourceSplitByCount(part, ctypes.byref(n), res, rest, 0, 16),
                 lambda: cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
                 lambda: cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, device, 1),
                 lambda: cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, 1, 0)]
        for i, s in enumerate(steps):
            r = s()
            if r:
                pytest.skip(f"no green contexts here (step {i}: {r})")
    except AttributeError as e:
        pytest.skip(str(e))
    yield torch.cuda.ExternalStream(stream.value, device=DEV)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


def basis(atoms, ladder):
    c = W.ball_centres(atoms, 1.5 * atoms ** (1.0 / 3.0) + 1.0, 0.7, np.random.default_rng(5))
    return W.make_basis(c, W.geometric_exponents(0.15, 6.0, ladder))


def args(b):
    return dev(b.xyz), dev(b.alpha), dev(b.atom.astype(np.int32))


@pytest.mark.parametrize("precision,atoms", [("fp64", 4), ("fp64", 12), ("ozaki", 4), ("ozaki", 20)])
def test_decomposition(few, precision, atoms):
    a = args(basis(atoms, 10))
    ref = G.cds_cd_decompose(*a, 1e-2, max_rank=300, precision=precision)
    torch.cuda.synchronize()
    with torch.cuda.stream(few):
        L, piv, D, de = G.cds_cd_decompose(*a, 1e-2, max_rank=300, precision=precision)
    few.synchronize()
    assert torch.equal(piv, ref[1]) and de == ref[3]
    tol = 1e-11 if precision == "fp64" else 0.0
    assert (L - ref[0]).abs().max().item() <= tol
    assert (D - ref[2]).abs().max().item() <= tol


def test_batch(few):
    bs = [basis(k, 6) for k in (3, 8, 20, 5)]
    mols = [(b.nbf, 4, 2, 4, min(G.npair(b.nbf), 400)) for b in bs]
    flat = [dev(np.concatenate([x.ravel() for x in v])) for v in zip(
        *[(b.xyz, b.alpha, b.atom.astype(np.int32)) for b in bs])]
    out = []
    for s in (torch.cuda.current_stream(), few):
        with torch.cuda.stream(s):
            batch = G.cdsigma.Batch(mols, DEV, "bf16x3")
            batch.L.zero_()
            ranks = batch.cd_decompose(*flat, 1e-2)
            out.append((list(ranks), batch.L.clone(), batch.D.clone()))
        torch.cuda.synchronize()
    assert out[0][0] == out[1][0]
    assert (out[0][1] - out[1][1]).abs().max().item() <= 1e-11
    assert (out[0][2] - out[1][2]).abs().max().item() <= 1e-11
