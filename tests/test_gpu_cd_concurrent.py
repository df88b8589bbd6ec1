"""Two host threads, each on a stream of its own, decompose at the same time: both
cooperative launches want the whole device.  Every row that one CTA hands to another
has to arrive whole whatever runs beside it, so the results are those of the calls
alone, bit for bit, also when repeated."""
import threading

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


def basis(atoms, ladder, seed):
    c = W.ball_centres(atoms, 1.5 * atoms ** (1.0 / 3.0) + 1.0, 0.7, np.random.default_rng(seed))
    b = W.make_basis(c, W.geometric_exponents(0.15, 6.0, ladder))
    return dev(b.xyz), dev(b.alpha), dev(b.atom.astype(np.int32))


@pytest.mark.parametrize("forms", [("fp64", "fp64"), ("fp64", "ozaki"), ("ozaki", "ozaki")])
def test_two_threads(forms):
    mols = [basis(14, 10, 1), basis(20, 12, 2)]
    alone = [G.cds_cd_decompose(*m, 1e-4, max_rank=512, precision=f) for m, f in zip(mols, forms)]
    out, errors = [[], []], []

    def work(i):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(4):
                    L, piv, D, de = G.cds_cd_decompose(*mols[i], 1e-4, max_rank=512, precision=forms[i])
                    out[i].append((L.clone(), piv.clone(), D.clone(), de))
            s.synchronize()
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for ref, runs in zip(alone, out):
        for L, piv, D, de in runs:
            assert torch.equal(L, ref[0]) and torch.equal(piv, ref[1])
            assert torch.equal(D, ref[2]) and de == ref[3]
