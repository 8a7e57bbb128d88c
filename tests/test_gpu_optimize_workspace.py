"""donof_optimize and what its workspace holds when it is called: the workspace is the caller's memory,
undefined on entry, so that a run from a given diagonal (whose first orbital step comes before any
eigendecomposition) gives the same bits whatever is in it."""
import numpy as np
import pytest

import synth
from oracle import pnof

from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()


@pytest.fixture
def optimize(monkeypatch):
    import torch
    import paper_2004_06142_gb300 as dn
    import paper_2004_06142_gb300.binding as bd
    alloc = bd.alloc_workspace

    def run(nbf, naux, npair, ncwo, fill, given=True):
        """(E, energies, C, gamma, diagonal) of a few iterations, every workspace filled."""
        monkeypatch.setattr(bd, "alloc_workspace", lambda n, dev: alloc(n, dev).fill_(fill))
        prob = synth.Problem(nbf, naux, npair, ncwo, seed=5)
        d = synth.generate(prob)
        b = dn.Builder(nbf, naux, npair, ncwo, pnof.PNOF7, dn.B_DENSE, dn.FP64)
        b.prepare(to_dev(d["B"]))
        C, g = to_dev(d["C"]).clone(), to_dev(d["gamma"]).clone()
        F = torch.linspace(9.0, -9.0, nbf, dtype=torch.float64, device="cuda") if given else None
        out, energies = b.optimize(to_dev(d["h"]), C, g, to_dev(d["pair_map"].astype(np.int32)),
                                   Fdiag=F, max_outer=2, max_inner=2)
        torch.cuda.synchronize()
        return [np.asarray(out["E"]), np.asarray(energies)] + [
            x.cpu().numpy() for x in (C, g, out["Fdiag"])]

    return run


@pytest.mark.parametrize("size", [(24, 96, 5, 1), (330, 60, 8, 4)])
def test_given_diagonal_whatever_the_workspace_holds(optimize, size):
    for a, b in zip(optimize(*size, fill=0), optimize(*size, fill=0xFF)):
        assert np.isfinite(a).all()
        np.testing.assert_array_equal(a, b)
