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


@pytest.fixture
def timeouts():
    """Lets the next n products of this thread's orbital steps end as if a wait had run out."""
    import ctypes
    import paper_2004_06142_gb300.binding as bd
    f = bd.lib().donof_testing_orbital_timeouts
    f.argtypes, f.restype = [ctypes.c_int32], ctypes.c_int
    yield lambda n: f(n)
    f(0)


@pytest.mark.parametrize("given", [True, False])
def test_timed_out_wait_of_the_loop_is_reported(optimize, timeouts, given):
    import paper_2004_06142_gb300.binding as bd
    good = optimize(24, 96, 5, 1, fill=0, given=given)
    timeouts(1)  # the first product, which comes before an eigendecomposition with a given diagonal
    with pytest.raises(bd.DonofError) as e:
        optimize(24, 96, 5, 1, fill=0, given=given)
    assert e.value.code == -6
    for a, b in zip(good, optimize(24, 96, 5, 1, fill=0, given=given)):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("nbf", [5, 140])
def test_timed_out_wait_of_the_update_leaves_nan(timeouts, nbf):
    import torch
    import paper_2004_06142_gb300.binding as bd
    rng = np.random.default_rng(nbf)
    C = to_dev(np.linalg.qr(rng.standard_normal((nbf, nbf)))[0])
    lam, F = to_dev(rng.standard_normal((nbf, nbf))), to_dev(rng.standard_normal(nbf))

    def update():
        C_new, eps = torch.zeros_like(C), torch.zeros_like(F)
        bd.donof_orbital_update(lam, F, C, C_new, eps)
        return C_new.cpu().numpy(), eps.cpu().numpy()

    good = update()
    for product in (1, 2, 3):  # C V, T^T T, T M
        timeouts(product)
        assert all(np.isnan(x).all() for x in update())
        timeouts(0)
    for a, b in zip(good, update()):
        assert np.isfinite(a).all()
        np.testing.assert_array_equal(a, b)
