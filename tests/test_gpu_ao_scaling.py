"""The double path and the norms of the AO functions.

With B^P and h scaled by w_mu w_nu and C by 1 / w_nu the energy, J, K, lambda and dE/dgamma are the
same numbers and dE/dC is scaled by w.  The powers of two w change no rounding of a double
contraction, so the build's errors against the oracle's unscaled one stay those of an evenly scaled
build (1e-12 of the largest element, the bound of test_gpu_digits.py) whatever w spans; fixed point
relative to unscaled rows would lose up to 8 digits of 16 at a spread of 1e8."""
import numpy as np
import pytest

import synth
from oracle import pnof

from helpers import gpu_build, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()


def _norms(nbf, spread, order):
    """Powers of two from 10^(-spread / 2) to 10^(spread / 2)."""
    e = np.random.default_rng(nbf).uniform(-spread / 2, spread / 2, nbf)
    e[:2] = -spread / 2, spread / 2
    if order == "sorted":
        e.sort()
    return 2.0 ** np.rint(e * np.log2(10.0))


def _scaled(d, w):
    return dict(d, B=d["B"] * w[:, None] * w[None, :], h=d["h"] * w[:, None] * w[None, :],
                C=d["C"] / w[:, None])


def _oracle(d, npair, ncwo):
    return pnof.build(d["h"], d["B"], d["C"], d["gamma"], d["pair_map"], npair, ncwo, pnof.PNOF7)


def _check(out, ref, w, keys=("J", "K", "lam", "dE_dgamma", "dE_dC")):
    assert abs(out["E"] - ref["E"]) <= 1e-12 * abs(ref["E"])
    for k in keys:
        x = out[k] / w[:, None] if k == "dE_dC" else out[k]
        assert np.abs(x - ref[k]).max() <= 1e-12 * np.abs(ref[k]).max(), k


# below and above the size up to which exponents and digits are made in one launch; packed slices
# by rows and a CTA each; one block of slices and several
@pytest.mark.parametrize("nbf,naux,npair,ncwo,packed,blocks", [
    (24, 96, 5, 1, False, 1), (24, 96, 5, 1, True, 3), (97, 60, 4, 3, True, 1),
    (120, 300, 8, 4, False, 4), (161, 110, 3, 2, True, 1), (41, 703, 4, 2, True, 1),
    (320, 12, 6, 3, False, 1), (321, 12, 6, 3, True, 1), (700, 12, 6, 3, False, 1)])
@pytest.mark.parametrize("spread", [2, 8, 20])
@pytest.mark.parametrize("order", ["random", "sorted"])
def test_errors_do_not_depend_on_the_norms(nbf, naux, npair, ncwo, packed, blocks, spread, order):
    prob = synth.Problem(nbf, naux, npair, ncwo, seed=nbf)
    d = synth.generate(prob)
    w = _norms(nbf, spread, order)
    budget = naux * nbf * prob.nact * 16 // blocks if blocks > 1 else 0
    out = gpu_build(prob, _scaled(d, w), 0, pnof.PNOF7, packed=packed, budget=budget)
    assert out["status"] == 0
    _check(out, _oracle(d, npair, ncwo), w)


@pytest.mark.parametrize("packed", [False, True])
def test_functions_outside_B_and_odd_diagonals(packed):
    # functions without integrals in B (any scale), and slices without diagonals (the rows' largest
    # elements decide)
    prob = synth.Problem(64, 80, 5, 2, seed=2)
    d = synth.generate(prob)
    w = _norms(64, 8, "random")
    zero = dict(d, B=d["B"].copy())
    zero["B"][:, [0, 31, 63], :] = 0.0
    zero["B"][:, :, [0, 31, 63]] = 0.0
    bare = dict(d, B=d["B"] * (1.0 - np.eye(64)))
    for x in (zero, bare):
        out = gpu_build(prob, _scaled(x, w), 0, pnof.PNOF7, packed=packed)
        assert out["status"] == 0
        _check(out, _oracle(x, 5, 2), w)


def test_one_norm_for_all_changes_no_bit():
    prob = synth.Problem(50, 70, 5, 2, seed=4)
    d = synth.generate(prob)
    w = np.full(50, 2.0 ** -40)
    a = gpu_build(prob, d, 0, pnof.PNOF7)
    b = gpu_build(prob, _scaled(d, w), 0, pnof.PNOF7)
    for k in ("E", "J", "K", "lam", "dE_dgamma"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("nbf,naux", [(60, 50), (650, 9)])
def test_shards_and_their_finish(nbf, naux):
    """Two shards' partial sums, finished in a workspace that no B was prepared in."""
    import torch
    import paper_2004_06142_gb300 as dn
    prob = synth.Problem(nbf, naux, 5, 2, seed=7)
    d = synth.generate(prob)
    w = _norms(nbf, 8, "random")
    x = _scaled(d, w)
    h, C, g = to_dev(x["h"]), to_dev(x["C"]), to_dev(d["gamma"])
    pm = to_dev(d["pair_map"].astype(np.int32))
    total = 0.0
    for rank in range(2):
        p0, p1 = dn.shard_range(naux, rank, 2)
        b = dn.Builder(nbf, p1 - p0, 5, 2, pnof.PNOF7, dn.B_DENSE, dn.FP64)
        b.prepare(to_dev(x["B"][p0:p1]))
        total = total + b.forward_partial(h, C, g, pm)
        assert b.status() == 0
    b = dn.Builder(nbf, 1, 5, 2, pnof.PNOF7, dn.B_DENSE, dn.FP64)
    b.ws.fill_(0xFF)
    b.ws[:256] = 0  # the status words
    E, lam, dEdg = b.finish(h, C, g, pm, total)
    dC, _ = b.backward(torch.ones(1, dtype=torch.float64, device="cuda"))
    assert b.status() == 0
    out = dict(E=E.item(), lam=lam.cpu().numpy(), dE_dgamma=dEdg.cpu().numpy(), dE_dC=dC.cpu().numpy())
    _check(out, _oracle(d, 5, 2), w, keys=("lam", "dE_dgamma", "dE_dC"))
