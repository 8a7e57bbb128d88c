"""The double build on the FP64 pipe (strided DGEMMs, k_jk, k_build_Y), which carries it where its
workspace has no room for digit products: against the oracle at 1e-10, over blocks of slices, dense
and packed, few orbitals and many."""
import ctypes

import numpy as np
import pytest

import synth
from oracle import pnof

from helpers import gpu_build, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [  # nbf, naux, npair, ncwo, packed, x_budget_bytes
    (7, 5, 3, 1, False, 4864), (6, 5, 3, 1, True, 5888),
    (22, 1560, 1, 1, False, 65536),    # 10 blocks
    (9, 1251, 1, 1, True, 8192),       # 139 blocks
    (46, 999, 1, 1, False, 4096),      # 200 blocks
    (737, 1, 120, 5, False, 0),        # one slice, wide: every tile of the DGEMMs, split sums
    (724, 1, 362, 1, False, 0), (709, 1, 353, 1, True, 0)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()


def _on_the_pipe(nbf, naux, npair, ncwo, packed, budget):
    from paper_2004_06142_gb300 import binding as bd
    prob = bd.make_problem(nbf, naux, npair, ncwo, b_layout=int(packed), x_budget_bytes=budget)
    digits = ctypes.c_int32(-1)
    assert bd.lib().donof_testing_fp64_digits(ctypes.byref(prob), ctypes.byref(digits)) == 0
    return digits.value == 0


def _check(out, ref, keys=("lam", "dE_dgamma", "dE_dC", "J", "K")):
    assert abs(out["E"] - ref["E"]) <= 1e-10 * max(1.0, abs(ref["E"]))
    for k in keys:
        assert np.abs(out[k] - ref[k]).max() <= 1e-10 * np.abs(ref[k]).max(), k


@pytest.mark.parametrize("nbf,naux,npair,ncwo,packed,budget", SHAPES)
@pytest.mark.parametrize("functional", [pnof.PNOF7, pnof.PNOF7S])
def test_build_on_the_fp64_pipe(nbf, naux, npair, ncwo, packed, budget, functional):
    assert _on_the_pipe(nbf, naux, npair, ncwo, packed, budget)
    prob = synth.Problem(nbf, naux, npair, ncwo, seed=nbf)
    d = synth.generate(prob)
    ref = pnof.build(d["h"], d["B"], d["C"], d["gamma"], d["pair_map"], npair, ncwo, functional)
    out = gpu_build(prob, d, 0, functional, packed=packed, budget=budget)
    assert out["status"] == 0
    _check(out, ref)


def test_shards_and_finish_on_the_fp64_pipe():
    import torch
    import paper_2004_06142_gb300 as dn
    nbf, naux, npair, budget = 22, 3120, 1, 65536
    prob = synth.Problem(nbf, naux, npair, 1, seed=1)
    d = synth.generate(prob)
    h, C, g = to_dev(d["h"]), to_dev(d["C"]), to_dev(d["gamma"])
    pm = to_dev(d["pair_map"].astype(np.int32))
    total = 0.0
    for rank in range(2):
        p0, p1 = dn.shard_range(naux, rank, 2)
        assert _on_the_pipe(nbf, p1 - p0, npair, 1, False, budget)
        b = dn.Builder(nbf, p1 - p0, npair, 1, pnof.PNOF7, dn.B_DENSE, dn.FP64, budget)
        b.prepare(to_dev(d["B"][p0:p1]))
        total = total + b.forward_partial(h, C, g, pm)
    E, lam, dEdg = b.finish(h, C, g, pm, total)
    dC, _ = b.backward(torch.ones(1, dtype=torch.float64, device="cuda"))
    J, K = b.jk()
    assert b.status() == 0
    ref = pnof.build(d["h"], d["B"], d["C"], d["gamma"], d["pair_map"], npair, 1, pnof.PNOF7)
    _check(dict(E=E.item(), lam=lam.cpu().numpy(), dE_dgamma=dEdg.cpu().numpy(),
                dE_dC=dC.cpu().numpy(), J=J.cpu().numpy(), K=K.cpu().numpy()), ref)


def test_non_finite_C_on_the_fp64_pipe():
    nbf, naux, npair, ncwo, packed, budget = SHAPES[2]
    prob = synth.Problem(nbf, naux, npair, ncwo, seed=3)
    d = synth.generate(prob)
    d["C"][4, 1] = np.nan
    assert gpu_build(prob, d, 0, pnof.PNOF7, budget=budget)["status"] == -3
