"""The conversion of B (donof_prepare_B, mixed precision).  Dense and packed slices take different
passes (a warp per row; a warp per stored row with partial column sums), which must find the same
scales and planes: the builds agree bit for bit, over sizes at the edges of the passes' warps and
of the 64- and 128-wide storage tiles, with slices and AO indices of very different magnitude and
a slice of zeros.  (The mixed path's accuracy is test_gpu_parity.py's subject.)"""
import numpy as np
import pytest

import synth
from oracle import pnof

from helpers import gpu_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()


@pytest.mark.parametrize("nbf,naux,npair,ncwo", [
    (4, 1, 2, 1), (8, 3, 2, 2), (31, 5, 3, 2), (33, 160, 4, 1), (255, 7, 5, 2), (256, 6, 5, 2),
    (257, 6, 5, 2), (301, 9, 6, 3), (385, 5, 6, 3)])
@pytest.mark.parametrize("uneven", [False, True])
def test_dense_and_packed_agree(nbf, naux, npair, ncwo, uneven):
    prob = synth.Problem(nbf, naux, npair, ncwo, seed=nbf)
    d = synth.generate(prob)
    if uneven:
        rng = np.random.default_rng(nbf)
        w = 10.0 ** rng.uniform(-4, 0, nbf)
        d["B"] = d["B"] * w[:, None] * w[None, :] * (10.0 ** rng.uniform(-12, 0, naux))[:, None, None]
        if naux > 2:
            d["B"][1] = 0.0
    dense = gpu_build(prob, d, 1, pnof.PNOF7)
    packed = gpu_build(prob, d, 1, pnof.PNOF7, packed=True)
    assert dense["status"] == 0 and packed["status"] == 0
    for k in ("E", "lam", "dE_dgamma", "dE_dC"):
        np.testing.assert_array_equal(dense[k], packed[k], err_msg=k)


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_B_is_reported(packed, bad):
    prob = synth.Problem(40, 12, 3, 2, seed=1)
    d = synth.generate(prob)
    d["B"][5, 7, 3] = d["B"][5, 3, 7] = bad
    assert gpu_build(prob, d, 1, pnof.PNOF7, packed=packed)["status"] == -3
