"""The conversion of B at the ends of its ranges (csrc/tc.cu): slices whose rows' norms are too far
up for the scale of the sums to be bounded from them, beside the same slices further down.  A
common factor 2^56 of B changes no rounding of the mixed path (its fp32 parts stay normal), so J
and K are 2^112 times those of B itself, bit for bit; sizes of both storage forms, ragged rows and
tiles, both layouts, AO indices of different magnitude."""
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


@pytest.mark.parametrize("packed", [False, True])
@pytest.mark.parametrize("nbf,naux,npair,ncwo,spread", [
    (5, 3, 2, 1, 0), (37, 20, 4, 2, 3), (130, 9, 5, 2, 0), (257, 6, 5, 2, 2), (301, 9, 6, 3, 0),
    (390, 5, 6, 3, 3)])
def test_common_factor(nbf, naux, npair, ncwo, spread, packed):
    prob = synth.Problem(nbf, naux, npair, ncwo, seed=nbf)
    d = synth.generate(prob)
    w = 10.0 ** np.random.default_rng(nbf).uniform(-spread, 0, nbf)
    d["B"] = d["B"] * w[:, None] * w[None, :]
    low = gpu_build(prob, d, 1, pnof.PNOF7, packed=packed)
    high = gpu_build(prob, d, 1, pnof.PNOF7, packed=packed, B=d["B"] * 2.0 ** 56)
    assert low["status"] == 0 and high["status"] == 0
    for k in ("J", "K"):
        assert (low[k] != 0).any()
        np.testing.assert_array_equal(low[k] * 2.0 ** 112, high[k], err_msg=k)
