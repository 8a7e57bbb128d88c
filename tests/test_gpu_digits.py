"""Double products by exact digit products on the tensor cores (csrc/digits.cu), against the
same products in extended precision.

Derived error bound.  With |a| < 2^EA over a row and |b| < 2^EB over a column, an element is
represented to 2^-57 of its bound (truncation), so a product of two loses at most
2 * 2^-57 * 2^(EA + EB); the digit products left out (i + j >= 8, digits of at most 64 units of
2^(49 - 7 i) of 57 bits) add less than 2^-57 * 2^(EA + EB); the sum is exact and rounded once:

    |error| <= K 2^-55 2^(EA + EB) + 2^-52 |c|

(2^-52: half an ulp, doubled for the truncation of the sum to 62 bits before the rounding).
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def product():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2004_06142_gb300.build as b
    b.build()
    import paper_2004_06142_gb300.binding as bd
    L = bd.lib()
    vp, i64, i32 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int32
    L.donof_testing_digit_product.argtypes = [vp, i64, i64, vp, i64, vp, i64, i32, i32, i32, vp,
                                              ctypes.c_size_t, vp]

    def run(A, B, k_contiguous, pad=0):
        """A (M x K) stored with k or m contiguous, rows `pad` elements further apart."""
        M, K = A.shape
        N = B.shape[1]
        S = A if k_contiguous else A.T
        st = np.zeros((S.shape[0], S.shape[1] + pad))
        st[:, :S.shape[1]] = S
        bs = np.zeros((K, N + pad))
        bs[:, :N] = B
        dA, dB = torch.from_numpy(st).cuda(), torch.from_numpy(bs).cuda()
        dC = torch.full((M, N + pad), np.nan, dtype=torch.float64, device="cuda")
        nb = 4096 + 4 * (M + N) + 16 * (N + 64) * (K + 32)
        ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        ld = S.shape[1] + pad
        rc = L.donof_testing_digit_product(
            dA.data_ptr(), *((ld, 1) if k_contiguous else (1, ld)), dB.data_ptr(), N + pad,
            dC.data_ptr(), N + pad, M, N, K, ws.data_ptr(), nb,
            torch.cuda.current_stream().cuda_stream)
        assert rc == 0
        torch.cuda.synchronize()
        assert ws[:4].view(torch.int32).item() == 0
        out = dC.cpu().numpy()
        assert np.isnan(out[:, N:]).all()  # nothing written past the columns
        return out[:, :N]

    return run


def _check(C, A, B):
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    ea = np.frexp(np.abs(A).max(1))[1].astype(float)
    eb = np.frexp(np.abs(B).max(0))[1].astype(float)
    bound = A.shape[1] * 2.0 ** -55 * 2.0 ** (ea[:, None] + eb[None, :]) + 2.0 ** -52 * np.abs(ref)
    err = np.abs(C - ref)
    assert (err <= bound).all(), float((err / np.where(bound > 0, bound, 1)).max())


# edges of the 128-row and 16..64-column tiles, of the 32-wide stages and the 256-wide chunks
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (5, 3, 7), (127, 16, 31), (128, 17, 32),
                                   (129, 48, 33), (257, 64, 255), (130, 65, 256), (64, 80, 257),
                                   (300, 130, 512), (131, 150, 1201)])
@pytest.mark.parametrize("k_contiguous,pad", [(True, 0), (True, 1), (False, 0), (False, 3)])
def test_against_extended_precision(product, M, N, K, k_contiguous, pad):
    rng = np.random.default_rng(M * 7 + N * 3 + K + pad)
    A = rng.standard_normal((M, K)) * 10.0 ** rng.uniform(-6, 6, (M, 1))
    A *= np.exp(-rng.uniform(0, 30, (M, K)))
    B = rng.standard_normal((K, N)) * 10.0 ** rng.uniform(-6, 6, (1, N))
    _check(product(A, B, k_contiguous, pad), A, B)


@pytest.mark.parametrize("K", [256, 511, 4096])
def test_coherent_digits_accumulate_exactly(product, K):
    # every element just below a power of two, all products of one sign: the largest partial
    # sums there are; and integers, whose products are exact in double
    v = np.nextafter(2.0, 0.0)
    A, B = np.full((130, K), v), np.full((K, 20), -v)
    _check(product(A, B, True), A, B)
    rng = np.random.default_rng(K)
    Ai = rng.integers(-1 << 20, 1 << 20, (130, K)).astype(np.float64)
    Bi = rng.integers(-1 << 19, 1 << 19, (K, 20)).astype(np.float64)
    np.testing.assert_array_equal(product(Ai, Bi, False), Ai @ Bi)


def test_zeros_extremes_and_non_finite(product):
    rng = np.random.default_rng(3)
    A, B = rng.standard_normal((140, 70)), rng.standard_normal((70, 33))
    A[3] = 0.0
    B[:, 5] = 0.0
    A[7] *= 1e200
    B[:, 6] *= 1e120     # row 7 x column 6 overflows
    A[8] *= 1e-200
    B[:, 8] *= 1e-120    # row 8 x column 8 underflows
    A[9, 4], A[10, 4] = np.nan, np.inf
    B[2, 9] = -np.inf
    with np.errstate(all="ignore"):
        C = product(A, B, True)
    assert (C[3, np.arange(33) != 9] == 0).all() and (C[np.arange(140) > 10][:, 5] == 0).all()
    assert np.isinf(C[7, 6]) and C[8, 8] == 0
    assert np.isnan(C[9]).all() and np.isnan(C[10]).all() and np.isnan(C[:, 9]).all()
    ok = [i for i in range(140) if i not in (7, 8, 9, 10)]
    cols = [j for j in range(33) if j not in (6, 8, 9)]
    _check(C[np.ix_(ok, cols)], A[ok], B[:, cols])


@pytest.mark.parametrize("kc", [True, False])
@pytest.mark.parametrize("N,K", [(64, 33), (120, 120), (80, 300), (33, 64), (200, 32), (49, 600)])
def test_result_does_not_depend_on_the_tiles(product, N, K, kc):
    """A product's sums are exact up to one rounding, so the rows of a tall product (wide tiles) are
    those of a short one of the same rows (tiles of a divisor of the width), bit for bit."""
    rng = np.random.default_rng(N + K)
    A = rng.standard_normal((128 * 160, K))
    B = rng.standard_normal((K, N))
    tall = product(A, B, kc)
    for rows in (1, 130):
        np.testing.assert_array_equal(tall[:rows], product(A[:rows], B, kc))


@pytest.mark.parametrize("nbf,naux,npair,ncwo,packed,blocks", [
    (500, 300, 20, 3, False, 1),   # several row and column tiles, two chunks of k
    (97, 150, 4, 3, True, 3),      # packed slices, blocks of slices, odd sizes
    (24, 96, 5, 1, False, 1), (16, 2, 8, 1, False, 1)])
def test_fp64_build_error_is_that_of_double(nbf, naux, npair, ncwo, packed, blocks):
    """The whole FP64 build against the oracle: within the differences that the oracle's own
    contraction order makes (an accumulated rounding of 1e-13 relative to |E| at most), two
    orders below the path's 1e-10 requirement."""
    import synth
    from oracle import pnof
    from helpers import gpu_build
    prob = synth.Problem(nbf, naux, npair, ncwo, seed=11)
    d = synth.generate(prob)
    ref = pnof.build(d["h"], d["B"], d["C"], d["gamma"], d["pair_map"], npair, ncwo, pnof.PNOF7)
    budget = naux * nbf * prob.nact * 16 // blocks if blocks > 1 else 0
    out = gpu_build(prob, d, 0, pnof.PNOF7, packed=packed, budget=budget)
    assert out["status"] == 0
    assert abs(out["E"] - ref["E"]) <= 1e-12 * abs(ref["E"])
    for k in ("lam", "dE_dgamma", "dE_dC", "J", "K"):
        scale = np.abs(ref[k]).max()
        assert np.abs(out[k] - ref[k]).max() <= 1e-12 * scale, k
