"""The eigensolver's forms (csrc/eigh.cu) at the sizes where they change: the reduction in one
cluster of 1, 2, 4, 8 and 16 CTAs, on the whole grid from 129 on, with rows in registers up to 1216
and in memory beyond; reflector blocks of 64; eigenvalue brackets that hit zero minors exactly (a
path graph's adjacency matrix has the eigenvalue 0 and principal minors 0); blocks split by zero
couplings; repeated calls on one workspace.  Bounds: those of a backward-stable solver, as for the
solver's other tests: eigenvalues and residuals within 8 max(n, 8) eps ||A||."""
import numpy as np
import pytest

from test_gpu_eigh import _check, _eigh, _lib  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 4, 8, 9, 16, 17, 31, 32, 33, 63, 66, 127, 128, 129, 288, 289, 1216,
                               1217])
def test_sizes(n):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, n))
    w, V, st, ws = _eigh(X + X.T)
    assert st == 0
    _check(X + X.T, w, V)
    again = _eigh(X + X.T, ws)
    np.testing.assert_array_equal(w, again[0])
    np.testing.assert_array_equal(V, again[1])


@pytest.mark.parametrize("n", [9, 10, 17, 33, 65, 128, 129, 257])
def test_zero_minors(n):
    A = np.zeros((n, n))
    i = np.arange(n - 1)
    A[i, i + 1] = A[i + 1, i] = 1.0
    w, V, st, _ = _eigh(A)
    assert st == 0
    _check(A, w, V)


@pytest.mark.parametrize("n,cuts", [(40, (1, 2, 31, 32, 33)), (120, (64,)), (130, (5, 127, 128)),
                                    (300, (32, 64, 96, 250))])
def test_split_blocks(n, cuts):
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, n))
    A = X + X.T
    for c in cuts:
        A[c:, :c] = 0.0
        A[:c, c:] = 0.0
    w, V, st, _ = _eigh(A)
    assert st == 0
    _check(A, w, V)
