"""The dense inverse of the pressure hierarchy's coarsest level: in shared
memory, in block steps, and column by column where the block steps' row
exchanges (inside 16 rows) do not do, against the inverse that numpy forms.
Tolerance: 10 n eps cond of the inverted matrix, relative to the largest entry
of the inverse."""
import ctypes as C
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fvs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1810_08572_gb300 import LIB_PATH, build
    if not os.path.exists(LIB_PATH):
        build()
    from paper_1810_08572_gb300 import fvs as f
    return f


def inverse(fvs, A):
    """fvs_dense_inverse of a matrix, its non-zeros packed to the left."""
    n = len(A)
    w = max(1, int((A != 0).sum(1).max()))
    col = np.repeat(np.arange(n, dtype=np.int32)[None, :], w, 0)
    val = np.zeros((w, n))
    for i in range(n):
        j = np.flatnonzero(A[i])
        col[:len(j), i], val[:len(j), i] = j, A[i, j]
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    X = np.zeros((n, n))
    by = C.c_int32(-1)
    r = fvs.fvs_dense_inverse(ptr(col), ptr(val), n, w, ptr(X), C.byref(by))
    return r, X, by.value


def close(X, A):
    want = np.linalg.inv(A)
    return np.abs(X - want).max() <= 10 * len(A) * np.finfo(float).eps * np.linalg.cond(A) * np.abs(want).max()


def banded(n, seed):
    """Diagonally dominant, not symmetric, couplings near and far."""
    rng = np.random.default_rng(seed)
    A = np.zeros((n, n))
    for d in (1, 2, 17, n // 2):
        if 0 < d < n:
            A[np.arange(n), (np.arange(n) + d) % n] = -rng.uniform(0.5, 1.0, n)
    A[np.arange(n), np.arange(n)] = np.abs(A).sum(1) + rng.uniform(0.1, 1.0, n)
    return A


def shifted(n, seed):
    """The same with every row moved 37 places down: no pivot near the diagonal."""
    return np.roll(banded(n, seed), 37, axis=0)


@pytest.mark.parametrize("n", [1, 100, 160, 161, 300, 1000])
def test_inverse_of_a_dominant_matrix(fvs, n):
    A = banded(n, n)
    r, X, by = inverse(fvs, A)
    assert r == fvs.FVS_OK and by == 0
    assert close(X, A)


@pytest.mark.parametrize("n", [100, 161, 300, 1000])
def test_inverse_that_needs_pivots_from_outside_the_blocks(fvs, n):
    A = shifted(n, n)
    r, X, by = inverse(fvs, A)
    assert r == fvs.FVS_OK and by == (1 if n > 160 else 0)
    assert close(X, A)


@pytest.mark.parametrize("n", [161, 300])
def test_inverse_of_singular_and_other_parts_by_columns(fvs, n):
    """A part whose rows sum to zero, its non-zeros far from the diagonal (its
    first row pinned, its mean projected out), beside one that is regular."""
    m = n - 61
    A = np.zeros((n, n))
    i = np.arange(m)
    A[i, (i + 37) % m], A[i, (i + 74) % m] = 1.0, -1.0
    A[m:, m:] = shifted(n - m, 7)
    pinned = A.copy()
    pinned[0] = np.eye(n)[0]
    P = np.eye(n)
    P[:m, :m] -= 1.0 / m
    r, X, by = inverse(fvs, A)
    assert r == fvs.FVS_OK and by == 1
    want = P @ np.linalg.inv(pinned) @ P
    # (the projections amplify by no more than the part's inverse does)
    scale = np.abs(np.linalg.inv(pinned)).max()
    assert np.abs(X - want).max() <= 10 * n * np.finfo(float).eps * np.linalg.cond(pinned) * scale


@pytest.mark.parametrize("n", [100, 200])
def test_no_inverse_is_reported(fvs, n):
    A = np.eye(n)
    A[40:42, 40:42] = 1.0
    r, _, _ = inverse(fvs, A)
    assert r == fvs.FVS_ERR_NOT_CONVERGED and "zero pivot" in fvs.fvs_last_error()


def test_bad_arguments_are_refused(fvs):
    X, by = np.zeros((2, 2)), C.c_int32()
    col, val = np.array([0, 2], np.int32), np.ones(2)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    for args in ((ptr(col), ptr(val), 2, 1, ptr(X)), (None, ptr(val), 2, 1, ptr(X)), (ptr(col), ptr(val), 1001, 1, ptr(X)),
                 (ptr(col), ptr(val), 2, 0, ptr(X)), (ptr(col), ptr(val), 2, 1, None)):
        assert fvs.fvs_dense_inverse(*args, C.byref(by)) == fvs.FVS_ERR_ARG
        assert fvs.fvs_last_error().startswith("fvs_dense_inverse")
