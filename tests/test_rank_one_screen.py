"""The discard without the SVD, checked directly: for the bounds of the
two-level truncated SVD (whatever its ranks), U <= max P~ + 53 e and
L >= min P~ - 53 e, with P~ enclosed by its trilinear part's corner values
and the sum of the other coefficients, and e the tensor's distance from the
rank-one tensor through its fibres at 000.  On the oracle's bounds for the
cubes of a molecule on every level, for tensors of random spectra, and for
tensors made of a strong rank-one term and a random rest; and every cube the
screen discards is one the oracle discards."""
import numpy as np
import pytest

import oracle
import synth

HIGH = np.maximum(np.maximum(np.arange(4)[:, None, None], np.arange(4)[None, :, None]),
                  np.arange(4)[None, None, :]) >= 2
SIGN = np.array([[(-1.0) ** n for n in range(4)], [1.0] * 4])


def screen(A):
    """(lower, upper) that the screen proves for L and U"""
    A = A.reshape(4, 4, 4)
    corners = np.einsum("abc,ia,jb,kc->ijk", np.where(HIGH, 0.0, A), SIGN, SIGN, SIGN)
    high = np.abs(A[HIGH]).sum()
    T = np.einsum("a,b,c->abc", A[:, 0, 0], A[0, :, 0] / A[0, 0, 0], A[0, 0, :] / A[0, 0, 0])
    e = np.sqrt(((A - T) ** 2).sum())
    return corners.min() - high - 53.0 * e, corners.max() + high + 53.0 * e


@pytest.mark.parametrize("level", [0, 1, 2, 3])
@pytest.mark.parametrize("D", [0.5, 0.9])
def test_molecule_cubes(level, D):
    xyz, r = synth.globular(150, seed=3)
    rng = np.random.default_rng(level)
    o, nroot, _ = oracle.root_grid(xyz, r, D, 1.0, 0.25, 3)
    h = 0.25 * 2 ** (3 - level)
    p = xyz[rng.integers(0, len(r), 400)] + rng.normal(0, 2.5, (400, 3))
    q = np.clip(np.floor((p - np.asarray(o)) / h).astype(np.int64), 0, (np.asarray(nroot) << level) - 1)
    keys = np.unique(np.array([int(a) | int(b) << 18 | int(c) << 36 | 30 << 54 | level << 59 for a, b, c in q],
                              dtype=np.uint64))
    A, b, d = oracle.cube_batch(xyz, r, D, 1.0, 1e-3, 0.25, 3, keys)
    proved = 0
    for a, bb, dd in zip(A, b, d):
        if a[0] == 0.0:
            continue
        lo, hi = screen(a)
        tol = 1e-9 * np.abs(a).sum()
        assert bb[0] >= lo - tol and bb[1] <= hi + tol
        if hi < 1.0 or lo > 1.0:
            assert dd == 0
            proved += 1
    assert proved > 0


@pytest.mark.parametrize("seed", range(6))
def test_random_tensors(seed):
    rng = np.random.default_rng(seed)
    for _ in range(300):
        rest = rng.standard_normal((4, 4, 4)) * rng.choice([1.0, 0.3, 0.05, 1e-3])
        a, b, c = (np.concatenate([[1.0], rng.normal(0, rng.choice([0.1, 0.6]), 3)]) for _ in range(3))
        A = 5.0 * np.einsum("a,b,c->abc", a, b, c) + rest
        if abs(A[0, 0, 0]) < 1e-3 * np.abs(A).sum():
            continue
        bb = oracle.bounds(A.reshape(64))
        lo, hi = screen(A)
        tol = 1e-9 * np.abs(A).sum()
        assert bb[0] >= lo - tol and bb[1] <= hi + tol
