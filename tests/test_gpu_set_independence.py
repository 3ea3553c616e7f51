"""A cube's or a point's result does not depend on what else is in the call:
the same tensors whatever the number of octets in a launch (one warp per
octet, or a block's four when there are few)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")

D, C, PREC, EDGE, DEPTH = 0.5, 1.0, 1e-3, 0.25, 3


def _keys(xyz, r, level, n, seed):
    """n cubes of one level near the atoms"""
    rng = np.random.default_rng(seed)
    o, nroot, _ = oracle.root_grid(xyz, r, D, C, EDGE, DEPTH)
    h = EDGE * 2 ** (DEPTH - level)
    p = xyz[rng.integers(0, len(r), n)] + rng.normal(0, 2.0, (n, 3))
    q = np.clip(np.floor((p - np.asarray(o)) / h).astype(np.int64), 0, (np.asarray(nroot) << level) - 1)
    return np.array([int(a) | int(b) << 18 | int(c) << 36 | 30 << 54 | level << 59 for a, b, c in q], dtype=np.uint64)


def _parts(xyz, r, keys, cuts):
    ends = list(cuts) + [len(keys)]
    res = [gs.gs_cube_decisions(xyz, r, D, C, PREC, EDGE, DEPTH, keys[a:b]) for a, b in zip([0] + ends, ends)]
    return tuple(np.concatenate([x[i] for x in res]) for i in range(3))


@pytest.mark.parametrize("level", [0, 1, 2, 3])
@pytest.mark.parametrize("atoms", [5, 600])
def test_tensors_of_a_set_and_its_parts(level, atoms):
    xyz, r = synth.globular(atoms, seed=31)
    keys = _keys(xyz, r, level, 700, seed=level)   # every key is an octet: more than four per SM
    A, _, _ = gs.gs_cube_decisions(xyz, r, D, C, PREC, EDGE, DEPTH, keys)
    Ap, _, _ = _parts(xyz, r, keys, (1, 90, 608))
    assert np.abs(A).sum() > 0
    assert np.array_equal(A, Ap)
