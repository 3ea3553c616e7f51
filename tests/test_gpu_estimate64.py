"""The FP64 estimate (bounds, ranks, decisions) against the oracle at the list
sizes where its two kernels change over (each key is an octet of eight cubes
to them, seven invalid: 192 keys are 1536 cubes, the last size of the
warp-per-cube kernel) and on tensors of low rank, whose small rows are
rounding noise."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")

D, C, PREC, EDGE, DEPTH = 0.5, 1.0, 1e-3, 0.25, 3


def _keys(xyz, r, n, seed):
    """n cubes near the atoms, on all levels"""
    rng = np.random.default_rng(seed)
    o, nroot, _ = oracle.root_grid(xyz, r, D, C, EDGE, DEPTH)
    out = []
    for i in range(n):
        l = int(rng.integers(0, DEPTH + 1))
        h = EDGE * 2 ** (DEPTH - l)
        p = xyz[rng.integers(0, len(r))] + rng.normal(0, 2.0, 3)
        q = np.clip(np.floor((p - np.asarray(o)) / h).astype(np.int64), 0, np.asarray(nroot) * 2 ** l - 1)
        out.append(int(q[0]) | int(q[1]) << 18 | int(q[2]) << 36 | 30 << 54 | l << 59)
    return np.array(out, dtype=np.uint64)


def _compare(xyz, r, keys):
    A, b, d = gs.gs_cube_decisions(xyz, r, D, C, PREC, EDGE, DEPTH, keys)
    rA, rb, rd = oracle.cube_batch(xyz, r, D, C, PREC, EDGE, DEPTH, keys)
    scale = np.abs(rA).sum(axis=1)
    assert np.all(np.abs(A - rA).max(axis=1) <= 1e-12 * scale + 1e-300)
    # L, U and sum|R|: rounding of the factors, 1e-9 of sum|A| (the bar of the other parity tests)
    assert np.all(np.abs(b[:, :4] - rb[:, :4]).max(axis=1) <= 1e-9 * scale + 1e-300)
    assert np.array_equal(b[:, 4:], rb[:, 4:])
    assert np.array_equal(d, rd)


@pytest.mark.parametrize("n", [1, 7, 191, 192, 193, 700])
def test_estimate_sizes(n):
    xyz, r = synth.globular(300, seed=7)
    _compare(xyz, r, _keys(xyz, r, n, seed=n))


@pytest.mark.parametrize("n", [40, 400])
@pytest.mark.parametrize("case", ["one", "line", "pair", "far"])
def test_estimate_low_rank(case, n):
    xyz = {"one": [[0.3, 0.2, 0.1]],                                   # rank one
           "line": [[0.0, 0.0, 0.0], [1.1, 0.0, 0.0], [2.4, 0.0, 0.0]],   # rank one in y and z
           "pair": [[0.1, 0.2, 0.3], [0.1, 0.2, 0.3]],
           "far": [[0.0, 0.0, 0.0], [6.0, 5.5, 5.0]]}[case]
    xyz = np.array(xyz)
    r = np.linspace(1.2, 1.8, len(xyz))
    _compare(xyz, r, _keys(xyz, r, n, seed=n))
