"""The FP64 estimate at isovalues whose tensors' squares leave FP64's range:
its bounds against the oracle's of the same tensor scaled by a power of two
(which changes nothing but the exponents), from both kernels (short lists and
long ones)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")

D, EDGE, DEPTH = 0.5, 0.5, 2


@pytest.mark.parametrize("n", [150, 400])   # an octet of eight cubes each: 1200 and 3200
@pytest.mark.parametrize("c", [1.0, 1e-90, 1e-125, 1e-135, 1e-145, 1e-200])
def test_bounds(c, n):
    xyz, r = synth.globular(12, seed=2)
    o, nroot, _ = oracle.root_grid(xyz, r, D, c, EDGE, DEPTH)
    rng = np.random.default_rng(4)
    h = EDGE * 2.0 ** DEPTH
    v = rng.standard_normal((n, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    # about the surface, which lies where exp(-D rho^2) has c's size
    p = xyz.mean(axis=0) + v * (np.sqrt(-np.log(c) / D) + rng.uniform(-2, 5, n))[:, None]
    q = np.clip(np.floor((p - np.asarray(o)) / h).astype(np.int64), 0, np.asarray(nroot) - 1)
    keys = np.array([int(x) | int(y) << 18 | int(z) << 36 | 30 << 54 for x, y, z in q], dtype=np.uint64)
    A, b, _ = gs.gs_cube_decisions(xyz, r, D, c, 1e-3 * c, EDGE, DEPTH, keys)
    tot = np.abs(A).sum(axis=1)
    assert (tot > 0).sum() > n // 2
    for a, bb, t in zip(A, b, tot):
        if t == 0.0:
            continue
        e = int(np.floor(np.log2(t)))
        ref = np.array(oracle.bounds(np.ldexp(a, -e)), dtype=np.float64)
        # rounding of the factors, 1e-9 of sum|A| (the bar of the other parity tests)
        assert np.abs(np.ldexp(bb[:4], -e) - ref[:4]).max() <= 1e-9 * np.ldexp(t, -e)
        assert np.array_equal(bb[4:], ref[4:6])
