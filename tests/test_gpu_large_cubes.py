"""Membership in cubes far larger than the cutoff: atoms just inside the
cutoff distance of a cube face are counted as terms of the cube beyond it in
the mixed form as in the FP64 form, whose test is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


@pytest.mark.parametrize("side", [-1, 1])
@pytest.mark.parametrize("h", [16.0, 64.0, 256.0, 1024.0])
def test_pairs_near_the_cutoff(h, side):
    n = 4000
    rng = np.random.default_rng(int(h))
    r = rng.uniform(1.0, 1.8, n)   # the distance to the face takes many roundings
    R = np.sqrt(r * r - np.log(1e-8) / 0.5)
    # the root lattice's planes are multiples of h
    xyz = rng.uniform(7.0, h - 7.0, (n, 3))
    xyz[:, 0] = h * rng.integers(1, 3, n) + side * (R - rng.uniform(1e-5, 1e-4, n))
    pairs = [gs.mesh_gaussian_surface(xyz, r, 0.5, 1.0, 1e-3, 0, min_edge=h, precision_mode=mode).stats["pair_terms"]
             for mode in (gs.GS_PREC_FP64, gs.GS_PREC_MIXED)]
    assert pairs == [2 * n, 2 * n]
