"""The discard without the SVD in the level loops: on one level of cubes the
FP64 mesh (which screens) keeps exactly the cubes that gs_cube_decisions
(which does not) keeps, also for isovalues whose squares leave FP64's range;
and the mixed form's screen drops no cube that the FP64 form keeps where FP32
squares underflow."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


@pytest.mark.parametrize("c", [1.0, 1e-3, 1e-20, 1e-120, 1e-150, 1e-156, 1e-158, 1e-160, 1e-161])
def test_fp64_screen_against_the_svd(c):
    D, h = 2.0, 1.0
    xyz, r = synth.globular(30, seed=6)
    m = gs.mesh_gaussian_surface(xyz, r, D, c, 1e-3 * c, 0, min_edge=h)
    _, nroot, _ = oracle.root_grid(xyz, r, D, c, h, 0)
    x, y, z = np.meshgrid(*[np.arange(k, dtype=np.uint64) for k in nroot], indexing="ij")
    keys = (x | y << np.uint64(18) | z << np.uint64(36) | np.uint64(30 << 54)).ravel()
    _, b, d = gs.gs_cube_decisions(xyz, r, D, c, 1e-3 * c, h, 0, keys)
    # a margin within rounding of the threshold is not compared (none is expected)
    clear = np.minimum(np.abs(c - b[:, 0]), np.abs(b[:, 1] - c)) > 1e-9 * np.abs(b[:, :2]).max(axis=1)
    kept = np.isin(keys, m.cube_keys)
    assert kept.sum() > 100 and (~kept).sum() > 1000
    assert np.array_equal(kept[clear], d[clear] != 0)
    assert (~clear).sum() < 5


def test_mixed_screen_where_squares_underflow():
    xyz, r = synth.globular(30, seed=30)
    k = [gs.mesh_gaussian_surface(xyz, r, 0.1, 1e-20, 1e-23, 0, min_edge=1.6, precision_mode=mode).cube_keys
         for mode in (gs.GS_PREC_FP64, gs.GS_PREC_MIXED)]
    assert len(k[0]) > 1000 and np.isin(k[0], k[1]).all()
