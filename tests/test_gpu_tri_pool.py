"""The triangulation's staging slots and the pool behind them against the
oracle: grids whose cubes fit their slots, grids of random values whose cubes
overflow them (within the pool's room for small grids, past it for larger
ones, whose remaining cubes are traced again), and cubes of different sizes."""
import numpy as np
import pytest

import oracle
import synth
from meshcheck import canonical_triangles

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


def _same(m, ref, tol):
    assert np.array_equal(np.sort(m.vertex_keys), ref["vkeys"])
    order = np.argsort(m.vertex_keys)
    assert np.abs(m.vertices[order] - ref["vertices"]).max(initial=0.0) < tol
    assert np.array_equal(canonical_triangles(m.vertex_keys, m.triangles),
                          canonical_triangles(ref["vkeys"], ref["triangles"]))


@pytest.mark.parametrize("n", [3, 8, 17, 26, 34])
@pytest.mark.parametrize("smooth", [False, True])
def test_grids(n, smooth):
    rng = np.random.default_rng(n)
    if smooth:
        z, y, x = np.meshgrid(*[np.linspace(-1.3, 1.2, n)] * 3, indexing="ij")
        vals = 0.8 - x * x - 1.1 * y * y - 0.7 * z * z + 0.1 * x * y
    else:
        vals = rng.standard_normal((n, n, n))
    vals[0], vals[-1], vals[:, 0], vals[:, -1], vals[:, :, 0], vals[:, :, -1] = -1, -1, -1, -1, -1, -1
    _same(gs.gs_triangulate_grid(vals, 0.0), oracle.mesh_grid(vals, 0.0), 1e-12)


@pytest.mark.parametrize("mode", ["GS_PREC_FP64", "GS_PREC_MIXED"])
def test_cubes_of_different_sizes(mode):
    xyz, r = synth.globular(120, seed=12)
    m = gs.mesh_gaussian_surface(xyz, r, 0.5, 1.0, 5e-2, 3, precision_mode=getattr(gs, mode))
    assert m.stats["mixed_cubes"] > 0
    _same(m, oracle.mesh(xyz, r, 0.5, 1.0, 5e-2, 0.25, 3), 1e-5)
