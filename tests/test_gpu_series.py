"""The 1-D Legendre coefficients of the two accumulation kernels over the
range of interval widths and cutoff radii: every polynomial length of the
series and the quadrature that takes over beyond it (wide cubes, very large
D R^2).  FP64 tensors against the oracle, mixed ones against the FP64 kernel
(the debug mode), at the bars of the other parity tests."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


def _cubes(xyz, r, D, h, n, rng):
    """n level-0 cubes of edge h around the atoms, out to their cutoff radii"""
    o, nroot, pad = oracle.root_grid(xyz, r, D, 1.0, h, 0)
    p = xyz[rng.integers(0, len(r), n)] + rng.normal(0, 0.4 * pad, (n, 3))
    q = np.clip(np.floor((p - np.asarray(o)) / h).astype(np.int64), 0, np.asarray(nroot) - 1)
    return np.array([int(a) | int(b) << 18 | int(c) << 36 | 30 << 54 for a, b, c in q], dtype=np.uint64)


@pytest.mark.parametrize("D", [0.05, 0.5, 0.9, 3.0])
@pytest.mark.parametrize("h", [0.03, 0.1, 0.25, 0.4, 0.5, 0.75, 1.0, 1.5, 2.0, 3.0, 5.0, 9.0])
def test_tensors_over_widths(D, h):
    xyz, r = synth.globular(120, seed=3)
    keys = _cubes(xyz, r, D, h, 60, np.random.default_rng(5))
    A, _, _ = gs.gs_cube_decisions(xyz, r, D, 1.0, 1e-3, h, 0, keys)
    rA, _, _ = oracle.cube_batch(xyz, r, D, 1.0, 1e-3, h, 0, keys)
    scale = np.abs(rA).sum(axis=1, keepdims=True) + 1e-300
    assert np.abs(rA).sum() > 0
    assert np.all(np.abs(A - rA) <= 1e-12 * scale)


@pytest.mark.parametrize("radius", [0.0, 1.5, 12.0, 30.0])
@pytest.mark.parametrize("h", [0.25, 1.0, 4.0])
def test_tensors_of_large_atoms(radius, h):
    """D R^2 from 18 to 470 (at 700 the weight exp(D r^2) leaves FP64)"""
    rng = np.random.default_rng(8)
    xyz = rng.uniform(-2, 2, (3, 3))
    r = np.full(3, radius)
    keys = _cubes(xyz, r, 0.5, h, 40, rng)
    A, _, _ = gs.gs_cube_decisions(xyz, r, 0.5, 1.0, 1e-3, h, 0, keys)
    rA, _, _ = oracle.cube_batch(xyz, r, 0.5, 1.0, 1e-3, h, 0, keys)
    scale = np.abs(rA).sum(axis=1, keepdims=True) + 1e-300
    assert np.all(np.abs(A - rA) <= 1e-12 * scale)


@pytest.mark.parametrize("D,edge,depth,n", [(0.5, 0.25, 3, 400), (0.9, 0.25, 3, 400), (0.9, 0.25, 5, 60),
                                            (0.5, 0.06, 3, 6), (0.5, 0.3, 4, 100), (3.0, 0.2, 4, 100),
                                            (0.05, 0.5, 3, 60), (0.02, 1.0, 5, 30), (0.5, 2.0, 2, 200)])
def test_mixed_tensors_against_fp64(D, edge, depth, n):
    xyz, r = synth.globular(n, seed=9)
    m = gs.mesh_gaussian_surface(xyz, r, D, 1.0, 1e-3, depth, min_edge=edge, precision_mode=gs.GS_PREC_MIXED,
                                 debug_flags=1)
    assert m.mismatches == 0
    assert 0 < m.stats["mixed_err_ratio"] < 1.5e-6


def test_batch_of_unequal_cutoffs():
    """molecules of one batch share the coefficients of the largest cutoff
    radius: the meshes of single calls all the same"""
    mols = []
    for i, (n, big) in enumerate([(40, 1.0), (90, 2.0), (30, 1.4)]):
        xyz, r = synth.globular(n, seed=20 + i)
        mols.append((xyz, r * big, 0.5))
    for mode in (gs.GS_PREC_FP64, gs.GS_PREC_MIXED):
        both = gs.mesh_gaussian_surface_batch(mols, 1.0, 1e-3, 3, precision_mode=mode)
        for (xyz, r, D), b in zip(mols, both):
            s = gs.mesh_gaussian_surface(xyz, r, D, 1.0, 1e-3, 3, precision_mode=mode)
            assert np.array_equal(b.cube_keys, s.cube_keys) and np.array_equal(b.triangles, s.triangles)
            assert np.array_equal(b.vertex_keys, s.vertex_keys) and np.array_equal(b.vertices, s.vertices)
