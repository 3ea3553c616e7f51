"""The triangulation without room: no staging slots (every cube is traced
twice), no pool or a pool that fills at once (cubes that overflow their slot
are traced again, those of both kinds), and an allocation that fails beside
the pool (which is then given back).  Injected on the host through GS_FAULT;
every call gives the same mesh or, where it cannot go on, GS_ERR_OOM."""
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


@pytest.fixture()
def fault():
    def set_to(spec):
        os.environ["GS_FAULT"] = spec
    yield set_to
    os.environ.pop("GS_FAULT", None)


def _grid(n):
    rng = np.random.default_rng(n)
    vals = rng.standard_normal((n, n, n))
    vals[0], vals[-1], vals[:, 0], vals[:, -1], vals[:, :, 0], vals[:, :, -1] = -1, -1, -1, -1, -1, -1
    m = gs.gs_triangulate_grid(vals, 0.0)
    c = [slice(0, n - 1), slice(1, n)]
    inside = np.stack([vals[i, j, k] > 0 for i in c for j in c for k in c])
    surface = (inside.any(axis=0) & ~inside.all(axis=0)).sum()
    assert len(m.triangles) > 4 * surface   # so some cubes overflow their slot of four
    return m


def _mixed_sizes():
    xyz, r = synth.globular(120, seed=12)
    m = gs.mesh_gaussian_surface(xyz, r, 0.5, 1.0, 5e-2, 3, precision_mode=gs.GS_PREC_MIXED)
    assert m.stats["mixed_cubes"] > 0
    return m


def _one_size(atoms=25):
    xyz, r = synth.globular(atoms, seed=13)
    return gs.mesh_gaussian_surface(xyz, r, 0.5, 1.0, 1e-3, 3)


def _same(a, b):
    assert np.array_equal(a.vertex_keys, b.vertex_keys) and np.array_equal(a.vertices, b.vertices)
    assert np.array_equal(a.triangles, b.triangles)
    assert a.stats["degenerate_ears"] == b.stats["degenerate_ears"]


@pytest.mark.parametrize("spec", ["staging", "pool@0", "pool@9", "pool@300"])
@pytest.mark.parametrize("make", [lambda: _grid(9), lambda: _grid(26), _mixed_sizes, _one_size],
                         ids=["grid9", "grid26", "mixed_sizes", "one_size"])
def test_no_room_for_slots_or_pool(fault, make, spec):
    ref = make()
    fault(spec)
    _same(make(), ref)


def _sweep(fault, make, ref):
    """(calls refused, calls served before the last refused one) as the first,
    second, ... allocation of the call fails"""
    refused, served, k = [], [], 1
    while k - (refused[-1] if refused else 0) <= 400:
        fault("alloc@%d" % k)
        try:
            _same(make(), ref)
            served.append(k)
        except gs.GsError as e:
            assert e.code == -2
            refused.append(k)
        k += 1
    return len(refused), sum(1 for x in served if x < refused[-1])


@pytest.mark.parametrize("make", [lambda: _one_size(6), lambda: _grid(17)], ids=["molecule", "grid"])
def test_failing_allocation_beside_the_pool(fault, make):
    refused, served = _sweep(fault, make, make())
    assert refused > 0
    # the tracing order's three are optional; the scans' two, the results' three and the redo list's two go on without the
    # pool
    assert served >= 3 + 7


def test_failing_allocation_with_cubes_of_two_sizes(fault):
    """(the list of the cubes with neighbours of another size among them)"""
    xyz, r = synth.globular(14, seed=3)

    def make():
        return gs.mesh_gaussian_surface(xyz, r, 0.5, 1.0, 5e-2, 3)

    ref = make()
    assert ref.stats["mixed_cubes"] > 0
    refused, served = _sweep(fault, make, ref)
    assert refused > 50 and served >= 3 + 9
