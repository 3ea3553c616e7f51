"""A cube's or a point's result does not depend on what else is in the call:
the same tensors whatever the number of octets in a launch (one warp per
octet, or a block's four when there are few), the same bounds whatever the
length of the list (one warp per cube, or four lanes in longer ones), and the same cubes in a
batch as alone, also where a decision is a tie; the same field at a point
whatever the other points (a warp carries the last members of one point into
the batches of the next)."""
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
    keys = _keys(xyz, r, level, 2600, seed=level)   # every key is an octet: more than sixteen per SM
    A, _, _ = gs.gs_cube_decisions(xyz, r, D, C, PREC, EDGE, DEPTH, keys)
    Ap, _, _ = _parts(xyz, r, keys, (1, 150, 2582))
    assert np.abs(A).sum() > 0
    assert np.array_equal(A, Ap)


@pytest.mark.parametrize("level", [0, 1, 2, 3])
@pytest.mark.parametrize("atoms", [5, 600])
def test_bounds_of_a_set_and_its_parts(level, atoms):
    xyz, r = synth.globular(atoms, seed=32)
    keys = _keys(xyz, r, level, 600, seed=10 + level)   # 4800 cubes (an octet of eight per key), seven invalid of eight
    _, b, d = gs.gs_cube_decisions(xyz, r, D, C, PREC, EDGE, DEPTH, keys)
    _, bp, dp = _parts(xyz, r, keys, (1, 60, 252, 444))   # up to 1536 cubes each
    assert len(np.unique(b[:, 4:], axis=0)) > 1   # several ranks
    assert np.array_equal(b, bp) and np.array_equal(d, dp)


@pytest.mark.parametrize("case", ["one", "line", "cross"])
def test_bounds_of_symmetric_tensors(case):
    """equal singular values and exact zeros: cubes centred on an atom, or
    with atoms placed symmetrically about them"""
    xyz = {"one": [[0.0, 0.0, 0.0]], "line": [[-1.0, 0.0, 0.0], [1.0, 0.0, 0.0]],
           "cross": [[-1.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.0, -1.0, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, -1.0],
                     [0.0, 0.0, 1.0]]}[case]
    xyz = np.array(xyz)
    r = np.full(len(xyz), 1.5)
    o, nroot, _ = oracle.root_grid(xyz, r, D, C, EDGE, DEPTH)
    # on the lattice's own planes and between them
    xyz = xyz + (np.asarray(o) + np.floor((0.5 - np.asarray(o)) / 0.125) * 0.125)
    keys = np.concatenate([_keys(xyz, r, 3, 400, seed=5), _keys(xyz, r, 2, 300, seed=6)])
    A, b, d = gs.gs_cube_decisions(xyz, r, D, C, PREC, EDGE, DEPTH, keys)
    Ap, bp, dp = _parts(xyz, r, keys, range(50, 700, 50))
    assert np.array_equal(A, Ap) and np.array_equal(b, bp) and np.array_equal(d, dp)


def _bound_ties(seed, which):
    """An atom in the root cube [0, 2]^3 and the isovalue equal to that
    cube's own bound L or U as gs_cube_decisions gives it."""
    rng = np.random.default_rng(seed)
    xyz, r = rng.uniform(0.1, 1.9, (1, 3)), np.array([1.5])
    c = 1.0
    for _ in range(3):   # the tensor depends on c through nothing but the lattice's origin
        o, _, _ = oracle.root_grid(xyz, r, D, c, EDGE, DEPTH)
        q = [int(round(-x / 2.0)) for x in o]
        key = np.array([q[0] | q[1] << 18 | q[2] << 36 | 30 << 54], dtype=np.uint64)
        _, b, _ = gs.gs_cube_decisions(xyz, r, D, c, PREC, EDGE, DEPTH, key)
        last, c = c, float(b[0, which])
    assert c == last
    return xyz, r, c


@pytest.mark.parametrize("mode", ["GS_PREC_FP64", "GS_PREC_MIXED"])
@pytest.mark.parametrize("which", [0, 1])
def test_ties_in_a_batch(mode, which):
    """beside a molecule whose larger cutoff radius selects other polynomials"""
    other = (np.array([[0.0, 0.0, 0.0], [1.5, 0.3, 0.2]]), np.array([2.6, 1.2]), D)
    kw = dict(min_edge=EDGE, precision_mode=getattr(gs, mode))
    for seed in range(12):
        xyz, r, c = _bound_ties(seed, which)
        one = gs.mesh_gaussian_surface(xyz, r, D, c, PREC, DEPTH, **kw)
        assert one.stats["near_threshold"][0] >= 1
        b = gs.mesh_gaussian_surface_batch([other, (xyz, r, D)], c, PREC, DEPTH, **kw)[1]
        for k in ("examined", "discarded", "accepted", "forced", "split"):
            assert b.stats[k] == one.stats[k], k
        assert np.array_equal(b.cube_keys, one.cube_keys)
        assert np.array_equal(b.vertices, one.vertices) and np.array_equal(b.triangles, one.triangles)


def _points(n, seed):
    """runs of points with no member, with a few and with more than 64"""
    xyz, r = synth.globular(500, seed=40)
    rng = np.random.default_rng(seed)
    p = xyz[rng.integers(0, len(r), n)] + rng.normal(0, 1.0, (n, 3)) * rng.choice([0.5, 3.0, 12.0, 60.0], (n, 1))
    p[100:400] += 500.0
    return xyz, r, p


@pytest.mark.parametrize("grad", [False, True])
@pytest.mark.parametrize("n", [90001, 1300017])   # 2 and 32 points per warp, neither a multiple
def test_field_of_a_set_and_its_parts(n, grad):
    xyz, r, p = _points(n, seed=n)
    whole = gs.gs_eval_field(xyz, r, D, C, p, grad=grad)
    phi = whole[0] if grad else whole
    assert (phi == 0).sum() > 300 and (phi > 0).sum() > n // 2
    some = np.unique(np.concatenate([np.arange(0, n, 23), np.arange(90, 420), [n - 1]]))   # one point per warp
    for take in (slice(0, 70003), slice(70003, n), some, np.random.default_rng(1).permutation(n)):
        part = gs.gs_eval_field(xyz, r, D, C, np.ascontiguousarray(p[take]), grad=grad)
        if grad:
            assert np.array_equal(part[1], whole[1][take])
            assert np.array_equal(part[0], phi[take])
        else:
            assert np.array_equal(part, phi[take])
    assert np.array_equal(phi, gs.gs_eval_field(xyz, r, D, C, p))   # with and without the gradient
    ref = oracle.field(xyz, r, D, C, p[some], grad=grad)
    rphi = ref[0] if grad else ref
    assert np.all(np.abs(phi[some] - rphi) <= 1e-13 * np.abs(rphi))
    if grad:
        # |dphi| <= 2 D R phi termwise
        assert np.all(np.abs(whole[1][some] - ref[1]) <= 1e-12 * (np.abs(rphi)[:, None] + 1e-300) * 7.0)
