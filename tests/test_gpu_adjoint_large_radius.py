"""The adjoint at the ends of its range: dL/dD for one atom far larger than the lattice spacing, where d^2 and r^2
nearly cancel in every term t (d^2 - r^2): against the same sum in numpy.

All coordinates are multiples of 1/8, D is a power of two and D r^2 an
integer, so d^2 - r^2 and the exponents are exact on both sides and a term's
error is a few units of the exponentials' rounding.  And atoms so far apart
that the vertices are sorted into cells of twice the edge."""
import math

import numpy as np
import pytest

import oracle
from meshcheck import key_normal_weights

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


def test_decay_rate_gradient():
    r, D, c, h, depth, prec = 112.0, 1.0 / 32.0, 1.0, 0.5, 2, 1e-9
    xyz = np.array([[0.125, -0.25, 0.375]])
    radii = np.array([r])
    m = gs.mesh_gaussian_surface(xyz, radii, D, c, prec, depth, min_edge=h)
    k = m.vertex_keys.astype(np.uint64)
    typ = ((k >> np.uint64(54)) & np.uint64(31)).astype(np.int64)
    edge = typ < 3
    assert edge.sum() > 500000 and m.stats["accepted"] == [0, 0, 0]   # every cube on the finest level
    o = np.asarray(oracle.root_grid(xyz, radii, D, c, h, depth)[0])
    i0 = np.stack([((k >> np.uint64(s)) & np.uint64(0x3FFFF)).astype(np.int64) for s in (0, 18, 36)], axis=1)[edge]
    i1 = i0.copy()
    i1[np.arange(len(i0)), typ[edge]] += 1
    q = [((o + h * i - xyz[0]) ** 2).sum(axis=1) - r * r for i in (i0, i1)]   # exact
    f = [np.exp(-D * x) for x in q]
    # the vertex moves outwards when the field grows: L counts that motion
    out = np.where(f[0] > f[1], 1.0, -1.0)
    g = np.zeros_like(m.vertices)
    g[np.flatnonzero(edge), typ[edge]] = out
    lam = [h * out * (c - f[1]) / (f[1] - f[0]) ** 2, -h * out * (c - f[0]) / (f[1] - f[0]) ** 2]
    terms = np.concatenate([-lam[t] * f[t] * q[t] for t in range(2)])
    assert lam[0].min() >= 0 and lam[1].min() >= 0
    ref, size = math.fsum(terms), math.fsum(np.abs(terms))
    _, _, gD = gs.gs_mesh_backward(xyz, radii, D, c, prec, depth, g, min_edge=h)
    # per term: two exponentials of the field and one of the term, a division and eight products, about 16 roundings of
    # 1.1e-16, were they all to point one way (they do not: sums of 500,000 terms leave 1e-16)
    assert abs(gD - ref) <= 16 * 1.2e-16 * size


def test_atoms_far_apart():
    xyz = np.array([[0.0, 0.0, 0.0], [900.2, 910.1, 905.3], [450.1, 3.0, 880.2]])
    r, D, h, depth = np.array([1.7, 1.2, 1.5]), 0.5, 0.5, 4
    _, nroot, pad = oracle.root_grid(xyz, r, D, 1.0, h, depth)
    # more than 2^24 cells of half the cutoff radius
    assert np.prod(np.ceil(np.asarray(nroot) * h * 2.0 ** depth / (0.5 * pad)) + 1) > 1 << 24
    m = gs.mesh_gaussian_surface(xyz, r, D, 1.0, 1e-3, depth, min_edge=h)
    om = oracle.mesh(xyz, r, D, 1.0, 1e-3, h, depth)
    assert np.array_equal(np.sort(m.vertex_keys), np.sort(om["vkeys"]))
    ga, gr, gD = gs.gs_mesh_backward(xyz, r, D, 1.0, 1e-3, depth, key_normal_weights(m.vertex_keys), min_edge=h)
    ox, orr, oD = oracle.mesh_grad(xyz, r, D, 1.0, 1e-3, h, depth, key_normal_weights(om["vkeys"]))
    scale = max(np.abs(ox).max(), np.abs(orr).max(), abs(oD))
    assert scale > 0.1
    # the bar of the other adjoint tests
    assert np.abs(ga - ox).max() <= 1e-9 * scale and np.abs(gr - orr).max() <= 1e-9 * scale
    assert abs(gD - oD) <= 1e-9 * max(1.0, abs(oD))
