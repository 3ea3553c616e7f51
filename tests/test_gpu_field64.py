"""The FP64 field at points (one warp per point, members queued) and the
field's adjoint (one warp per atom over the vertices sorted into a grid)
against the oracle, at the sizes where their loops change: fewer members than
a warp, several queue fills, more points than warps, no member at all; one
atom and few atoms (several warps share an atom), and a sparse grid."""
import numpy as np
import pytest

import oracle
import synth
from meshcheck import key_normal_weights, surface_loss_grad

pytestmark = pytest.mark.gpu

gs = pytest.importorskip("paper_1611_03474_gb300")


@pytest.mark.parametrize("atoms", [1, 3, 60, 700])
@pytest.mark.parametrize("points", [1, 5, 333])
@pytest.mark.parametrize("grad", [False, True])
def test_field_sizes(atoms, points, grad):
    xyz, r = synth.globular(atoms, seed=atoms)
    rng = np.random.default_rng(points)
    pts = xyz[rng.integers(0, atoms, points)] + rng.normal(0, 4.0, (points, 3))
    pts[0] = xyz[0] + 1000.0   # no atom reaches it
    out = gs.gs_eval_field(xyz, r, 0.5, 1.0, pts, grad=grad)
    ref = oracle.field(xyz, r, 0.5, 1.0, pts, grad=grad)
    phi, rphi = (out[0], ref[0]) if grad else (out, ref)
    assert phi[0] == 0.0
    assert np.all(np.abs(phi - rphi) <= 1e-13 * np.abs(rphi))
    if grad:
        # |dphi| <= 2 D R phi termwise
        assert np.all(np.abs(out[1] - ref[1]) <= 1e-12 * (np.abs(rphi)[:, None] + 1e-300) * 7.0)


def test_field_more_points_than_warps():
    xyz, r = synth.globular(200, seed=5)
    rng = np.random.default_rng(1)
    pts = xyz[rng.integers(0, 200, 60001)] + rng.normal(0, 3.0, (60001, 3))
    phi = gs.gs_eval_field(xyz, r, 0.9, 1.0, pts)
    ref = oracle.field(xyz, r, 0.9, 1.0, pts)
    assert np.all(np.abs(phi - ref) <= 1e-13 * np.abs(ref))


@pytest.mark.parametrize("case", ["one", "four", "apart", "many"])
def test_adjoint_sizes(case):
    xyz, r = {"one": lambda: (np.array([[0.1, 0.2, 0.3]]), np.array([1.5])),
              "four": lambda: synth.chain(4, seed=2),
              "apart": lambda: (np.array([[0.0, 0.0, 0.0], [150.0, 90.0, 40.0]]), np.array([1.7, 1.2])),
              "many": lambda: synth.globular(150, seed=6)}[case]()
    D, prec, me, md = 0.5, 1e-3, 0.5, 2
    m = gs.mesh_gaussian_surface(xyz, r, D, 1.0, prec, md, min_edge=me)
    g = surface_loss_grad(m.vertices, m.triangles, key_normal_weights(m.vertex_keys))
    ga, gr, gD = gs.gs_mesh_backward(xyz, r, D, 1.0, prec, md, g, min_edge=me)
    om = oracle.mesh(xyz, r, D, 1.0, prec, me, md)
    og = surface_loss_grad(om["vertices"], om["triangles"], key_normal_weights(om["vkeys"]))
    ox, orr, oD = oracle.mesh_grad(xyz, r, D, 1.0, prec, me, md, og)
    scale = max(np.abs(ox).max(), np.abs(orr).max(), abs(oD))
    assert np.abs(ga - ox).max() <= 1e-9 * scale
    assert np.abs(gr - orr).max() <= 1e-9 * scale
    assert abs(gD - oD) <= 1e-9 * max(1.0, abs(oD))
