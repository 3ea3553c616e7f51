"""Host meshes are the library's own memory: writable, alive as long as any
view of them, released once, each array on its own."""
import ctypes
import gc

import numpy as np

from paper_1611_03474_gb300 import _native as nat


class _Lib:
    """stands for the library: meshes from malloc-like buffers, frees counted"""

    def __init__(self):
        self.freed = []

    def mesh_free(self, ref):
        m = ref._obj
        for f in ("vertices", "triangles", "vertex_keys", "cube_keys"):
            p = ctypes.cast(getattr(m, f), ctypes.c_void_p).value
            if p:
                self.freed.append(p)
                setattr(m, f, type(getattr(m, f))())


def _mesh(bufs, nv, nt, nc):
    m = nat.MeshC()
    for (field, kind), b in zip((("vertices", ctypes.c_double), ("triangles", ctypes.c_int32),
                                 ("vertex_keys", ctypes.c_uint64), ("cube_keys", ctypes.c_uint64)), bufs):
        setattr(m, field, ctypes.cast(b.ctypes.data, ctypes.POINTER(kind)))
    m.n_vertices, m.n_triangles, m.n_cubes = nv, nt, nc
    return m


def test_host_arrays_own_their_memory():
    bufs = [np.arange(15, dtype=np.float64), np.arange(12, dtype=np.int32), np.arange(5, dtype=np.uint64),
            np.arange(7, dtype=np.uint64)]
    lib = _Lib()
    m = _mesh(bufs, 5, 4, 7)
    r = nat._mesh_from_c(m, lib, nat.Stats(), 3)
    assert lib.freed == []
    assert np.array_equal(r.vertices, bufs[0].reshape(5, 3)) and r.vertices.dtype == np.float64
    assert np.array_equal(r.triangles, bufs[1].reshape(4, 3)) and r.triangles.dtype == np.int32
    assert np.array_equal(r.vertex_keys, bufs[2]) and np.array_equal(r.cube_keys, bufs[3])
    r.vertices[0, 0] = -1.0   # writable
    view = r.vertices[1:]
    keys = r.vertex_keys
    del r
    gc.collect()
    # triangles and cube keys are gone, the other two are still in use
    assert sorted(lib.freed) == sorted([bufs[1].ctypes.data, bufs[3].ctypes.data])
    assert view[0, 0] == 3.0 and keys[4] == 4
    del view, keys
    gc.collect()
    assert sorted(lib.freed) == sorted(b.ctypes.data for b in bufs)


def test_empty_mesh_releases_everything():
    bufs = [np.zeros(3), np.zeros(3, dtype=np.int32), np.zeros(1, dtype=np.uint64), np.zeros(1, dtype=np.uint64)]
    lib = _Lib()
    r = nat._mesh_from_c(_mesh(bufs, 0, 0, 0), lib, nat.Stats(), 3)
    assert r.vertices.shape == (0, 3) and r.triangles.shape == (0, 3) and len(r.cube_keys) == 0
    assert sorted(lib.freed) == sorted(b.ctypes.data for b in bufs)
