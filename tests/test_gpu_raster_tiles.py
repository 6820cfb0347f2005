"""The rasteriser at the edges of its 64 x 64 pixel tiles: face sizes around
one and two tiles, a mesh whose triangles fit the tiles' lists and one (few
large triangles over many tiles) whose do not, a source close to a wall
(triangles that cross the near plane), and batches of every size.  Flux against
the FP64 ray-cast oracle within the flux it marks ambiguous."""
import numpy as np
import pytest

import paper_2103_14137_gb300 as uvc
from synth import tiny_room
from synth.scenes import line_lamp, point_lamp
from tests.gpu_util import T, build, build_arrays, lamp_of
from tests.test_gpu_plates import _box
from tests.test_gpu_raster import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 63, 64, 65, 130])
@pytest.mark.parametrize("mesh", ["tiny", "cube"])
def test_tile_edges(R, mesh):
    if mesh == "tiny":
        s = tiny_room()
        verts, tris, nrm, sc = s.verts, s.tris, s.normal, build(s)
        cand = np.array([[2.0, 1.9, 1.0], [0.004, 3.0, 1.2], [1.0, 0.5, 2.996]], np.float32)
        lamp = point_lamp(80.0)
    else:
        V = _box([0, 0, 0], [2, 3, 2.5], 1, -1).astype(np.float32)
        verts, inv = np.unique(V.reshape(-1, 3), axis=0, return_inverse=True)
        tris = inv.reshape(-1, 3).astype(np.int32)
        nrm = np.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
        nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
        n = tris.shape[0]
        sc = build_arrays(verts, tris, V.mean(1), nrm, np.ones(n, np.float32), np.stack([np.arange(n), np.full(n, -1)], 1))
        cand = np.array([[0.7, 1.1, 0.3], [1.99, 2.5, 0.6]], np.float32)
        lamp = line_lamp(0.8, 3, 80.0)
    check(verts, tris, nrm, sc, cand, lamp, R)
    sc.free()


def test_batches_of_any_size_agree():
    s = tiny_room()
    sc, lamp = build(s), lamp_of(line_lamp(0.5, 2, 80.0))
    cand, nrm = T(s.cand[:7]), T(s.normal)
    A = [uvc.irradiance_raster(sc, nrm, cand, lamp, R=100, cand_per_batch=b).cpu() for b in (1, 2, 3, 5, 7)]
    assert all(np.array_equal(A[0].numpy(), x.numpy()) for x in A[1:])
    sc.free()
