"""The rasteriser where a tile's work is cut into units: tiles of thousands of
triangles (few cubes, small faces), triangles that do not fit the tiles' list
(sheets that cover every tile), and more tiles of several units than have a
place for their depths.  Flux against the FP64 ray-cast oracle within the flux
it marks ambiguous, and bit for bit whatever the batch."""
import numpy as np
import pytest

import paper_2103_14137_gb300 as uvc
from synth.scenes import line_lamp, point_lamp
from tests.gpu_util import T, build_arrays, lamp_of
from tests.test_gpu_plates import _box, _face
from tests.test_gpu_raster import check

pytestmark = pytest.mark.gpu


def _arrays(V):
    V = V.astype(np.float32)
    verts, inv = np.unique(V.reshape(-1, 3), axis=0, return_inverse=True)
    tris, n = inv.reshape(-1, 3).astype(np.int32), V.shape[0]
    nrm = np.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
    nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
    sc = build_arrays(verts, tris, V.mean(1), nrm, np.ones(n, np.float32), np.stack([np.arange(n), np.full(n, -1)], 1))
    return verts, tris, nrm, sc


def _sheets(n):
    """n sheets across a room, alternately facing either way."""
    return np.concatenate([_box([0, 0, 0], [4, 3, 2.5], 2, -1)] + [
        _face([0.1 + 3.8 * q / n, 0.05, 0.05], *(([0, 2.9, 0], [0, 0, 2.4]) if q % 2 else ([0, 0, 2.4], [0, 2.9, 0])), 1, 1)
        for q in range(n)])


@pytest.mark.parametrize("R", [16, 64, 65])
@pytest.mark.parametrize("n", [3, 20])      # 108 triangles, a unit or three a tile; 4,800
def test_many_triangles_in_a_tile(R, n):
    verts, tris, nrm, sc = _arrays(np.concatenate([_box([0, 0, 0], [4, 3, 2.5], n, -1), _box([1, 1, 0.25], [2, 2, 0.75], n)]))
    check(verts, tris, nrm, sc, np.array([[3.1, 0.7, 0.5]], np.float32), point_lamp(80.0), R)
    check(verts, tris, nrm, sc, np.array([[0.4, 2.2, 0.3], [2.6, 2.9, 1.2]], np.float32), line_lamp(0.8, 2, 80.0), R)
    sc.free()


@pytest.mark.parametrize("n", [20, 70])     # 64 triangles and 164: lists of both are too short
def test_triangles_past_the_list(n):
    verts, tris, nrm, sc = _arrays(_sheets(n))
    check(verts, tris, nrm, sc, np.array([[2.03, 1.1, 0.9]], np.float32), point_lamp(80.0), 200)
    sc.free()


@pytest.mark.parametrize("R, nc", [(64, 9), (200, 5), (1024, 4)])   # the last: 6,144 tiles, 4,096 places
def test_batches_agree(R, nc):
    verts, tris, nrm, sc = _arrays(_sheets(70))
    rng = np.random.default_rng(R)
    cand, nrm = T(rng.uniform([0.2, 0.2, 0.2], [3.8, 2.8, 2.3], (nc, 3)).astype(np.float32)), T(nrm)
    lamp = lamp_of(point_lamp(80.0))
    A = [uvc.irradiance_raster(sc, nrm, cand, lamp, R=R, cand_per_batch=b).cpu().numpy() for b in (1, 2, nc)]
    assert (A[0] > 0).any()
    assert all(np.array_equal(A[0], x) for x in A[1:])
    sc.free()
