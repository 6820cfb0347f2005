"""Patch points a few micrometres from a sloping sheet, which is no plate, and a
little farther from a triangle of their own plane that is not their own.  The
sheet is nearer, so the clearance says nothing about that triangle, and the segment
test may or may not hit it: the plates must leave such points to the search of the
whole hierarchy, bit for bit."""
import numpy as np
import pytest
import torch

import paper_2103_14137_gb300 as uvc
from tests.gpu_util import T, build_arrays, lamp_of
from tests.test_gpu_plates import _box, _face, _lamps

pytestmark = pytest.mark.gpu

CELLS = 8


def _room(scale):
    """A room 4 x 3 x 2.5 (times `scale`) with a box and a sheet that rises from the floor's line x = 5/32; the
    floor's cells are cut from (1, 0) to (0, 1), so the other triangle of a corner's cell is far from it."""
    V = np.concatenate([_box([0, 0, 0], [4, 3, 2.5], CELLS, -1), _box([1, 1, 0.25], [2, 2, 0.75], 3)])
    V = V[~(V[:, :, 2] == 0).all(1)]
    F = []
    for i in range(CELLS):
        for j in range(CELLS):
            p = [np.array([4.0 * a / CELLS, 3.0 * b / CELLS, 0.0]) for a, b in ((i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1))]
            F += [[p[0], p[1], p[3]], [p[1], p[2], p[3]]]
    sheet = _face([0.15625, 0, 0], [1.0, 0, 2.0], [0, 3, 0], 2, 6)
    return (scale * np.concatenate([np.array(F), V, sheet])).astype(np.float32)


def _points(scale):
    """On the floor, a little before the sheet's line, delta past the cell border y = 3 j / 8: in the first triangle
    of cell (0, j), the triangles of cell (0, j - 1) farther off than the sheet."""
    rng = np.random.default_rng(3)
    j = rng.integers(1, CELLS, 2000)
    border = np.float32(3.0 * scale / CELLS) * j.astype(np.float32)          # exact
    y = (border + np.exp(rng.uniform(np.log(3e-7), np.log(6e-6 * scale), j.size))).astype(np.float32)
    x = (0.15625 * scale - 0.25 * (y.astype(np.float64) - border)).astype(np.float32)
    ok = (x < np.float32(0.15625 * scale)) & (y > border)
    return np.stack([x, y, np.zeros_like(x)], 1)[ok], j[ok]


@pytest.mark.parametrize("scale", [1, 16])
@pytest.mark.parametrize("lamp", ["line2", "line16", "point", "tube"])
def test_points_next_to_a_sheet_and_a_coplanar_triangle(scale, lamp):
    V = _room(scale)
    verts, inv = np.unique(V.reshape(-1, 3), axis=0, return_inverse=True)
    tris = inv.reshape(-1, 3).astype(np.int32)
    cen, j = _points(scale)
    own = 2 * j                                           # cells of i = 0 come first
    n = j.size
    sc = build_arrays(verts, tris, cen, np.tile([[0, 0, 1]], (n, 1)), np.ones(n), np.stack([own, np.full(n, -1)], 1))
    rng = np.random.default_rng(4)
    src = T((scale * rng.uniform([0.1, 0.1, 0.1], [3.9, 2.9, 1.2], (60, 3))).astype(np.float32))
    L = lamp_of(_lamps()[lamp])
    A, vis = uvc.irradiance_matrix(sc, src, L, with_vis=True)
    old = uvc.set_wedge_traversal(False)
    A0, vis0 = uvc.irradiance_matrix(sc, src, L, with_vis=True)
    uvc.set_wedge_traversal(old)
    torch.cuda.synchronize()
    assert uvc.scene_status(sc) == 0
    differ = (uvc.vis_to_bool(vis, n) != uvc.vis_to_bool(vis0, n)).any(-1)
    assert not differ.any(), f"{int(differ.sum())} of {differ.size} pairs"
    assert torch.equal(A, A0)
    sc.free()
