"""The build where its launches change form: sort tiles of 512 and of 2048 keys
(the line between them, ragged last tiles), and the four-wide tree whose first
and last levels one block makes (shallow, balanced and chain-like trees)."""
import numpy as np
import pytest

import paper_2103_14137_gb300 as uvc
from tests.gpu_util import build_arrays
from tests.test_gpu_bvh import _check

pytestmark = pytest.mark.gpu


def _soup(n, points):
    verts = np.repeat(points.astype(np.float32), 3, axis=0)
    verts += np.tile(np.array([[0, 0, 0], [0.01, 0, 0], [0, 0.01, 0.002]], np.float32), (n, 1))
    return verts, np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


def _built(verts, tris, **kw):
    return build_arrays(verts, tris, np.zeros((1, 3), np.float32), [[0, 0, 1]], [1.0], [[-1, -1]], **kw)


@pytest.mark.parametrize("n", [511, 512, 513, 1537, 311295, 311296, 313345])
def test_sort_tiles(n):
    rng = np.random.default_rng(n)
    verts, tris = _soup(n, rng.uniform(0, 5, (n, 3)))
    sc = _built(verts, tris, lbvh_only=True)
    _check(verts, tris, sc)
    sc.free()


@pytest.mark.parametrize("shape", ["even", "chain", "cluster"])
@pytest.mark.parametrize("n", [2, 3, 300, 1500, 40000])
def test_four_wide_tree_reaches_every_triangle_once(n, shape):
    rng = np.random.default_rng(n)
    p = rng.uniform(0, 5, (n, 3))
    if shape == "chain":
        p[:, 0] = 5.0 * 0.5 ** np.linspace(0, 20, n)     # ever smaller cells: a deep, narrow tree
    if shape == "cluster":
        p[n // 2:] = p[0]
    verts, tris = _soup(n, p)
    sc = _built(verts, tris)
    r = uvc.scene_export_traversal(sc)["nodes4"][:, 24:28].astype(np.int64).astype(np.int32)
    seen, level, levels = np.zeros(n, np.int64), np.array([0]), 0
    while level.size:
        kids = r[level].ravel()
        leaves = ~kids[kids < 0]
        np.add.at(seen, leaves, 1)
        level = kids[(kids >= 0) & (kids < n)]
        levels += 1
        assert levels <= sc.depth + 1
    assert (seen == 1).all()
    sc.free()
