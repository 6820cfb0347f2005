"""Segments decided at whole rectangles (plates) against the plain search.

A scene's flat, fully tiled rectangles decide most segments without the
hierarchy; with uvc_set_wedge_traversal(0) every source is searched in the
hierarchy instead.  Both must give the same entries and visibility bits, on
scenes chosen for what a plate must not be (a wall with a window, a doubled
triangle, a rotated or sloping face, a T-junction), for mixes of plates and
other triangles, and for segments at a plate's borders and in its plane.
A pair may only differ where the oracle flags it as grazing."""
import numpy as np
import pytest
import torch

import oracle
import paper_2103_14137_gb300 as uvc
from synth.scenes import Lamp, line_lamp, point_lamp
from tests.gpu_util import build_arrays, lamp_of
from tests.test_gpu_wedge import _area, _same_as_per_source

pytestmark = pytest.mark.gpu


def _face(o, eu, ev, nu, nv, skip=()):
    """Triangles (n, 3, 3) of the parallelogram o + s eu + t ev in nu x nv cells, normal along eu x ev."""
    out = []
    for i in range(nu):
        for j in range(nv):
            if (i, j) in skip:
                continue
            p = [np.asarray(o, float) + np.asarray(eu) * a / nu + np.asarray(ev) * b / nv
                 for a, b in ((i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1))]
            out += [[p[0], p[1], p[2]], [p[0], p[2], p[3]]]
    return np.array(out)


def _box(lo, hi, n, sign=1, turn=0.0, skip_top=()):
    """Faces of a box (sign -1: seen from inside), turned about its vertical axis."""
    lo, hi = np.asarray(lo, float), np.asarray(hi, float)
    d, f = hi - lo, []
    for k in range(3):
        u, v = np.eye(3)[(k + 1) % 3] * d, np.eye(3)[(k + 2) % 3] * d
        for side in (0, 1):
            o = lo + np.eye(3)[k] * d * side
            a, b = (u, v) if (side == 1) == (sign > 0) else (v, u)
            f.append(_face(o, a, b, n, n, skip_top if (k, side) == (2, 1) else ()))
    T = np.concatenate(f)
    if turn:
        c, s, m = np.cos(turn), np.sin(turn), (lo + hi) / 2
        T = (T - m) @ np.array([[c, s, 0], [-s, c, 0], [0, 0, 1]]) + m
    return T


def _scenes():
    room = _box([0, 0, 0], [4, 3, 2.5], 6, -1)
    bed, chest = _box([1, 1, 0.25], [2, 2, 0.75], 3), _box([2.5, 0.5, 0], [3, 1.25, 1.5], 2)
    return {
        "plates_only": (np.concatenate([room, bed, chest]), False),
        "window_in_a_wall": (np.concatenate([room, bed, _face([3, 0, 0], [0, 3, 0], [0, 0, 2.5], 6, 5, {(2, 2), (3, 2)})]), True),
        "turned_box": (np.concatenate([room, bed, _box([2.4, 0.6, 0], [3.2, 1.3, 1.5], 3, 1, 0.4)]), True),
        "sloping_face": (np.concatenate([room, _face([1, 1, 0.5], [1, 0, 0], [0, 1, 0.125], 4, 4)]), True),
        "doubled_triangle": (np.concatenate([room, bed, bed[:1]]), True),
        # two rectangles whose cells do not match along their common border: each is a plate by itself
        "abutting_plates": (np.concatenate([room, _face([1, 1, 1], [1, 0, 0], [0, 1, 0], 2, 2),
                                            _face([2, 1, 1], [1, 0, 0], [0, 1, 0], 2, 3)]), False),
        # joined along half of that border, with a T-junction in the other half
        "t_junction": (np.concatenate([room, _face([1, 1, 1], [1, 0, 0], [0, 1, 0], 2, 2),
                                       _face([2, 1, 1], [1, 0, 0], [0, 0.5, 0], 2, 1),
                                       _face([2, 1.5, 1], [1, 0, 0], [0, 0.5, 0], 2, 2)]), True),
        # the scene keeps its plates while the loose triangles are at most 8 times the 48 of the inner ones
        "loose_at_the_line": (np.concatenate([room, _box([1, 1, 0.25], [2, 2, 0.75], 2), _face([2.2, 1, 0.5], [1, 0, 0.2], [0, 1, 0], 12, 16)]), True),
        "loose_over_the_line": (np.concatenate([room, _box([1, 1, 0.25], [2, 2, 0.75], 2), _face([2.2, 1, 0.5], [1, 0, 0.2], [0, 1, 0], 193, 1)]), True),
        "walls_and_turned_box": (np.concatenate([room, _box([1.4, 0.6, 0.1], [3.2, 1.3, 1.5], 3, 1, 0.4)]), True),
        "thin_triangles": (np.concatenate([room, _face([1, 1, 1], [1.5, 0, 0], [0, 0.5, 0], 1, 40)]), True),
        "over_32_plates": (np.concatenate([room] + [_box([0.3 + 0.5 * i, 0.4 + 0.6 * j, 0.1], [0.6 + 0.5 * i, 0.7 + 0.6 * j, 0.5 + 0.2 * j], 2)
                                                    for i in range(7) for j in range(4)]), False),
        "over_1024_plates": (np.concatenate([room] + [_box([0.1 + 0.2 * i, 0.1 + 0.2 * j, 0.1], [0.2 + 0.2 * i, 0.2 + 0.2 * j, 0.3], 2)
                                                      for i in range(19) for j in range(14)]), True),
    }


def _lamps():
    tube = Lamp(np.stack([np.linspace(-0.4, 0.4, 5), np.zeros(5), np.zeros(5)], 1).astype(np.float32),
                np.full(5, 0.2, np.float32), 90.0)
    return {"line2": line_lamp(0.5, 2, 60.0), "line16": line_lamp(1.2, 16, 120.0), "point": point_lamp(80.0), "tube": tube}


def _patches(T, name):
    """The scene's arrays and 300 patches on its triangles: (verts, tris, points, normals, excl), and the
    patches' own triangles."""
    verts, inv = np.unique(T.reshape(-1, 3).astype(np.float32), axis=0, return_inverse=True)
    tris = inv.reshape(-1, 3).astype(np.int32)
    rng = np.random.default_rng(len(name))
    V = verts.astype(np.float64)[tris]
    n = np.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
    n = (n / np.linalg.norm(n, axis=1, keepdims=True))
    own = rng.permutation(T.shape[0])[:300]           # a ragged number of warps
    w = rng.dirichlet([2, 2, 2], own.size)
    cen = np.einsum("ij,ijk->ik", w, V[own]).astype(np.float32)
    for a in range(3):                                # points of flat faces lie in their plane exactly
        flat = (V[own][:, :, a] == V[own][:, :1, a]).all(1)
        cen[flat, a] = V[own][flat, 0, a]
    excl = np.stack([own, np.full(own.size, -1)], 1).astype(np.int32)
    excl[::17, 1] = rng.integers(0, T.shape[0], excl[::17].shape[0])   # an excluded triangle elsewhere
    nrm = n[own].astype(np.float32)
    nrm[np.abs(nrm) < 1e-7] = 0.0
    cand = rng.uniform([0.1, 0.1, 0.1], [3.9, 2.9, 1.2], (24, 3)).astype(np.float32)
    cand[:8, 0] = [1.0, 2.0, 2.5, 3.0, 0.5, 1.5, 2.25, 1.0]            # in the planes of faces, above their edges
    cand[:8, 1] = [0.5, 1.0, 1.25, 2.0, 2.0, 0.75, 0.5, 2.0]
    cand[8:12, 2] = [0.25, 0.5, 0.75, 1.0]
    return (verts, tris, cen, nrm, excl), V[own].astype(np.float32), cand


@pytest.mark.parametrize("name", list(_scenes()))
def test_plates_give_the_search_results(name):
    T, loose = _scenes()[name]
    arrays, _, cand = _patches(T, name)
    sc = build_arrays(*arrays[:4], np.ones(300, np.float32), arrays[4])
    assert (uvc.scene_export_traversal(sc)["nodes4"][0, 30] != 0) == loose
    for L in _lamps().values():
        _same_as_per_source(arrays, sc, cand, L)
    torch.cuda.synchronize()
    sc.free()


@pytest.mark.parametrize("shift", [(64.0, -32.0, 16.0), (-300.0, 500.0, 100.0)])
@pytest.mark.parametrize("name", ["plates_only", "over_32_plates"])
def test_plates_far_from_the_origin(name, shift):
    """The decisions rest on differences of coordinates, as the search's triangle tests do."""
    T, _ = _scenes()[name]
    (verts, tris, cen, nrm, excl), _, cand = _patches(T, name)
    verts, cen, cand = (np.float32(x + np.float32(shift)) for x in (verts, cen, cand))
    sc = build_arrays(verts, tris, cen, nrm, np.ones(300, np.float32), excl)
    for L in _lamps().values():
        _same_as_per_source((verts, tris, cen, nrm, excl), sc, cand, L)
    sc.free()


@pytest.mark.parametrize("name", ["plates_only", "window_in_a_wall", "doubled_triangle", "over_32_plates"])
@pytest.mark.parametrize("lamp", ["line2", "line16"])
def test_area_mean_at_plates_gives_the_search_results(name, lamp):
    """Check points, too, are decided at plates: patches that are their excluded triangle, the half of it, a
    part reaching outside of it, and patches that exclude nothing."""
    T, _ = _scenes()[name]
    arrays, own, cand = _patches(T, name)
    verts, tris, cen, nrm, excl = arrays
    s = cen[:, None, :]
    ptri = np.zeros((300, 2, 3, 3), np.float32)
    ptri[:, 0] = own
    ptri[1::4, 0, 2] = 0.5 * (own[1::4, 1] + own[1::4, 2])
    ptri[2::4, 0] = s[2::4] + 1.5 * (own[2::4] - s[2::4])
    excl[3::4, 0] = -1
    area = np.full(300, 0.1, np.float32)
    sc = build_arrays(verts, tris, cen, nrm, area, excl)
    L = _lamps()[lamp]
    Aw, cw = _area(sc, cand, lamp_of(L), ptri, True)
    Ap, cp = _area(sc, cand, lamp_of(L), ptri, False)
    differ = ((Aw != Ap) | (cw != cp)).cpu().numpy()
    if differ.any():
        pairs = np.argwhere(differ)
        _, _, flag = oracle.area_mean(verts, tris, cen, nrm, area, excl, ptri, cand, L.offsets, L.weights, L.power,
                                      pairs=pairs)
        assert np.all(flag != 0), f"{int((flag == 0).sum())} of {pairs.shape[0]} differing pairs are not grazing"
    assert (cw > 0).any()
    sc.free()
