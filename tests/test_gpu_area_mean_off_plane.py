"""Area means of patches whose geometry lies off the plane of their excluded
triangle while their sample point lies in it: the segments to the check points
cross the excluded triangle, which never occludes, and the triangles around it,
which do."""
import numpy as np
import pytest
import torch

import paper_2103_14137_gb300 as uvc
from tests.gpu_util import build_arrays, lamp_of
from tests.test_gpu_plates import _lamps, _patches, _scenes
from tests.test_gpu_wedge import _area

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["plates_only", "window_in_a_wall"])
@pytest.mark.parametrize("depth", [1e-6, 0.002, 0.05])
@pytest.mark.parametrize("lamp", ["line2", "line16"])
def test_geometry_behind_the_excluded_triangle(name, depth, lamp):
    T, _ = _scenes()[name]
    (verts, tris, cen, nrm, excl), own, cand = _patches(T, name)
    ptri = np.zeros((300, 2, 3, 3), np.float32)
    ptri[:, 0] = cen[:, None] + 0.4 * (own - cen[:, None]) - np.float32(depth) * nrm[:, None]
    ptri[::3, 0] = own[::3]                               # and some in it
    area = np.full(300, 0.1, np.float32)
    sc = build_arrays(verts, tris, cen, nrm, area, excl)
    Aw, cw = _area(sc, cand, lamp_of(_lamps()[lamp]), ptri, True)
    Ap, cp = _area(sc, cand, lamp_of(_lamps()[lamp]), ptri, False)
    torch.cuda.synchronize()
    assert uvc.scene_status(sc) == 0 and (cp > 0).any()
    differ = (Aw != Ap) | (cw != cp)
    assert not differ.any(), f"{int(differ.sum())} of {differ.numel()} entries"
    sc.free()
