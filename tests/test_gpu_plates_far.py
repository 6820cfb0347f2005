"""Plates in small scenes far from the origin, where the rounding of a coordinate is
more than the boxes' widening (0.05 m at 150 m): lamps that are searched source by
source get the search's results all the same."""
import numpy as np
import pytest

from synth.scenes import Lamp
from tests.gpu_util import build_arrays
from tests.test_gpu_plates import _lamps, _patches, _scenes
from tests.test_gpu_wedge import _same_as_per_source

pytestmark = pytest.mark.gpu


def _lamp(name):
    if name == "long":   # a vertical line of more sources than the merged search takes
        off = np.zeros((20, 3), np.float32)
        off[:, 2] = np.linspace(0.05, 0.9, 20)
        return Lamp(off, np.full(20, 0.05, np.float32), 90.0)
    return _lamps()[name]


@pytest.mark.parametrize("scale, shift", [(0.01, (-82.4, -104.6, -45.4)), (0.01, (193.7, -138.0, -139.4)), (1.0, (3000.0, 2500.0, 900.0))])
@pytest.mark.parametrize("name", ["plates_only", "over_32_plates"])
@pytest.mark.parametrize("lamp", ["point", "tube", "long"])
def test_small_scenes_far_away(scale, shift, name, lamp):
    T, _ = _scenes()[name]
    rng = np.random.default_rng(len(name))
    for trial in range(4):
        (verts, tris, cen, nrm, excl), _, _ = _patches(T, name + "x" * trial)
        cand = rng.uniform([0.1, 0.1, 0.1], [3.9, 2.9, 2.2], (200, 3))
        far = [np.float32(x.astype(np.float64) * scale + np.array(shift)) for x in (verts, cen, cand)]
        V = far[0][tris]
        own = excl[:, 0]
        for a in range(3):   # points of flat faces stay in their plane
            flat = (V[own][:, :, a] == V[own][:, :1, a]).all(1)
            far[1][flat, a] = V[own][flat, 0, a]
        L = _lamp(lamp)
        L = Lamp((L.offsets * np.float32(scale)).astype(np.float32), L.weights, L.power)
        sc = build_arrays(far[0], tris, far[1], nrm, np.ones(300, np.float32), excl)
        _same_as_per_source((far[0], tris, far[1], nrm, excl), sc, far[2], L)
        sc.free()
