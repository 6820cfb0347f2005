"""Device memory of a build, which it maps and gives back each time: the scene's own
arrays and the temporaries of its steps, with none for the search for plates
beside those it finds spent."""
import ctypes

import numpy as np
import pytest
import torch

from tests.test_gpu_build_edges import _built, _soup

pytestmark = pytest.mark.gpu

# tri 48, nodes 64, four-wide nodes 128, keys 8, order 4, place 8; boxes and
# reference points 48, keys 8, values 8, heights, depths, costs and parents 16,
# children and parents 16, leaf and node boxes 64, flags 4, marks 8, level counts 4
SCENE, TEMPORARY = 260, 176


def _used_high(reset):
    rt = ctypes.CDLL("libcudart.so.13")
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    v = ctypes.c_uint64(0)
    if reset:
        assert rt.cudaMemPoolSetAttribute(pool, 8, ctypes.byref(v)) == 0   # cudaMemPoolAttrUsedMemHigh
    assert rt.cudaMemPoolGetAttribute(pool, 8, ctypes.byref(v)) == 0
    return v.value


@pytest.mark.parametrize("n", [200000, 500000])
def test_plates_search_takes_no_memory_of_its_own(n):
    verts, tris = _soup(n, np.random.default_rng(n).uniform(0, 5, (n, 3)))
    torch.cuda.synchronize()
    before = _used_high(True)
    sc = _built(verts, tris)
    used = _used_high(False) - before
    sc.free()
    # and 2 MB for the radix sort's histograms, the plates and the arrays' alignment
    assert used <= (SCENE + TEMPORARY) * n + (2 << 20), used / n
