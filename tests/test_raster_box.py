"""The pixels that the rasteriser tests a triangle at (csrc/raster_box.h, compiled
here without CUDA): all centres inside the projection, and next to the source's own
plane the next centre outwards and one more on either side, never a third, as
there the ray test hits pixels anywhere."""
import ctypes
import subprocess

import numpy as np
import pytest


@pytest.fixture(scope="module")
def pixel_range(tmp_path_factory):
    d = tmp_path_factory.mktemp("box")
    (d / "box.cpp").write_text('#include "raster_box.h"\nextern "C" void range(int n, const float* lo, const float* hi, int R, '
                               "int deep, int* o) {\n    for (int k = 0; k < n; ++k) {\n"
                               "        const uvc::PixelRange p = uvc::pixel_range(lo[k], hi[k], R, deep != 0);\n"
                               "        o[2 * k] = p.first; o[2 * k + 1] = p.last;\n    }\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I", "paper_2103_14137_gb300/csrc",
                    str(d / "box.cpp"), "-o", str(d / "box.so")], check=True)
    lib = ctypes.CDLL(str(d / "box.so"))

    def call(lo, hi, R, deep):
        o = np.empty((lo.size, 2), np.int32)
        lib.range(lo.size, lo.ctypes.data_as(ctypes.c_void_p), hi.ctypes.data_as(ctypes.c_void_p), R, int(deep),
                  o.ctypes.data_as(ctypes.c_void_p))
        return o.T
    return call


@pytest.mark.parametrize("R", [1, 2, 5, 16, 33, 64, 511, 512, 4096])
def test_pixels_of_a_projection(pixel_range, R):
    c = (2 * np.arange(R) + 1) / R - 1
    rng = np.random.default_rng(R)
    ends = np.concatenate([c, c + 0.3 / R, [0.0, -1.0, 1.0, 0.25, -0.5], rng.uniform(-1, 1, 200)]).clip(-1, 1)
    lo, hi = np.sort(rng.choice(ends, (3000, 2)), axis=1).astype(np.float32).T.copy()
    hi[:1000] = lo[:1000]                          # edge-on: no extent, on a centre and off
    a, b = ((x.astype(np.float64) + 1) * R / 2 - 0.5 for x in (lo, hi))   # in pixels
    tol = 1e-3 if R < 1000 else 0.02               # FP32 of the range's own arithmetic, in pixels
    f, l = pixel_range(lo, hi, R, False)
    assert np.all(f <= np.maximum(0, np.ceil(a - tol))) and np.all(l >= np.minimum(R - 1, np.floor(b + tol)))
    assert np.all(f >= np.maximum(0, np.floor(a - tol) - 1)) and np.all(l <= np.minimum(R - 1, np.ceil(b + tol) + 1))
    on = (a == np.round(a)) & (a >= 2)             # exactly on a centre: that one and one more outwards
    assert np.all(f[on] >= a[on] - 1 - (tol > 0.01))
    f, l = pixel_range(lo, hi, R, True)
    assert np.all(f <= np.maximum(0, np.ceil(a))) and np.all(l >= np.minimum(R - 1, np.floor(b)))
    assert np.all(f >= np.maximum(0, np.ceil(a - 0.032 - tol))) and np.all(l <= np.minimum(R - 1, np.floor(b + 0.032 + tol)))
