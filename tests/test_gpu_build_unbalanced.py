"""The last levels of the four-wide tree, which hold most of an unbalanced tree's
nodes: the launch that makes them has a thread for each (on the CPU), and a hall
with one densely meshed object gets its whole tree (on a GPU)."""
import ctypes
import subprocess

import numpy as np
import pytest


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text('#include "collapse_plan.h"\nextern "C" int blocks(long long n, int resident) '
                                "{ return uvc::collapse_blocks(n, resident); }\n"
                                'extern "C" int threads() { return uvc::kCollapseThreads; }\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", "paper_2103_14137_gb300/csrc",
                    str(d / "plan.cpp"), "-o", str(d / "plan.so")], check=True)
    lib = ctypes.CDLL(str(d / "plan.so"))
    return lambda n, resident: (lib.blocks(ctypes.c_longlong(n), ctypes.c_int(resident)), lib.threads())


@pytest.mark.parametrize("resident", [1, 152, 304, 456])
def test_a_thread_for_every_node_of_a_level(blocks, resident):
    for n in [2, 3, 1024, 1025, 30604, 311296, 10 ** 6, 2 * 10 ** 6, 2 ** 31 - 1]:
        b, threads = blocks(n, resident)
        assert 1 <= b <= resident                       # a cooperative launch of more would be refused
        assert b == resident or b * threads >= n // 2   # a level has at most n / 2 nodes
        assert b == 1 or (b - 1) * threads < n // 2     # and no block has nothing


@pytest.mark.gpu
@pytest.mark.parametrize("n", [5, 2000, 60000, 300000])
@pytest.mark.parametrize("size", [0.3, 0.01])
def test_hall_with_a_dense_object(n, size):
    import paper_2103_14137_gb300 as uvc
    from tests.test_gpu_build_edges import _built, _soup
    rng = np.random.default_rng(n)
    p = rng.uniform(0, 60, (n, 3))
    m = int(0.95 * n)
    p[:m] = np.array([20.3, 11.7, 1.0]) + size * rng.uniform(0, 1, (m, 3))
    sc = _built(*_soup(n, p))
    r = uvc.scene_export_traversal(sc)["nodes4"][:, 24:28].astype(np.int64).astype(np.int32)
    seen, level = np.zeros(n, np.int64), np.array([0])
    while level.size:
        kids = r[level].ravel()
        np.add.at(seen, ~kids[kids < 0], 1)
        level = kids[(kids >= 0) & (kids < n)]
    assert (seen == 1).all()
    sc.free()
