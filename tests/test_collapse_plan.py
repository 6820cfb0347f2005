"""The launches that make the four-wide tree: no level may be launched whose
node count nothing wrote.  The plan is host arithmetic (csrc/collapse_plan.h),
compiled here without CUDA; on a GPU, scenes of two to five triangles, whose
trees are shallower than the plan's first launch, are built with a large scene
alive and another one just freed, so that their memory is not fresh."""
import ctypes
import subprocess

import numpy as np
import pytest

CSRC = "paper_2103_14137_gb300/csrc"


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text('#include "collapse_plan.h"\nextern "C" void plan(int depth, long long n, int* o) {\n'
                                "    const uvc::CollapsePlan p = uvc::collapse_plan(depth, n);\n"
                                "    o[0] = p.levels; o[1] = p.counters; o[2] = p.top; o[3] = p.tail;\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(d / "plan.cpp"), "-o",
                    str(d / "plan.so")], check=True)
    lib = ctypes.CDLL(str(d / "plan.so"))

    def call(depth, n):
        o = (ctypes.c_int * 4)()
        lib.plan(ctypes.c_int(depth), ctypes.c_longlong(n), o)
        return list(o)
    return call


def test_every_launched_level_has_its_counter_cleared(plan):
    for depth in range(1, 200):
        for n in {depth + 1, depth + 2, 4 * depth, 1000, 30604, 311296, 10 ** 6, 10 ** 7, min(2 ** depth, 2 ** 31 - 1)}:
            if n < depth + 1 or (depth < 31 and n > 2 ** depth):
                continue   # no binary tree of n leaves has this depth
            levels, counters, top, tail = plan(depth, n)
            assert levels == depth + 1
            assert 0 <= top <= tail <= levels
            read = list(range(top)) + list(range(top, tail)) + list(range(tail, levels))
            assert read == list(range(levels))           # every level once, none past the tree
            assert max(read) + 1 < counters <= n + 2     # the counter a level adds to is cleared and allocated


@pytest.mark.gpu
@pytest.mark.parametrize("n", [2, 3, 4, 5])
def test_small_scenes_in_used_memory(n):
    import paper_2103_14137_gb300 as uvc
    from tests.test_gpu_build_edges import _built, _soup

    def nodes(sc):
        return uvc.scene_export_traversal(sc)["nodes4"].copy()

    rng = np.random.default_rng(n)
    small = _soup(n, rng.uniform(0, 5, (n, 3)))
    sc = _built(*small)
    want = nodes(sc)
    sc.free()
    big = _soup(60000, rng.uniform(0, 5, (60000, 3)))
    alive, gone = _built(*big), _built(*big)
    before = nodes(alive)
    gone.free()
    sc = _built(*small)
    got = nodes(sc)
    r = want[:, 24:28].astype(np.int64).astype(np.int32)
    level, leaves = np.array([0]), []
    while level.size:
        assert np.array_equal(got[level], want[level])   # the other rows are not nodes
        kids = r[level].ravel()
        leaves += list(~kids[kids < 0])
        level = kids[(kids >= 0) & (kids < n)]
    assert sorted(leaves) == list(range(n))
    assert np.array_equal(nodes(alive), before)
    sc.free()
    alive.free()
