"""A batch of rooms with plates and rooms without, in any order: each job's matrix
and visibility words are those of the single call, in a launch, after autotuning,
and replayed from a graph, and jobs of no candidates take no part."""
import numpy as np
import pytest
import torch

import paper_2103_14137_gb300 as uvc
from synth.scenes import line_lamp
from tests.gpu_util import T, build_arrays, lamp_of
from tests.test_gpu_plates import _patches, _scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", ["plates first", "plates last", "mixed", "plates only", "none"])
def test_jobs_with_and_without_plates(order):
    scenes = []
    turn = np.array([[0.8, -0.6, 0], [0.6, 0.8, 0], [0, 0, 1]]) @ np.array([[1, 0, 0], [0, 0.96, -0.28], [0, 0.28, 0.96]])
    kinds = {"plates first": [1, 1, 0, 0], "plates last": [0, 0, 1], "mixed": [0, 1, 0, 1, 1], "plates only": [1, 1], "none": [0, 0]}[order]
    for q, flat in enumerate(kinds):
        V, _ = _scenes()[("plates_only", "over_32_plates")[q % 2]]
        (verts, tris, cen, nrm, excl), _, cand = _patches(V, "room" * (q + 1))
        if not flat:
            verts, cen, nrm, cand = (np.float32(x.astype(np.float64) @ turn.T) for x in (verts, cen, nrm, cand))
        sc = build_arrays(verts, tris, cen, nrm, np.ones(300, np.float32), excl)
        scenes.append((sc, T(cand)))
    lamps = [lamp_of(line_lamp(0.5, 2, 60.0)), lamp_of(line_lamp(1.2, 8, 120.0))]
    jobs = []
    for q, (sc, cand) in enumerate(scenes):
        for d in range(2):
            n = 0 if (q, d) == (1, 1) else cand.shape[0]
            jobs.append((sc, cand[:n], d, torch.full((n, sc.np), -1.0, device="cuda"),
                         torch.zeros((lamps[d].K, n, (sc.np + 31) // 32), dtype=torch.int32, device="cuda")))
    want = [uvc.irradiance_matrix(sc, cand, lamps[d], with_vis=True) for sc, cand, d, _, _ in jobs]

    def check():
        torch.cuda.synchronize()
        for (_, _, _, A, vis), (A0, v0) in zip(jobs, want):
            assert torch.equal(A, A0) and torch.equal(vis, v0)
            A.fill_(-1.0)
            vis.zero_()

    b = uvc.Batch(jobs, lamps)
    b.launch()
    check()
    b.autotune(0.3)
    b.launch()
    check()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.launch()
    g.replay()
    check()
    b.free()
    for sc, _ in scenes:
        sc.free()
