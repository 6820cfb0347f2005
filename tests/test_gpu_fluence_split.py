"""The fluence kernels' splits: the CUDA-core kernel's row splits over clusters
of 1 to 8 blocks (narrow matrices; few and many candidates; passes of 16
vectors), the line between narrow matrices and the tensor cores, the
tensor-core kernel's stages and passes on matrices wide enough for it, and
coverage over one to many of its clusters' strides.  Bounds: 1e-5 relative as in
tests/test_gpu_fluence.py (terms are non-negative); coverage 1e-6."""
import numpy as np
import pytest
import torch

import oracle
import paper_2103_14137_gb300 as uvc
from synth.scenes import line_lamp, point_lamp
from tests.gpu_util import T, build_arrays, lamp_of
from tests.test_gpu_fluence import MU_TOL, _rel, _rows_of

pytestmark = pytest.mark.gpu


def _points(n, seed):
    rng = np.random.default_rng(seed)
    nrm = np.tile(np.array([[0, 0, 1]], np.float32), (n, 1))
    area = rng.uniform(0.1, 1.0, n).astype(np.float32)
    sc = build_arrays(np.zeros((0, 3)), np.zeros((0, 3)), rng.uniform(0, 1, (n, 3)), nrm, area, -np.ones((n, 2)))
    return rng, sc, area


@pytest.mark.parametrize("n", [1, 63, 65, 1000, 9728, 9729, 9852])
@pytest.mark.parametrize("nc,nvec", [(1, 1), (31, 16), (33, 17), (255, 2), (256, 33), (1025, 3)])
def test_row_splits_and_the_line_to_the_tensor_cores(n, nc, nvec):
    rng, sc, _ = _points(n, n + nc)
    A = np.exp(rng.uniform(np.log(1e-4), np.log(1e2), size=(nc, n))).astype(np.float32)
    A[rng.uniform(size=A.shape) < 0.3] = 0.0
    t = rng.uniform(0, 60, size=(nvec, nc)).astype(np.float32)
    ref = oracle.fluence(A, t)
    out = []
    for lda in ((n + 3) // 4 * 4, n + 1 - n % 2):      # rows on 16-byte boundaries, odd rows
        Ab = _rows_of(nc, n, lda)
        Ab.copy_(T(A))
        out.append(uvc.fluence(sc, Ab, T(t)).cpu().numpy())
        assert np.all(out[-1][ref == 0] == 0) and _rel(out[-1], ref) <= MU_TOL, (lda, _rel(out[-1], ref))
    assert uvc.scene_status(sc) == 0
    if n <= 9728:
        assert np.array_equal(out[0], out[1])          # narrow matrices take one kernel whatever their rows
    sc.free()


@pytest.mark.parametrize("n,nvec", [(1, 1), (511, 3), (4096, 2), (4097, 1), (70000, 5)])
def test_coverage_over_clusters(n, nvec):
    rng, sc, area = _points(n, n)
    mu = rng.uniform(0.0, 200.0, (nvec, n)).astype(np.float32)
    mu[0] = 100.0                                       # the threshold itself counts
    ca, cc = uvc.coverage(sc, T(mu), 100.0)
    torch.cuda.synchronize()
    ok = mu >= np.float32(100.0)
    a = area.astype(np.float64)
    np.testing.assert_allclose(ca.cpu().numpy(), (ok * a).sum(1) / a.sum(), rtol=1e-6)
    np.testing.assert_allclose(cc.cpu().numpy(), ok.mean(1), rtol=1e-6)
    sc.free()


@pytest.mark.parametrize("nvec", [1, 31, 32, 33, 70])
@pytest.mark.parametrize("nc", [1, 3, 19, 20, 21, 45])
def test_streamed_stages_of_candidates_and_vectors(nc, nvec):
    """Stages of 20 candidates by 32 vectors, whole and ragged, against the product of the stored entries: non-negative
    sums of at most 45 terms in FP32, so within 50 x 2^-24 = 3e-6."""
    rng, sc, _ = _points(100, nc + nvec)
    cand = T(rng.uniform([0, 0, 1], [1, 1, 2], (nc, 3)).astype(np.float32))
    t = rng.uniform(0, 60, size=(nvec, nc)).astype(np.float32)
    t[:, ::4] = 0.0
    for lamp in (lamp_of(point_lamp(80.0)), lamp_of(line_lamp(0.5, 3, 60.0))):
        A, _ = uvc.irradiance_matrix(sc, cand, lamp)
        ref = t.astype(np.float64) @ A[:, :100].cpu().numpy().astype(np.float64)
        mu = uvc.fluence_streamed(sc, cand, lamp, T(t)).cpu().numpy()
        assert _rel(mu, ref) <= 3e-6, _rel(mu, ref)
    sc.free()


@pytest.mark.parametrize("n", [1, 1023, 1025, 9000, 70001])
def test_area_sums_keep_their_order(n):
    """Coverage and the scene's area: 1024 compensated chains, then trees of 32 and 32, bit for bit."""
    rng, sc, area = _points(n, n)
    mu = rng.uniform(0, 2, (2, n)).astype(np.float32)

    def total(a):   # masked patches leave their chain as it is
        a = np.concatenate([a, np.full(-n % 1024, np.nan, np.float32)]).reshape(-1, 1024)
        s, c = np.zeros(1024, np.float32), np.zeros(1024, np.float32)
        for row in a:
            ok = ~np.isnan(row)
            y = row - c
            t = s + y
            c, s = np.where(ok, (t - s) - y, c), np.where(ok, t, s)
        s = (s - c).reshape(32, 32)
        for w in (16, 8, 4, 2, 1):
            s = s[:, :w] + s[:, w:2 * w]
        s = s[:, 0]
        for w in (16, 8, 4, 2, 1):
            s = s[:w] + s[w:2 * w]
        return s[0]

    got = uvc.coverage(sc, T(mu), 1.0)[0].cpu().numpy()
    assert np.array_equal(got, np.float32([total(np.where(m >= 1.0, area, np.nan)) / total(area) for m in mu]))
    sc.free()
