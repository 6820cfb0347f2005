"""Candidate features and selection where their kernels can go wrong: patches on
the very edges of the distance bins and next to them in FP32, no patch, one
candidate; scenes of no, one and many triangles for the nearest distance; the
selection over all byte patterns of the scores, with ties, NaN and
infinities, at one score and at the most it takes."""
import numpy as np
import pytest

import paper_2103_14137_gb300 as uvc
from tests.gpu_util import T, build_arrays

pytestmark = pytest.mark.gpu


def _edges():
    return np.array([np.float32((0.1 * 250.0 ** (b / 64)) ** 2) for b in range(1, 64)], np.float32)


@pytest.mark.parametrize("nc", [1, 3])
def test_bins_at_their_edges(nc):
    e = _edges()
    x = np.concatenate([np.sqrt(e.astype(np.float64)), [0.0, 1e-6, 1e3]]).astype(np.float32)
    x = np.unique(np.concatenate([x, np.nextafter(x, np.float32(np.inf)), np.nextafter(x, np.float32(0))]))
    cen = np.stack([x, np.zeros_like(x), np.zeros_like(x)], 1)
    n = x.size
    area = np.exp2(-np.arange(n) % 24).astype(np.float32)      # sums of a bin's few areas are exact
    sc = build_arrays(np.zeros((0, 3)), np.zeros((0, 3)), cen, np.tile([[0, 0, 1]], (n, 1)), area, -np.ones((n, 2)))
    cand = np.zeros((nc, 3), np.float32)
    cand[1:, 2] = 0.75
    f = uvc.candidate_features(sc, T(cand)).cpu().numpy()
    d2 = (x * x).astype(np.float32)                            # one rounding on the axis
    want = np.bincount(np.searchsorted(e, d2, side="right"), weights=area.astype(np.float64), minlength=64)
    np.testing.assert_allclose(f[0, :64], want / area.astype(np.float64).sum(), rtol=2e-6, atol=0)
    assert np.all(np.abs(f[:, :64].sum(1) - 1) < 1e-5) and np.all(f[:, 64] > 1e38) and np.array_equal(f[:, 65], cand[:, 2])
    sc.free()


@pytest.mark.parametrize("nt", [1, 2, 3, 700])
def test_nearest_triangle(nt):
    rng = np.random.default_rng(nt)
    V = (rng.uniform(0, 4, (nt, 1, 3)) + rng.uniform(-0.2, 0.2, (nt, 3, 3))).astype(np.float32)
    sc = build_arrays(V.reshape(-1, 3), np.arange(3 * nt).reshape(-1, 3), np.ones((1, 3)), [[0, 0, 1]], [1.0], [[-1, -1]])
    c = rng.uniform(-1, 5, (37, 3)).astype(np.float32)
    got = uvc.candidate_features(sc, T(c)).cpu().numpy()[:, 64]
    s = np.linspace(0, 1, 41)                                  # a dense sample of every triangle bounds it from above
    u, v = (a.ravel() for a in np.meshgrid(s, s))
    u, v = u[u + v <= 1], v[u + v <= 1]
    P = V[:, :1].astype(np.float64) + u[None, :, None] * (V[:, 1:2] - V[:, :1]) + v[None, :, None] * (V[:, 2:] - V[:, :1])
    near = np.array([np.linalg.norm(P - x, axis=-1).min() for x in c.astype(np.float64)])
    step = np.linalg.norm(V[:, 1:] - V[:, :1], axis=-1).max() / 40
    assert np.all(got <= near + 1e-5) and np.all(got >= near - step)
    sc.free()


@pytest.mark.parametrize("n,k", [(1, 1), (2, 1), (255, 256 - 1), (1023, 77), (4096, 4000), (16384, 1), (16384, 8191), (16384, 16384)])
@pytest.mark.parametrize("what", ["bits", "ties", "few"])
def test_selection(n, k, what):
    rng = np.random.default_rng(n + k)
    if what == "bits":
        s = rng.integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32).view(np.float32)
    elif what == "ties":
        s = rng.integers(-3, 4, n).astype(np.float32)
        s[rng.random(n) < 0.1] = np.nan
    else:
        s = np.where(rng.random(n) < 0.5, -np.inf, np.inf).astype(np.float32)
    key = np.where(np.isnan(s), -np.inf, s.astype(np.float64))
    key = np.where(s == 0, np.where(np.signbit(s), -1e-46, 0.0), key)         # -0 ranks below +0
    order = np.lexsort((np.arange(n), np.isnan(s), -key))                       # NaN last, then the lower index
    cand = rng.uniform(size=(n, 3)).astype(np.float32)
    idx, kept = uvc.select_top(T(s), k, cand=T(cand))
    want = np.sort(order[:k])
    assert np.array_equal(idx.cpu().numpy(), want) and np.array_equal(kept.cpu().numpy(), cand[want])
