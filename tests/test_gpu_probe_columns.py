"""The probe-column kernels over their three shapes: column counts at the lines
between them and off the blocks' widths, row counts off the slices and the batches
of rows.  Marks, lost areas and the features of padded matrices are exact."""
import numpy as np
import pytest
import torch

import paper_2103_14137_gb300 as uvc
from tests.gpu_util import T

pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("nc", [1, 7, 31, 33, 257, 1025])
@pytest.mark.parametrize("cols", ["one", "few", "few_end", "mid", "mid_end", "many"])
def test_shapes(cols, nc):
    n = {"one": 1, "few": 511, "few_end": 8 * _sms(), "mid": 8 * _sms() + 1, "mid_end": 64 * _sms(), "many": 64 * _sms() + 1}[cols]
    rng = np.random.default_rng(n + nc)
    A = rng.uniform(0.1, 1.0, (nc, n)).astype(np.float32)
    A[rng.random(A.shape) < (0.6 if nc < 100 else 0.995)] = 0.0
    A[:, rng.random(n) < 0.1] = 0.0                        # unlit columns
    if nc > 40:
        A[nc - 30:, ::7] = np.maximum(A[nc - 30:, ::7], np.float32(0.5))   # ties
        A[nc - 9:, ::7] = np.where(A[nc - 9:, ::7] > 0, np.float32(1.0), 0)
    area = rng.uniform(0.1, 1.0, n).astype(np.float32)
    dA, rare = T(A), 2
    want = np.zeros(nc, np.float32)
    lit = A > 0
    want[A.argmax(0)[lit.any(0)]] = 5.0                    # argmax: the lowest row among equals
    few = lit.any(0) & (lit.sum(0) <= rare)
    want[lit[:, few].any(1)] = 5.0
    score = torch.zeros(nc, device="cuda")
    uvc.mark_best(dA, score, value=5.0, rare=rare)
    assert np.array_equal(score.cpu().numpy(), want)
    idx = np.sort(rng.choice(nc, max(1, nc // 3), replace=False)).astype(np.int32)
    lost = torch.empty(n, device="cuda")
    total = uvc.probe_lost(dA, T(idx), T(area), lost=lost)
    keep = lit.any(0) & ~lit[idx].any(0)
    assert np.array_equal(lost.cpu().numpy(), np.where(keep, area, np.float32(0)))
    np.testing.assert_allclose(total.cpu().numpy(), (keep * area.astype(np.float64)).sum() / area.astype(np.float64).sum(), rtol=1e-5)
    # unlit columns add nothing: the same features, bit for bit, from a matrix of the widest shape
    wide = torch.zeros((nc, 64 * _sms() + 1), device="cuda")
    wide[:, :n] = dA
    warea = torch.ones(wide.shape[1], device="cuda")
    warea[:n] = T(area)
    assert torch.equal(uvc.probe_features(dA, T(area)), uvc.probe_features(wide, warea))
