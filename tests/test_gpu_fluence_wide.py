"""Wide matrices whose rows allow no tensor map: the same bits as the tensor-map
copies give on 16-byte rows (both sum in one order), at the edges of the 128-column
blocks, the passes of 16 vectors and the chunks of rows, and narrow ones of few
rows, whose dwell times are staged in part."""
import numpy as np
import pytest

import oracle
import paper_2103_14137_gb300 as uvc
from tests.gpu_util import T
from tests.test_gpu_fluence import MU_TOL, _rel, _rows_of
from tests.test_gpu_fluence_split import _points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9729, 9856, 9857, 30001])
@pytest.mark.parametrize("nc,nvec", [(1, 1), (33, 16), (130, 17), (513, 40)])
def test_odd_rows_give_the_bits_of_aligned_ones(n, nc, nvec):
    rng, sc, _ = _points(n, n + nc)
    A = np.exp(rng.uniform(np.log(1e-4), np.log(1e2), size=(nc, n))).astype(np.float32)
    A[rng.uniform(size=A.shape) < 0.3] = 0.0
    t = rng.uniform(0, 60, size=(nvec, nc)).astype(np.float32)
    old = uvc.set_fluence_tensor_cores(False)
    out = []
    for lda in ((n + 3) // 4 * 4, n + 1 - n % 2, n + 2 - n % 2):   # 16-byte rows, odd rows, 8-byte rows or odd ones
        Ab = _rows_of(nc, n, lda)
        Ab.copy_(T(A))
        out.append(uvc.fluence(sc, Ab, T(t)).cpu().numpy())
    uvc.set_fluence_tensor_cores(old)
    assert _rel(out[0], oracle.fluence(A, t)) <= MU_TOL
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    sc.free()


@pytest.mark.parametrize("nc", [2, 32, 33, 64, 65, 127, 128, 129, 257])
def test_few_rows_of_a_narrow_matrix(nc):
    rng, sc, _ = _points(70, nc)
    A = rng.uniform(1e-3, 1e2, (nc, 70)).astype(np.float32)
    t = rng.uniform(0, 60, size=(19, nc)).astype(np.float32)
    assert _rel(uvc.fluence(sc, T(A), T(t)).cpu().numpy(), oracle.fluence(A, t)) <= MU_TOL
    sc.free()
