"""Coverage by one block a vector and by a cluster: either side of the line in
patches and in vectors gives the same bits (one order of additions)."""
import numpy as np
import pytest
import torch

import paper_2103_14137_gb300 as uvc
from tests.gpu_util import T
from tests.test_gpu_fluence_split import _points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 49152, 49153, 60001])
def test_block_and_cluster_agree(n):
    rng, sc, _ = _points(n, n)
    many = torch.cuda.get_device_properties(0).multi_processor_count + 1     # vectors past which no cluster is used
    mu = rng.uniform(0, 2, (many, n)).astype(np.float32)
    a, c = (x.cpu().numpy() for x in uvc.coverage(sc, T(mu), 1.0))
    for v in (0, many - 1):
        a1, c1 = (x.cpu().numpy() for x in uvc.coverage(sc, T(mu[v:v + 1]), 1.0))
        assert a1[0] == a[v] and c1[0] == c[v]
    sc.free()
