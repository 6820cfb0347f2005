"""The scorer's tensor-core products at the edges of their tiles (128 rows, 64
columns, slices of 128 along K, slices of the batch): logits and gradients
against the FP64 oracle of the BF16 network, with the tolerances of
tests/test_gpu_proposal.py (logits: 2^-8 of the terms' magnitude; gradients: 1 %
in norm, as BF16 rounds each activation by up to 2^-9)."""
import numpy as np
import pytest

import paper_2103_14137_gb300 as uvc
from oracle import mlp as OM
from tests.gpu_util import T
from tests.test_gpu_proposal import logit_tol, seeded_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,H,B", [(1, 8, 1), (16, 8, 129), (17, 64, 127), (114, 136, 128), (130, 72, 300), (300, 264, 2049)])
def test_products_at_tile_edges(d, H, B):
    rng = np.random.default_rng(d + H + B)
    m = uvc.Mlp(d, H, max_batch=B)
    flat = seeded_params(d, H, 3)
    m.set_params(flat)
    x = rng.uniform(-1.0, 1.0, (B, d)).astype(np.float32)
    got = m.forward(T(x)).cpu().numpy().astype(np.float64)
    want, tol = logit_tol(flat, x, d, H)
    assert np.all(np.abs(got - want) <= tol), np.max(np.abs(got - want) / tol)
    y, w = rng.uniform(size=B).astype(np.float32), rng.uniform(0.5, 2.0, B).astype(np.float32) / B
    m.train_step(T(x), T(y), T(w), 1e-3)
    _, g = OM.gradients(flat, x, y, w, d, H, quant=True)
    gp, go = m.split(m.grads().astype(np.float64)), m.split(g)
    for name in gp:
        err = np.linalg.norm(gp[name] - go[name]) / max(np.linalg.norm(go[name]), 1e-30)
        assert err <= 1e-2, (name, err)
    assert np.all(gp["W1"][d:] == 0)
    m.close()
