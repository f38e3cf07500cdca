"""Gradients at the edges of the products' chunks of 64 rows: one row, one
chunk (no split products: the bias gradients' launch alone), split products
beside the bias gradients, and a ragged last chunk, against the FP64 oracle.
Tolerances as in test_gpu_surrogate.py."""
import numpy as np
import pytest

from gpu_common import require_gpu
from oracle import mlp as M

pytestmark = pytest.mark.gpu

LO = np.array([0.0, 0.0, 100.0, -80.0, 1.0])
HI = np.array([0.9, 120.0, 1000.0, -60.0, 16.0])


@pytest.mark.parametrize("rows,n_out", [(1, 24), (7, 3), (64, 24), (65, 33), (1000, 24)])
def test_gradients_at_chunk_edges(rows, n_out):
    tvbx = require_gpu()
    s = tvbx.Surrogate(LO, HI, n_out, n_members=3, seed=rows)
    rng = np.random.default_rng(rows)
    X = (LO + (HI - LO) * rng.uniform(size=(rows, 5))).astype(np.float32)
    Y = rng.standard_normal((rows, n_out)).astype(np.float32)
    dims = [5, 256, 256, 256, n_out]
    layers = M.unflatten(np.asarray(s.params(2), dtype=np.float64), dims)
    loss, g = s.gradients(X, Y, member=2)
    rloss, ref = M.loss_and_grads(layers, M.normalise_inputs(X.astype(np.float64), LO, HI), Y.astype(np.float64))
    assert abs(loss - rloss) <= 1e-5 * rloss
    for got, want in zip(M.unflatten(np.asarray(g, dtype=np.float64), dims), ref):
        for a, r in zip(got, want):
            assert np.linalg.norm(a - r) <= 1e-4 * max(np.linalg.norm(r), 1e-30)
            assert np.abs(a - r).max() <= 1e-3 * max(np.abs(r).max(), 1e-30)
    s.close()
