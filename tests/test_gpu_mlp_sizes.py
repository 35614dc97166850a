"""The learned closure's kernels at the batch sizes where their split changes: one row, a
warp's four rows, a block's 16, the largest batch of 16-row tiles (152 of them) and the
smallest of 32-row ones, several tiles per block, and the weight gradient's row ranges (128
rows up to 32 of them).  Against the FP64 oracle with the tolerances of test_gpu_mlp.py."""
import numpy as np
import pytest

import gsis_inputs as gi
from oracle import mlp as M
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import create
from test_gpu_mlp import _bf16_params, _blob

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 16, 17, 128, 129, 2432, 2433, 4097, 9999])
def test_loss_gradient_and_prediction(n):
    build.build()
    c = create(gi.workloads.with_solver(gi.workloads.slab(8), precision="fp64"))
    try:
        params = M.init_params(3)
        G.gsis_mlp_set_params(c, _blob(params))
        rng = np.random.default_rng(n)
        X = rng.normal(size=(n, 16)).astype(np.float32)
        Y = rng.normal(size=(n, 12)).astype(np.float32)
        loss, g = G.gsis_mlp_loss_grad(c, X, Y)
        pred = G.gsis_mlp_predict(c, X)
    finally:
        G.gsis_destroy(c)
    p16 = _bf16_params(params)
    lo, go = M.loss_and_grad(p16, X.astype(np.float64), Y.astype(np.float64))
    assert abs(loss - lo) <= 1e-4 * lo
    off = 0
    for (gW, gb) in go:
        for ref in (gW, gb):
            got = g[off:off + ref.size].reshape(ref.shape)
            off += ref.size
            assert np.all(np.abs(got - ref) <= 1e-3 * np.abs(ref) + 1e-4 * np.abs(ref).max())
    out, _ = M.forward(p16, X.astype(np.float64))
    assert np.abs(pred - out).max() <= 1e-4 * np.abs(out).max()
