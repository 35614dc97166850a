"""GSIS steps given to the device in a row, without a read between them, are the steps that a
program waits for one by one, bit for bit: also with so few inner iterations that a solve polls
nothing and returns while the one before it still runs."""
import numpy as np
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import create

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("macro_fp32,max_inner", [(0, 8), (1, 8), (2, 8), (2, 3), (2, 17)])
def test_steps_in_a_row(macro_fp32, max_inner):
    import torch
    build.build()
    wl = gi.workloads.with_solver(gi.workloads.cavity(n_side=12, n_v=16), precision="fp32", order=1, relax_block=16,
                                  macro_fp32=macro_fp32, max_inner=max_inner, tol_inner=0.0)
    M = gi.fields.smooth_random_fields(wl.mesh.cell_centroid, 3, u_scale=0.1)
    out = []
    for wait in (True, False):
        stream = torch.cuda.Stream()
        ctx = create(wl, stream.cuda_stream)
        try:
            G.gsis_init_fields(ctx, M)
            for _ in range(4):
                G.gsis_step_async(ctx, G.GSIS_MODE_GSIS)
                if wait:
                    stream.synchronize()
            G.gsis_last_eps(ctx)
            out.append((G.gsis_get_fields(ctx, wl.mesh.n_cells), G.gsis_macro_stats(ctx)[0]))
        finally:
            G.gsis_destroy(ctx)
    assert out[0][1] == out[1][1] == max_inner
    assert np.array_equal(out[0][0], out[1][0])
