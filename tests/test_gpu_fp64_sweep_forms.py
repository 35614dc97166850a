"""The FP64 sweep on both sides of each line between its forms, against the FP64 oracle (1e-10, as
the other parity tests): a cluster of eight CTAs per (block, chunk) pair, one CTA of eight rows, one
of two.  One chunk of velocities, so that the pairs are the relaxation blocks; the last one ragged."""
import pytest

import gsis_inputs as gi
from oracle import kinetic as K
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

import test_gpu_gsis_parity as P
from _ctx import assert_fields_close, assert_planes_close, create

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("block,pairs", [(1, 4), (3, 5), (4, 5), (4, 16), (4, 17), (16, 51), (16, 52), (16, 152), (32, 36),
                                         (32, 37), (64, 15), (64, 16)])
def test_forms_match_oracle(block, pairs, order):
    build.build()
    cells = block * pairs - block // 3
    wl = gi.workloads.with_solver(gi.workloads.slab(cells, n_xi=20, n_mu=8, Kn=0.05), precision="fp64", order=order,
                                  relax_block=block)
    f, I = P._inputs(wl, 8, "fp64")
    ctx = create(wl)
    try:
        G.gsis_set_distributions(ctx, f, I)
        G.gsis_step(ctx, G.GSIS_MODE_CIS)
        fg, Ig = G.gsis_get_distributions(ctx, cells, wl.xi.shape[0], wl.omega.shape[0])
        rec = G.gsis_get_fields(ctx, cells)
    finally:
        G.gsis_destroy(ctx)
    fo, Io = K.kinetic_sweep(f, I, wl, relax_block=block)
    assert_planes_close(fg, fo, P.TOL["fp64"], "f")
    assert_planes_close(Ig, Io, P.TOL["fp64"], "I")
    assert_fields_close(rec, K.moments(fo, Io, wl.xi, wl.w, wl.omega, wl.wo, 1, wl.model), P.TOL["fp64"], 1)
