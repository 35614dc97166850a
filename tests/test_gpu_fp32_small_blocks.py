"""The FP32 sweep's one-warp form (relaxation blocks of one and two cells) and the next larger
block, against the FP64 oracle with the FP32 path's 1e-5: segments, triangles and tetrahedra, both
orders, an odd number of cells, and the form that sums the residual's moments."""
import numpy as np
import pytest

import gsis_inputs as gi
from oracle import kinetic as K
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

import test_gpu_defect_correction as DC
import test_gpu_gsis_parity as P
from _ctx import assert_fields_close, assert_planes_close, create

pytestmark = pytest.mark.gpu

CASES = {"slab17": lambda: gi.workloads.slab(17, n_xi=33, n_mu=8, Kn=0.05),
         "cavity50": lambda: gi.workloads.cavity(n_side=5, n_v=9, n_polar=4, n_azim=8),
         "box162": DC.CASES["box162"]}


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("block", [1, 2, 3])
@pytest.mark.parametrize("case", sorted(CASES))
def test_step_matches_oracle(case, block, order):
    build.build()
    wl = gi.workloads.with_solver(CASES[case](), precision="fp32", order=order, relax_block=block, tc_moments=0)
    f, I = P._inputs(wl, 4, "fp32")
    ctx = create(wl)
    try:
        G.gsis_set_distributions(ctx, f, I)
        G.gsis_step(ctx, G.GSIS_MODE_CIS)
        fg, Ig = G.gsis_get_distributions(ctx, wl.mesh.n_cells, wl.xi.shape[0], wl.omega.shape[0])
        rec = G.gsis_get_fields(ctx, wl.mesh.n_cells)
    finally:
        G.gsis_destroy(ctx)
    fo, Io = K.kinetic_sweep(f, I, wl, relax_block=block)
    assert_planes_close(fg, fo, P.TOL["fp32"], "f")
    assert_planes_close(Ig, Io, P.TOL["fp32"], "I")
    ref = K.moments(fo, Io, wl.xi, wl.w, wl.omega, wl.wo, wl.dim, wl.model)
    assert_fields_close(rec, ref, P.TOL["fp32"], wl.dim)


@pytest.mark.parametrize("block", [1, 2])
def test_residual_moments_match_oracle(block):
    build.build()
    wl = gi.workloads.with_solver(DC._wl("cavity72", "fp32", 2), relax_block=block)
    f, I = DC._inputs(wl, 23, "fp32")
    fg, Ig, rec, _ = DC._gpu(wl, f, I, [G.GSIS_MODE_GSIS])
    fo, Io, Fo, _ = P._oracle(wl, f, I, 1)
    assert_planes_close(fg, fo, DC.TOL["fp32"], "f^{k+1}")
    assert_fields_close(rec, Fo, DC.TOL["fp32"], wl.dim, "fields")
    assert np.isfinite(Ig).all()
