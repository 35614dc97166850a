"""Forms of the synthetic solver and of the FP64 sweep that the other parity tests do not reach,
against the FP64 oracle with their tolerances (FP64 1e-10, FP32 1e-5):

* one and two relaxation sweeps (the only sweep applied by itself; the first one, made by the
  residual kernel, followed by the last), at a CFL number at which a single sweep damps;
* the FP32 residual side in 1-D and at a far field;
* the FP64 sweep on fewer and on as many (block, chunk) pairs as the line between a cluster and a
  single CTA per pair (152), also in the form that only sums the residual's moments."""
import pytest

import gsis_inputs as gi
from oracle import kinetic as K
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

import test_gpu_defect_correction as DC
import test_gpu_gsis_parity as P
from _ctx import assert_fields_close, assert_planes_close, create

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    G.load()


def _step_matches(wl, precision, seed):
    f, I = P._inputs(wl, seed, precision)
    fg, Ig, rec, _ = P._run(wl, f, I, 1)
    fo, Io, Fo, _ = P._oracle(wl, f, I, 1)
    tol = P.TOL[precision]
    assert_planes_close(fg, fo, tol, "f^{k+1}")
    assert_planes_close(Ig, Io, tol, "I^{k+1}")
    assert_fields_close(rec, Fo, tol, wl.dim, "moments of f^{k+1}")


@pytest.mark.parametrize("precision,macro_fp32", [("fp64", 0), ("fp32", 1), ("fp32", 2)])
@pytest.mark.parametrize("sweeps", [1, 2])
@pytest.mark.parametrize("case", ["slab16", "cavity72", "cylinder64"])
def test_few_relaxation_sweeps(case, sweeps, precision, macro_fp32):
    _step_matches(gi.workloads.with_solver(P.CASES[case](), precision=precision, order=2, relax_block=16, max_inner=20,
                                           tol_inner=0.0, macro_sweeps=sweeps, cfl_macro=5.0, macro_fp32=macro_fp32),
                  precision, 21)


@pytest.mark.parametrize("macro_fp32", [1, 2])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("case", ["slab16", "cylinder64"])
def test_fp32_residual_side(case, order, macro_fp32):
    _step_matches(gi.workloads.with_solver(P.CASES[case](), precision="fp32", order=order, relax_block=16, max_inner=24,
                                           tol_inner=0.0, macro_sweeps=4, cfl_macro=200.0, macro_fp32=macro_fp32),
                  "fp32", 5)


# cells, cells per block: pairs with one chunk of 64 velocities
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("cells,block", [(151, 1), (152, 1), (303, 2), (304, 2)])
def test_sweep_around_the_cluster_line_1d(cells, block, order):
    wl = gi.workloads.with_solver(gi.workloads.slab(cells, Kn=0.05), precision="fp64", order=order, relax_block=block)
    f, I = P._inputs(wl, 8, "fp64")
    ctx = create(wl)
    try:
        G.gsis_set_distributions(ctx, f, I)
        G.gsis_step(ctx, G.GSIS_MODE_CIS)
        fg, Ig = G.gsis_get_distributions(ctx, cells, wl.xi.shape[0], wl.omega.shape[0])
    finally:
        G.gsis_destroy(ctx)
    fo, Io = K.kinetic_sweep(f, I, wl, relax_block=block)
    assert_planes_close(fg, fo, P.TOL["fp64"], "f")
    assert_planes_close(Ig, Io, P.TOL["fp64"], "I")


# 72 triangles x 13 chunks, 162 tetrahedra x 4 chunks: clusters, then single CTAs
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("case,block", [("cavity72", 8), ("cavity72", 4), ("box162", 8), ("box162", 4)])
def test_residual_moments_around_the_cluster_line(case, block, order):
    wl = gi.workloads.with_solver(DC._wl(case, "fp64", order), relax_block=block)
    f, I = DC._inputs(wl, 12, "fp64")
    fg, Ig, rec, _ = DC._gpu(wl, f, I, [G.GSIS_MODE_GSIS])
    fo, Io, Fo, _ = P._oracle(wl, f, I, 1)
    assert_planes_close(fg, fo, DC.TOL["fp64"], "f^{k+1}")
    assert_planes_close(Ig, Io, DC.TOL["fp64"], "I^{k+1}")
    assert_fields_close(rec, Fo, DC.TOL["fp64"], wl.dim, "moments of f^{k+1}")
