"""A value that is not finite spreads as the scheme transports it: after a step at order 1 it is
found in its cell and in the neighbours that its velocity enters, not in those it comes from."""
import numpy as np
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import create

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", ["slab", "cavity", "capsule"])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_upstream_cells_stay_finite(name, precision, bad):
    build.build()
    base = {"slab": lambda: gi.workloads.slab(n_cells=12, n_xi=16, n_mu=8),
            "cavity": lambda: gi.workloads.cavity(n_side=6, n_v=10),
            "capsule": lambda: gi.workloads.capsule(n=4, n_v=6, n_polar=4, n_azim=4)}[name]()
    # one cell per relaxation block: no relaxation between cells
    wl = gi.workloads.with_solver(base, precision=precision, order=1, relax_block=1)
    m, n = wl.mesh, wl.mesh.n_cells
    M = gi.fields.uniform_fields(n)
    f, I = gi.fields.noisy_equilibrium(M, wl.xi, wl.omega, wl.dim, wl.model.d_r, wl.model.d_v, wl.model.sigma_R, 1)
    inner = np.ones(n, bool)                       # a cell without boundary faces
    inner[m.face_owner[m.face_nbr < 0]] = False
    c = int(np.flatnonzero(inner)[inner.sum() // 2])
    v = int(np.argmax((wl.xi[:, :wl.dim] * [0.9, 0.7, 0.4][:wl.dim]).sum(1)))
    f[c, v, :] = bad
    ctx = create(wl)
    try:
        G.gsis_set_distributions(ctx, f, I)
        with pytest.raises(G.GsisError) as e:
            G.gsis_step(ctx, G.GSIS_MODE_CIS)
        assert e.value.code == G.GSIS_ERR_DIVERGED
        got, _ = G.gsis_get_distributions(ctx, n, wl.xi.shape[0], wl.omega.shape[0])
    finally:
        G.gsis_destroy(ctx)
    expect = np.zeros((n, wl.xi.shape[0]), bool)
    expect[c] = True                               # its moments, and with them its source
    for face in range(m.n_faces):
        o, j = int(m.face_owner[face]), int(m.face_nbr[face])
        if j < 0 or c not in (o, j):
            continue
        xn = float(m.face_normal[face, :wl.dim] @ wl.xi[v, :wl.dim]) * (1 if o == c else -1)
        if xn > 1e-6:
            expect[j if o == c else o, v] = True
    assert np.array_equal(~np.isfinite(got).all(2), expect)
