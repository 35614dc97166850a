"""The FP32 slope pass, sweep and field pass where their tiling can go wrong, against the FP64
oracle: triangles and quadrilaterals (their two compiled forms), relaxation blocks of one
cell, ragged ones and the largest, velocity sets that fill less than half a chunk of 64, end
just past a half and a whole chunk, or give the field pass fewer, as many and more chunks than
its four warps.  Tolerance: the FP32 path's 1e-5 (the inputs are FP32-rounded, so the
comparison measures arithmetic only).
"""
import numpy as np
import pytest

import gsis_inputs as gi
from oracle import kinetic as K
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import assert_fields_close, assert_planes_close, create


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    G.load()


def _polygons(n_side, quads, seed):
    """A jittered grid of squares, whole or each cut in two."""
    r = np.random.default_rng(seed)
    g = np.stack(np.meshgrid(np.linspace(0, 1, n_side + 1), np.linspace(0, 1, n_side + 1), indexing="ij"), -1)
    g[1:-1, 1:-1] += 0.15 / n_side * r.uniform(-1, 1, (n_side - 1, n_side - 1, 2))
    v = g.reshape(-1, 2)
    cells = []
    for i in range(n_side):
        for j in range(n_side):
            a, b, c, d = (i * (n_side + 1) + j, (i + 1) * (n_side + 1) + j, (i + 1) * (n_side + 1) + j + 1,
                          i * (n_side + 1) + j + 1)
            cells += [[a, b, c, d]] if quads else [[a, b, c], [a, c, d]]
    cc, vol, faces = np.zeros((len(cells), 2)), np.zeros(len(cells)), {}
    for k, p in enumerate(cells):
        x, y = v[p].T
        cr = x * np.roll(y, -1) - np.roll(x, -1) * y
        vol[k] = 0.5 * cr.sum()
        cc[k] = [((x + np.roll(x, -1)) * cr).sum(), ((y + np.roll(y, -1)) * cr).sum()]
        cc[k] /= 6.0 * vol[k]
        for a, b in zip(p, p[1:] + p[:1]):
            faces.setdefault((min(a, b), max(a, b)), []).append(k)
    own, nbr, nrm, area, fc = [], [], [], [], []
    for (a, b), owners in faces.items():
        d, m = v[b] - v[a], 0.5 * (v[a] + v[b])
        n = np.array([d[1], -d[0]]) / np.hypot(*d)
        own.append(owners[0])
        nbr.append(owners[1] if len(owners) > 1 else -1 - (1 if m[1] > 1 - 1e-9 else 0))
        nrm.append(n if n @ (m - cc[owners[0]]) > 0 else -n)
        area.append(np.hypot(*d))
        fc.append(m)
    P = gi.mesh.Patch
    return gi.mesh.Mesh(dim=2, n_cells=len(cells), face_owner=np.asarray(own, np.int32),
                        face_nbr=np.asarray(nbr, np.int32), face_normal=np.asarray(nrm), face_area=np.asarray(area),
                        face_centroid=np.asarray(fc), cell_volume=vol, cell_centroid=cc,
                        patches=[P(gi.mesh.WALL), P(gi.mesh.WALL, u=(0.2, 0.0, 0.0), T_t=2.0)])


@pytest.mark.gpu
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("quads,block,n_v", [(True, 16, 4), (True, 1, 6), (True, 7, 9), (True, 64, 17), (False, 33, 16),
                                             (False, 5, 5)])
def test_fp32_step_on_polygons(quads, block, n_v, order):
    """Velocities: 16, 36, 81, 289 (five chunks), 256 (four chunks), 25."""
    wl = gi.workloads.cavity(n_side=9, n_v=n_v)
    wl.mesh = _polygons(9, quads, 5)
    wl.xi, wl.w = gi.quadrature.trapezoid_nd(n_v, min(8.0, 0.8 * (n_v - 1)), 2)   # spacings of at most 1.6
    wl = gi.workloads.with_solver(wl, precision="fp32", order=order, relax_block=block)
    M = gi.fields.random_macro_fields(wl.mesh.n_cells, 2, 3, u_scale=0.3)
    f, I = gi.fields.noisy_equilibrium(M, wl.xi, wl.omega, 2, wl.model.d_r, wl.model.d_v, wl.model.sigma_R, 4)
    f, I = f.astype(np.float32).astype(np.float64), I.astype(np.float32).astype(np.float64)
    ctx = create(wl)
    try:
        G.gsis_set_distributions(ctx, f, I)
        G.gsis_step(ctx, G.GSIS_MODE_CIS)
        fg, Ig = G.gsis_get_distributions(ctx, wl.mesh.n_cells, wl.xi.shape[0], wl.omega.shape[0])
        rec = G.gsis_get_fields(ctx, wl.mesh.n_cells)
    finally:
        G.gsis_destroy(ctx)
    fo, Io = K.kinetic_sweep(f, I, wl, relax_block=block)
    assert_planes_close(fg, fo, 1e-5, "f")
    assert_planes_close(Ig, Io, 1e-5, "I")
    # the fields of the step's own distributions
    F1 = K.moments(fg.astype(np.float64), Ig.astype(np.float64), wl.xi, wl.w, wl.omega, wl.wo, 2, wl.model)
    assert_fields_close(rec, F1, 1e-5, 2, "fields")
