"""The FP32 equilibrium that a run starts from: a value is an FP32 rounding of a two-word result
whose own error is below 2^-7 units in the last place, so it lies within 0.51 units of the FP64
value (whose error is about |argument| 2^-52); below the smallest normal number within one
denormal step.  Meshes of fewer and more cells than a thread block takes, 1-D to 3-D.
"""
import numpy as np
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import create


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    G.load()


@pytest.mark.gpu
@pytest.mark.parametrize("case", ["slab1", "slab40", "cavity", "box"])
def test_fp32_equilibrium_is_rounded(case):
    """Cold and fast cells too: arguments of the exponential from 0 to past underflow."""
    wl = {"slab1": lambda: gi.workloads.slab(3, n_xi=17), "slab40": lambda: gi.workloads.slab(701, n_xi=32),
          "cavity": lambda: gi.workloads.cavity(n_side=50, n_v=9),
          "box": lambda: gi.workloads.capsule(n=5, n_v=8)}[case]()
    wl = gi.workloads.with_solver(wl, precision="fp32")
    n, dim = wl.mesh.n_cells, wl.dim
    r = np.random.default_rng(9)
    M = gi.fields.uniform_fields(n)
    M[:, 0] = np.exp(r.uniform(-2, 2, n))
    M[:, 1:1 + dim] = r.uniform(-2, 2, (n, dim))
    M[:, 4:8] = np.exp(r.uniform(-3, 1.5, (n, 4)))
    ctx = create(wl)
    try:
        G.gsis_init_fields(ctx, M)
        f, I = G.gsis_get_distributions(ctx, n, wl.xi.shape[0], wl.omega.shape[0])
    finally:
        G.gsis_destroy(ctx)
    xi = wl.xi[:, :dim].astype(np.float32).astype(np.float64)
    T = M[:, 4:5]
    c2 = ((xi[None] - M[:, None, 1:1 + dim]) ** 2).sum(-1)
    F0 = M[:, :1] * (2 * np.pi * T) ** (-0.5 * dim) * np.exp(-c2 / (2 * T))
    ref = np.stack([F0, (3 - dim) * T * F0, 0.5 * wl.model.d_r * M[:, 5:6] * F0, 0.5 * wl.model.d_v * M[:, 6:7] * F0], -1)
    ulp = 2.0 ** (np.floor(np.log2(np.maximum(ref, 2.0 ** -126))) - 23)
    slack = np.where(ref < 2.0 ** -126, 1.01, 0.51) * ulp + 1e-13 * ref
    err = np.abs(f - ref)
    assert (err <= slack).all(), (err / ulp).max()
    B = wl.model.sigma_R * M[:, 7] ** 4 / np.pi
    assert np.abs(I - B[:, None]).max() <= 1e-6 * B.max()
