"""The FP32 equilibrium is the FP64 one rounded to FP32, as nearly as its two-word arithmetic
gives: half a unit in the last place, plus the errors of the two-word value: the r^2/2 term of
the exponential's sum (|r| <= ln 2 / 128, three roundings of 1.5e-5: 4.4e-5 units), the argument
(|y| <= 150, five roundings of its second word, 2^-49 |y| each: 3e-5) and the factors' second
words (1e-6): 1e-4 units, taken twice."""
import numpy as np
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import create


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["slab", "cavity", "capsule"])
def test_values_are_rounded_once(name):
    build.build()
    wl = {"slab": lambda: gi.workloads.slab(2000, n_xi=64, n_mu=8), "cavity": lambda: gi.workloads.cavity(n_side=40, n_v=20),
          "capsule": lambda: gi.workloads.capsule(n=6, n_v=12, n_polar=4, n_azim=4)}[name]()
    wl = gi.workloads.with_solver(wl, precision="fp32")
    n, dim = wl.mesh.n_cells, wl.dim
    r = np.random.default_rng(17)
    M = gi.fields.uniform_fields(n)
    M[:, 0] = np.exp(r.uniform(-2, 2, n))
    M[:, 1:1 + dim] = r.uniform(-1, 1, (n, dim))
    M[:, 4:8] = np.exp(r.uniform(-1, 1.5, (n, 4)))
    ctx = create(wl)
    try:
        G.gsis_init_fields(ctx, M)
        f, _ = G.gsis_get_distributions(ctx, n, wl.xi.shape[0], wl.omega.shape[0])
    finally:
        G.gsis_destroy(ctx)
    xi = wl.xi[:, :dim].astype(np.float32).astype(np.float64)
    T = M[:, 4:5]
    c2 = ((xi[None] - M[:, None, 1:1 + dim]) ** 2).sum(-1)
    F0 = M[:, :1] * (2 * np.pi * T) ** (-0.5 * dim) * np.exp(-c2 / (2 * T))
    ref = np.stack([F0, (3 - dim) * T * F0, 0.5 * wl.model.d_r * M[:, 5:6] * F0, 0.5 * wl.model.d_v * M[:, 6:7] * F0], -1)
    normal = ref >= 2.0 ** -126
    ulps = np.abs(f - ref)[normal] / 2.0 ** (np.floor(np.log2(ref[normal])) - 23)
    assert ulps.size > 100000 and ulps.max() <= 0.5002, ulps.max()
