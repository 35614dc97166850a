"""The far tails of the velocity set, where FP32 values are subnormal: a gas in uniform
equilibrium with its walls keeps them through steps.

A tail value is 2^y with |y| up to 130: y carries three roundings (|y| ln 2 3 2^-24 = 1.7e-5),
the exponential 2^-22, and the moments' own rounding, a temperature off by 1e-7, moves the tail
by half of c^2 times that (1e-5).  Per step 1e-4, and two units of the subnormal spacing for
each of the roundings of source and update."""
from dataclasses import replace

import numpy as np
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import create

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("dim", [1, 2])
def test_equilibrium_tails_are_kept(dim, order):
    build.build()
    if dim == 1:
        wl = gi.workloads.slab(n_cells=12, n_mu=8, T_right=1.0)
        reach, n_v = 13.4, 64
    else:
        wl = gi.workloads.couette(n_side=3, n_polar=4, n_azim=8)
        reach, n_v = 9.5, 40
    wl.mesh.patches = [replace(p, u=(0.0, 0.0, 0.0), T_t=1.0) for p in wl.mesh.patches]
    xi, w = gi.quadrature.trapezoid_nd(n_v, reach, dim)
    wl = replace(wl, xi=xi, w=w)
    wl = gi.workloads.with_solver(wl, precision="fp32", order=order, relax_block=4)
    n = wl.mesh.n_cells
    ctx = create(wl)
    try:
        G.gsis_init_fields(ctx, gi.fields.uniform_fields(n))
        f0, _ = G.gsis_get_distributions(ctx, n, w.size, wl.wo.size)
        steps = 2
        for _ in range(steps):
            G.gsis_step(ctx, G.GSIS_MODE_CIS)
        f1, _ = G.gsis_get_distributions(ctx, n, w.size, wl.wo.size)
    finally:
        G.gsis_destroy(ctx)
    tiny = (f0[..., 0] > 0) & (f0[..., 0] < 2.0 ** -126)
    assert tiny.any()
    off = np.abs(f1 - f0) - steps * (1e-4 * f0 + 4 * 2.0 ** -149)
    assert off.max() <= 0.0, (f0.ravel()[off.argmax()], f1.ravel()[off.argmax()])
