"""An infinite value among the distributions makes its cell's moments infinite, as the plain sum
does, wherever in the velocity set it stands (also where a lane of the last run has no velocity of
its own), and no other cell's."""
import numpy as np
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n_v", [("fp32", 20), ("fp32", 60), ("fp64", 10), ("fp64", 20)])
@pytest.mark.parametrize("at", [0, -1])
def test_infinite_density(precision, n_v, at):
    import torch
    build.build()
    dev = torch.device("cuda", 0)
    real = torch.float32 if precision == "fp32" else torch.float64
    xi, w = gi.quadrature.trapezoid_nd(n_v, 6.0, 2)
    om, wo = gi.quadrature.photon_product(4, 8)
    q = [torch.from_numpy(a.copy()).to(dev) for a in (xi, w, om, wo)]
    f = torch.exp(-(q[0] ** 2).sum(1) / 2).to(real)[None, :, None].repeat(5, 1, 4)
    f[2, at, 0] = float("inf")
    I = torch.ones(5, wo.size, device=dev, dtype=real)
    out = torch.zeros(5, G.GSIS_NF, dtype=torch.float64, device=dev)
    assert G.gsis_moments_static(2, precision, 5, w.size, q[0].data_ptr(), q[1].data_ptr(), wo.size, q[2].data_ptr(),
                                 q[3].data_ptr(), f.contiguous().data_ptr(), I.data_ptr(), 2.0, 1.16, 0.01,
                                 out.data_ptr(), torch.cuda.current_stream(dev).cuda_stream) == G.GSIS_OK
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert got[2, 0] == np.inf
    others = np.delete(got, 2, axis=0)
    assert np.isfinite(others).all() and np.array_equal(others, others[:1].repeat(4, 0))
