"""gsis_moments_static at the sizes where its work split changes: velocities around a lane
row (32), an FP32 run (128) and the largest shared tables (about 3 200 velocities in 2-D);
cells around a warp's and a block's share; f off its record alignment.  Against the FP64
oracle, with the tolerances of the other moment tests (1e-5 in FP32, 1e-10 in FP64)."""
import numpy as np
import pytest

import gsis_inputs as gi
from oracle import kinetic as K
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import assert_fields_close

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp64": 1e-10}


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,n_cells,n_v,n_omega,offset", [
    (1, 1, 31, 8, 0), (1, 9, 128, 128, 1), (1, 7, 129, 136, 0), (2, 33, 13, 64, 3), (2, 2432, 8, 16, 0),
    (2, 2440, 9, 8, 1), (2, 9728, 8, 8, 0), (2, 17, 56, 64, 0), (2, 5, 57, 64, 2)])
def test_sizes_match_oracle(dim, n_cells, n_v, n_omega, offset, precision):
    import torch
    build.build()
    model = gi.workloads.ModelParams(sigma_R=0.01)
    M = gi.fields.random_macro_fields(n_cells, dim, 5, u_scale=2.0, q_scale=0.0)
    xi, w = gi.quadrature.trapezoid_nd(n_v, 12.0, dim)
    om, wo = gi.quadrature.photon_product(8, n_omega // 8)
    f, I = gi.fields.noisy_equilibrium(M, xi, om, dim, model.d_r, model.d_v, model.sigma_R, 6)
    real = torch.float32 if precision == "fp32" else torch.float64
    dev = torch.device("cuda", 0)
    buf = torch.zeros(f.size + offset, dtype=real, device=dev)       # f `offset` values off the allocation's start
    buf[offset:] = torch.from_numpy(f.ravel()).to(dev, real)
    fd, Id = buf[offset:], torch.from_numpy(I).to(dev, real)
    q = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in (xi, w, om, wo)]
    out = torch.full((n_cells, G.GSIS_NF), float("nan"), dtype=torch.float64, device=dev)
    rc = G.gsis_moments_static(dim, precision, n_cells, w.size, q[0].data_ptr(), q[1].data_ptr(), wo.size,
                               q[2].data_ptr(), q[3].data_ptr(), fd.data_ptr(), Id.data_ptr(), model.d_r, model.d_v,
                               model.sigma_R, out.data_ptr(), torch.cuda.current_stream(dev).cuda_stream)
    assert rc == G.GSIS_OK
    torch.cuda.synchronize()
    f8, I8 = (x.double().cpu().numpy().reshape(s) for x, s in ((fd, f.shape), (Id, I.shape)))
    ref = K.moments(f8, I8, xi, w, om, wo, dim, model)
    assert_fields_close(out.cpu().numpy(), ref, TOL[precision], dim)
