"""gsis_moments_static where a cell is split among CTAs: sets around a run (128) and the smallest
and largest cluster, one cell and the numbers at which a cluster has half the CTAs, the last
count that is split and the first that is not, more directions than velocities, f off its
record alignment.  Against the FP64 oracle, with the tolerances of the other moment tests
(1e-5 in FP32, 1e-10 in FP64)."""
import numpy as np
import pytest

import gsis_inputs as gi
from oracle import kinetic as K
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

from _ctx import assert_fields_close

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp64": 1e-10}


@pytest.mark.parametrize("precision,dim,n_cells,n_v,n_omega,offset", [
    ("fp64", 1, 1, 255, 8, 0), ("fp64", 1, 1, 256, 8, 1), ("fp64", 1, 3, 1025, 8, 0), ("fp64", 2, 19, 46, 136, 0),
    ("fp64", 2, 38, 64, 64, 3), ("fp64", 2, 39, 64, 8, 0), ("fp64", 2, 77, 33, 8, 2), ("fp64", 1, 700, 257, 8, 0),
    ("fp64", 1, 701, 257, 8, 0), ("fp64", 2, 2, 10, 264, 0), ("fp32", 2, 1, 57, 64, 0), ("fp32", 2, 1, 96, 8, 1),
    ("fp32", 1, 5, 5459, 8, 0), ("fp32", 1, 38, 5600, 8, 2), ("fp32", 2, 153, 58, 64, 0), ("fp32", 2, 2, 10, 8200, 0)])
def test_split_cells_match_oracle(precision, dim, n_cells, n_v, n_omega, offset):
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
