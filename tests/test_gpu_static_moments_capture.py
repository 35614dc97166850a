"""gsis_moments_static in a captured graph, its first call on the process included: a replay
gives the direct call's fields bit for bit, in the form of a warp per cell and in that of a
cluster per cell."""
import pytest

import gsis_inputs as gi
from paper_2601_03935_gb300 import build
from paper_2601_03935_gb300 import gsis as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n_cells,n_v", [("fp32", 50, 20), ("fp32", 3, 60), ("fp64", 5, 30), ("fp64", 900, 8)])
def test_replay_equals_the_direct_call(precision, n_cells, n_v):
    import torch
    build.build()
    dev = torch.device("cuda", 0)
    real = torch.float32 if precision == "fp32" else torch.float64
    xi, w = gi.quadrature.trapezoid_nd(n_v, 6.0, 2)
    om, wo = gi.quadrature.photon_product(4, 8)
    q = [torch.from_numpy(a.copy()).to(dev) for a in (xi, w, om, wo)]
    gen = torch.Generator(device=dev).manual_seed(2)
    f = torch.rand(n_cells, w.size, 4, generator=gen, device=dev, dtype=real) * torch.exp(-(q[0] ** 2).sum(1) / 2).to(real)[:, None]
    I = torch.rand(n_cells, wo.size, generator=gen, device=dev, dtype=real)
    out = [torch.zeros(n_cells, G.GSIS_NF, dtype=torch.float64, device=dev) for _ in range(2)]

    def call(o):
        assert G.gsis_moments_static(2, precision, n_cells, w.size, q[0].data_ptr(), q[1].data_ptr(), wo.size,
                                     q[2].data_ptr(), q[3].data_ptr(), f.data_ptr(), I.data_ptr(), 2.0, 1.16, 0.01,
                                     o.data_ptr(), torch.cuda.current_stream(dev).cuda_stream) == G.GSIS_OK

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(out[0])
    for _ in range(2):
        out[0].zero_()
        graph.replay()
    call(out[1])
    torch.cuda.synchronize()
    assert torch.isfinite(out[1]).all() and (out[1][:, 0] > 0).all()
    assert torch.equal(out[0], out[1])
