"""What the host gives to the device and in which order, on the CPU: libgsis is linked with a
runtime that records instead of running (fake_cudart.cpp)."""
import ctypes as C

import numpy as np
import pytest

import gsis_inputs as gi

import _fake

STREAM = 0x1000          # a stream of the caller's own


@pytest.fixture(scope="module")
def G(tmp_path_factory):
    return _fake.load(str(tmp_path_factory.mktemp("fake")))


def _create(G, wl, stream=STREAM):
    m = wl.mesh
    return G.gsis_create(m.dim, m.face_owner, m.face_nbr, m.face_normal, m.face_area, m.face_centroid,
                         m.cell_volume, m.cell_centroid, m.patches, wl.xi[:, :m.dim], wl.w, wl.omega, wl.wo,
                         wl.model, wl.solver, stream, period=getattr(m, "period", 0.0))


@pytest.mark.parametrize("max_inner", [3, 8, 9, 16, 17, 40])
@pytest.mark.parametrize("macro_fp32", [0, 1, 2])
def test_solver_state_is_not_rewritten_under_a_copy(G, macro_fp32, max_inner):
    # steps in a row without a read between them, and two pre-solves
    wl = gi.workloads.with_solver(gi.workloads.slab(n_cells=12, n_xi=16, n_mu=8), precision="fp32",
                                  macro_fp32=macro_fp32, max_inner=max_inner)
    ctx = _create(G, wl)
    G.fake.fake_reset()
    try:
        for _ in range(3):
            assert G.load().gsis_step_async(ctx, G.GSIS_MODE_GSIS) == G.GSIS_OK
        G.load().gsis_warm_start(ctx, 2, 0)
    finally:
        G.gsis_destroy(ctx)
    assert _fake.report(G, "rewritten") == []


@pytest.mark.parametrize("precision,macro_fp32", [("fp64", 0), ("fp32", 0), ("fp32", 2)])
@pytest.mark.parametrize("name,order,defect", [("slab", 1, 0), ("cavity", 2, 1), ("capsule", 2, 0)])
def test_the_context_stream_orders_all_work(G, name, order, defect, precision, macro_fp32):
    # nothing that a kernel reads or overwrites is left to the default stream
    base = {"slab": lambda: gi.workloads.slab(n_cells=12, n_xi=16, n_mu=8),
            "cavity": lambda: gi.workloads.cavity(n_side=4, n_v=8),
            "capsule": lambda: gi.workloads.capsule(n=4, n_v=6, n_polar=4, n_azim=4)}[name]()
    wl = gi.workloads.with_solver(base, precision=precision, order=order, macro_fp32=macro_fp32, max_inner=10,
                                  defect_correction=defect)
    lib = G.load()
    G.fake.fake_reset()
    ctx = _create(G, wl)
    try:
        n = wl.mesh.n_cells
        for mode in (G.GSIS_MODE_CIS, G.GSIS_MODE_GSIS):
            assert lib.gsis_step_async(ctx, mode) == G.GSIS_OK
        G.gsis_set_distributions(ctx, np.ones((n, wl.w.size, 4)), np.ones((n, wl.wo.size)))
        image = G.gsis_export_state(ctx)
        G.gsis_import_state(ctx, image)
        assert lib.gsis_step_async(ctx, G.GSIS_MODE_CIS) == G.GSIS_OK
        if wl.dim < 3 and not defect:
            G.gsis_shard_setup(ctx, wl.xi[:, :wl.dim], wl.w, wl.omega, wl.wo)
            assert lib.gsis_shard_begin(ctx, G.GSIS_MODE_GSIS) == G.GSIS_OK
    finally:
        G.gsis_destroy(ctx)
    assert _fake.report(G, "unordered") == []


def test_kernel_attributes_are_the_same_for_every_caller(G):
    # a kernel's shared-memory limit belongs to the process: calls of other threads, with other
    # velocity sets or relaxation blocks, may come between one call's setting and its launch
    G.fake.fake_reset()
    a = np.zeros(64)
    p = a.ctypes.data
    for dim, precision in ((1, "fp32"), (2, "fp32"), (1, "fp64"), (2, "fp64")):
        for n_xi in (100, 900, 2000, 3000, 5000):
            for f in (p, p + 8):
                assert G.gsis_moments_static(dim, precision, 40, n_xi, p, p, 64, p, p, f, p, 2.0, 2.0, 0.01, p,
                                             STREAM) == G.GSIS_OK
    cases = [(gi.workloads.slab(n_cells=70, n_xi=16, n_mu=8), "fp64"), (gi.workloads.cavity(n_side=9, n_v=8), "fp32"),
             (gi.workloads.cavity(n_side=9, n_v=40), "fp64"), (gi.workloads.capsule(n=4, n_v=6, n_polar=4, n_azim=4), "fp32")]
    for base, precision in cases:
        for order in (1, 2):
            for block in (1, 16, 48):
                ctx = _create(G, gi.workloads.with_solver(base, precision=precision, order=order, relax_block=block))
                try:
                    assert G.load().gsis_step_async(ctx, G.GSIS_MODE_CIS) == G.GSIS_OK
                finally:
                    G.gsis_destroy(ctx)
    G.gsis_mlp_init(ctx := _create(G, gi.workloads.slab(n_cells=8, n_xi=16, n_mu=8)), 1)
    try:
        for n in (1, 2000, 5000):
            G.gsis_mlp_predict(ctx, np.zeros((n, 16), np.float32))
            G.gsis_mlp_loss_grad(ctx, np.zeros((n, 16), np.float32), np.zeros((n, 12), np.float32))
    finally:
        G.gsis_destroy(ctx)
    assert _fake.report(G, "attribute") == []


def _network_calls(G, ctx):
    X, Y = np.ones((40, 16), np.float32), np.ones((40, 12), np.float32)
    G.gsis_mlp_init(ctx, 1)
    G.gsis_mlp_loss_grad(ctx, X, Y)
    G.gsis_mlp_train(ctx, X, Y, epochs=1, batch=20)
    G.gsis_mlp_train(ctx, X[:20], Y[:20], epochs=1, batch=20)


def test_closure_buffers_after_a_failed_allocation(G):
    # whichever allocation fails, the call is refused and a later one finds every buffer there
    wl = gi.workloads.slab(n_cells=8, n_xi=16, n_mu=8)
    G.fake.fake_reset()
    ctx = _create(G, wl)
    _network_calls(G, ctx)
    whole = G.fake.fake_device_bytes()
    G.gsis_destroy(ctx)
    for k in range(100):
        ctx = _create(G, wl)
        try:
            G.fake.fake_fail_malloc_after(k)
            failed = False
            for _ in range(2):
                try:
                    _network_calls(G, ctx)
                except G.GsisError as e:
                    assert e.code == G.GSIS_ERR_OUT_OF_MEMORY
                    failed = True
                    G.fake.fake_fail_malloc_after(-1)
            G.fake.fake_fail_malloc_after(-1)
            assert G.fake.fake_device_bytes() == whole, k
            if not failed:
                break
        finally:
            G.fake.fake_fail_malloc_after(-1)
            G.gsis_destroy(ctx)
    assert k > 20 and _fake.report(G, "freed") == []


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_face_values_are_defined_before_the_first_sweep(G, precision):
    # an upwind value is written where xi . n > 0 on one side; in 3-D the sweep's S/V xi . n may
    # round to something else than zero where xi . n is zero, and then reads what nobody wrote
    wl = gi.workloads.with_solver(gi.workloads.capsule(n=4, n_v=6, n_polar=4, n_azim=4), precision=precision, order=2)
    faces, real = int((wl.mesh.face_nbr >= 0).sum()), 4 if precision == "fp32" else 8
    pad = lambda n: (n + 63) // 64 * 64  # noqa: E731
    G.fake.fake_reset()
    G.gsis_destroy(_create(G, wl))
    assert G.fake.fake_cleared(faces * pad(wl.w.size) * 4 * real) == 1       # gas
    assert G.fake.fake_cleared(faces * pad(wl.wo.size) * real) == 1          # photons


@pytest.mark.parametrize("dim,precision,n_cells,n_xi,ctas", [
    (2, "fp32", 1, 9216, 8), (2, "fp32", 16, 16384, 128), (2, "fp32", 152, 4096, 152), (2, "fp32", 4000, 4096, 4000),
    (1, "fp32", 1, 9216, 8), (2, "fp64", 1, 9216, 8), (2, "fp64", 64, 4096, 128), (2, "fp64", 300, 784, 300),
    (1, "fp64", 64, 784, 64)])
def test_few_cells_of_large_sets_fill_the_chip(G, dim, precision, n_cells, n_xi, ctas):
    # one CTA of eight warps per eight cells, whatever the set, left all but a few SMs idle
    G.fake.fake_reset()
    a = np.zeros(64)
    p = a.ctypes.data
    assert G.gsis_moments_static(dim, precision, n_cells, n_xi, p, p, 64, p, p, p, p, 2.0, 2.0, 0.01, p, STREAM) == G.GSIS_OK
    grid, block = C.c_int(), C.c_int()
    assert G.fake.fake_launch_count() == 1
    G.fake.fake_launch(0, C.byref(grid), C.byref(block))
    assert grid.value >= ctas and block.value == 256


@pytest.mark.parametrize("block,pairs,clusters", [
    (1, 4, False), (3, 10, False), (2, 100, False), (4, 16, True), (4, 17, False), (16, 51, True), (16, 52, False),
    (16, 151, False), (16, 152, False), (32, 36, True), (32, 37, False), (64, 15, True), (64, 16, False), (64, 52, False)])
def test_fp64_sweep_takes_clusters_while_the_chip_holds_them(G, block, pairs, clusters):
    # one chunk of velocities: as many pairs as relaxation blocks.  More clusters than fit at once
    # (or with more CTAs than cells) took up to 4.6 times as long as one CTA per pair
    wl = gi.workloads.with_solver(gi.workloads.slab(n_cells=block * pairs, n_xi=16, n_mu=8), precision="fp64",
                                  order=1, relax_block=block)
    ctx = _create(G, wl)
    G.fake.fake_reset()
    try:
        assert G.load().gsis_step_async(ctx, G.GSIS_MODE_CIS) == G.GSIS_OK
    finally:
        G.gsis_destroy(ctx)
    grid, threads, grids = C.c_int(), C.c_int(), []
    for k in range(G.fake.fake_launch_count()):
        if b"7k_sweepIdLi4" in G.fake.fake_launch(k, C.byref(grid), C.byref(threads)):
            grids.append(grid.value)
    assert grids == [8 * pairs if clusters else pairs]


@pytest.mark.parametrize("name", ["slab", "cavity", "capsule"])
@pytest.mark.parametrize("block,threads", [(1, 32), (2, 32), (3, 128), (16, 128)])
def test_fp32_sweep_has_no_idle_warps_on_small_blocks(G, name, block, threads):
    # four warps on a block of one cell left three of them idle, and the SM short of warps
    base = {"slab": lambda: gi.workloads.slab(n_cells=12, n_xi=16, n_mu=8),
            "cavity": lambda: gi.workloads.cavity(n_side=4, n_v=8),
            "capsule": lambda: gi.workloads.capsule(n=4, n_v=6, n_polar=4, n_azim=4)}[name]()
    ctx = _create(G, gi.workloads.with_solver(base, precision="fp32", order=2, relax_block=block))
    G.fake.fake_reset()
    try:
        assert G.load().gsis_step_async(ctx, G.GSIS_MODE_CIS) == G.GSIS_OK
    finally:
        G.gsis_destroy(ctx)
    grid, n, found = C.c_int(), C.c_int(), []
    for k in range(G.fake.fake_launch_count()):
        if b"k_sweep_gas32" in G.fake.fake_launch(k, C.byref(grid), C.byref(n)):
            found.append(n.value)
    assert found == [threads]
