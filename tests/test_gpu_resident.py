"""The many-steps launch (k_resident) against one launch per step.

A default handle whose lattices fit the SMs' shared memory advances many
steps in one launch, a larger one two steps (FP32 storage) or one;
kernel_variant=LBM_KERNEL_TMA keeps it on the tile kernel, one launch per
step.  All run the same operations on the same values, so every output is
equal bit for bit.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2003_07968_gb300 import build, capi

    build.build()
    capi.load()
    return capi


def _desc(P, nx, ny, storage, mrt, T=0.8, **kw):
    if mrt:
        kw.update(collision=P.LBM_COLL_MRT, tau=0.7, mrt_rates=[1.0] * 7 + [1.0 / 0.7] * 2)
    return P.lbm_desc_default(nx, ny, T=T, storage=storage, **kw)


def _field(nx, ny, k=0):
    rng = np.random.default_rng(17 + k)
    rho = synth.droplet(nx, ny, 0.3 * min(nx, ny) + 1, 0.8)
    return rho + 1e-3 * rng.standard_normal(rho.shape)


def _run(P, descs, fields, chunks, **kw):
    h = P.lbm_create(descs, **kw)
    for i, f in enumerate(fields):
        P.lbm_init(h, i, f)
    l0 = P.lbm_launch_count(h)
    for n in chunks:
        P.lbm_step(h, n)
    launches = P.lbm_launch_count(h) - l0
    out = [P.lbm_moments(h, i) for i in range(len(fields))]
    P.lbm_destroy(h)
    return out, launches


def _same(a, b):
    for x, y in zip(a, b):
        for k in ("rho", "ux", "uy"):
            assert np.array_equal(x[k], y[k]), k
        assert x["mass"] == y["mass"]


# edges of strips (60 columns), of rounds (8 rows) and of packets (3 values),
# the narrowest lattices, the largest of the FP32 range
SHAPES = [(2, 2), (3, 5), (5, 3), (60, 8), (61, 9), (119, 31), (120, 33), (121, 34), (64, 64),
          (203, 77), (7, 150), (1500, 4), (181, 181), (777, 611)]


@pytest.mark.parametrize("storage,mrt", [(1, 0), (0, 1), (2, 0), (2, 1)])
def test_many_steps_equal_single_launches(P, storage, mrt):
    for nx, ny in SHAPES:
        d, f = _desc(P, nx, ny, storage, mrt, sigma=0.5), _field(nx, ny)
        chunks = (2, 1, 3, 17)
        a, la = _run(P, [d], [f], chunks)
        b, lb = _run(P, [d], [f], chunks, kernel_variant=P.LBM_KERNEL_TMA)
        assert (la, lb) == (4, 23), (nx, ny)
        _same(a, b)


def test_batches_of_resident_lattices(P):
    sizes = [(64, 64), (2, 3), (130, 40), (61, 100), (33, 7)]
    descs = [_desc(P, nx, ny, 1, 0, T=0.75 + 0.03 * k) for k, (nx, ny) in enumerate(sizes)]
    descs[2] = _desc(P, 130, 40, 1, 0, T=0.9, eos_kind=P.LBM_EOS_KIND_VDW)
    fields = [_field(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    fields[2] = synth.droplet(130, 40, 12.0, 0.9, densities=(0.42574, 1.65727))
    a, la = _run(P, descs, fields, (40,))
    b, lb = _run(P, descs, fields, (40,), kernel_variant=P.LBM_KERNEL_TMA)
    assert (la, lb) == (1, 40)
    _same(a, b)


def test_handles_on_many_streams_at_once(P):
    # blocks of a launch wait for one another, so launches that could run at
    # the same time must fit the GPU together: handles that do not are queued
    sizes = [(400, 400), (64, 64), (256, 256), (500, 300), (64, 64), (200, 200), (400, 410), (90, 90)]
    hs = [P.lbm_create(_desc(P, nx, ny, 1, 0)) for nx, ny in sizes]
    for k, (h, (nx, ny)) in enumerate(zip(hs, sizes)):
        P.lbm_init(h, 0, _field(nx, ny, k))
    for n in (50, 2, 101):
        for h in hs:
            P.lbm_step(h, n)
    got = [P.lbm_moments(h, 0) for h in hs]
    for h in hs:
        P.lbm_destroy(h)
    for k, (nx, ny) in enumerate(sizes):
        want, _ = _run(P, [_desc(P, nx, ny, 1, 0)], [_field(nx, ny, k)], (153,),
                       kernel_variant=P.LBM_KERNEL_TMA)
        _same([got[k]], want)


# ------------------------------------------------------- one step a launch on rows
# lattices beyond the resident range: edges of strips and items, ragged sizes,
# the narrowest and the flattest, one wave of items and several
ROW_SHAPES = [(901, 1403), (1200, 1100), (3, 40011), (61, 21001), (16001, 85), (2500, 1931)]


@pytest.mark.parametrize("storage,mrt", [(1, 0), (0, 1), (2, 0), (2, 1)])
def test_row_kernels_equal_tile_kernel(P, storage, mrt):
    for nx, ny in ROW_SHAPES:
        d, f = _desc(P, nx, ny, storage, mrt, sigma=0.5), _field(nx, ny)
        for kw in ({}, {"graph_steps": 2}, {"graph_steps": -1}):
            # not resident: FP32 two steps a launch and the odd ones single
            a, la = _run(P, [d], [f], (5, 1, 4), **kw)
            assert la == (10 if storage == 2 else 6), (nx, ny)
            b, lb = _run(P, [d], [f], (10,), kernel_variant=P.LBM_KERNEL_TMA) if not kw else (b, 10)
            assert lb == 10
            _same(a, b)


@pytest.mark.parametrize("storage", [1, 2])
def test_row_kernel_batches(P, storage):
    sizes = [(700, 651), (3, 5), (61, 300), (2, 2), (800, 701), (33, 7), (640, 640), (57, 1)]
    sizes = [(nx, max(ny, 2)) for nx, ny in sizes]
    descs = [_desc(P, nx, ny, storage, 0, T=0.7 + 0.02 * k) for k, (nx, ny) in enumerate(sizes)]
    fields = [_field(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    a, la = _run(P, descs, fields, (35,))
    b, lb = _run(P, descs, fields, (35,), kernel_variant=P.LBM_KERNEL_TMA)
    assert (la, lb) == (35 if storage == 2 else 18, 35)
    _same(a, b)


@pytest.mark.parametrize("storage", [1, 2])
def test_served_results_equal_a_plain_handle(P, storage):
    # the server's requests run on row items with step quotas: two steps a
    # launch in FP32 storage, odd quotas ending among even ones
    import time

    srv = P.lbm_server_create(P.lbm_server_opts_default(
        arena_bytes=1 << 30, max_request_sites=512 * 512, max_width=512, chunk_steps=7,
        storage=storage))
    reqs = [(100, 37, 20), (512, 300, 31), (61, 130, 5), (2, 3, 1), (400, 512, 13), (57, 9, 2)]
    todo = {}
    for k, (nx, ny, n) in enumerate(reqs):
        d, f = _desc(P, nx, ny, storage, 0), _field(nx, ny, k)
        todo[P.lbm_submit(srv, d, f, n)] = (d, f, n)
    while todo:
        for t in list(todo):
            got = P.lbm_poll(srv, t)
            if got is not None:
                d, f, n = todo.pop(t)
                want, _ = _run(P, [d], [f], (n,), kernel_variant=P.LBM_KERNEL_TMA)
                for key in ("rho", "ux", "uy"):
                    assert np.array_equal(got[key], want[0][key]), (key, d.nx, d.ny)
        time.sleep(0.001)
    P.lbm_server_destroy(srv)


# ------------------------------------------------------------ fields read back
def test_fields_read_back_into_any_host_array(P):
    # page-locked arrays are written by the kernel itself up to 2^20 sites,
    # others through copies: the same values, whichever each field lies in
    import torch

    for nx, ny in ((5, 3), (77, 41), (1024, 1024), (1025, 1024)):
        h = P.lbm_create(_desc(P, nx, ny, 1, 0))
        P.lbm_init(h, 0, _field(nx, ny))
        P.lbm_step(h, 4)
        pin = lambda: torch.full((ny, nx), -1.0, dtype=torch.float64, pin_memory=True).numpy()
        page = lambda: np.full((ny, nx), -1.0)
        want = P.lbm_moments(h, 0, out={k: page() for k in ("rho", "ux", "uy")})
        # one field alone, an array inside a larger page-locked one, a mixture
        big = torch.full((2 * ny * nx + 3,), -1.0, dtype=torch.float64, pin_memory=True).numpy()
        rho = big[3:3 + nx * ny].reshape(ny, nx)
        P.lbm_moments(h, 0, u=False, mass=False, out={"rho": rho})
        assert np.array_equal(rho, want["rho"])
        assert np.all(big[:3] == -1.0) and np.all(big[3 + nx * ny:] == -1.0)
        for mix in ((pin(), pin(), pin()), (pin(), page(), pin())):
            got = P.lbm_moments(h, 0, out=dict(zip(("rho", "ux", "uy"), mix)))
            _same([got], [want])
        P.lbm_destroy(h)


def test_steps_captured_by_the_caller_replay(P):
    # into a caller's capture goes one launch per step, so that a replay of an
    # even number of steps ends in the buffer it started from
    import torch

    for nx, ny in ((64, 50), (1100, 901)):
        d, f = _desc(P, nx, ny, 1, 0), _field(nx, ny)
        h = P.lbm_create(d)
        P.lbm_init(h, 0, f)
        P.lbm_step(h, 4)
        P.lbm_sync(h)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=h.stream):
            P.lbm_step(h, 2)
        with torch.cuda.stream(h.stream):
            for _ in range(3):
                g.replay()
        got = P.lbm_moments(h, 0)
        P.lbm_destroy(h)
        want, _ = _run(P, [d], [f], (10,), kernel_variant=P.LBM_KERNEL_TMA)
        _same([got], want)
