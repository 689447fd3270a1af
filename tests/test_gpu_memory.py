"""Device memory of contexts: what a call's buffers may take, and that the library's own count of it is the device's."""
import time

import numpy as np
import pytest

from gpu_util import gpu_run, to_dev
from paper_1802_03972_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1802_03972_gb300 import build as _build  # noqa: E402

_build.build()
from paper_1802_03972_gb300 import rad  # noqa: E402

BLOCKS = 2 * torch.cuda.get_device_properties(0).multi_processor_count  # resident blocks of the default variant
TILE_BINS = 512                                                         # bins of its tile


def workload(n, n_omega, nx, ny):
    return inputs.Workload("memory", inputs.omega_log(1e14, 1e20, n_omega), inputs.dirs_grid(0.01, nx, ny),
                           inputs.BetatronBunch(n, seed=71), 4, 1e-16, inputs.FF_GAUSS, 0.1e-6)


@pytest.mark.parametrize("n,n_omega,nx,ny", [(100000, 512, 16, 16), (400000, 1024, 16, 16), (300000, 4096, 16, 16),
                                             (150000, 512, 8, 8)])
def test_partial_sums_stay_within_the_work_items(n, n_omega, nx, ny):
    """Every alternative of a call's low band cuts its own bins into chunks: about 8 items of a tile's bins per resident
    block (at most 2048 particles' worth of rounding apart, so allow 24 as without the band), plus one chunk of all bins."""
    wl = workload(n, n_omega, nx, ny)
    bins = n_omega * nx * ny
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    base = ctx.selftest_memory()
    free0 = torch.cuda.mem_get_info()[0]
    st = wl.step(0)
    arrs = [to_dev(a) for a in (st.r, st.beta, st.beta_dot, st.w)]
    torch.cuda.synchronize()
    taken = free0 - torch.cuda.mem_get_info()[0]
    free0 = torch.cuda.mem_get_info()[0]
    ctx.accumulate(*arrs, st.t, st.dt)
    ctx.sync()
    held = ctx.selftest_memory() - base
    records = n * (80 + 13 + 80) + (64 << 10)          # records, sort buffers, records in cell order
    fine = 32 * TILE_BINS * (6 * BLOCKS + 40 * 24)     # the fine-chunked last tiles
    low = 32 * 8 * n_omega * (2 * BLOCKS + (nx * ny + 7) // 8)
    assert held <= records + 32 * (24 * BLOCKS * TILE_BINS + bins) + fine + low, held
    # the count is the device's (allocations are rounded up to 2 MB), and nothing is missing from it
    got = free0 - torch.cuda.mem_get_info()[0]
    assert held - (2 << 20) <= got <= held + 12 * (2 << 20), (held, got, taken)
    print("held", n, n_omega, nx * ny, held)
    assert np.all(np.isfinite(ctx.spectrum()[2]))
    ctx.close()


def test_growing_calls_of_a_band_context_equal_fresh_ones():
    """Calls of growing and shrinking sizes through one context: the partial sums' layout is each call's own."""
    ctx = None
    for n in (20000, 150000, 3000, 90000):
        wl = workload(n, 512, 8, 8)
        if ctx is None:
            ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
        ctx.reset()
        gpu_run(wl, [0], ctx=ctx)
        for x, y in zip(ctx.spectrum(), gpu_run(wl, [0]).spectrum()):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("n,n_omega,nx,ny", [(300, 64, 2, 2), (3000, 128, 4, 4), (20000, 300, 5, 3), (60000, 512, 8, 8),
                                             (150000, 1024, 9, 9), (40000, 64, 1, 1), (30000, 2048, 32, 32)])
def test_a_limited_context_stays_within_its_limit(n, n_omega, nx, ny):
    """Calls of up to the stated number of particles, in sizes that make the buffers grow again and again, leave the
    context within the bytes a server would count for it."""
    wl = workload(n, n_omega, nx, ny)
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    limit = ctx.selftest_limit(n)
    assert ctx.selftest_memory() <= limit
    st = wl.step(0)
    arrs = [a.reshape(3, n) for a in (st.r, st.beta, st.beta_dot)]
    rng = np.random.default_rng(5)
    sizes = sorted({1, 32, 128, 256, 257, *(int(x) for x in np.geomspace(1, n, 25)), *rng.integers(1, n, 10), n} & set(range(n + 1)))
    for m in [int(x) for x in sizes]:
        ctx.accumulate(*[to_dev(a[:, :m].copy()) for a in arrs], to_dev(st.w[:m]), st.t, st.dt)
        assert ctx.selftest_memory() <= limit, m
    ctx.sync()
    print("limit", n, n_omega, nx * ny, limit, "held", ctx.selftest_memory())
    ctx.close()


def test_small_jobs_are_counted_at_what_they_hold():
    """A job of 1000 particles on 64 x 4 bins holds some hundred kilobytes: a server of 200 MB accepts it, and one of 1 GB
    holds 30 at once."""
    omega, dirs = inputs.omega_log(1e14, 1e20, 64), inputs.dirs_grid(0.01, 2, 2)
    srv = rad.Server(hbm_budget=200 << 20, max_slots=4)
    srv.submit(omega, dirs, inputs.FF_GAUSS, 0.1e-6, max_particles=1000, max_queued=2)
    srv.close()
    srv = rad.Server(hbm_budget=1 << 30, max_slots=64)
    for _ in range(30):
        srv.submit(omega, dirs, inputs.FF_GAUSS, 0.1e-6, max_particles=1000, max_queued=2)
    deadline = time.time() + 30
    while srv.stats()["active"] < 30 and time.time() < deadline:
        time.sleep(0.005)
    s = srv.stats()
    assert s["active"] == 30 and s["footprint_bytes"] <= 30 * (2 << 20), s
    srv.close()


def test_a_job_that_fits_only_without_the_low_band_runs_without_it():
    """Between the job's bytes with the band's buffers and without them the server takes it, and its spectrum is the one
    the bin tiles give (a context whose band found no memory)."""
    wl = workload(150000, 512, 8, 8)
    grids = (wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    ctx = rad.Context(*grids)
    staging = 2 * 80 * 150000
    full = ctx.selftest_limit(150000) + staging
    ctx.selftest_fail_alloc(8)
    gpu_run(wl, range(2), ctx=ctx)
    tiles = ctx.spectrum()
    srv = rad.Server(hbm_budget=full - 1, max_slots=1)
    j = srv.submit(*grids, max_particles=150000, max_queued=2)
    for s in range(2):
        st = wl.step(s)
        while srv.feed(j, rad.make_step(st.n, st.r, st.beta, st.beta_dot, st.w, st.t, st.dt)) != rad.RAD_OK:
            time.sleep(0.001)
    srv.finish(j)
    got = srv.result(j, 64, 512, timeout=60)
    assert srv.stats()["peak_footprint_bytes"] < full
    srv.close()
    for x, y in zip(got[:3], tiles):
        np.testing.assert_array_equal(x, y)
    srv = rad.Server(hbm_budget=full, max_slots=1)
    j = srv.submit(*grids, max_particles=150000, max_queued=2)
    while srv.stats()["active"] < 1:
        time.sleep(0.001)
    assert srv.stats()["footprint_bytes"] == full
    srv.close()
