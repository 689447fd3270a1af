"""Device memory of contexts: what a call's buffers may take, and that the library's own count of it is the device's."""
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
