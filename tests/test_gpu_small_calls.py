"""Small calls: chunks of 128 particles, one chunk per tile, tiles of many chunks, grids that are no multiple of four
frequencies (the tile reduction's scalar path), ragged tiles and directions; alone, batched and replayed from a graph."""
import numpy as np
import pytest

from gpu_util import assert_parity, gpu_run, oracle_run, spectra_grid, to_dev
from paper_1802_03972_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1802_03972_gb300 import build as _build  # noqa: E402

_build.build()
from paper_1802_03972_gb300 import rad  # noqa: E402

# (particles, frequencies, directions): one particle; one chunk; many chunks of one tile; a
# frequency count that is no multiple of 4; one frequency; a tile's last directions and frequencies outside the grid
SIZES = [(1, 1, 1), (33, 64, 1), (5000, 64, 3), (300, 99, 5), (777, 1, 37), (2049, 130, 9), (20000, 257, 2)]


def workload(n, n_omega, n_dir):
    return inputs.Workload("small", inputs.omega_log(1e14, 1e20, n_omega), inputs.dirs_theta_line(0.012, n_dir),
                           inputs.BetatronBunch(n, seed=51), 2, 1e-16, inputs.FF_GAUSS, 0.1e-6)


@pytest.mark.parametrize("variant", [0, 9])
@pytest.mark.parametrize("n,n_omega,n_dir", SIZES)
def test_small_calls_against_the_oracle(n, n_omega, n_dir, variant):
    wl = workload(n, n_omega, n_dir)
    ctx = gpu_run(wl, range(2), tile=(variant, 0, 0))
    ref = spectra_grid(oracle_run(wl, range(2)), wl)
    for k, g in zip(("coh", "inc", "tot"), ctx.spectrum()):
        assert_parity(g, ref[k], what=k)


@pytest.mark.parametrize("n_omega", [64, 99])
def test_literal_sum_of_a_small_call(n_omega):
    wl = workload(700, n_omega, 5)
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width, ff_flags=rad.FF_LITERAL)
    gpu_run(wl, range(2), ctx=ctx)
    ref = oracle_run(wl, range(2)).spectra()["paper"].reshape(5, n_omega)
    assert_parity(ctx.spectrum_literal(), ref, what="literal")


def test_batch_of_small_jobs_equals_each_alone():
    """The batch hands out runs of the jobs' chunks; the chunks and the results are the jobs' own."""
    wls = [workload(*s) for s in SIZES]
    alone = [gpu_run(wl, range(2)).spectrum() for wl in wls]
    ctxs = [rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width) for wl in wls]
    batch, keep = rad.Batch(ctxs), []
    for s in range(2):
        keep.append([[to_dev(a) for a in (st.r, st.beta, st.beta_dot, st.w)] for st in (wl.step(s) for wl in wls)])
        batch.accumulate([rad.make_step(wl.n_particles, *a, s * wl.dt, wl.dt) for wl, a in zip(wls, keep[-1])])
    batch.sync()
    for a, c in zip(alone, ctxs):
        for x, y in zip(a, c.spectrum()):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("n", [64, 3000, 20000])
def test_accumulate_replayed_from_a_captured_graph(n):
    """A program may capture its step: every replay leaves the counters ready for the next one."""
    wl = workload(n, 96, 4)
    st = wl.step(1)
    arrs = [to_dev(a) for a in (st.r, st.beta, st.beta_dot, st.w)]
    stream = torch.cuda.Stream()
    direct = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width, stream=stream)
    for _ in range(4):
        direct.accumulate(*arrs, st.t, st.dt)
    torch.cuda.synchronize()
    ctx.accumulate(*arrs, st.t, st.dt)  # sizes the context's buffers
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.accumulate(*arrs, st.t, st.dt)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for x, y in zip(direct.spectrum(), ctx.spectrum()):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("variant", [0, 2, 7, 9])
@pytest.mark.parametrize("n_omega,n_dir", [(65, 8), (150, 3), (300, 9), (330, 2), (450, 1), (520, 5), (800, 11), (850, 1)])
def test_frequency_segments_of_every_width(n_omega, n_dir, variant):
    """Frequency counts that leave 1 to 7 warps' worth past the last full tile: covered by narrower tiles."""
    wl = workload(500, n_omega, n_dir)
    ctx = gpu_run(wl, range(2), tile=(variant, 0, 0))
    ref = spectra_grid(oracle_run(wl, range(2)), wl)
    for k, g in zip(("coh", "inc", "tot"), ctx.spectrum()):
        assert_parity(g, ref[k], what=k)
