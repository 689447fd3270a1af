"""The autotuner and the low band: a tile that switches the band off is kept only where it is faster than the band, and a
cache file from before the band does not decide for calls that may take it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1802_03972_gb300 import build as _build  # noqa: E402

_build.build()
from paper_1802_03972_gb300 import inputs, rad  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def tuned(n, n_omega, side, cache, descending=False):
    """The tile that a fresh process (the cache file is read once) tunes."""
    code = ("import sys\nfrom paper_1802_03972_gb300 import rad, inputs\n"
            f"om = inputs.omega_log(1e14, 1e20, {n_omega}){'[::-1].copy()' if descending else ''}\n"
            f"print(*rad.Context(om, inputs.dirs_grid(0.01, {side}, {side}), rad.FF_GAUSS, 1e-7).tune({n}))\n")
    env = dict(os.environ, RAD_TUNE_CACHE=str(cache), PYTHONPATH=ROOT)
    p = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0, p.stderr[-2000:]
    return tuple(int(x) for x in p.stdout.split())


def test_cache_lines_from_before_the_band(tmp_path):
    cache = tmp_path / "tiles"
    cache.write_text("512 256 16 8 256 0\n")  # 512 frequencies, 256 directions, 65536-131071 particles: variant 8
    assert tuned(100000, 512, 16, cache) == (9, 512, 0)
    lines = cache.read_text().splitlines()
    assert lines[1:] == ["512 256 16 9 512 0 1"]
    assert tuned(100000, 512, 16, cache, descending=True) == (8, 256, 0)  # a grid without the band: the line holds
    cache.write_text("512 256 16 8 256 0 1\n")  # a choice made with the band in mind
    assert tuned(100000, 512, 16, cache) == (8, 256, 0)


@pytest.mark.parametrize("n,n_omega,side", [(40000, 1024, 32), (100000, 512, 16), (60000, 512, 8)])
def test_tuned_contexts_keep_the_band(n, n_omega, side):
    """The trials' particles are fewer than the band needs at these sizes; the band saves a fifth of the call and more."""
    ctx = rad.Context(inputs.omega_log(1e14, 1e20, n_omega), inputs.dirs_grid(0.01, side, side), rad.FF_GAUSS, 1e-7)
    assert ctx.tune(n) == (9, 512, 0)
    ctx.close()


@pytest.mark.parametrize("nth", range(6, 16))
def test_a_shortage_during_the_trials_does_not_outlast_them(nth):
    """The nth buffer that a trial allocates is refused, a band buffer at some nth: the tuner goes on without the band, and
    the caller's next call, with memory for it, takes it."""
    from gpu_util import gpu_run
    n_omega = 512 + 4 * nth  # (a shape of its own: results are cached)
    wl = inputs.Workload("tune", inputs.omega_log(1e14, 1e20, n_omega), inputs.dirs_grid(0.01, 8, 8),
                         inputs.BetatronBunch(60000, seed=81), 4, 1e-16, inputs.FF_GAUSS, 1e-7)
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    ctx.selftest_fail_alloc(nth)
    try:
        ctx.tune(60000)
    except rad.RadError as e:  # a buffer of a candidate without the band
        assert e.status == rad.RAD_ENOMEM
    ctx.selftest_fail_alloc(0)
    ctx.set_tile(9, 0, 0)
    assert gpu_run(wl, [0], ctx=ctx).selftest_band()[0] > 0
    ctx.close()
