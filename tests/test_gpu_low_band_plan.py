"""Which calls take the low band, and with which alternative (rad_selftest_band), beside their results against the oracle:
the calls that test_gpu_low_band.py means to take it do, those outside the rule do not, the particle count from which it is
considered, and bunches that grow until fewer and fewer frequencies, and then none, have wide enough cells."""
import numpy as np
import pytest

from gpu_util import gpu_run, to_dev
from paper_1802_03972_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_low_band import check, workload  # noqa: E402  (builds the library)
from paper_1802_03972_gb300 import rad  # noqa: E402

NONE = (0, 0)


def band_of(wl, steps=(0,), ctx=None):
    return gpu_run(wl, steps, ctx=ctx).selftest_band()


@pytest.mark.parametrize("n,n_omega,nx,ny,bins", [(100000, 512, 16, 16, 256), (300000, 256, 9, 7, 128),
                                                  (250000, 1024, 5, 5, 512), (200000, 700, 6, 5, 320),
                                                  (150000, 512, 8, 8, 256), (120000, 512, 4, 4, 256),
                                                  (400000, 512, 3, 1, 0), (50000, 256, 8, 8, 0)])
def test_frequencies_from_nodes(n, n_omega, nx, ny, bins):
    """(Three directions, or few particles on a small grid, do not pay for the sort and the nodes.)"""
    got, cells = band_of(workload(n, n_omega, nx, ny))
    assert got == bins and (cells > 0) == (bins > 0) and 64 * cells <= n + 64


@pytest.mark.parametrize("case,bins", [("coherent", 256), ("invalid last", 256), ("invalid first", 0), ("tilted", 256)])
def test_the_special_calls(case, bins):
    """(With the first particle invalid the reference point is the origin, a millimetre off: a wide call.)"""
    wl = workload(150000, 512, 8, 8)
    st = wl.step(0)
    r, b, bd = (v.reshape(3, -1).copy() for v in (st.r, st.beta, st.beta_dot))
    if case == "coherent":
        bd[0], bd[1] = np.abs(bd[0]), np.abs(bd[1])
    elif case.startswith("invalid"):
        r += np.array([[1e-3], [2e-3], [-1e-3]])
        at = 0 if case.endswith("first") else r.shape[1] - 3
        r[:, at:at + 2] = np.nan
        b[2, at + 2] = 1.5
    else:
        c, s = np.cos(0.4), np.sin(0.4)
        R = np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]])
        wl.dirs = wl.dirs @ R.T
        r, b, bd = R @ r + 1e-3, R @ b, R @ bd
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    ctx.accumulate(*[to_dev(a) for a in (r, b, bd, st.w)], st.t, st.dt)
    assert ctx.selftest_band()[0] == bins


def test_calls_outside_the_rule_do_not_take_it():
    base = workload(120000, 512, 4, 4)
    down = workload(120000, 512, 4, 4)
    down.omega = down.omega[::-1].copy()
    cone = workload(120000, 512, 4, 4, hi=1e18)
    cone.dirs = inputs.dirs_grid(1.2, 4, 4)
    long = workload(120000, 512, 4, 4, seed=63, sigma_z=2e-4)
    assert band_of(down) == band_of(cone) == band_of(long) == NONE
    ctx = rad.Context(base.omega, base.dirs, base.ff_kind, base.ff_width)
    seen = [band_of(wl, ctx=ctx)[0] for wl in (base, long, base)]  # one context, call by call
    assert seen == [256, 0, 256]
    ctx.set_tile(9, 512, 2048)  # chunks of the caller's
    assert band_of(base, ctx=ctx) == NONE
    ctx.set_tile(9, 256, 0)     # another width
    assert band_of(base, ctx=ctx) == NONE
    ctx.set_tile(9, 512, 0)
    assert band_of(base, ctx=ctx)[0] == 256
    lit = rad.Context(base.omega, base.dirs, base.ff_kind, base.ff_width, ff_flags=rad.FF_LITERAL)
    assert band_of(base, ctx=lit) == NONE


@pytest.mark.parametrize("n,bins", [(16383, 0), (16384, 512), (16385, 512)])
def test_particle_count_from_which_it_is_considered(n, bins):
    """Below it the call's sort is one cluster's kernel, from it on four kernels."""
    ctx = check(workload(n, 1024, 32, 32), per_dir=2)
    assert ctx.selftest_band()[0] == bins
    ctx.close()


@pytest.mark.parametrize("n,nx,n_omega,want", [(100000, 16, 512, [384, 384, 320, 256, 256, 192]),
                                               (20000, 32, 1024, [704, 704, 576, 448, 320, 0])])
def test_longer_bunches_take_fewer_frequencies(n, nx, n_omega, want):
    """Frequencies up to 1e18 rad/s: the cells of an alternative are at least 64 particles on average, so a longer bunch
    takes one of fewer frequencies, whose cells are wider, and in the end none."""
    got = []
    for k, sigma in enumerate((1e-6, 1e-5, 3e-5, 1e-4, 2e-4, 5e-4)):
        ctx = check(workload(n, n_omega, nx, nx, hi=1e18, sigma_z=sigma), per_dir=1)
        bins, cells = ctx.selftest_band()
        assert 64 * cells <= n + 64 and cells <= 4000
        got.append(bins)
        ctx.close()
    assert got == want


def test_jobs_of_a_batch_decide_for_themselves():
    wls = [workload(150000, 512, 8, 8), workload(2000, 128, 4, 4), workload(150000, 512, 8, 8, sigma_z=2e-4)]
    ctxs = [rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width) for wl in wls]
    batch = rad.Batch(ctxs)
    keep = [[to_dev(a) for a in (st.r, st.beta, st.beta_dot, st.w)] for st in (wl.step(0) for wl in wls)]
    batch.accumulate([rad.make_step(wl.n_particles, *a, 0.0, 1e-16) for wl, a in zip(wls, keep)])
    batch.sync()
    assert [c.selftest_band()[0] for c in ctxs] == [256, 0, 0]
