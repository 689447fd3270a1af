"""The low band (interpolated from evenly spaced nodes per cell of particles) against the oracle: calls large enough to
take it, on log grids of several sizes, ragged directions, shifted, tilted and invalid particles; determinism, the same
results alone and in a batch, and calls just outside the rule."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_sampled_bins, to_dev
from paper_1802_03972_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1802_03972_gb300 import build as _build  # noqa: E402

_build.build()
from paper_1802_03972_gb300 import rad  # noqa: E402


def workload(n, n_omega, nx, ny, seed=61, lo=1e14, hi=1e20, **bunch):
    return inputs.Workload("low", inputs.omega_log(lo, hi, n_omega), inputs.dirs_grid(0.01, nx, ny),
                           inputs.BetatronBunch(n, seed=seed, **bunch), 4, 1e-16, inputs.FF_GAUSS, 0.1e-6)


def check(wl, arrays=None, per_dir=5, seed=3):
    """One step and a second of the same context, against the oracle on sampled bins of several directions, most in the
    band: its first bins, its last ones and the first past it."""
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    rng = np.random.default_rng(seed)
    n_dir, n_om = wl.dirs.shape[0], wl.omega.shape[0]
    dirs = sorted({0, n_dir - 1, n_dir // 2})
    bins = [(d, int(o)) for d in dirs for o in
            [0, 1, n_om // 3, n_om // 2 - 1, n_om // 2, n_om - 1] + list(rng.integers(0, n_om, per_dir))]
    bo, bd = oracle.grid_bins(wl.omega, wl.dirs, bins)
    acc = oracle.Accumulator(bo, bd, wl.ff_kind, wl.ff_width)
    for s in range(2):
        st = wl.step(s) if arrays is None else arrays(s)
        ctx.accumulate(*[to_dev(a) for a in (st.r, st.beta, st.beta_dot, st.w)], st.t, st.dt)
        acc.accumulate(st.r, st.beta, st.beta_dot, st.w, st.t, st.dt)
    got = dict(zip(("coh", "inc", "tot"), ctx.spectrum()))
    ref = acc.spectra()
    assert_sampled_bins(got, {k: ref[k] for k in got}, bins)
    return ctx


@pytest.mark.parametrize("n,n_omega,nx,ny", [(100000, 512, 16, 16), (300000, 256, 9, 7), (250000, 1024, 5, 5),
                                             (200000, 700, 6, 5), (400000, 512, 3, 1)])
def test_low_band_against_the_oracle(n, n_omega, nx, ny):
    check(workload(n, n_omega, nx, ny))


def test_low_band_far_from_the_origin_and_off_axis():
    """A bunch a millimetre off, seen along a tilted cone: the cells' references and the grid's frame carry it."""
    wl = workload(200000, 512, 8, 8)
    c, s = np.cos(0.4), np.sin(0.4)
    R = np.array([[c, 0, s], [0, 1, 0], [-s, 0, c]])
    wl.dirs = wl.dirs @ R.T

    def arrays(k):
        st = wl.step(k)
        turn = lambda v: R @ v.reshape(3, -1)  # noqa: E731
        return inputs.Step(turn(st.r) + np.array([[1e-3], [-2e-3], [5e-4]]), turn(st.beta), turn(st.beta_dot), st.w,
                           st.t + 3e-12, st.dt)
    check(wl, arrays)


@pytest.mark.parametrize("first", [False, True])
def test_low_band_with_invalid_particles(first):
    """Invalid particles at the end, or first (the call's reference is then the origin, a millimetre from the bunch)."""
    wl = workload(150000, 512, 8, 8)
    good = wl.step(0)
    if first:
        good.r = good.r.reshape(3, -1) + np.array([[1e-3], [2e-3], [-1e-3]])
    ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    ref = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
    ref.accumulate(*[to_dev(a) for a in (good.r, good.beta, good.beta_dot, good.w)], 0.0, 1e-16)
    order = (lambda v, b: [b, v]) if first else (lambda v, b: [v, b])
    pad = lambda v, bad: np.concatenate(order(v.reshape(3, -1), np.array(bad, dtype=float).T), axis=1)  # noqa: E731
    ctx.accumulate(to_dev(pad(good.r, [[np.nan, 0, 0], [0, 1.0, 0], [0, 0, np.inf]])),
                   to_dev(pad(good.beta, [[0, 0, .5], [0, 0, 1.5], [0, 0, .5]])),
                   to_dev(pad(good.beta_dot, [[1e13, 0, 0]] * 3)), to_dev(np.concatenate(order(good.w, [10.0, 10.0, 10.0]))),
                   0.0, 1e-16)
    with pytest.raises(rad.RadError) as ei:
        ctx.spectrum()
    assert ei.value.status == rad.RAD_EDATA
    for a, b in zip(ctx.spectrum(), ref.spectrum()):  # (other chunks: rounding only)
        np.testing.assert_allclose(np.linalg.norm(a - b, axis=1), 0.0, atol=1e-5 * np.linalg.norm(b, axis=1).max())


def test_low_band_is_deterministic_and_the_same_in_a_batch():
    wls = [workload(150000, 512, 8, 8), workload(2000, 128, 4, 4), workload(300000, 300, 9, 9, seed=62)]
    alone = []
    for wl in wls:
        runs = []
        for _ in range(2):
            ctx = rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width)
            for s in range(2):
                st = wl.step(s)
                ctx.accumulate(*[to_dev(a) for a in (st.r, st.beta, st.beta_dot, st.w)], st.t, st.dt)
            runs.append(ctx.spectrum())
        for x, y in zip(*runs):
            np.testing.assert_array_equal(x, y)
        alone.append(runs[0])
    ctxs = [rad.Context(wl.omega, wl.dirs, wl.ff_kind, wl.ff_width) for wl in wls]
    batch, keep = rad.Batch(ctxs), []
    for s in range(2):
        st = [wl.step(s) for wl in wls]
        keep.append([[to_dev(a) for a in (x.r, x.beta, x.beta_dot, x.w)] for x in st])
        batch.accumulate([rad.make_step(x.n, *a, x.t, x.dt) for x, a in zip(st, keep[-1])])
    batch.sync()
    for a, c in zip(alone, ctxs):
        for x, y in zip(a, c.spectrum()):
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("case", ["descending", "wide angles", "long", "alternating"])
def test_calls_outside_the_rule(case):
    """Frequencies in another order, directions over a wide cone and bunches too long for the cells take the bin tiles; a
    context that changes between the two keeps both right."""
    wl = workload(120000, 512, 4, 4)
    arrays = None
    if case == "descending":
        wl.omega = wl.omega[::-1].copy()
    elif case == "wide angles":
        wl.dirs = inputs.dirs_grid(1.2, 4, 4)
        wl.omega = inputs.omega_log(1e14, 1e18, 512)
    elif case == "long":
        wl.bunch = inputs.BetatronBunch(120000, seed=63, sigma_z=2e-4)
    else:
        long = inputs.BetatronBunch(120000, seed=63, sigma_z=2e-4)
        arrays = lambda s: (long if s else wl.bunch).step(s * wl.dt, wl.dt)  # noqa: E731
    check(wl, arrays, per_dir=2)


def test_low_band_of_a_coherent_bunch():
    """All accelerations the same way: the cells' sums are coherent and cancel beyond the bunch's roll-off."""
    wl = workload(150000, 512, 8, 8)
    b = wl.bunch
    b.x0, b.y0 = np.abs(b.x0), np.abs(b.y0)
    b.phx[:], b.phy[:] = 1.0, 0.5
    check(wl, per_dir=40)
