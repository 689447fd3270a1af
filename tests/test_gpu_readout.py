"""The readout kernels on a given state (a checkpoint), bin by bin against NumPy in 64 bits: one and several bins per
thread, ragged grids, zeros and subnormal values in the state, every shape, two species."""
import struct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1802_03972_gb300 import build as _build  # noqa: E402

_build.build()
from paper_1802_03972_gb300 import inputs, rad  # noqa: E402

C = 299792458.0
K0 = 1.602176634e-19**2 / (16.0 * np.pi**3 * 8.8541878128e-12 * C)


def form(kind, width, x):
    if kind == rad.FF_GAUSS:
        return np.exp(-0.5 * (x * width / C) ** 2)
    h = x * width / (2 * C)
    s = np.where(h == 0.0, 1.0, np.sin(h) / np.where(h == 0.0, 1.0, h))
    return {rad.FF_POINT: np.ones_like(x), rad.FF_CIC: s, rad.FF_TSC: s**2, rad.FF_QSC: s**3}[kind]


def factor(ff, omega, dirs):
    if len(ff) > 2 and ff[0] not in (rad.FF_POINT, rad.FF_GAUSS):
        return np.stack([np.prod([form(ff[0], ff[1], omega * x) for x in d], axis=0) for d in dirs])
    return np.broadcast_to(form(ff[0], ff[1], omega), (len(dirs), len(omega)))


@pytest.mark.parametrize("n_omega,nx,ny", [(1, 1, 1), (7, 3, 1), (1, 40, 33), (333, 15, 10), (512, 16, 16), (1000, 9, 13)])
def test_readouts_of_a_given_state(n_omega, nx, ny):
    rng = np.random.default_rng(n_omega + nx)
    omega, dirs = inputs.omega_log(1e14, 3e17, n_omega), inputs.dirs_grid(0.01, nx, ny)
    dirs = dirs / np.linalg.norm(dirs, axis=1, keepdims=True)
    shape = (len(dirs), n_omega)
    ctxs, states = [], []
    for _ in range(2):
        v = (rng.normal(0, 1, (8, *shape)) * 10.0 ** rng.uniform(-3, 6, shape)).astype(np.float32)
        v[:, rng.random(shape) < 0.1] = 0.0
        v.reshape(8, -1)[:, 0] = np.float32(1e-41)  # subnormal
        comp = (v * rng.uniform(-3e-8, 3e-8, v.shape)).astype(np.float32)
        a = np.concatenate([v, comp])
        c = rad.Context(omega, dirs, rad.FF_GAUSS, 1e-7)
        c.state_import(struct.pack("<IIiiiiiiQ", 0x52414453, 1, 0, n_omega, len(dirs), 16, 4, 0, a.nbytes) + a.tobytes())
        ctxs.append(c)
        states.append(a[:8].astype(np.float64) - a[8:].astype(np.float64))
    f3 = (rad.FF_QSC, 2e-9, rad.FF_3D)
    # (allowed: 1e-11 of the value, from rounding in FP64 and, near a shape's zeros, of the sines' arguments: 1e-13 of |S|^2)
    for ff in [(rad.FF_POINT, 0.0), (rad.FF_CIC, 1e-8), (rad.FF_TSC, 3e-9), (rad.FF_GAUSS, 1e-9), f3, (rad.FF_TSC, 5e-9, rad.FF_3D)]:
        f = factor(ff, omega, dirs)
        u2, v2 = (states[0][:4] ** 2).sum(0), (states[0][4:] ** 2).sum(0)
        ref = [K0 * f**2 * u2, K0 * (1 - f**2) * v2]
        ref.append(ref[0] + ref[1])
        for g, r in zip(ctxs[0].spectrum(ff), ref):
            assert np.all(np.abs(g - r) <= 1e-11 * np.abs(r) + 1e-13 * K0 * (u2 + v2)), ff
    ffs = [(rad.FF_GAUSS, 1e-9), f3]
    fs = [factor(ff, omega, dirs) for ff in ffs]
    amp = sum(f * s[:4] for f, s in zip(fs, states))
    ref = [K0 * (amp**2).sum(0), K0 * sum((1 - f**2) * (s[4:] ** 2).sum(0) for f, s in zip(fs, states))]
    ref.append(ref[0] + ref[1])
    scale = sum((s**2).sum(0) for s in states)
    for g, r in zip(rad.spectrum_species(ctxs, ffs), ref):
        assert np.all(np.abs(g - r) <= 1e-11 * np.abs(r) + 1e-12 * K0 * scale)
