"""The FP64 kernel at the edges of its blocks: bins that do not fill a block, many directions in one block, one
frequency, particle counts around its chunks and staged records, against the FP64 oracle."""
import numpy as np
import pytest

from gpu_util import TOL_FP64, assert_parity, gpu_run, oracle_run, spectra_grid
from paper_1802_03972_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1802_03972_gb300 import build as _build  # noqa: E402

_build.build()
from paper_1802_03972_gb300 import rad  # noqa: E402


@pytest.mark.parametrize("n,n_omega,n_dir", [(1, 1, 1), (65, 1, 131), (3, 5, 27), (64, 128, 1), (257, 127, 2), (700, 129, 3)])
def test_fp64_block_edges(n, n_omega, n_dir):
    wl = inputs.Workload("edges", inputs.omega_log(1e14, 1e20, n_omega), inputs.dirs_theta_line(0.01, n_dir),
                         inputs.BetatronBunch(n, seed=41), 3, 1e-16, inputs.FF_GAUSS, 0.1e-6)
    ctx = gpu_run(wl, range(3), prec=rad.PREC_FP64)
    ref = spectra_grid(oracle_run(wl, range(3)), wl)
    for k, g in zip(("coh", "inc", "tot"), ctx.spectrum()):
        assert_parity(g, ref[k], tol=TOL_FP64, what=k, fp64=True)


@pytest.mark.parametrize("t", [1e-9, 1e-6, 1.0])
def test_fp64_phase_of_any_size_has_unit_modulus(t):
    """One particle's spectrum does not depend on its phase, however many turns that is (up to 1.6e19 here)."""
    wl = inputs.lwfa_bunch(n_particles=1, n_omega=64, n_side=2, seed=42)
    st = wl.step(1)
    out = []
    for at in (0.0, t):
        ctx = rad.Context(wl.omega, wl.dirs, rad.FF_GAUSS, 0.1e-6, prec=rad.PREC_FP64)
        ctx.accumulate(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (st.r, st.beta, st.beta_dot, st.w)], at, st.dt)
        out.append(ctx.spectrum()[2])
    np.testing.assert_allclose(out[1], out[0], rtol=1e-13)
