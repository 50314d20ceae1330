"""FP32 face solvers on packed (left, right) pairs: against the FP64 path, whose
solvers are scalar, and a gas without field against the same gas in an MHD
context with B = 0 (every field term is a product with zero, so bit for bit),
with supersonic, still and strongly sheared regions and tiles with remainders."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from tests.gpu_helpers import RECON, RIEMANN

pytestmark = pytest.mark.gpu

N = (35, 9, 6)   # flux faces 36 x 10 x 7: tiles of 32 x 4 with remainders each way


def _state(mhd):
    nx, ny, nz = N
    rng = np.random.default_rng(11)
    cons = np.zeros((5, nz, ny, nx))
    cons[0] = 0.3 + rng.random((nz, ny, nx))
    v = rng.standard_normal((3, nz, ny, nx))
    v[:, :, :, :6] = 0.0                       # contact and shear only
    v[0, :, :, 20:] += 6.0                     # supersonic both ways
    v[0, :, :, 28:] -= 12.0
    cons[1:4] = cons[0] * v
    b = [np.zeros((nz, ny, nx + 1)), np.zeros((nz, ny + 1, nx)), np.zeros((nz + 1, ny, nx))]
    if mhd:   # each component constant along its own axis: divergence-free
        b[0][:] = 0.4 * rng.standard_normal((nz, ny, 1))
        b[1][:] = 0.4 * rng.standard_normal((nz, 1, nx))
        b[2][:] = 0.4 * rng.standard_normal((1, ny, nx))
        b[0][:, :3] = 0.0                      # degenerate: no normal field
    bb = (b[0][:, :, :-1] ** 2 + b[1][:, :-1] ** 2 + b[2][:-1] ** 2) / 2
    cons[4] = (0.2 + rng.random((nz, ny, nx))) / 0.4 + 0.5 * (cons[1:4] ** 2).sum(0) / cons[0] + bb
    # values FP32 holds exactly: both precisions start from the same state
    f = lambda a: a.astype(np.float32).astype(np.float64)
    return f(cons), [f(x) for x in b]


def _one_step(cons, b, recon, riemann, prec, mhd):
    import torch
    cfg = A.make_config(gamma=1.4, recon=RECON[recon][1], integrator=A.RK2, precision=prec,
                        mhd=mhd, riemann=RIEMANN[riemann][1])
    sv = A.Solver(cfg, [A.make_block(N, (0.0,) * 3, (N[0] / 35.0, N[1] / 35.0, N[2] / 35.0))],
                  stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, cons, *b) if mhd else sv.set_state(0, cons)
        sv.step(2e-4)
        return sv.get_state(0)
    finally:
        sv.close()


@pytest.mark.parametrize("recon", ["donor", "plm", "ppm"])
@pytest.mark.parametrize("riemann", ["hlld", "lhlld", "hlle"])
def test_hydro_context_equals_mhd_context_without_field(recon, riemann):
    cons, b = _state(False)
    hydro = _one_step(cons, b, recon, riemann, A.FP32, False)[0]
    mhd = _one_step(cons, b, recon, riemann, A.FP32, True)
    np.testing.assert_array_equal(hydro, mhd[0])
    assert all(not f.any() for f in mhd[1:])


@pytest.mark.parametrize("recon", ["donor", "plm", "ppm"])
@pytest.mark.parametrize("riemann", ["hlld", "lhlld", "hlle"])
def test_fp32_pairs_against_fp64(recon, riemann):
    """One RK2 step of dt/dx = 7e-3 over fluxes up to about 500: roundings of
    the state (energies up to 40, 2^-24 each) and of some thirty operations a
    flux times dt/dx stay under 1e-4; a wrong term is off by 1e-2 and more."""
    cons, b = _state(True)
    got = _one_step(cons, b, recon, riemann, A.FP32, True)
    ref = _one_step(cons, b, recon, riemann, A.FP64, True)
    for x, y in zip(got, ref):
        assert np.abs(x - y).max() < 2e-4
        assert np.abs(x - y).mean() < 1e-5
