"""The isothermal HLLD solver on packed (left, right) pairs: against the FP64 path, and
a gas without field against the same gas with B = 0, on the states of
test_gpu_pair_solvers.py."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from tests.gpu_helpers import RECON
from tests.test_gpu_pair_solvers import N, _state

pytestmark = pytest.mark.gpu


def _one_step(cons, b, recon, prec, mhd):
    import torch
    cfg = A.make_config(recon=RECON[recon][1], integrator=A.RK2, precision=prec, mhd=mhd, riemann=A.HLLD,
                        iso=True, cs=0.7)
    sv = A.Solver(cfg, [A.make_block(N, (0.0,) * 3, (N[0] / 35.0, N[1] / 35.0, N[2] / 35.0))],
                  stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, cons, *b) if mhd else sv.set_state(0, cons)
        sv.step(2e-4)
        return sv.get_state(0)
    finally:
        sv.close()


@pytest.mark.parametrize("recon", ["donor", "plm", "ppm", "ppm5"])
def test_hydro_context_equals_mhd_context_without_field(recon):
    cons, b = _state(False)
    hydro = _one_step(cons, b, recon, A.FP32, False)[0]
    mhd = _one_step(cons, b, recon, A.FP32, True)
    # without field there are no Alfven waves: the transverse momentum fluxes of the two
    # solvers are the same upwind values by other sums, up to 16 roundings of fluxes of
    # at most 100 times dt / dx = 7e-3
    np.testing.assert_array_equal(hydro[0], mhd[0][0])
    assert np.abs(hydro[:4] - mhd[0][:4]).max() <= 16 * 2.0 ** -24 * 100 * 7e-3
    assert all(not f.any() for f in mhd[1:])


@pytest.mark.parametrize("recon", ["donor", "plm", "ppm", "ppm5"])
def test_fp32_pairs_against_fp64(recon):
    """Bounds as in test_gpu_pair_solvers.py (momentum fluxes here stay under 200)."""
    cons, b = _state(True)
    got, ref = _one_step(cons, b, recon, A.FP32, True), _one_step(cons, b, recon, A.FP64, True)
    for q, (x, y) in enumerate(zip(got, ref)):
        x, y = (x[:4], y[:4]) if q == 0 else (x, y)
        assert np.abs(x - y).max() < 2e-4
        assert np.abs(x - y).mean() < 1e-5
