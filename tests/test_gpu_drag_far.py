"""Cells that the FP32 pairs of the drag solve leave to FP64: no dearer than the
constant-coefficient law, which solves every cell in FP64, and none for the sake of
a species that is solved in FP32."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _step_us(n, ts, scale=1.0, drag=A.DRAG_FP64, law=0):
    """A step of a dust box in units of `scale` (densities, momenta, energies)."""
    import torch
    nd = len(ts)
    gas, dust, _ = I.dust_box(I.Block(n), 7, nd=nd, t_stop=list(ts))
    cfg = A.make_config(gamma=gas.gamma, recon=A.PLM, integrator=A.IMEX2P, precision=A.FP32, mhd=False,
                        t_stop=[scale] * nd if law else list(ts), drag_precision=drag, drag_law=law,
                        rho_floor=1e-30, p_floor=1e-34)
    sv = A.Solver(cfg, [A.make_block(n)], stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, gas.cons * scale)
        for k in range(nd):
            A.aeth_set_dust(sv.ctx, 0, k, np.ascontiguousarray(dust[k] * scale))
        sv.run(2)
        best = 1e30
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sv.run(4)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / 4)
        return best
    finally:
        sv.close()


# densities of 1e-20 put every cell outside the pairs' range; the other law has
# two divisions a species, the solve here one a cell (nd <= 8) or a species
@pytest.mark.parametrize("n,nd", [((61, 100, 37), 3), ((96, 96, 96), 4), ((64, 64, 64), 8), ((48, 48, 48), 12)])
def test_cells_outside_the_range_cost_no_more_than_an_fp64_solve(n, nd):
    ts = np.logspace(-3, 0, nd)
    far, coeff = _step_us(n, ts, 1e-20), _step_us(n, ts, 1e-20, law=1)
    assert far <= coeff, (far, coeff)


# an uncoupled species (h / t_k about 1e-15) is below SEL64's threshold: FP32
def test_an_fp32_species_keeps_the_pairs():
    n, ts = (64, 64, 64), [1e-4, 1e-3, 1e-2, 1.0]
    base = _step_us(n, ts, drag=A.DRAG_SEL64)
    loose = _step_us(n, ts[:3] + [1e12], drag=A.DRAG_SEL64)
    assert loose <= 1.15 * base, (loose, base)
