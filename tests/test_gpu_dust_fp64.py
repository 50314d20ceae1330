"""FP64 dust transport: a flux pass per direction, each face once."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _step_us(n, nd, recon):
    import torch
    gas, dust, ts = I.dust_box(I.Block(n), 7, nd=nd, t_stop=list(np.logspace(-3, 0, nd)))
    cfg = A.make_config(gamma=gas.gamma, recon=recon, integrator=A.IMEX2P, precision=A.FP64, mhd=False, t_stop=ts)
    sv = A.Solver(cfg, [A.make_block(n)], stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, gas.cons)
        for k in range(nd):
            A.aeth_set_dust(sv.ctx, 0, k, np.ascontiguousarray(dust[k]))
        sv.run(2)
        best = 1e30
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sv.run(3)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / 3)
        return best
    finally:
        sv.close()


# The FP64 pipe bounds a dust step, and the species' fluxes are most of it: PLM
# forms 32 slopes a cell and species more than donor cells when every face is
# computed once, 20 more again when both cells of an x or y face compute it (a
# step of this box then took 2.83 times the donor step, against 2.44).
def test_plm_faces_are_computed_once():
    n = (61, 100, 37)
    donor, plm = _step_us(n, 12, A.DONOR), _step_us(n, 12, A.PLM)
    assert plm <= 2.6 * donor, (plm, donor)
