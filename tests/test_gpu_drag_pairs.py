"""The FP64 drag of FP32 transport in FP32 pairs, and the cells and constants
that it leaves to FP64, against the FP64 oracle."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I
from tests.gpu_helpers import rel_l1
from tests.test_gpu_dust import _oracle

pytestmark = pytest.mark.gpu


# one species; the 4- and 8-species kernels and their neighbours; implicit
# weights beyond the pairs' range (t = 1e-14); thin: one species at 1e-14 of the
# gas in half of the box, where its cells are solved in FP64
@pytest.mark.parametrize("drag", [A.DRAG_FP64, A.DRAG_SEL64])
@pytest.mark.parametrize("ts,thin", [([1e-2], False), ([1e-5, 1e-2, 1.0], True),
                                     ([1e-4, 1e-3, 1e-2, 1.0], False),
                                     ([1e-14, 1e-4, 1e-3, 1e-2, 1.0], False),
                                     (list(np.logspace(-6, 0, 8)), True),
                                     (list(np.logspace(-4, 0, 9)), False)])
def test_drag_pairs_match_oracle(ts, thin, drag):
    import torch
    b = I.Block((33, 6, 5))
    gas, dust, ts = I.dust_box(b, 7, nd=len(ts), t_stop=ts)
    if thin:
        dust[0][:, :, :, : b.n[0] // 2] *= 1e-14
    rc, rd, dts = _oracle(gas, dust, ts, 3)
    cfg = A.make_config(gamma=gas.gamma, recon=A.PLM, integrator=A.IMEX2P, precision=A.FP32, mhd=False,
                        t_stop=ts, drag_precision=drag)
    sv = A.Solver(cfg, [A.make_block(b.n)], stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, gas.cons)
        for k in range(len(ts)):
            A.aeth_set_dust(sv.ctx, 0, k, np.ascontiguousarray(dust[k]))
        for dt in dts:
            sv.step(dt)
        cons = sv.get_state(0)[0]
        d = np.empty_like(dust)
        for k in range(len(ts)):
            A.aeth_get_dust(sv.ctx, 0, k, d[k])
    finally:
        sv.close()
    # the bound of FP32 transport: 1e-5 relative L1 per variable, momenta
    # against their vector
    for v in (0, 4):
        assert rel_l1(cons[v], rc[v]) < 1e-5
    assert rel_l1(cons[1:4], rc[1:4]) < 1e-5
    for k in range(len(ts)):
        assert rel_l1(d[k, 0], rd[k, 0]) < 1e-5
        assert rel_l1(d[k, 1:], rd[k, 1:]) < 1e-5
