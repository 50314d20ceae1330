"""The one-launch ghost fill and the packed dust divergence at their edge
sizes.  Every cell of a replicated or split domain goes through the same
arithmetic, so the states must agree: extents below the ghost
width, linked blocks of the smallest allowed size (their ghosts reach through
two neighbours), outflow edges, and z marches with a remainder."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I
from tests.test_gpu_blocks import _run_blocks

pytestmark = pytest.mark.gpu


# two steps of states of order one: a few dozen roundings; a wrong ghost is off
# by the differences between cells, 1e-2 and more
EPS = {"fp32": 64 * 2.0 ** -24, "fp64": 64 * 2.0 ** -53}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("splits", [((2, 3, 2), (2, 4), (3, 2, 2)), ((7,), (2, 2, 2), (7,))])
@pytest.mark.parametrize("bc", [(0, 0, 0), (1, 0, 1), (1, 1, 1)])
def test_smallest_linked_blocks_match_one_block(prec, splits, bc):
    n = tuple(sum(s) for s in splits)
    st = I.smooth_random_mhd(I.Block(n, (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), bc=bc), 5)
    dts = [1e-3, 2e-3]
    got, _, dt = _run_blocks(st, splits, dts, prec=prec)
    ref, _, dt_ref = _run_blocks(st, tuple((m,) for m in n), dts, prec=prec)
    for a, b in zip(got, ref):
        np.testing.assert_allclose(a, b, rtol=EPS[prec], atol=EPS[prec])
    assert dt == pytest.approx(dt_ref, rel=EPS[prec])


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("recon,drag", [(A.PLM, A.DRAG_FP32), (A.PLM, A.DRAG_FP64), (A.DONOR, A.DRAG_FP64),
                                        (A.PPM, A.DRAG_FP64), (A.PPM5, A.DRAG_SEL64)])
def test_thin_dusty_blocks_match_replicated_ones(bc, recon, drag):
    """A state that varies along x only: blocks of 1 x 1 and of 5 x 19 (z march
    16 + 3) cells across evolve alike."""
    import torch
    nx, nd, rng = 33, 3, np.random.default_rng(3)
    line = np.empty((5 + 4 * nd, nx))
    line[0], line[1:4], line[4] = 1 + rng.random(nx), rng.standard_normal((3, nx)), 8.0
    for k in range(nd):
        line[5 + 4 * k] = 0.1 + rng.random(nx)
        line[6 + 4 * k:9 + 4 * k] = rng.standard_normal((3, nx)) * 0.2
    out = []
    for ny, nz in ((1, 1), (5, 19)):
        full = np.ascontiguousarray(np.broadcast_to(line[:, None, None, :], (len(line), nz, ny, nx)))
        cfg = A.make_config(gamma=1.4, recon=recon, integrator=A.IMEX2P, precision=A.FP32,
                            mhd=False, t_stop=[0.1, 0.01, 1.0], drag_precision=drag)
        sv = A.Solver(cfg, [A.make_block((nx, ny, nz), (0.0, 0.0, 0.0), (1.0, ny / nx, nz / nx),
                                         A.CART, (bc, bc, bc))], stream=torch.cuda.current_stream())
        try:
            sv.set_state(0, full[:5])
            for k in range(nd):
                A.aeth_set_dust(sv.ctx, 0, k, np.ascontiguousarray(full[5 + 4 * k:9 + 4 * k]))
            for _ in range(3):
                sv.step(1e-3)
            r = [sv.get_state(0)[0]]
            for k in range(nd):
                buf = np.empty((4, nz, ny, nx))
                A.aeth_get_dust(sv.ctx, 0, k, buf)
                r.append(buf)
        finally:
            sv.close()
        out.append(np.concatenate(r))
    np.testing.assert_array_equal(out[1], np.broadcast_to(out[0], out[1].shape))
    assert np.abs(out[0] - line[:, None, None, :]).max() > 1e-3
