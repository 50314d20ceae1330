"""States at the floors: the count of floored cells, and what counting them costs."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _solver(st, rho_floor, path=A.FUSED):
    import torch
    cfg = A.make_config(gamma=st.gamma, precision=A.FP32, rho_floor=rho_floor, path=path)
    sv = A.Solver(cfg, [A.make_block(st.block.n)], stream=torch.cuda.current_stream())
    sv.set_state(0, st.cons, st.b1, st.b2, st.b3)
    return sv


def _state(n):
    return I.smooth_random_mhd(I.Block(n), 5, v_rms=0.2, b_rms=0.2)


# an uneven box, the floor at the median density: warps with idle lanes and with
# lanes that have no hit.  The unfused conversion takes every cell of the padded
# range once a stage, and a step of 1e-12 moves no density across the floor.
def test_floored_cells_are_counted():
    st = _state((35, 9, 6))
    rho = st.cons[0].astype(np.float32)
    floor = float(np.median(rho)) * (1 + 1e-4)
    sv = _solver(st, floor, A.UNFUSED)
    try:
        sv.step(1e-12)
        hits = sv.diagnostics()["floor_hits"]
    finally:
        sv.close()
    low = (rho < np.float32(floor)).astype(int)
    want = {g: 2 * int(np.pad(low, g, mode="wrap").sum()) for g in (2, 3, 4)}   # g ghost layers
    assert hits in want.values(), (hits, want)


# every cell below the density floor: a step may take half as long again as without
# hits (one atomic a warp and tile, against one a thread: 2.2 times as long)
def test_counting_floors_is_cheap():
    import torch
    t = []
    for floor in (1e-12, 5.0):
        sv = _solver(_state((64, 64, 64)), floor)
        try:
            sv.run(4)
            best = 1e30
            for _ in range(7):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                sv.run(8)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) * 1e3 / 8)
            t.append(best)
        finally:
            sv.close()
    assert t[1] <= 1.5 * t[0], t
