"""A box of one block linked to itself on all sides: the state of the periodic box, at
about its speed."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _run(n, linked):
    """The state after the warm-up steps and us a step."""
    import torch
    st = I.smooth_random_mhd(I.Block(n), 8, v_rms=0.5, b_rms=0.5)
    blocks, links, _ = A.decompose(n, [[m] for m in n])
    assert len(blocks) == 1 and len(links) == 3
    sv = A.Solver(A.make_config(gamma=st.gamma, precision=A.FP32), blocks,
                  stream=torch.cuda.current_stream(), links=links if linked else ())
    try:
        sv.set_state(0, st.cons, st.b1, st.b2, st.b3)
        sv.run(4)
        state = sv.get_state(0)
        best = 1e30
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            sv.run(8)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3 / 8)
        return state, best
    finally:
        sv.close()


# the fill of a linked block looks its neighbours up in the block table, a few us a
# step; 1.2 leaves room for that (with the parameters on the stack: 1.45)
def test_linked_box_is_the_periodic_box():
    periodic, tp = _run((64, 64, 64), False)
    linked, tl = _run((64, 64, 64), True)
    for x, y in zip(periodic, linked):
        np.testing.assert_array_equal(x, y)
    assert tl <= 1.2 * tp, (tl, tp)
