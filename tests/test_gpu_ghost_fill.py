"""The one-launch ghost fill at its edge sizes: linked blocks of the smallest
allowed size (their ghosts reach through two neighbours) between outflow and
periodic edges, against one block."""
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
