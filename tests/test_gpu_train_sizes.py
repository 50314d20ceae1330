"""Training gradient of the learned flux at the edges of its row tiles and
batch chunks, against the FP64 oracle's backpropagation."""
import numpy as np
import pytest

import oracle as O
from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# 1 row; one tile of 16 and its neighbours; one and two chunks of the weight
# gradients (the workspace holds one per 133 rows); the tile heights of
# larger batches, with a remainder.  shift: every array 4 bytes off a
# 16-byte boundary (the call asks for no alignment).
@pytest.mark.parametrize("n,shift", [(1, 0), (15, 1), (16, 0), (17, 0), (132, 0), (267, 1), (2433, 0),
                                     (4871, 0), (8203, 1)])
def test_gradient_at_tile_edges(n, shift):
    import torch
    rng = np.random.default_rng(n)
    p = I.mlp_init_params(11, bias_scale=0.1)
    X = np.full((n, 16), np.nan, np.float32)     # the padding columns are not read
    Y = np.full((n, 8), np.nan, np.float32)
    X[:, :14] = rng.normal(size=(n, 14))
    Y[:, :7] = rng.normal(size=(n, 7))

    def dev(a):
        t = torch.empty(a.size + shift, dtype=torch.float32, device="cuda")[shift:]
        return t.copy_(torch.from_numpy(np.ascontiguousarray(a).ravel()))

    wf = A.aeth_mlp_work_floats(n)
    dp, dX, dY, g, work = dev(p), dev(X), dev(Y), dev(np.full(p.shape, 7, np.float32)), dev(np.zeros(wf, np.float32))
    loss = torch.full((1,), 5.0, device="cuda")
    A.aeth_mlp_grad(dp.data_ptr(), dX.data_ptr(), dY.data_ptr(), n, g.data_ptr(), work.data_ptr(), wf,
                    loss.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    l_ref, g_ref = O.mlp_grad(A.MLP_DIMS, p.astype(np.float64), X[:, :14].astype(np.float64),
                              Y[:, :7].astype(np.float64))
    # eight products (forward and backward of four layers) of 128-term FP32
    # sums, each within sqrt(128) roundings of 6e-8: 6e-6; 1e-5 with SiLU
    assert abs(loss.item() - l_ref) <= 1e-5 * abs(l_ref)
    gg = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(gg - g_ref) <= 1e-5 * np.linalg.norm(g_ref)
