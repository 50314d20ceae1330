"""Weight gradients of the learned flux where the workspace first holds partial sums
(35,847 floats a chunk out of 264 a row: two chunks from 272 rows, three from 408), and
nothing written past the workspace."""
import numpy as np
import pytest

import oracle as O
from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [135, 271, 272, 407, 408])
def test_gradient_at_the_first_chunks(n, shift):
    import torch
    rng = np.random.default_rng(n)
    p = I.mlp_init_params(11, bias_scale=0.1)
    X, Y = np.zeros((n, 16), np.float32), np.zeros((n, 8), np.float32)
    X[:, :14] = rng.normal(size=(n, 14))
    Y[:, :7] = rng.normal(size=(n, 7))
    wf, guard = A.aeth_mlp_work_floats(n), 4096
    assert wf == 1040 * n and (1040 - 776) * 272 >= 2 * A.MLP_NPARAM > 264 * 271

    def dev(a):
        t = torch.empty(a.size + shift, dtype=torch.float32, device="cuda")[shift:]
        return t.copy_(torch.from_numpy(np.ascontiguousarray(a).ravel()))

    dp, dX, dY, g = dev(p), dev(X), dev(Y), dev(np.full(p.shape, 7, np.float32))
    work = dev(np.full(wf + guard, 123.0, np.float32))
    loss = torch.full((1,), 5.0, device="cuda")
    A.aeth_mlp_grad(dp.data_ptr(), dX.data_ptr(), dY.data_ptr(), n, g.data_ptr(), work.data_ptr(), wf,
                    loss.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert bool((work[wf:] == 123.0).all())
    l_ref, g_ref = O.mlp_grad(A.MLP_DIMS, p.astype(np.float64), X[:, :14].astype(np.float64),
                              Y[:, :7].astype(np.float64))
    # as in test_gpu_train_sizes.py: eight products of 128-term FP32 sums, 6e-6; 1e-5 with SiLU
    assert abs(loss.item() - l_ref) <= 1e-5 * abs(l_ref)
    gg = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(gg - g_ref) <= 1e-5 * np.linalg.norm(g_ref)
