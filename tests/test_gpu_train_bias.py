"""Bias gradients of the learned flux: sums over the batch that keep their digits."""
import numpy as np
import pytest

import oracle as O
from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# The output bias sums (yhat - y) / n over the rows: each term is rounded to half an ulp
# at random, and a sum that loses nothing rounds once, 2^-24 of the result each; 2^-23 in
# the mean of eight batches.  (One running sum of 256 rows: 2.5e-7.)
@pytest.mark.parametrize("n", [256, 271, 1000])
def test_output_bias_gradient(n):
    import torch
    err = []
    for seed in range(8):
        rng = np.random.default_rng(1000 * n + seed)
        p = I.mlp_init_params(11, bias_scale=0.1)
        X, Y = np.zeros((n, 16), np.float32), np.zeros((n, 8), np.float32)
        X[:, :14] = rng.normal(size=(n, 14))
        Y[:, :7] = 0.1 * rng.normal(size=(n, 7))
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()
        wf = A.aeth_mlp_work_floats(n)
        dp, dX, dY = dev(p), dev(X), dev(Y)
        g, work, loss = torch.zeros_like(dp), torch.zeros(wf, device="cuda"), torch.zeros(1, device="cuda")
        A.aeth_mlp_grad(dp.data_ptr(), dX.data_ptr(), dY.data_ptr(), n, g.data_ptr(), work.data_ptr(), wf,
                        loss.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        _, ref = O.mlp_grad(A.MLP_DIMS, p.astype(np.float64), X[:, :14].astype(np.float64),
                            Y[:, :7].astype(np.float64))
        e = g.cpu().numpy().astype(np.float64)[-7:] - ref[-7:]
        err.append(np.linalg.norm(e) / np.linalg.norm(ref[-7:]))
    assert np.mean(err) <= 2.0 ** -23, err
