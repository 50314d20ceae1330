"""The flux-tile tuner against the untuned context, and the cache key's kernels."""
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I
from tests.gpu_helpers import RECON


def test_cache_key_follows_the_kernels(monkeypatch):
    cfg, b = A.make_config(precision=A.FP32), [A.make_block((64, 64, 64))]
    k = A.tile_cache_key(cfg, b, "GB300")[0]
    assert A.tile_cache_key(cfg, b, "GB300")[0] == k
    monkeypatch.setattr(A, "tile_kernels", lambda: "other")
    assert A.tile_cache_key(cfg, b, "GB300")[0] != k


def _step_us(sv):
    import torch
    sv.run(4)
    best = 1e30
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        sv.run(4)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / 4)
    return best


# contexts whose default chunk is short (FP64: 2 planes) and long; tuning may not
# cost more than the 5% that single timings of three steps differ by
@pytest.mark.gpu
@pytest.mark.parametrize("prec,n,recon", [(A.FP64, (64, 64, 64), "ppm"), (A.FP64, (64, 64, 64), "plm"),
                                          (A.FP32, (96, 96, 96), "plm"), (A.FP32, (190, 131, 77), "ppm")])
def test_a_tuned_context_is_no_slower(prec, n, recon):
    import torch
    st = I.smooth_random_mhd(I.Block(n), 8, v_rms=0.5, b_rms=0.5)
    cfg = A.make_config(gamma=st.gamma, precision=prec, recon=RECON[recon][1])
    sv = A.Solver(cfg, [A.make_block(n)], stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, st.cons, st.b1, st.b2, st.b3)
        shape, untuned = A.aeth_get_flux_tile(sv.ctx), _step_us(sv)
        tuned_shape = A.aeth_autotune(sv.ctx)
        sv.set_state(0, st.cons, st.b1, st.b2, st.b3)
        tuned = _step_us(sv)
    finally:
        sv.close()
    assert tuned <= 1.05 * untuned, (shape, untuned, tuned_shape, tuned)
