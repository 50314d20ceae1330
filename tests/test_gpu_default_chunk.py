"""The default z-chunk of the flux pass where the FP64 pipe bounds it (FP64 contexts
and the FP64 pressure recovery of FP32_P64): no slower than plain chunks of 4, 8,
16 and 32 planes."""
import pytest

from paper_2608_14048_gb300 import aether as A
from paper_2608_14048_gb300 import inputs as I
from tests.gpu_helpers import RECON

pytestmark = pytest.mark.gpu


def _step_us(sv):
    import torch
    sv.run(4)
    best = 1e30
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        sv.run(8)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / 8)
    return best


# boxes whose tiles make parts of waves of the chip (a chunk too short spends
# itself on the planes below it, a long one leaves SMs idle); the bound is 10%
# over the best plain chunk, ten times what repeated runs differ by
@pytest.mark.parametrize("prec,n,recon,mhd", [
    (A.FP32_P64, (64, 64, 64), "plm", True), (A.FP32_P64, (150, 20, 60), "plm", True),
    (A.FP32_P64, (34, 124, 42), "plm", False), (A.FP32_P64, (80, 80, 80), "ppm", True),
    (A.FP32_P64, (20, 20, 20), "donor", True), (A.FP64, (17, 160, 24), "plm", False),
    (A.FP64, (30, 50, 90), "donor", True), (A.FP64, (40, 40, 40), "ppm", True)])
def test_default_chunk_is_no_slower_than_plain_chunks(prec, n, recon, mhd):
    import torch
    st = I.smooth_random_mhd(I.Block(n), 5, v_rms=0.5, b_rms=0.5)
    cfg = A.make_config(gamma=st.gamma, precision=prec, recon=RECON[recon][1], mhd=mhd)
    sv = A.Solver(cfg, [A.make_block(n)], stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, st.cons, st.b1, st.b2, st.b3) if mhd else sv.set_state(0, st.cons)
        kc = A.aeth_get_flux_tile(sv.ctx)[1]
        own = _step_us(sv)
        plain = {}
        for k in (4, 8, 16, 32):
            A.aeth_set_flux_tile(sv.ctx, 32, k)
            plain[k] = _step_us(sv)
    finally:
        sv.close()
    assert own <= 1.10 * min(plain.values()), (kc, own, plain)
