"""The flux of a dust face is one value, whichever of its two cells computes it (FP32
dust passes compute x and y faces in both, z faces at the ends of a march too): a
profile along x or y, where each cell evaluates its own pair of faces, moves bit
for bit like the same profile along z, where a march hands each face on."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A
from tests.gpu_helpers import RECON

pytestmark = pytest.mark.gpu

N = 75   # marches of 4 to 16 cells along z: several seams and a remainder


def _profile():
    """rho, the normal and two transverse velocities: smooth waves, a density jump and a
    strong shear, all signs of the normal velocity."""
    r = np.random.default_rng(3)
    x = (np.arange(N) + 0.5) / N
    rho = 0.3 + 0.2 * np.sin(2 * np.pi * x) + 0.6 * (x > 0.4) * (x < 0.6) + 0.01 * r.random(N)
    v = [np.sin(4 * np.pi * x + 0.3), 0.7 * np.cos(2 * np.pi * x) + 0.2 * r.random(N), np.where(x < 0.5, 0.9, -0.4)]
    return rho, v


def _run(axis, recon, nd):
    """(density, normal, first and second transverse momentum) of each species after six
    steps, along `axis`; no species feels the gas."""
    import torch
    n = [5, 5, 5]
    n[axis] = N
    hi = [1.0 if d == axis else 5.0 / N for d in range(3)]
    shape = (n[2], n[1], n[0])
    rho, v = _profile()
    line = lambda f: np.broadcast_to(f.reshape([-1 if 2 - q == axis else 1 for q in range(3)]), shape)
    gas = np.zeros((5,) + shape)
    gas[0], gas[4] = 1.0, 1.0
    cfg = A.make_config(gamma=1.4, recon=RECON[recon][1], integrator=A.IMEX2P, precision=A.FP32, mhd=False,
                        t_stop=[1e25] * nd)
    sv = A.Solver(cfg, [A.make_block(tuple(n), (0.0,) * 3, tuple(hi))], stream=torch.cuda.current_stream())
    try:
        sv.set_state(0, gas)
        for s in range(nd):
            d = np.zeros((4,) + shape)
            d[0] = line(rho) * (1 + s)
            for t in range(3):
                d[1 + (axis + t) % 3] = d[0] * line(v[t])
            A.aeth_set_dust(sv.ctx, 0, s, np.ascontiguousarray(d))
        for _ in range(6):
            sv.step(1e-3)
        out = []
        for s in range(nd):
            d = np.empty((4,) + shape)
            A.aeth_get_dust(sv.ctx, 0, s, d)
            d = d[[0] + [1 + (axis + t) % 3 for t in range(3)]]
            out.append(np.moveaxis(d, 3 - axis, 1).reshape(4, N, -1))
        return np.stack(out)
    finally:
        sv.close()


@pytest.mark.parametrize("nd", [1, 2])
@pytest.mark.parametrize("recon", ["donor", "plm", "ppm", "ppm5"])
def test_a_face_has_one_flux(recon, nd):
    z = _run(2, recon, nd)
    assert np.all(np.isfinite(z)) and np.ptp(z[0, 0, :, 0]) > 0.1
    np.testing.assert_array_equal(z, np.broadcast_to(z[..., :1], z.shape))   # still one profile
    for axis in (0, 1):
        np.testing.assert_array_equal(_run(axis, recon, nd), z)
