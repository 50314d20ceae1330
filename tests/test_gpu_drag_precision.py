"""The drag solve by itself, cell by cell, against the closed form in FP64: uniform
blocks (no divergence), each with a state of its own, one IMEX2P step.

The dust is heavy and fast and couples weakly, so the heat is a small difference of
large kinetic energies: an FP32 solve loses it (shown below), FP32 pairs must not."""
import numpy as np
import pytest

from paper_2608_14048_gb300 import aether as A

pytestmark = pytest.mark.gpu

GAMMA, DT, NB = 1.4, 1e-3, 24
G = 1.0 + np.sqrt(0.5)
D = 1.0 - 1.0 / (2.0 * G)


def _states(nd, thin):
    """Gas (rho, M, E) and dust (rho, M) of NB blocks, values that FP32 holds exactly.  thin:
    the first species of every other block at 1e-14 of the others (solved in FP64)."""
    r = np.random.default_rng(100 * nd + thin)
    rho = r.uniform(0.5, 2.0, NB)
    v = r.standard_normal((NB, 3))
    gas = np.concatenate([rho[:, None], rho[:, None] * v, (1.0 / 0.4 + 0.5 * rho * (v ** 2).sum(1))[:, None]], 1)
    rk = 10.0 ** r.uniform(-1.0, 2.0, (NB, nd))
    if thin:
        rk[::2, 0] *= 1e-14
    dust = np.concatenate([rk[..., None], rk[..., None] * 10.0 * r.standard_normal((NB, nd, 3))], 2)
    f = lambda a: a.astype(np.float32).astype(np.float64)
    return f(gas), f(dust)


def _drag(gas, dust, a):
    gas, dust = gas.copy(), dust.copy()
    w = a / (1 + a)
    den = gas[:, 0] + dust[:, :, 0] @ w
    vg = (gas[:, 1:4] + np.einsum("bkq,k->bq", dust[:, :, 1:], w)) / den[:, None]
    m0, rk = dust[:, :, 1:].copy(), dust[:, :, :1]
    dust[:, :, 1:] = (m0 + rk * a[:, None] * vg[:, None]) / (1 + a[:, None])
    gas[:, 1:4] = gas[:, :1] * vg
    gas[:, 4] -= 0.5 * ((dust[:, :, 1:] - m0) * (dust[:, :, 1:] + m0) / rk).sum((1, 2))
    return gas, dust


def _step(gas, dust, a):
    """One IMEX2P step without divergence."""
    g2, d2 = _drag(gas, dust, a)
    return _drag(gas + (1 - G) / G * (g2 - gas), dust + (1 - G) / G * (d2 - dust), a)


def _gpu(gas, dust, a, drag):
    import torch
    n, nd = (4, 4, 4), len(a)
    cfg = A.make_config(gamma=GAMMA, recon=A.PLM, integrator=A.IMEX2P, precision=A.FP32, mhd=False,
                        t_stop=[G * DT / x for x in a], drag_precision=drag, drag_ratio=1e-12)
    sv = A.Solver(cfg, [A.make_block(n)] * NB, stream=torch.cuda.current_stream())
    full = lambda s: np.ascontiguousarray(np.broadcast_to(s[:, None, None, None], s.shape + n))
    try:
        for b in range(NB):
            sv.set_state(b, full(gas[b]))
            for k in range(nd):
                A.aeth_set_dust(sv.ctx, b, k, full(dust[b, k]))
        sv.step(DT)
        og, od = np.empty_like(gas), np.empty_like(dust)
        for b in range(NB):
            cons = sv.get_state(b)[0]
            assert np.all(cons == cons[:, :1, :1, :1])    # still uniform: no divergence entered
            og[b] = cons[:, 0, 0, 0]
            for k in range(nd):
                d = np.empty((4,) + n)
                A.aeth_get_dust(sv.ctx, b, k, d)
                assert np.all(d == d[:, :1, :1, :1])
                od[b, k] = d[:, 0, 0, 0]
        return og, od
    finally:
        sv.close()


def _errors(nd, thin, drag):
    """Errors of the gas momentum, gas energy and dust momenta in units of FP32's half ulp of
    what enters them: the momenta that couple, the energy and the heat, the species' own
    momentum (a thin species by its own scale)."""
    gas, dust = _states(nd, thin)
    a = np.logspace(-5.0, -3.0, nd) if nd > 1 else np.array([1e-4])
    rg, rd = _step(gas, dust, a)
    og, od = _gpu(gas, dust, a, drag)
    u = 2.0 ** -24
    w = a / (1 + a)
    mom = np.abs(gas[:, 1:4]).max(1) + np.einsum("bkq,k->bq", np.abs(dust[:, :, 1:]), w).max(1)
    np.testing.assert_array_equal(og[:, 0], gas[:, 0])
    np.testing.assert_array_equal(od[:, :, 0], dust[:, :, 0])
    return (np.abs(og[:, 1:4] - rg[:, 1:4]).max(1) / mom / u,
            np.abs(og[:, 4] - rg[:, 4]) / (gas[:, 4] + np.abs(rg[:, 4] - gas[:, 4])) / u,
            np.abs(od[:, :, 1:] - rd[:, :, 1:]).max(2) / np.abs(dust[:, :, 1:]).max(2) / u)


# Bound: each of the two solves rounds its results once (1), the combination between
# them takes three products and sums of terms up to 1.4 times the values (5), and what
# that leaves in the second solve's inputs comes out once: 8 half ulps.
BOUND = 8.0


@pytest.mark.parametrize("drag", [A.DRAG_FP64, A.DRAG_SEL64])
@pytest.mark.parametrize("nd,thin", [(1, False), (3, True), (4, False), (5, True), (8, False), (9, True)])
def test_drag_to_the_last_bits(nd, thin, drag):
    for e in _errors(nd, thin, drag):
        assert e.max() <= BOUND, e.max()


def test_fp32_drag_is_told_apart():
    assert _errors(4, False, A.DRAG_FP32)[1].max() > 20 * BOUND
