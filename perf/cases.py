"""Performance cases of the MHD library: what is timed, on which inputs, and what
the results are in 64 bits.

Two kinds of work make up the library's use.  A simulation advances a state
held on the GPU by some steps, with the CFL time step on the device
(`Solver.run`) or a given one (`Solver.step`), and takes a snapshot into the
program's own tensors in its working precision ("gas", "boxes" and "dust"
cases).  The learned Riemann flux is evaluated on a set of faces ("faces")
and trained on a batch ("train").

  listed()        the cases by name
  draw(rng)       another case of the same ranges
  prepare(c, s)   inputs from the seed s alone, on the GPU, and the handle a
                  program keeps (solver, snapshot buffers, network)
  run(state)      one pass
  work(c)         bytes and operations of one pass that cannot be avoided
  exact(c, s)     the pass in plain torch FP64
"""
import math

import numpy as np
import torch

from paper_2608_14048_gb300 import aether as A

RECON = {"donor": A.DONOR, "plm": A.PLM, "ppm": A.PPM, "ppm5": A.PPM5}
RIEMANN = {"hlld": A.HLLD, "hlle": A.HLLE, "lhlld": A.LHLLD}
INTEGRATOR = {"vl2": A.VL2, "rk2": A.RK2, "rk3": A.RK3}
PRECISION = {"fp64": A.FP64, "fp32": A.FP32, "fp32_p64": A.FP32_P64, "fp32_sel64": A.FP32_SEL64}
DRAG = {"fp64": A.DRAG_FP64, "fp32": A.DRAG_FP32, "sel64": A.DRAG_SEL64}
CFL = 0.3
BOX_DT = 5e-4     # common step of the uneven boxes, below every box's limit
DIMS = A.MLP_DIMS


def _gas(name, n, steps, *, flow="smooth", recon="plm", riemann="hlld", integrator="vl2", eos="mhd",
         precision="fp32", gamma=5.0 / 3.0, split=1, outflow="", dual=False):
    """A box of n cells as split^3 linked blocks, advanced by `steps`.  flow: "turbulence" (shell
    spectrum, rms Mach 2), "smooth" (low-k random fields) or "vortex" (Taylor-Green, Mach 0.1)."""
    return {"name": name, "kind": "gas", "nx": n[0], "ny": n[1], "nz": n[2], "steps": steps, "flow": flow,
            "recon": recon, "riemann": riemann, "integrator": integrator, "eos": eos, "precision": precision,
            "gamma": gamma, "split": split, "outflow": outflow, "dual": dual}


def _dust(name, n, steps, species, drag, recon="plm", precision="fp32"):
    return {"name": name, "kind": "dust", "nx": n[0], "ny": n[1], "nz": n[2], "steps": steps, "species": species,
            "drag": drag, "recon": recon, "precision": precision, "gamma": 5.0 / 3.0}


def listed():
    return [
        # the 32^3 wave-sized box of a convergence study: tiny kernels, launches and their gaps count
        _gas("box32_fp32", (32, 32, 32), 20),
        # the default workload: decaying Mach-2 turbulence on one 256^3 box
        _gas("turb256_fp32", (256, 256, 256), 20, flow="turbulence", gamma=1.0001),
        # the paper's throughput set-up: PLM + HLLE + RK2 on a mesh of linked 128^3 blocks
        _gas("blocks256_hlle_rk2", (256, 256, 256), 50, riemann="hlle", integrator="rk2", split=2),
        # a production box whose sizes divide nothing, third-order reconstruction and time steps
        _gas("ragged_ppm_rk3", (190, 131, 77), 20, recon="ppm", integrator="rk3"),
        # the FP64 path that results are validated with
        _gas("turb96_fp64", (96, 96, 96), 4, flow="turbulence", gamma=1.0001, precision="fp64"),
        # isothermal turbulence, the paper's weak-scaling problem at one device's share of a small run
        _gas("iso128_fp32", (128, 128, 128), 40, flow="turbulence", eos="iso"),
        # low-Mach hydro (Taylor-Green) with the low-dissipation solver
        _gas("vortex128_hydro", (128, 128, 128), 40, flow="vortex", eos="hydro", riemann="lhlld", integrator="rk2"),
        # many independent uneven boxes (16 to 64 cells a side, every third spherical) in one context, with
        # one time step that the program gives
        {"name": "boxes512_uneven", "kind": "boxes", "blocks": 512, "steps": 20, "gamma": 5.0 / 3.0},
        # gas and eight dust species, the drag solved in FP64
        _dust("dust128_fp64drag", (128, 128, 128), 10, 8, "fp64"),
        # a small ragged dust box, the drag in FP64 only for the stiff species
        _dust("dust_ragged_sel64", (61, 100, 37), 20, 3, "sel64", recon="ppm"),
        # the learned flux on the faces of a subdomain
        {"name": "faces_2m", "kind": "faces", "faces": 1 << 21, "gamma": 1.0001},
        # one training step of the learned flux (gradient and Adam) at the training batch
        {"name": "train_8192", "kind": "train", "batch": 8192},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gas"] * 6 + ["boxes", "dust", "dust", "faces", "train"])
    if kind == "faces":
        return {"kind": kind, "faces": _log_int(rng, 1 << 10, 1 << 21), "gamma": rng.choice([1.0001, 5.0 / 3.0])}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 256, 32768)}
    if kind == "boxes":
        return {"kind": kind, "blocks": _log_int(rng, 8, 384), "steps": rng.randint(4, 10), "gamma": 5.0 / 3.0}
    if kind == "dust":
        n = [_log_int(rng, 12, 112) for _ in range(3)]
        c = _dust(None, n, rng.randint(4, 12), rng.randint(1, 8), rng.choice(["fp64", "fp64", "sel64", "fp32"]),
                  recon=rng.choice(["plm", "ppm"]))
    else:
        eos = rng.choice(["mhd", "mhd", "mhd", "iso", "hydro"])
        precision = rng.choice(["fp32"] * 5 + ["fp64", "fp32_p64", "fp32_sel64"])
        split = rng.choice([1, 1, 1, 2])
        hi = 64 if precision == "fp64" else 192
        n = [split * _log_int(rng, 12, hi // split) for _ in range(3)]
        c = _gas(None, n, rng.randint(10, 30), flow=rng.choice(["smooth", "turbulence"]),
                 recon=rng.choice(["plm", "plm", "plm", "ppm", "ppm5", "donor"]),
                 riemann=rng.choice(["hlld", "hlld", "hlle"] + (["lhlld"] if eos != "iso" else [])),
                 integrator=rng.choice(["vl2", "vl2", "rk2", "rk3"]), eos=eos, precision=precision, split=split,
                 outflow=rng.choice(["", "", "", "x", "xz"]), dual=eos != "iso" and precision == "fp32" and rng.random() < 0.1)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs, in FP64 on the GPU; arrays are [z][y][x]
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _random_field(n, g, kmin, kmax, slope, count=1):
    """`count` Gaussian random periodic fields of unit variance, shell spectrum k^slope on kmin <= k <= kmax."""
    k = [torch.fft.fftfreq(m, d=1.0 / m, device="cuda", dtype=torch.float64) for m in (n[2], n[1])]
    k.append(torch.fft.rfftfreq(n[0], d=1.0 / n[0], device="cuda", dtype=torch.float64))
    kk = torch.sqrt(k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2)
    amp = torch.where((kk >= kmin) & (kk <= kmax), kk.clamp(min=1.0) ** ((slope - 2.0) / 2.0), torch.zeros_like(kk))
    out = []
    for _ in range(count):
        f = torch.complex(torch.randn(kk.shape, generator=g, device="cuda", dtype=torch.float64),
                          torch.randn(kk.shape, generator=g, device="cuda", dtype=torch.float64))
        f = torch.fft.irfftn(f * amp, s=(n[2], n[1], n[0]))
        out.append(f / f.std().clamp(min=1e-300))
    return out


def _wrap(f):
    """The periodic field with its first layer repeated after the last along each axis."""
    for d in range(3):
        f = torch.cat([f, f.narrow(d, 0, 1)], dim=d)
    return f


def _curl_faces(pot, length, area):
    """Face fields [z][y][x] with one more face along their own axis: the circulation of the vector
    potential (edge values times edge lengths) over the face area, so that div B = 0 to round-off."""
    I = [_wrap(p) * length[d] for d, p in enumerate(pot)]
    b1 = I[2][:-1, 1:, :] - I[2][:-1, :-1, :] - (I[1][1:, :-1, :] - I[1][:-1, :-1, :])
    b2 = I[0][1:, :, :-1] - I[0][:-1, :, :-1] - (I[2][:-1, :, 1:] - I[2][:-1, :, :-1])
    b3 = I[1][:, :-1, 1:] - I[1][:, :-1, :-1] - (I[0][:, 1:, :-1] - I[0][:, :-1, :-1])
    return [b1 / area[0], b2 / area[1], b3 / area[2]]


def _mean_faces(b):
    return [0.5 * (b[0][:, :, 1:] + b[0][:, :, :-1]), 0.5 * (b[1][:, 1:, :] + b[1][:, :-1, :]),
            0.5 * (b[2][1:, :, :] + b[2][:-1, :, :])]


def _conserved(gamma, rho, v, p, bc):
    e = p / (gamma - 1.0) + 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
    if bc is not None:
        e = e + 0.5 * (bc[0] ** 2 + bc[1] ** 2 + bc[2] ** 2)
    return torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], e])


def _unit(f):
    return (f - f.min()) / (f.max() - f.min()).clamp(min=1e-300)


def _smooth_fields(n, g):
    """rho in [0.5, 2], p in [0.1, 1] and a velocity of rms 0.5 from low-k random fields."""
    f = _random_field(n, g, 1.0, 3.0, -2.0, 5)
    return 2.0 ** (2.0 * _unit(f[0]) - 1.0), 0.1 * 10.0 ** _unit(f[1]), [0.5 / math.sqrt(3.0) * q for q in f[2:]]


def _random_faces(n, g, length, area, rms):
    b = _curl_faces(_random_field(n, g, 1.0, 3.0, -2.0, 3), length, area)
    r = torch.sqrt(sum((q ** 2).mean() for q in _mean_faces(b))).clamp(min=1e-300)
    return [q * (rms / r) for q in b]


def _gas_state(c, seed):
    """(cons [5][nz][ny][nx], [b1, b2, b3] or None) of a box on the unit cube."""
    n, g = (c["nx"], c["ny"], c["nz"]), _generator(seed)
    h = [1.0 / m for m in n]
    gamma, mhd = c["gamma"], c["eos"] != "hydro"
    one = torch.ones((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    cell = [(torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m for m in n]
    area = [h[1] * h[2], h[0] * h[2], h[0] * h[1]]
    if c["flow"] == "vortex":
        # Taylor-Green vortex at Mach 0.1 with a phase from the seed
        ph = 2 * math.pi * torch.rand(3, generator=g, device="cuda", dtype=torch.float64)
        x, y, z = (2 * math.pi * cell[d].reshape([-1 if q == 2 - d else 1 for q in range(3)]) + ph[d] for d in range(3))
        v = [torch.sin(x) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(y) * torch.cos(z), 0.0 * one]
        p = 100.0 / gamma + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
        rho, b = one, None
    elif c["flow"] == "turbulence":
        # decaying turbulence: uniform gas with c_s = 1, rms Mach 2, beta = 1 along x
        v = [2.0 / math.sqrt(3.0) * q for q in _random_field(n, g, 2.0, 8.0, -2.0, 3)]
        rho, p = one, one / gamma
        b = [torch.zeros((n[2] + (d == 2), n[1] + (d == 1), n[0] + (d == 0)), dtype=torch.float64, device="cuda")
             for d in range(3)]
        b[0] += math.sqrt(2.0 / gamma)
    else:
        rho, p, v = _smooth_fields(n, g)
        b = _random_faces(n, g, h, area, 0.5)
    b = b if mhd else None
    return _conserved(gamma, rho, v, p, _mean_faces(b) if mhd else None), b


def _box_state(seed, spherical, n, gamma):
    """One of the uneven boxes: a periodic unit box or a spherical wedge."""
    g = _generator(seed)
    if not spherical:
        length, area = [1.0 / m for m in n], [1.0 / (n[1] * n[2]), 1.0 / (n[0] * n[2]), 1.0 / (n[0] * n[1])]
    else:
        f = [torch.linspace(lo, hi, n[d] + 1, dtype=torch.float64, device="cuda")
             for d, (lo, hi) in enumerate(zip(WEDGE["lo"], WEDGE["hi"]))]
        r, th = f[0][None, None, :], f[1][None, :, None]
        dr, dth, dph = (f[d][1] - f[d][0] for d in range(3))
        length = [dr, r * dth, r * torch.sin(th) * dph]
        half = 0.5 * (r[:, :, 1:] ** 2 - r[:, :, :-1] ** 2)
        area = [r ** 2 * (torch.cos(th[:, :-1]) - torch.cos(th[:, 1:])) * dph, half * torch.sin(th) * dph, half * dth]
    rho, p, v = _smooth_fields(n, g)
    b = _random_faces(n, g, length, area, 0.5)
    return _conserved(gamma, rho, v, p, _mean_faces(b)), b


WEDGE = {"lo": (1.0, math.pi / 4, 0.0), "hi": (2.0, 3 * math.pi / 4, math.pi / 2)}


def _box_sizes(c):
    """(spherical, (nx, ny, nz)) of each box, the Cartesian ones first."""
    r = np.random.default_rng(20260818)
    sizes = [tuple(int(x) for x in r.choice((16, 24, 32, 48, 64), size=3)) for _ in range(c["blocks"])]
    return [(False, n) for i, n in enumerate(sizes) if i % 3 != 2] + [(True, n) for i, n in enumerate(sizes) if i % 3 == 2]


def _exact_boxes(c):
    """How many of the boxes exact() gives."""
    return min(16, sum(not s for s, _ in _box_sizes(c)))


def _stopping_times(nd):
    return [float(t) for t in np.logspace(-4.0, 0.0, nd)] if nd > 1 else [1e-2]


def _dust_state(c, seed):
    """Gas rho = 1, c_s = 1 and the species: density ratios 10^U(-3, 0), velocities near the gas's."""
    n, g = (c["nx"], c["ny"], c["nz"]), _generator(seed)
    low = [0.5 / math.sqrt(3.0) * q for q in _random_field(n, g, 1.0, 3.0, -2.0, 3)]
    one = torch.ones((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    cons = _conserved(c["gamma"], one, low, one / c["gamma"], None)
    dust = []
    for _ in range(c["species"]):
        eps = 10.0 ** (-3.0 * torch.rand(1, generator=g, device="cuda", dtype=torch.float64))
        dv = _random_field(n, g, 1.0, 3.0, -2.0, 3)
        dust.append(torch.stack([eps * one] + [eps * (low[d] + 0.1 / math.sqrt(3.0) * dv[d]) for d in range(3)]))
    return cons, torch.stack(dust)


def _face_states(c, seed):
    """Face states [n][15] (left 7, right 7, normal field) with the jump sizes of turbulent flow: mostly
    smooth, some strong gradients, a few shock-like jumps."""
    n, g, gamma = c["faces"], _generator(seed), c["gamma"]

    def rand(*shape):
        return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    rho = torch.exp(math.log(0.3) + math.log(10.0) * rand(n))
    p = rho ** gamma / gamma * (0.5 + 1.5 * rand(n))
    v = randn(n, 3) * (2.0 / math.sqrt(3.0))
    b = randn(n, 3)
    bmag = torch.sqrt(2.0 * p / 10.0 ** (2.0 * rand(n) - 1.0))
    b = b * (bmag / b.norm(dim=1))[:, None]
    wl = torch.cat([rho[:, None], v, p[:, None], b[:, 1:]], dim=1)
    u = rand(n)
    cls = (u > 0.70).long() + (u > 0.95).long()
    lo, hi = (torch.tensor(t, device="cuda", dtype=torch.float64).log()[cls] for t in ((1e-3, 2e-2, 0.3), (2e-2, 0.3, 1.5)))
    size = torch.exp(lo + (hi - lo) * rand(n))
    cs = torch.sqrt(gamma * p / rho)
    scale = torch.stack([rho, cs, cs, cs, p, bmag, bmag], dim=1)
    wr = wl + size[:, None] * scale * randn(n, 7)
    for q in (0, 4):
        wr[:, q] = torch.maximum(wr[:, q], 0.2 * wl[:, q])
    return torch.cat([wl, wr, b[:, :1]], dim=1).float().contiguous()


def _network(seed, last=1.0):
    """Packed FP32 parameters (per layer W[out][in], then b[out]); `last` scales the output layer (a
    trained correction is small)."""
    r = np.random.default_rng(seed)
    parts = []
    for k in range(4):
        s = last if k == 3 else 1.0
        parts += [s * r.normal(size=(DIMS[k + 1], DIMS[k])) / math.sqrt(DIMS[k]), 0.1 * s * r.normal(size=DIMS[k + 1])]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _batch(c, seed):
    """A training batch: 14 features and 7 targets of order one, padded to 16 and 8 columns, and the
    optimiser's state in the middle of a training."""
    n, g = c["batch"], _generator(seed)
    X = torch.randn((n, 16), generator=g, device="cuda")
    X[:, 14:] = 0.0
    Y = torch.randn((n, 8), generator=g, device="cuda") * 0.1
    Y[:, 7] = 0.0
    p = torch.from_numpy(_network(seed, 0.1)).cuda()
    m = 1e-3 * torch.randn(p.shape, generator=g, device="cuda")
    v = 1e-6 * (0.5 + torch.rand(p.shape, generator=g, device="cuda"))
    return X, Y, p, m, v


ADAM_STEP, ADAM_LR, BETA1, BETA2, ADAM_EPS = 1000, 1e-3, 0.9, 0.999, 1e-8


# ---------------------------------------------------------------------------
# a program's set-up and one pass
# ---------------------------------------------------------------------------

def _config(c):
    kw = {"gamma": c["gamma"], "cfl": CFL, "precision": PRECISION[c.get("precision", "fp32")],
          "recon": RECON[c.get("recon", "plm")]}
    if c["kind"] == "dust":
        return A.make_config(mhd=False, integrator=A.IMEX2P, t_stop=_stopping_times(c["species"]),
                             drag_precision=DRAG[c["drag"]], **kw)
    eos = c.get("eos", "mhd")
    return A.make_config(mhd=eos != "hydro", iso=eos == "iso", cs=1.0, dual=c.get("dual", False),
                         riemann=RIEMANN[c.get("riemann", "hlld")], integrator=INTEGRATOR[c.get("integrator", "vl2")], **kw)


def _cut(cons, b, c):
    """The packed parts (cons, b1, b2, b3) of each linked block of the whole box, in block order."""
    s, parts = c["split"], []
    m = [c["nx"] // s, c["ny"] // s, c["nz"] // s]
    for kz in range(s):
        for ky in range(s):
            for kx in range(s):
                x, y, z = kx * m[0], ky * m[1], kz * m[2]
                parts.append(cons[:, z:z + m[2], y:y + m[1], x:x + m[0]])
                if b is not None:
                    parts += [b[d][z:z + m[2] + (d == 2), y:y + m[1] + (d == 1), x:x + m[0] + (d == 0)] for d in range(3)]
    return parts


def _pack(parts):
    return torch.cat([p.reshape(-1) for p in parts])


def _split_outputs(c, packed):
    """The packed state as the program's fields: density, momentum, energy, face fields and dust of a
    single box; whole blocks of a mesh of several."""
    if c["kind"] == "boxes":
        q = 0
        for _, (nx, ny, nz) in _box_sizes(c)[:_exact_boxes(c)]:
            q += 8 * nx * ny * nz + ny * nz + nx * nz + nx * ny
        return [packed[:q], packed[q:]]
    nc = c["nx"] * c["ny"] * c["nz"]
    if c.get("split", 1) > 1:
        return [packed]
    cuts = [nc, 4 * nc, 5 * nc] + ([packed.numel()] if packed.numel() > 5 * nc else [])
    return [packed[a:b] for a, b in zip([0] + cuts[:-1], cuts)]


def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "train":
        X, Y, p, m, v = _batch(case, seed)
        wf = A.aeth_mlp_work_floats(case["batch"])
        return {"case": case, "X": X, "Y": Y, "p": p, "m": m, "v": v, "grad": torch.zeros_like(p), "work_floats": wf,
                "work": torch.empty(wf, device="cuda"), "loss": torch.zeros(1, device="cuda"), "stream": stream}
    if kind == "faces":
        solver = A.Solver(A.make_config(gamma=case["gamma"], precision=A.FP32), [A.make_block((8, 8, 8))], stream=stream)
        A.aeth_load_mlp(solver.ctx, _network(7, 0.02))
        n = case["faces"]
        return {"case": case, "solver": solver, "states": _face_states(case, seed),
                "flux": torch.zeros((n, 7), device="cuda"), "accept": torch.zeros(n, dtype=torch.int32, device="cuda")}
    links = ()
    if kind == "boxes":
        blocks = [A.make_block(n, WEDGE["lo"], WEDGE["hi"], A.SPH, (A.OUTFLOW, A.OUTFLOW, A.PERIODIC)) if s else A.make_block(n)
                  for s, n in _box_sizes(case)]
        packed = _pack([p for i, (s, n) in enumerate(_box_sizes(case))
                        for cons, b in [_box_state(seed * 1009 + i, s, n, case["gamma"])] for p in [cons] + b])
    elif kind == "dust":
        blocks = [A.make_block((case["nx"], case["ny"], case["nz"]))]
        packed = _pack(_dust_state(case, seed))
    else:
        n = (case["nx"], case["ny"], case["nz"])
        bc = tuple(A.OUTFLOW if ax in case["outflow"] else A.PERIODIC for ax in "xyz")
        blocks, links, _ = A.decompose(n, [[m // case["split"]] * case["split"] for m in n], bc=bc)
        if case["split"] == 1:
            links = ()
        packed = _pack(_cut(*_gas_state(case, seed), case))
    solver = A.Solver(_config(case), blocks, stream=stream, links=links)
    host = torch.empty(packed.numel(), dtype=torch.float64, pin_memory=True)
    host.copy_(packed)
    A.aeth_set_state_all_async(solver.ctx, host)
    state = {"case": case, "solver": solver, "host": host, "dev": packed}
    if case.get("precision", "fp32") != "fp64":
        state["out"] = torch.empty(packed.numel(), dtype=torch.float32, device="cuda")
    stream.synchronize()
    return state


def run(state):
    c = state["case"]
    if c["kind"] == "train":
        s, sp = state, state["stream"].cuda_stream
        A.aeth_mlp_grad(s["p"].data_ptr(), s["X"].data_ptr(), s["Y"].data_ptr(), c["batch"], s["grad"].data_ptr(),
                        s["work"].data_ptr(), s["work_floats"], s["loss"].data_ptr(), sp)
        A.aeth_mlp_adam(s["p"].data_ptr(), s["grad"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(), s["p"].numel(),
                        ADAM_STEP, ADAM_LR, BETA1, BETA2, ADAM_EPS, sp)
        return {"loss": s["loss"], "grad": s["grad"], "params": s["p"], "m": s["m"], "v": s["v"]}
    if c["kind"] == "faces":
        A.aeth_mlp_face_flux(state["solver"].ctx, state["states"].data_ptr(), state["flux"].data_ptr(),
                             state["accept"].data_ptr(), c["faces"])
        return {"flux": state["flux"], "accept": state["accept"]}
    # advance, then the snapshot (an FP64 host array) into the program's tensors in its working precision
    if c["kind"] == "boxes":
        for _ in range(c["steps"]):
            state["solver"].step(BOX_DT)
    else:
        state["solver"].run(c["steps"])
    A.aeth_get_state_all_async(state["solver"].ctx, state["host"])
    out = state["dev"].copy_(state["host"], non_blocking=True)
    if "out" in state:
        out = state["out"].copy_(out)
    return _split_outputs(c, out)


def work(case):
    """Simulations: every stage of a step reads its state once and writes it once, and the snapshot is
    written once; about 900 operations a cell and stage of MHD (three faces of reconstruction and solver, the
    corner EMFs, the update), 500 of hydro, 150 a species and stage of dust.  Network: 35,840 multiply-adds a
    face and direction of the pass."""
    kind = case["kind"]
    if kind == "faces":
        return {"bytes": case["faces"] * (15 + 7 + 1) * 4.0, "flops": case["faces"] * 71680.0}
    if kind == "train":
        npar = A.MLP_NPARAM
        return {"bytes": case["batch"] * 24 * 4.0 + npar * 4.0 * 7, "flops": case["batch"] * 71680.0 * 3 + 10.0 * npar}
    if kind == "boxes":
        cells, words, flops, stages = sum(x * y * z for _, (x, y, z) in _box_sizes(case)), 8, 900, 2
    elif kind == "dust":
        cells, words, stages = case["nx"] * case["ny"] * case["nz"], 5 + 4 * case["species"], 2
        flops = 500 + 150 * case["species"]
    else:
        cells, stages = case["nx"] * case["ny"] * case["nz"], 3 if case["integrator"] == "rk3" else 2
        words = (5 if case["eos"] == "hydro" else 8) + bool(case["dual"])
        flops = 500 if case["eos"] == "hydro" else 900
    size = 8 if case.get("precision") == "fp64" else 4
    return {"bytes": float(cells * words * size * (2 * stages * case["steps"] + 1)),
            "flops": float(cells * flops * stages * case["steps"])}


# ---------------------------------------------------------------------------
# the same passes in plain torch FP64 (periodic Cartesian boxes)
# ---------------------------------------------------------------------------
# Cell arrays and lower-face arrays are [z][y][x]; index d = 0, 1, 2 is x, y, z.

RHO_FLOOR, P_FLOOR, DUST_FLOOR = 1e-12, 1e-10, 1e-20


def _up(a, d):
    return torch.roll(a, -1, dims=2 - d)     # the value at index + 1


def _dn(a, d):
    return torch.roll(a, 1, dims=2 - d)      # the value at index - 1


def _edges_of_cell(w, d, recon):
    """Reconstructed values at the lower and the upper face of each cell along d."""
    if recon == "donor":
        return w, w
    wm, wp = _dn(w, d), _up(w, d)
    if recon == "plm":
        a, b = w - wm, wp - w
        s = torch.where(a * b > 0, 2 * a * b / torch.where(a * b > 0, a + b, torch.ones_like(a)), torch.zeros_like(a))
        return w - 0.5 * s, w + 0.5 * s

    def clip(x, p, q):
        return torch.minimum(torch.maximum(x, torch.minimum(p, q)), torch.maximum(p, q))

    if recon == "ppm":
        f = clip(7.0 / 12.0 * (wm + w) - (_dn(wm, d) + wp) / 12.0, wm, w)
        lo, hi = f, _up(f, d)
    else:
        wmm, wpp = _dn(wm, d), _up(wp, d)
        lo = clip((-3 * wmm + 27 * wm + 47 * w - 13 * wp + 2 * wpp) / 60.0, wm, w)
        hi = clip((2 * wmm - 13 * wm + 47 * w + 27 * wp - 3 * wpp) / 60.0, w, wp)
    flat = (hi - w) * (w - lo) <= 0
    q, d2 = (hi - lo) * (w - 0.5 * (lo + hi)), (hi - lo) ** 2 / 6.0
    return (torch.where(flat, w, torch.where(q > d2, 3 * w - 2 * hi, lo)),
            torch.where(flat, w, torch.where(~(q > d2) & (-d2 > q), 3 * w - 2 * lo, hi)))


def _fast(gamma, rho, p, bn, b1, b2):
    a2, t = gamma * p / rho, (bn ** 2 + b1 ** 2 + b2 ** 2) / rho
    return torch.sqrt(0.5 * (a2 + t + torch.sqrt(torch.clamp((a2 + t) ** 2 - 4 * a2 * bn ** 2 / rho, min=0.0))))


def _side(gamma, w, bn):
    """Conserved vector and flux (rho, Mn, Mt1, Mt2, E, Bt1, Bt2) of w = (rho, vn, vt1, vt2, p, Bt1, Bt2)."""
    rho, u, v1, v2, p, b1, b2 = w
    bb = bn ** 2 + b1 ** 2 + b2 ** 2
    pt = p + 0.5 * bb
    e = p / (gamma - 1.0) + 0.5 * rho * (u ** 2 + v1 ** 2 + v2 ** 2) + 0.5 * bb if gamma > 1.0 else torch.zeros_like(rho)
    f4 = (e + pt) * u - bn * (u * bn + v1 * b1 + v2 * b2) if gamma > 1.0 else torch.zeros_like(rho)
    return [rho, rho * u, rho * v1, rho * v2, e, b1, b2], [rho * u, rho * u * u + pt - bn ** 2, rho * u * v1 - bn * b1,
                                                           rho * u * v2 - bn * b2, f4, b1 * u - bn * v1, b2 * u - bn * v2]


def _where(c, a, b):
    return [torch.where(c, x, y) for x, y in zip(a, b)]


def _speeds(gamma, wl, wr, bn):
    cm = torch.maximum(_fast(gamma, wl[0], wl[4], bn, wl[5], wl[6]), _fast(gamma, wr[0], wr[4], bn, wr[5], wr[6]))
    return torch.minimum(wl[1], wr[1]) - cm, torch.maximum(wl[1], wr[1]) + cm, cm


def _hlle(gamma, wl, wr, bn):
    (ul, fl), (ur, fr) = _side(gamma, wl, bn), _side(gamma, wr, bn)
    sl, sr, _ = _speeds(gamma, wl, wr, bn)
    m, p = sl.clamp(max=0.0), sr.clamp(min=0.0)
    return [(p * fl[q] - m * fr[q] + p * m * (ur[q] - ul[q])) / (p - m) for q in range(7)]


def _hlld(gamma, wl, wr, bn, low=False):
    """HLLD (Miyoshi & Kusano 2005); low: the pressure dissipation scaled with the local Mach number."""
    (ul, fl), (ur, fr) = _side(gamma, wl, bn), _side(gamma, wr, bn)
    sl, sr, cm = _speeds(gamma, wl, wr, bn)
    bb = [bn ** 2 + w[5] ** 2 + w[6] ** 2 for w in (wl, wr)]
    ptl, ptr = wl[4] + 0.5 * bb[0], wr[4] + 0.5 * bb[1]
    al, ar = wl[0] * (sl - wl[1]), wr[0] * (sr - wr[1])
    sm = (ar * wr[1] - al * wl[1] - ptr + ptl) / (ar - al)
    diss = al * ar * (wr[1] - wl[1]) / (ar - al)
    pts = (ar * ptl - al * ptr) / (ar - al) + diss
    sgn = torch.sign(bn)

    def star(w, u, s, pt):
        rho, un = w[0], w[1]
        dd = rho * (s - un) * (s - sm) - bn ** 2
        ok = dd.abs() >= 1e-12 * pts
        den = torch.where(ok, dd, torch.ones_like(dd))
        fv = torch.where(ok, bn * (sm - un) / den, torch.zeros_like(dd))
        fb = torch.where(ok, (rho * (s - un) ** 2 - bn ** 2) / den, torch.ones_like(dd))
        rs = rho * (s - un) / (s - sm)
        v1, v2, b1, b2 = w[2] - w[5] * fv, w[3] - w[6] * fv, w[5] * fb, w[6] * fb
        vb, vbs = un * bn + w[2] * w[5] + w[3] * w[6], sm * bn + v1 * b1 + v2 * b2
        e = ((s - un) * u[4] - pt * un + pts * sm + bn * (vb - vbs)) / (s - sm)
        return rs, v1, v2, b1, b2, e

    L, R = star(wl, ul, sl, ptl), star(wr, ur, sr, ptr)
    ql, qr = torch.sqrt(L[0]), torch.sqrt(R[0])
    degen = 0.5 * bn ** 2 < 1e-12 * pts
    ssl = torch.where(degen, sm, sm - bn.abs() / ql)
    ssr = torch.where(degen, sm, sm + bn.abs() / qr)
    iq = 1.0 / (ql + qr)
    vv = [(ql * L[k] + qr * R[k] + (R[k + 2] - L[k + 2]) * sgn) * iq for k in (1, 2)]
    bs = [(ql * R[k] + qr * L[k] + ql * qr * (R[k - 2] - L[k - 2]) * sgn) * iq for k in (3, 4)]
    vbss = sm * bn + vv[0] * bs[0] + vv[1] * bs[1]
    zero = torch.zeros_like(bn)
    out = []
    for sig, w, u, f, S, s, q, ss in ((-1.0, wl, ul, fl, L, sl, ql, ssl), (1.0, wr, ur, fr, R, sr, qr, ssr)):
        vbs = sm * bn + S[1] * S[3] + S[2] * S[4]
        U = [S[0], S[0] * sm, S[0] * S[1], S[0] * S[2], S[5], S[3], S[4]]
        one = [f[k] + s * (U[k] - u[k]) for k in range(7)]
        if low:
            vm = [torch.sqrt(x[1] ** 2 + x[2] ** 2 + x[3] ** 2) for x in (wl, wr)]
            phi = (torch.maximum(*vm) / cm).clamp(max=1.0)
            one[1], one[4] = one[1] + (phi - 1.0) * diss, one[4] + (phi - 1.0) * diss * sm
        d2 = [zero, zero, S[0] * (vv[0] - S[1]), S[0] * (vv[1] - S[2]), sig * q * (vbs - vbss) * sgn,
              bs[0] - S[3], bs[1] - S[4]]
        out.append((one, [one[k] + ss * d2[k] for k in range(7)]))
    (l1, l2), (r1, r2) = out
    f = _where(ssl >= 0, l1, _where(sm >= 0, l2, _where(ssr >= 0, r2, r1)))
    return _where(sl > 0, fl, _where(sr < 0, fr, f))


def _hlld_iso(wl, wr, bn):
    """Isothermal HLLD (Mignone 2007) with c_s = 1; w[4] = rho."""
    (ul, fl), (ur, fr) = _side(1.0, wl, bn), _side(1.0, wr, bn)
    sl, sr, _ = _speeds(1.0, wl, wr, bn)
    d = sr - sl
    rs = (sr * ur[0] - sl * ul[0] - (fr[0] - fl[0])) / d
    f0, f1 = ((sr * fl[k] - sl * fr[k] + sl * sr * (ur[k] - ul[k])) / d for k in (0, 1))
    us, q, sgn = f0 / rs, torch.sqrt(rs), torch.sign(bn)
    ssl, ssr = us - bn.abs() / q, us + bn.abs() / q

    def star(w, s):
        a = w[0] * (s - w[1])
        den = a * (s - us) - bn ** 2
        ok = den.abs() >= 1e-12 * (a * (s - w[1]) + bn ** 2)
        den = torch.where(ok, den, torch.ones_like(den))
        fv = torch.where(ok, bn * (us - w[1]) / den, torch.zeros_like(den))
        fb = torch.where(ok, (a * (s - w[1]) - bn ** 2) / den, torch.ones_like(den))
        return w[2] - w[5] * fv, w[3] - w[6] * fv, w[5] * fb, w[6] * fb

    L, R = star(wl, sl), star(wr, sr)
    mid = [0.5 * (L[k] + R[k]) + 0.5 * (R[k + 2] - L[k + 2]) * sgn / q for k in (0, 1)]
    mid += [0.5 * (L[k] + R[k]) + 0.5 * q * (R[k - 2] - L[k - 2]) * sgn for k in (2, 3)]

    def flux(S, u, f, s):
        t = [f[2] + s * (rs * S[0] - u[2]), f[3] + s * (rs * S[1] - u[3]), f[5] + s * (S[2] - u[5]), f[6] + s * (S[3] - u[6])]
        return [f0, f1, t[0], t[1], torch.zeros_like(f0), t[2], t[3]]

    l1, r1 = flux(L, ul, fl, sl), flux(R, ur, fr, sr)
    c = list(l1)
    for k, a, s in ((2, 0, rs), (3, 1, rs), (5, 2, 1.0), (6, 3, 1.0)):
        c[k] = l1[k] + ssl * s * (mid[a] - L[a])
    f = _where(ssl >= 0, l1, _where(ssr > 0, c, r1))
    return _where(sl >= 0, fl, _where(sr <= 0, fr, f))


def _primitives(gamma, U, B):
    """(rho, v1, v2, v3, p, B1, B2, B3) at cell centres; gamma = 1: isothermal with c_s = 1."""
    rho = U[0].clamp(min=RHO_FLOOR)
    v = [U[1 + d] / rho for d in range(3)]
    bc = [0.5 * (B[d] + _up(B[d], d)) for d in range(3)] if B is not None else [torch.zeros_like(rho)] * 3
    if gamma == 1.0:
        p = rho
    else:
        ke, me = 0.5 * rho * sum(q ** 2 for q in v), 0.5 * sum(q ** 2 for q in bc)
        p = ((gamma - 1.0) * (U[4] - ke - me)).clamp(min=P_FLOOR)
    return [rho] + v + [p] + bc


def _gas_rhs(gamma, U, B, h, recon, riemann):
    """-div F of the five conserved variables and -curl E of the faces."""
    w = _primitives(gamma, U, B)
    F, emf = [], []
    for d in range(3):
        t1, t2 = (d + 1) % 3, (d + 2) % 3
        lo, hi = zip(*(_edges_of_cell(w[q], d, recon) for q in (0, 1 + d, 1 + t1, 1 + t2, 4, 5 + t1, 5 + t2)))
        wl, wr = [_dn(q, d) for q in hi], list(lo)
        bn = B[d] if B is not None else torch.zeros_like(w[0])
        if gamma == 1.0:
            wl[4], wr[4] = wl[0], wr[0]
            f = _hlld_iso(wl, wr, bn) if riemann == "hlld" else _hlle(1.0, wl, wr, bn)
        else:
            f = _hlle(gamma, wl, wr, bn) if riemann == "hlle" else _hlld(gamma, wl, wr, bn, riemann == "lhlld")
        g = [None] * 5
        g[0], g[1 + d], g[1 + t1], g[1 + t2], g[4] = f[:5]
        F.append(g)
        emf.append((f[6], -f[5]))       # E along t1 and along t2
    dU = torch.stack([-sum((_up(F[d][v], d) - F[d][v]) / h[d] for d in range(3)) for v in range(5)])
    if B is None:
        return dU, None
    vel, bc, corner = w[1:4], w[5:8], []
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        er = -(vel[a] * bc[b] - vel[b] * bc[a])
        ea, eb, fa, fb = emf[a][1], emf[b][0], F[a][0], F[b][0]
        eam, ebm, fam, fbm = _dn(ea, b), _dn(eb, a), _dn(fa, b), _dn(fb, a)
        r01, r10 = _dn(er, b), _dn(er, a)
        r00 = _dn(r10, b)

        def upwind(m, x, y):
            return torch.where(m > 0, x, torch.where(m < 0, y, 0.5 * (x + y)))

        corner.append(0.25 * (eam + ea + ebm + eb + upwind(fam, ebm - r00, eb - r01) - upwind(fa, r10 - ebm, er - eb)
                              + upwind(fbm, eam - r00, ea - r10) - upwind(fb, r01 - eam, er - ea)))
    dB = []
    for d in range(3):
        e1, e2 = (d + 1) % 3, (d + 2) % 3
        dB.append(-((_up(corner[e2], e1) - corner[e2]) / h[e1] - (_up(corner[e1], e2) - corner[e1]) / h[e2]))
    return dU, dB


def _time_step(gamma, U, B, h):
    w = _primitives(gamma, U, B)
    return CFL * min(float((h[d] / (w[1 + d].abs() + _fast(gamma, w[0], w[4], w[5 + d], w[5 + (d + 1) % 3],
                                                            w[5 + (d + 2) % 3]))).min()) for d in range(3))


STAGES = {"vl2": ((0, 1.0, 0.0, 0.5, 1), (1, 1.0, 0.0, 1.0, 0)), "rk2": ((0, 1.0, 0.0, 1.0, 1), (1, 0.5, 0.5, 0.5, 0)),
          "rk3": ((0, 1.0, 0.0, 1.0, 1), (1, 0.75, 0.25, 0.25, 1), (1, 1 / 3, 2 / 3, 2 / 3, 0))}


def _exact_gas(gamma, cons, b, steps, recon, riemann, integrator, dt_given=None):
    h = [1.0 / cons.shape[3 - d] for d in range(3)]
    B = [b[0][:, :, :-1], b[1][:, :-1, :], b[2][:-1, :, :]] if b is not None else None
    reg = [(cons, B), (cons, B)]
    for _ in range(steps):
        dt = dt_given or _time_step(gamma, *reg[0], h)
        for k, (src, w0, w1, beta, out) in enumerate(STAGES[integrator]):
            first = integrator == "vl2" and k == 0
            dU, dB = _gas_rhs(gamma, *reg[src], h, "donor" if first else recon, riemann)
            U = w0 * reg[0][0] + w1 * reg[1][0] + beta * dt * dU
            nB = [w0 * p + w1 * q + beta * dt * r for p, q, r in zip(reg[0][1], reg[1][1], dB)] if B is not None else None
            reg[out] = (U, nB)
    U, B = reg[0]
    if B is not None:
        B = [torch.cat([q, q.narrow(2 - d, 0, 1)], dim=2 - d) for d, q in enumerate(B)]
    return U, B


def _dust_rhs(D, h, recon):
    """-div F of the species (rho, M1, M2, M3): pressureless Rusanov fluxes."""
    out = torch.zeros_like(D)
    for s in range(D.shape[0]):
        rho = D[s, 0].clamp(min=DUST_FLOOR)
        w = [rho] + [D[s, 1 + d] / rho for d in range(3)]
        for d in range(3):
            lo, hi = zip(*(_edges_of_cell(q, d, recon) for q in w))
            wl, wr = [_dn(q, d) for q in hi], list(lo)
            ul, ur = ([x[0], x[0] * x[1], x[0] * x[2], x[0] * x[3]] for x in (wl, wr))
            sp = torch.maximum(wl[1 + d].abs(), wr[1 + d].abs())
            for v in range(4):
                f = 0.5 * (ul[v] * wl[1 + d] + ur[v] * wr[1 + d]) - 0.5 * sp * (ur[v] - ul[v])
                out[s, v] -= (_up(f, d) - f) / h[d]
    return out


def _drag(U, D, hdt, ts):
    """The implicit drag of one stage: momenta after h dt, and the energy lost by drift as heat."""
    a = [hdt / t for t in ts]
    U, D0, D = U.clone(), D, D.clone()
    den = U[0] + sum(D0[k, 0] * a[k] / (1 + a[k]) for k in range(len(ts)))
    heat = torch.zeros_like(U[0])
    for q in (1, 2, 3):
        vg = (U[q] + sum(D0[k, q] * a[k] / (1 + a[k]) for k in range(len(ts)))) / den
        U[q] = U[0] * vg
        for k in range(len(ts)):
            D[k, q] = (D0[k, q] + D0[k, 0] * a[k] * vg) / (1 + a[k])
            heat += (D[k, q] ** 2 - D0[k, q] ** 2) / (2 * D0[k, 0])
    U[4] -= heat
    return U, D


def _exact_dust(c, cons, D):
    gamma, ts, h = c["gamma"], _stopping_times(c["species"]), [1.0 / c["nx"], 1.0 / c["ny"], 1.0 / c["nz"]]
    g = 1.0 + 1.0 / math.sqrt(2.0)
    d = 1.0 - 1.0 / (2.0 * g)
    U = cons
    for _ in range(c["steps"]):
        dt = _time_step(gamma, U, None, h) / CFL
        for k in range(c["species"]):
            for q in range(3):
                dt = min(dt, float((h[q] / (D[k, 1 + q] / D[k, 0]).abs().clamp(min=1e-300)).min()))
        dt *= CFL / g
        dU, dD = _gas_rhs(gamma, U, None, h, c["recon"], "hlld")[0], _dust_rhs(D, h, c["recon"])
        XU, XD = U + g * dt * dU, D + g * dt * dD
        U2, D2 = _drag(XU, XD, g * dt, ts)
        WU, WD = (W + d * dt * dW + (1 - g) / g * (Y - X) for W, dW, Y, X in ((U, dU, U2, XU), (D, dD, D2, XD)))
        dU, dD = _gas_rhs(gamma, U2, None, h, c["recon"], "hlld")[0], _dust_rhs(D2, h, c["recon"])
        U, D = _drag(WU + (1 - d) * dt * dU, WD + (1 - d) * dt * dD, g * dt, ts)
    return U, D


def _layers(params):
    p, out = torch.as_tensor(params).double().cuda(), []
    for k in range(4):
        w, p = p[:DIMS[k + 1] * DIMS[k]].reshape(DIMS[k + 1], DIMS[k]), p[DIMS[k + 1] * DIMS[k]:]
        out.append((w, p[:DIMS[k + 1]]))
        p = p[DIMS[k + 1]:]
    return out


def _exact_faces(c, seed):
    """F = F_HLLE + k J y of the network's output y where it is accepted, HLLD elsewhere."""
    st, gamma = _face_states(c, seed).double(), c["gamma"]
    wl, wr, bn = list(st[:, :7].T), list(st[:, 7:14].T), st[:, 14]
    sl, sr, cm = _speeds(gamma, wl, wr, bn)
    sq = torch.sqrt(wl[0])
    sc = [1.0 / wl[0]] + [1.0 / cm] * 3 + [1.0 / (wl[0] * cm ** 2)] + [1.0 / (sq * cm)] * 2
    dw = torch.stack([(wr[q] - wl[q]) * sc[q] for q in range(7)], dim=1)
    m = dw.norm(dim=1, keepdim=True)
    x = torch.cat([torch.stack([wl[q] * sc[q] for q in range(1, 7)] + [bn * sc[5]], dim=1),
                   dw * torch.where(m > 0, (1 + m) / m.clamp(min=1e-300), torch.zeros_like(m))], dim=1)
    for k, (w, b) in enumerate(_layers(_network(7, 0.02))):
        x = x @ w.T + b
        x = torch.nn.functional.silu(x) if k < 3 else x
    (ul, fl), (ur, fr) = _side(gamma, wl, bn), _side(gamma, wr, bn)
    rc2 = wl[0] * cm ** 2
    k7 = [wl[0] * cm, rc2, rc2, rc2, rc2 * cm * gamma / (gamma - 1.0), sq * cm ** 2, sq * cm ** 2]
    J = (sr - sl) * torch.sqrt(sum(((ur[q] - ul[q]) / k7[q]) ** 2 for q in range(7)))
    fe = _hlle(gamma, wl, wr, bn)
    F = [fe[q] + k7[q] * J * x[:, q] for q in range(7)]
    ok = torch.ones_like(bn, dtype=torch.bool)
    for q in range(7):
        ok &= (F[q] - fe[q]).abs() <= 0.25 * (sr - sl) * (ur[q] - ul[q]).abs() + 2e-2 * k7[q]
    for s, on, u, f in ((sl, sl < 0, ul, fl), (sr, sr > 0, ur, fr)):
        us = [u[q] + (F[q] - f[q]) / torch.where(on, s, torch.ones_like(s)) for q in range(7)]
        pr = us[4] - 0.5 * (us[1] ** 2 + us[2] ** 2 + us[3] ** 2) / us[0] - 0.5 * (bn ** 2 + us[5] ** 2 + us[6] ** 2)
        ok &= ~on | ((us[0] > 0) & (pr > 0))
    return {"flux": torch.stack(_where(ok, F, _hlld(gamma, wl, wr, bn)), dim=1), "accept": None}


def _exact_train(c, seed):
    X, Y, p, m, v = (t.double() for t in _batch(c, seed))
    L = [(w.requires_grad_(), b.requires_grad_()) for w, b in ((w.clone(), b.clone()) for w, b in _layers(p))]
    x = X[:, :14]
    for k, (w, b) in enumerate(L):
        x = x @ w.T + b
        x = torch.nn.functional.silu(x) if k < 3 else x
    loss = 0.5 * ((x - Y[:, :7]) ** 2).sum() / c["batch"]
    loss.backward()
    g = torch.cat([t.grad.reshape(-1) for wb in L for t in wb])
    m, v = BETA1 * m + (1 - BETA1) * g, BETA2 * v + (1 - BETA2) * g * g
    step = ADAM_LR * (m / (1 - BETA1 ** ADAM_STEP)) / (torch.sqrt(v / (1 - BETA2 ** ADAM_STEP)) + ADAM_EPS)
    return {"loss": loss.detach().reshape(1), "grad": g, "params": p - step, "m": m, "v": v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "faces":
        return _exact_faces(case, seed)
    if kind == "dust":
        return _split_outputs(case, _pack(_exact_dust(case, *_dust_state(case, seed))))
    if kind == "boxes":
        parts = []
        for i, (s, n) in enumerate(_box_sizes(case)[:_exact_boxes(case)]):
            cons, b = _box_state(seed * 1009 + i, s, n, case["gamma"])
            U, B = _exact_gas(case["gamma"], cons, b, case["steps"], "plm", "hlld", "vl2", BOX_DT)
            parts += [U] + B
        return [_pack(parts), None]
    if case["outflow"] or case["dual"]:
        return None
    cons, b = _gas_state(case, seed)
    U, B = _exact_gas(1.0 if case["eos"] == "iso" else case["gamma"], cons, b, case["steps"], case["recon"],
                      case["riemann"], case["integrator"])
    return _split_outputs(case, _pack(_cut(U, B, case)))
