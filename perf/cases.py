"""The work a planning service has this library do, as cases that can be timed.

Each case is one pass through the public entry points on inputs made from a
seed: the Rayleigh-Sommerfeld source plane of a placement, FDTD runs (FP32 and
scaled FP16 state, grids with and without whole 16-byte rows), one whole plan,
a batched sweep, the bioheat exposure, and the surrogate (planning-time
inference, BF16 inference, one training gradient).  `exact` gives what a pass
returns in 64 bits, from plain torch and numpy.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and the handles a program keeps
    run(state)           one pass, and its outputs
    work(case)           bytes and operations the pass cannot do without
    exact(case, seed)    the outputs in 64 bits
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2301_12727_gb300 import bvf, fno, plan, synth

DEV = "cuda"
F64 = torch.float64
COURANT = 6.0 / (7.0 * math.sqrt(3.0))
C0 = 1500.0
P0 = 6.0e4
PML = 8
N_BINS = 125
# surrogate of the benchmark and of the training tool
NET = dict(c_in=8, width=32, modes=12, n_layers=4, hidden=128, c_out=2)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the source plane of one placement on the benchmark's grid: the
        # smallest call of a plan, made again for each bowl pose a user tries
        dict(name="source_plane_240", path="rs", nx=240, ny=240, dx=0.5e-3, f0=5e5),
        # the 64^3 slab burst: a small domain stepped 400 times, where the
        # launches and the latency of a step are what a user waits for
        dict(name="fdtd_slab_64", path="fdtd", kind="slab", nx=64, ny=64, nz=64, dx=0.5e-3, f0=5e5,
             steps=400, window=0, storage="f32"),
        # the benchmark's skull: two periods of steps, the second one inside
        # the amplitude window (the bulk of every full-size plan)
        dict(name="fdtd_skull_240", path="fdtd", kind="skull", nx=240, ny=240, nz=200, dx=0.5e-3,
             f0=5e5, steps=92, window=46, storage="f32"),
        # the largest grid of the mixed-precision family (700 kHz at 9 points
        # per wavelength) with its scaled FP16 state
        dict(name="fdtd_skull_360_f16", path="fdtd", kind="skull", nx=360, ny=360, nz=300,
             dx=1500.0 / (9.0 * 7e5), f0=7e5, steps=46, window=16, storage="f16"),
        # a subject's bounding box as it comes: no axis a multiple of 8
        dict(name="fdtd_ragged_197", path="fdtd", kind="skull", nx=197, ny=211, nz=163, dx=0.5e-3,
             f0=5e5, steps=92, window=46, storage="f32"),
        # one whole plan as the training-data tool makes them by the thousand:
        # skull and water runs, E_L, scaling, the 40 s / 80 s exposure
        dict(name="plan_64x64x96", path="plan", nx=64, ny=64, nz=96, dx=1e-3, f0=2.5e5, cycles=6,
             storage="f32"),
        # a planning sweep over placements: 16 domains of 96..200 cells per
        # axis at 250 / 500 / 700 kHz, one recorded graph per sweep
        dict(name="sweep_16", path="sweep", domains=16, spec=4321, steps=46),
        # the bioheat exposure on the benchmark's grid (source on, then cooling)
        dict(name="bhte_240", path="bhte", nx=240, ny=240, nz=200, dx=0.5e-3, n_on=160, n_off=320),
        # planning-time inference of one placement on the trained grid:
        # feature volume and network
        dict(name="fno_64x64x96", path="fno", nx=64, ny=64, nz=96, features=1),
        # the same network on the benchmark's grid
        dict(name="fno_240", path="fno", nx=240, ny=240, nz=200, features=0),
        # its BF16 forward on the benchmark's grid
        dict(name="fno_bf16_240", path="fno16", nx=240, ny=240, nz=200, batch=1),
        # one training gradient of the tool's batch of four placements
        dict(name="train_64x64x96_b4", path="train", nx=64, ny=64, nz=96, batch=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["rs", "fdtd", "fdtd", "fdtd", "plan", "sweep", "bhte", "fno", "fno16", "train"])
    if path == "rs":
        n = _log_int(rng, 48, 240)
        f0 = rng.choice([2.5e5, 5e5])
        return dict(path="rs", nx=n, ny=_log_int(rng, 48, 240), dx=1500.0 / (6.0 * f0), f0=f0)
    if path == "fdtd":
        nx, ny, nz = (_log_int(rng, 40, 240) for _ in range(3))
        if rng.random() < 0.6:
            nx = max(40, nx // 8 * 8)
        f0 = rng.choice([2.5e5, 5e5, 7e5])
        cap = 240 * 240 * 200 * 92
        steps = int(min(400, max(24, cap // (nx * ny * nz)) * rng.uniform(0.3, 1.0)))
        return dict(path="fdtd", kind=rng.choice(["skull", "skull", "slab"]), nx=nx, ny=ny, nz=nz,
                    dx=1500.0 / (rng.choice([6.0, 9.0]) * f0), f0=f0, steps=steps,
                    window=int(steps * rng.choice([0.0, 0.3, 0.5])),
                    storage=rng.choice(["f32", "f32", "f16"]))
    if path == "plan":
        nx, ny, nz = (_log_int(rng, 40, 64) for _ in range(3))
        if rng.random() < 0.6:
            nx = nx // 8 * 8
        return dict(path="plan", nx=nx, ny=ny, nz=max(nz, 48), dx=1e-3, f0=2.5e5, cycles=4,
                    storage=rng.choice(["f32", "f16"]))
    if path == "sweep":
        return dict(path="sweep", domains=rng.randint(3, 12), spec=rng.randint(1, 10 ** 6), steps=46)
    if path == "bhte":
        nx, ny, nz = (_log_int(rng, 40, 220) for _ in range(3))
        if rng.random() < 0.5:
            nx = nx // 8 * 8
        n = rng.randint(60, 460)
        return dict(path="bhte", nx=nx, ny=ny, nz=nz, dx=0.5e-3, n_on=n // 3, n_off=n - n // 3)
    if path == "fno":
        nx, ny, nz = (_log_int(rng, 32, 200) for _ in range(3))
        return dict(path="fno", nx=nx, ny=ny, nz=nz, features=rng.randint(0, 1))
    if path == "fno16":
        nx, ny, nz = (_log_int(rng, 32, 180) for _ in range(3))
        return dict(path="fno16", nx=nx, ny=ny, nz=nz, batch=rng.randint(1, 2))
    nx, ny, nz = _log_int(rng, 32, 64), _log_int(rng, 32, 64), _log_int(rng, 32, 96)
    return dict(path="train", nx=nx, ny=ny, nz=nz, batch=rng.randint(1, 4))


# ------------------------------------------------------------ inputs (GPU, seeded)
def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + salt)


def _rand(gen, *shape):
    return torch.rand(shape, generator=gen, device=DEV, dtype=F64)


def _smooth(gen, shape, cell):
    """Smooth seeded field in [0, 1]: a coarse random lattice, interpolated."""
    n = [max(2, int(math.ceil(s / cell)) + 1) for s in shape]
    f = torch.nn.functional.interpolate(_rand(gen, 1, 1, *n), size=shape, mode="trilinear",
                                        align_corners=True)[0, 0]
    return (f - f.min()) / (f.max() - f.min())


def _table(f0):
    """Water, brain, skin, then bone by HU bin: rows as in bvf_material."""
    rows = [[1000.0, 1500.0, 0.0, 0.0, 0.0, 0.60, 4178.0, 0.0, 1.0],
            [1041.0, 1562.0, 0.0, 6.9 * f0 / 1e6, 0.0, 0.51, 3630.0, 0.008, 1.0],
            [1116.0, 1537.0, 0.0, 4.6 * f0 / 1e6, 0.0, 0.37, 3391.0, 0.008, 1.0]]
    for b in range(N_BINS):
        hu = 300.0 + (b + 0.5) * 1700.0 / N_BINS
        al = 85.0 * (hu / 2000.0) * (f0 / 5e5)
        rows.append([1000.0 + 0.425 * hu, 1500.0 + 0.65 * hu, 0.75 * hu, al, 2.0 * al, 0.32, 1313.0,
                     0.008, 0.16])
    return np.array(rows)


def _time_step(dx, f0, table):
    dt0 = 0.5 * COURANT * dx / table[:, 1].max()
    m = int(math.ceil(1.0 / (f0 * dt0)))
    return 1.0 / (f0 * m), m


def _skull(gen, nx, ny, nz, dx):
    """Ellipsoidal skull cap crossing the axis, 6-9 mm thick, skin outside and
    brain inside; cortical and trabecular HU from smooth noise, in bins."""
    a, b, c = 70e-3, 85e-3, 60e-3
    ax = torch.arange(nx, device=DEV, dtype=F64) * dx - 0.5 * (nx - 1) * dx
    ay = torch.arange(ny, device=DEV, dtype=F64) * dx - 0.5 * (ny - 1) * dx
    az = torch.arange(nz, device=DEV, dtype=F64) * dx - ((PML + 2) * dx + 5e-3 + c)
    x, y, z = ax[None, None, :], ay[None, :, None], az[:, None, None]
    r = torch.sqrt(x * x + y * y + z * z) + 1e-12
    depth = r / torch.sqrt((x / a) ** 2 + (y / b) ** 2 + (z / c) ** 2) - r
    thick = 6e-3 + 3e-3 * _smooth(gen, (nz, ny, nx), max(2, int(20e-3 / dx)))
    cell = max(2, int(round(4e-3 / dx)))
    frac = depth / thick
    cort = (frac < 0.1) | (frac >= 0.9)
    hu = torch.where(cort, 1500.0 + 500.0 * _smooth(gen, (nz, ny, nx), cell),
                     300.0 + 700.0 * _smooth(gen, (nz, ny, nx), cell))
    bins = torch.floor((hu - 300.0) / (1700.0 / N_BINS)).clamp(0, N_BINS - 1)
    index = torch.zeros((nz, ny, nx), device=DEV, dtype=F64)
    index = torch.where((depth < 0) & (depth >= -3e-3), torch.full_like(index, 2.0), index)
    index = torch.where(depth >= thick, torch.full_like(index, 1.0), index)
    index = torch.where((depth >= 0) & (depth < thick), 3.0 + bins, index)
    return index.to(torch.uint8).contiguous()


def _slab(gen, nx, ny, nz, dx):
    """A 6 mm cortical / trabecular / cortical slab across the whole plane."""
    z = torch.arange(nz, device=DEV, dtype=F64) * dx
    z0 = (PML + 2) * dx + 3e-3 + 4e-3 * float(_rand(gen, 1))
    m = torch.zeros(nz, device=DEV, dtype=F64)
    m = torch.where((z >= z0) & (z < z0 + 6e-3), torch.full_like(m, 3.0 + 110), m)
    m = torch.where((z >= z0 + 1.5e-3) & (z < z0 + 4.5e-3), torch.full_like(m, 3.0 + 30), m)
    return m.to(torch.uint8)[:, None, None].expand(nz, ny, nx).contiguous()


def _acoustic(case, seed, salt=0):
    """Everything one FDTD run takes: material volume and table, time step,
    a converging source plane (complex amplitudes as float pairs)."""
    nx, ny, nz, dx, f0 = case["nx"], case["ny"], case["nz"], case["dx"], case["f0"]
    gen = _gen(seed, salt)
    table = _table(f0)
    dt, per = _time_step(dx, f0, table)
    slab = case.get("kind") == "slab"
    index = (_slab if slab else _skull)(gen, nx, ny, nz, dx)
    x = (torch.arange(nx, device=DEV, dtype=F64) - 0.5 * (nx - 1))[None, :] * dx
    y = (torch.arange(ny, device=DEV, dtype=F64) - 0.5 * (ny - 1))[:, None] * dx
    if slab:       # plane burst, uneven across the plane
        amp = 1e5 * (0.8 + 0.4 * _smooth(gen, (1, ny, nx), 24)[0]) if min(nx, ny) >= 2 else 1e5
        phase = torch.zeros_like(amp)
    else:          # a focused beam with a wandering focus
        ox, oy, foc = (float(v) for v in _rand(gen, 3))
        r = torch.hypot(x - (ox - 0.5) * 8e-3, y - (oy - 0.5) * 8e-3)
        amp = P0 * torch.exp(-(r / (0.35 * min(nx, ny) * dx)) ** 4)
        phase = 2.0 * math.pi * f0 / C0 * (torch.sqrt(r * r + (40e-3 + 20e-3 * foc) ** 2))
    pl = torch.stack([amp * torch.cos(phase), amp * torch.sin(phase)], -1).float().contiguous()
    return dict(nx=nx, ny=ny, nz=nz, dx=dx, dt=dt, f0=f0, per=per, index=index, table=table,
                plane=pl, k_src=PML + 2, env=1 if slab else 2, cycles=3 if slab else 0)


def _bowl(case, seed):
    """A 64 mm / 63 mm bowl with a seeded tilt, its rim below the source plane."""
    gen = _gen(seed, 5)
    t = math.radians(30.0 * (float(_rand(gen, 1)) - 0.5))
    az = 2.0 * math.pi * float(_rand(gen, 1))
    a, roc = 32e-3, 63e-3
    h = roc - math.sqrt(roc * roc - a * a)
    z_src = (PML + 2) * case["dx"]
    top = h * math.cos(t) + a * abs(math.sin(t))
    return dict(aperture=2 * a, roc=roc, p0=P0 * (0.8 + 0.4 * float(_rand(gen, 1))),
                apex=(0.5 * (case["nx"] - 1) * case["dx"], 0.5 * (case["ny"] - 1) * case["dx"],
                      z_src - 2e-3 - top),
                dir=(math.sin(t) * math.cos(az), math.sin(t) * math.sin(az), math.cos(t)))


def _plan_case(case, seed):
    q = dict(case, kind="skull")
    a = _acoustic(q, seed)
    n = int(math.ceil(1.3 * case["nz"] * case["dx"] / C0 / a["dt"])) + case["cycles"] * a["per"]
    return a, n, case["cycles"] * a["per"], _bowl(case, seed)


def _sweep_domains(case):
    """Sizes and frequencies of a sweep's domains (96..200 cells per axis, nx
    a multiple of 16, 6 points per wavelength)."""
    rng = np.random.default_rng(case["spec"])
    out = []
    for _ in range(case["domains"]):
        nx, ny, nz = (int(v) for v in rng.integers(96, 201, size=3))
        f0 = float(rng.choice([2.5e5, 5e5, 7e5]))
        out.append(dict(nx=min(208, (nx + 15) // 16 * 16), ny=ny, nz=nz, f0=f0, kind="skull",
                        dx=C0 / f0 / 6.0))
    return out


def _heat(case, seed):
    """Tissue volume and a focal pressure amplitude that warms it by a few C."""
    nx, ny, nz, dx = case["nx"], case["ny"], case["nz"], case["dx"]
    gen = _gen(seed, 3)
    index = _skull(gen, nx, ny, nz, dx)
    f = _rand(gen, 3) * 0.3 + 0.35
    z, y, x = (torch.arange(n, device=DEV, dtype=F64) for n in (nz, ny, nx))
    r2 = ((x - f[0] * nx) ** 2)[None, None, :] + ((y - f[1] * ny) ** 2)[None, :, None]
    amp = 1.2e6 * torch.exp(-r2 / 60.0 - ((z - f[2] * nz) ** 2)[:, None, None] / 900.0)
    amp = amp + 2e5 * _smooth(gen, (nz, ny, nx), 16)
    return index, _table(5e5), amp.contiguous()


def _count(net):
    m3 = 4 * net["modes"] ** 3
    w = net["width"]
    return (w * net["c_in"] + w + net["n_layers"] * (m3 * w * w * 2 + w * w + w) +
            net["hidden"] * w + net["hidden"] + net["c_out"] * net["hidden"] + net["c_out"])


def _weights(seed, net, train=False):
    """Flat weight blob on the GPU (float32), scaled by fan-in."""
    gen = _gen(seed, 11)
    w, m3 = net["width"], 4 * net["modes"] ** 3
    spec = 1.0 / w ** (2 if train else 1)

    def part(n, scale):
        return torch.randn(n, generator=gen, device=DEV) * scale
    out = [part(w * net["c_in"], net["c_in"] ** -0.5), part(w, 0.1)]
    for _ in range(net["n_layers"]):
        out += [part(m3 * w * w * 2, spec), part(w * w, w ** -0.5), part(w, 0.1)]
    out += [part(net["hidden"] * w, w ** -0.5), part(net["hidden"], 0.1),
            part(net["c_out"] * net["hidden"], net["hidden"] ** -0.5), part(net["c_out"], 0.1)]
    return torch.cat(out)


def _volume(gen, c, nz, ny, nx):
    """Feature-like channels: a few low Fourier modes plus white noise."""
    out = torch.empty((c, nz, ny, nx), device=DEV)
    z, y, x = (torch.arange(n, device=DEV, dtype=torch.float32) / n for n in (nz, ny, nx))
    for i in range(c):
        f = 0.1 * torch.randn((nz, ny, nx), generator=gen, device=DEV)
        for _ in range(3):
            k = torch.randint(-3, 4, (3,), generator=gen, device=DEV).float()
            ph, s = 6.28 * torch.rand(2, generator=gen, device=DEV)
            f += 0.3 * s * torch.cos(6.2831853 * (k[0] * z[:, None, None] + k[1] * y[None, :, None] +
                                                  k[2] * x[None, None, :]) + ph)
        out[i] = f
    return out


def _target(gen, b, nz, ny, nx):
    """Amplitude-like target fields and transmission efficiencies of a batch."""
    z, y, x = (torch.arange(n, device=DEV, dtype=torch.float32) / n - 0.5 for n in (nz, ny, nx))
    t = torch.empty((b, nz, ny, nx), device=DEV)
    for i in range(b):
        o = 0.2 * torch.rand(3, generator=gen, device=DEV) - 0.1
        r2 = ((z - o[0]) ** 2)[:, None, None] / 0.08 + ((y - o[1]) ** 2)[None, :, None] / 0.01 + \
            ((x - o[2]) ** 2)[None, None, :] / 0.01
        t[i] = 4.0 * torch.exp(-r2) + 0.2
    return t, 0.2 + 0.5 * torch.rand(b, generator=gen, device=DEV)


EL_WEIGHT = 10.0


def _net_inputs(case, seed):
    gen = _gen(seed, 17)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["path"] == "fno" and case["features"]:
        a = _acoustic(dict(nx=nx, ny=ny, nz=nz, dx=1e-3, f0=2.5e5), seed)
        return dict(a=a)
    if case["path"] == "fno":
        return dict(x=_volume(gen, NET["c_in"], nz, ny, nx))
    b = case["batch"]
    q = dict(x=torch.stack([_volume(gen, NET["c_in"], nz, ny, nx) for _ in range(b)]))
    if case["path"] == "train":
        q["t"], q["el"] = _target(gen, b, nz, ny, nx)
    return q


# ------------------------------------------------------------------- a pass
def _solver(a, storage="f32"):
    s = bvf.Solver(a["nx"], a["ny"], a["nz"], a["dx"], a["dt"], a["f0"], n_pml=PML, storage=storage)
    s.set_materials(a["index"], a["table"])
    s.set_source(a["plane"], a["k_src"], C0, a["env"], a["cycles"])
    return s


def prepare(case, seed):
    path = case["path"]
    st = dict(path=path, case=case)
    if path == "rs":
        st["bowl"] = _bowl(case, seed)
    elif path == "fdtd":
        st["solver"] = _solver(_acoustic(case, seed), case["storage"])
    elif path == "plan":
        a, n, dft, bowl = _plan_case(case, seed)
        c = synth.Case("placement", a["nx"], a["ny"], a["nz"], a["dx"], a["f0"], a["dt"], a["per"], n,
                       None, a["table"], a["k_src"], 2, bowl=bowl, n_pml=PML, dft_cycles=case["cycles"])
        st.update(planner=plan.Planner(c, case["storage"]), index=a["index"], table=a["table"],
                  bowl=bowl)
    elif path == "sweep":
        doms = _sweep_domains(case)
        st["solvers"] = [_solver(_acoustic(d, seed, k + 100)) for k, d in enumerate(doms)]
        st["caps"] = [bvf.Capture(0, case["steps"] - 15, 16) for _ in doms]
        st["batch"] = bvf.Batch(st["solvers"])
    elif path == "bhte":
        index, table, amp = _heat(case, seed)
        s = bvf.Solver(case["nx"], case["ny"], case["nz"], case["dx"],
                       _time_step(case["dx"], 5e5, table)[0], 5e5, n_pml=PML)
        s.set_materials(index, table)
        st.update(solver=s, amp=amp)
    elif path == "fno":
        st.update(_net_inputs(case, seed))
        st["net"] = fno.Surrogate(NET, _weights(seed, NET).cpu().numpy())
    else:
        st.update(_net_inputs(case, seed))
        st["net"] = fno.Bf16Net(NET, _weights(seed, NET, path == "train").cpu().numpy(),
                                (case["nx"], case["ny"], case["nz"]), max_batch=case["batch"])
    return st


def run(st):
    path, case = st["path"], st["case"]
    if path == "rs":
        return bvf.rs_plane(st["bowl"], case["nx"], case["ny"], case["dx"], (PML + 2) * case["dx"],
                            case["f0"])
    if path == "fdtd":
        s, n, w = st["solver"], case["steps"], case["window"]
        s.reset()
        s.run(n, peak_from=0, dft_start=n - w + 1, dft_steps=w)
        out = dict(pressure=s.pressure(), peak=s.peak())
        if w:
            out["amp"], out["phase"] = s.amp_phase()
        return out
    if path == "plan":
        r = st["planner"].run(st["index"], st["table"], st["bowl"])
        return dict(peak=r.peak, amp=r.amp, Tmax=r.Tmax, cem43=r.cem43, EL=r.EL, TS=r.TS, z_m=r.z_m,
                    Iw_max=r.Iw_max, p_scale=r.p_scale)
    if path == "sweep":
        for s in st["solvers"]:
            s.reset()
        st["batch"].run_graph(case["steps"], caps=st["caps"], n_branches=8)
        return [(s.pressure(), s.peak(), s.amp_phase()[0]) for s in st["solvers"]]
    if path == "bhte":
        T, Tmax, cem = st["solver"].thermal(st["amp"], 0.1, case["n_on"], case["n_off"], 0.3)
        return dict(T=T, Tmax=Tmax, cem43=cem)
    if path == "fno":
        x = st.get("x")
        if x is None:
            a = st["a"]
            x = torch.empty((fno.N_FEATURES, a["nz"], a["ny"], a["nx"]), device=DEV)
            fno.bvf_fno_features(a["index"], a["table"], a["table"][0], a["f0"], a["k_src"],
                                 a["plane"], P0, x)
        return st["net"](x)
    if path == "fno16":
        return st["net"].forward(st["x"])
    loss, grad = st["net"].gradient(st["x"], st["t"], st["el"], EL_WEIGHT)
    return dict(loss=loss, grad=grad)


# -------------------------------------------------------------------- its work
def _net_work(nx, ny, nz, b):
    n, w, L, h, m = nx * ny * nz, NET["width"], NET["n_layers"], NET["hidden"], NET["modes"]
    # weights, input and output, and each layer's volume written and read once
    by = 4.0 * _count(NET) + 4.0 * b * n * (NET["c_in"] + NET["c_out"] + w * (2 * L + 2))
    # channel products, and the truncated transforms as products along each axis
    fl = 2.0 * b * n * (w * NET["c_in"] + L * w * w + h * w + NET["c_out"] * h)
    spec = 2.0 * w * (n * 2 * m + nz * m * 4 * ny * 2 * m + 2 * m * m * 4 * nz * 2 * m)
    fl += b * L * (2 * spec + 8.0 * 4 * m ** 3 * w * w)
    return by, fl


def _fdtd_work(n, steps, window, storage):
    # velocities, stresses and memory variables read and written each step, the
    # material index and the peak map; the two FP64 sums inside the window
    st = 168.0 if storage == "f32" else 84.0
    return n * (steps * (st + 9.0) + 32.0 * window), 260.0 * n * steps


def work(case):
    path = case["path"]
    if path == "rs":
        lam = C0 / case["f0"]
        area = 2.0 * math.pi * 63e-3 * (63e-3 - math.sqrt(63e-3 ** 2 - 32e-3 ** 2))
        ne = 16.0 * area / lam ** 2
        pts = case["nx"] * case["ny"]
        return dict(bytes=8.0 * pts + 16.0 * ne, flops=25.0 * pts * ne)
    if path == "sweep":
        tot = [_fdtd_work(d["nx"] * d["ny"] * d["nz"], case["steps"], 16, "f32")
               for d in _sweep_domains(case)]
        return dict(bytes=sum(t[0] for t in tot), flops=sum(t[1] for t in tot))
    n = case["nx"] * case["ny"] * case["nz"]
    if path == "fdtd":
        by, fl = _fdtd_work(n, case["steps"], case["window"], case["storage"])
        return dict(bytes=by, flops=fl)
    if path == "plan":
        dt, per = _time_step(case["dx"], case["f0"], _table(case["f0"]))
        dft = case["cycles"] * per
        steps = int(math.ceil(1.3 * case["nz"] * case["dx"] / C0 / dt)) + dft
        by, fl = _fdtd_work(n, steps, dft, case["storage"])
        return dict(bytes=2 * by + 1200 * 29.0 * n, flops=2 * fl + 1200 * 40.0 * n)
    if path == "bhte":
        steps = case["n_on"] + case["n_off"]
        return dict(bytes=29.0 * n * steps, flops=40.0 * n * steps)
    by, fl = _net_work(case["nx"], case["ny"], case["nz"], case.get("batch", 1))
    if path == "train":
        return dict(bytes=3.0 * by, flops=3.0 * fl)
    return dict(bytes=by, flops=fl)


# ------------------------------------------------------- the same in 64 bits
def _fit(rho, c, alpha, f0, ts):
    """Relaxed modulus and strength of the standard linear solid whose Q at f0
    is w / (2 c alpha) and whose phase speed there is c."""
    if c == 0.0:
        return 0.0, 0.0
    if alpha <= 0.0:
        return rho * c * c, 0.0
    x = 2.0 * math.pi * f0 * ts
    q = 2.0 * math.pi * f0 / (2.0 * c * alpha)
    tau = 1.0 / (q * (x / (1 + x * x)).sum() - (x * x / (1 + x * x)).sum())
    m = 1.0 + tau * (1j * x / (1.0 + 1j * x)).sum()
    return rho * c * c * ((1.0 / np.sqrt(m)).real) ** 2, tau


def _cpml(n, dx, dt, f0, cmax, half):
    pos = 2.0 * np.arange(n) + (1.0 if half else 0.0)
    xi = np.maximum((2.0 * PML - pos) / (2.0 * PML), (pos - 2.0 * (n - 1 - PML)) / (2.0 * PML))
    inside = xi > 0.0
    xi = np.clip(xi, 0.0, 1.0)
    d = (-3.0 * cmax * np.log(1e-4) / (2.0 * PML * dx)) * xi * xi
    al = np.pi * f0 * (1.0 - xi)
    b = np.where(inside, np.exp(-(d + al) * dt), 0.0)
    a = np.where(inside & (d + al > 0.0), d * (b - 1.0) / np.where(d + al > 0.0, d + al, 1.0), 0.0)
    return a, b


def _fdtd64(a, steps, dft_start, dft_steps):
    """Velocity-stress steps with two-mechanism standard linear solids and CPML
    slabs on fields padded by two zero layers; returns p, peak, C and S."""
    nx, ny, nz, dx, dt, f0 = (a[k] for k in ("nx", "ny", "nz", "dx", "dt", "f0"))
    size, L = (nz, ny, nx), 2
    ts = 1.0 / (2.0 * np.pi * f0 * np.array([1.0 / 3.0, 3.0]))
    tab = np.asarray(a["table"], dtype=np.float64)
    fits = np.array([_fit(r[0], r[1], r[3], f0, ts) + _fit(r[0], r[2], r[4], f0, ts) for r in tab])
    dev = lambda v: torch.as_tensor(v, dtype=F64, device=DEV)  # noqa: E731
    idx = a["index"].long()
    rho, piR, tP, muR, tS = (dev(v)[idx] for v in (tab[:, 0], fits[:, 0], fits[:, 1], fits[:, 2],
                                                   fits[:, 3]))
    prof = {}
    for ax in range(3):
        for half in (False, True):
            ab = _cpml(size[ax], dx, dt, f0, tab[:, 1].max(), half)
            sh = [1, 1, 1]
            sh[ax] = size[ax]
            prof[ax, half] = [dev(v).reshape(sh) for v in ab]

    def cutv(t, cut):
        return t[tuple(slice(0, n - c) if n > 1 else slice(None) for n, c in zip(t.shape, cut))]

    def view(F, cut, ax=0, o=0):
        return F[tuple(slice(2 + (o if i == ax else 0), 2 + (o if i == ax else 0) + size[i] - cut[i])
                       for i in range(3))]

    def nxt(t, ax):
        return torch.cat([t.narrow(ax, 1, size[ax] - 1), t.narrow(ax, size[ax] - 1, 1)], ax)

    pad = [n + 4 for n in size]
    F = [torch.zeros(pad, dtype=F64, device=DEV) for _ in range(9)]
    vx, vy, vz, sxx, syy, szz, sxy, sxz, syz = F
    psi = [torch.zeros(size, dtype=F64, device=DEV) for _ in range(18)]
    mem = [[torch.zeros(size, dtype=F64, device=DEV) for _ in range(6)] for _ in range(L)]
    zero = (0, 0, 0)

    def der(f, ax, half, q, cut):
        o = (1, 0, 2, -1) if half else (0, -1, 1, -2)
        d = (view(f, cut, ax, o[0]) - view(f, cut, ax, o[1])) * (9.0 / 8.0 / dx)
        d.add_(view(f, cut, ax, o[2]) - view(f, cut, ax, o[3]), alpha=-1.0 / 24.0 / dx)
        ka, kb = (v.narrow(ax, 0, size[ax] - cut[ax]) for v in prof[ax, half])
        p = cutv(psi[q], cut)
        p.mul_(kb).addcmul_(d, ka)
        return d.add_(p)

    Z, Y, X = 0, 1, 2
    vel = [(vx, (0, 0, 1), 0, ((sxx, X, True), (sxy, Y, False), (sxz, Z, False)), X),
           (vy, (0, 1, 0), 3, ((sxy, X, False), (syy, Y, True), (syz, Z, False)), Y),
           (vz, (1, 0, 0), 6, ((sxz, X, False), (syz, Y, False), (szz, Z, True)), Z)]
    buoy = [cutv(dt * 2.0 / (rho + nxt(rho, ax)), cut) for _, cut, _, _, ax in vel]
    piU, muU = piR * (1 + L * tP), 2.0 * muR * (1 + L * tS)
    piT, muT = piR * tP, 2.0 * muR * tS
    shear = []
    for c, sig, cut, q, terms, ax1, ax2 in (
            (3, sxy, (0, 1, 1), 12, ((vx, Y), (vy, X)), X, Y),
            (4, sxz, (1, 0, 1), 14, ((vx, Z), (vz, X)), X, Z),
            (5, syz, (1, 1, 0), 16, ((vy, Z), (vz, Y)), Y, Z)):
        u = [muR, nxt(muR, ax1), nxt(muR, ax2), nxt(nxt(muR, ax1), ax2)]
        t = [tS, nxt(tS, ax1), nxt(tS, ax2), nxt(nxt(tS, ax1), ax2)]
        inv = sum(1.0 / v for v in u)
        muh = torch.where(torch.isfinite(inv), 4.0 / inv, torch.zeros_like(inv))
        tsh = 0.25 * sum(t)
        shear.append((c, sig, cut, q, terms, cutv(muh * (1 + L * tsh), cut).contiguous(),
                      cutv(muh * tsh, cut).contiguous()))
    hh = dt / (2.0 * ts)
    ca, cb = (1.0 - hh) / (1.0 + hh), (dt / ts) / (1.0 + hh)

    def relax(c, cut, psi_, the):
        for m in range(L):
            r = cutv(mem[m][c], cut)
            psi_.add_(r, alpha=0.5)
            r.mul_(ca[m]).add_(the, alpha=-cb[m])
            psi_.add_(r, alpha=0.5)
        return psi_

    A = torch.complex(a["plane"][..., 0].double(), a["plane"][..., 1].double())
    amp, ang = A.abs(), A.angle()
    w = 2.0 * math.pi * f0
    peak = torch.zeros(size, dtype=F64, device=DEV)
    C, S = torch.zeros_like(peak), torch.zeros_like(peak)
    for n in range(steps):
        for (f, cut, q, terms, _), b in zip(vel, buoy):
            d = sum(der(g, ax, half, q + i, cut) for i, (g, ax, half) in enumerate(terms))
            view(f, cut).addcmul_(d, b)
        e = [der(f, ax, False, 9 + i, zero) for i, (f, ax) in enumerate(((vx, X), (vy, Y), (vz, Z)))]
        th = e[0] + e[1] + e[2]
        t = (n + 0.5) * dt
        if a["env"] == 1:
            env = 1.0 if t < a["cycles"] / f0 else 0.0
        else:
            env = 0.5 * (1.0 - math.cos(math.pi * f0 * t)) if t < 1.0 / f0 else 1.0
        src = (2.0 * C0 * dt / dx) * env * amp * torch.sin(w * t + ang)
        for c, f in enumerate((sxx, syy, szz)):
            dv = th - e[c]
            view(f, zero).add_(relax(c, zero, piU * th - muU * dv, piT * th - muT * dv), alpha=dt)
            view(f, zero)[a["k_src"]].sub_(src)
        for c, f, cut, q, terms, pU, pT in shear:
            ev = der(terms[0][0], terms[0][1], True, q, cut) + der(terms[1][0], terms[1][1], True,
                                                                  q + 1, cut)
            view(f, cut).add_(relax(c, cut, pU * ev, pT * ev), alpha=dt)
        p = -(view(sxx, zero) + view(syy, zero) + view(szz, zero)) / 3.0
        peak = torch.maximum(peak, p.abs())
        if dft_steps and dft_start <= n + 1 < dft_start + dft_steps:
            C.add_(p, alpha=math.cos(w * (n + 1) * dt))
            S.add_(p, alpha=math.sin(w * (n + 1) * dt))
    return p, peak, C, S


def _bhte64(index, table, dx, amp, dt, n_on, n_off, duty):
    """Forward-Euler bioheat steps with harmonic-mean faces, borders at 37 C."""
    idx = index.long()
    col = lambda c: torch.as_tensor(table[:, c], dtype=F64, device=DEV)[idx]  # noqa: E731
    k, perf = col(5), col(7) * (1050.0 * 3617.0)
    src = col(8) * col(3) * amp ** 2 / (col(0) * col(1))
    gain = dt / (col(0) * col(6))
    faces = [2.0 * k.narrow(ax, 0, k.shape[ax] - 1) * k.narrow(ax, 1, k.shape[ax] - 1) /
             (k.narrow(ax, 0, k.shape[ax] - 1) + k.narrow(ax, 1, k.shape[ax] - 1)) / dx ** 2
             for ax in range(3)]
    inner = tuple(slice(1, -1) for _ in range(3))
    T = torch.full(k.shape, 37.0, dtype=F64, device=DEV)
    Tmax, cem = T.clone(), torch.zeros_like(T)
    for n in range(n_on + n_off):
        rhs = -perf * (T - 37.0)
        if n < n_on:
            rhs.add_(src, alpha=duty)
        for ax in range(3):
            m = k.shape[ax] - 1
            flux = faces[ax] * (T.narrow(ax, 1, m) - T.narrow(ax, 0, m))
            rhs.narrow(ax, 0, m).add_(flux)
            rhs.narrow(ax, 1, m).sub_(flux)
        T[inner] += (gain * rhs)[inner]
        Tmax = torch.maximum(Tmax, T)
        cem += dt / 60.0 * torch.where(T >= 43.0, torch.exp2(T - 43.0), torch.exp2(2.0 * (T - 43.0)))
    return T, Tmax, cem


def _rs64(bowl, nx, ny, dx, z, f0):
    """Rayleigh-Sommerfeld sum over the cap's elements of lambda^2 / 16."""
    a, R = 0.5 * bowl["aperture"], bowl["roc"]
    k = 2.0 * math.pi * f0 / C0
    ds = 0.25 * C0 / f0
    th = math.asin(a / R)
    nr = max(1, math.ceil(R * th / ds))
    u = np.array(bowl["dir"]) / np.linalg.norm(bowl["dir"])
    sn, cs = math.hypot(u[0], u[1]), u[2]
    ax = np.array([-u[1], u[0], 0.0]) / (sn if sn > 0 else 1.0)
    rows = []
    for r in range(nr):
        t0, t1 = th * r / nr, th * (r + 1) / nr
        tc = 0.5 * (t0 + t1)
        naz = max(1, int(math.floor(2.0 * math.pi * R * math.sin(tc) / ds + 0.5)))
        ph = 2.0 * math.pi * (np.arange(naz) + 0.5) / naz
        p = np.stack([R * math.sin(tc) * np.cos(ph), R * math.sin(tc) * np.sin(ph),
                      np.full(naz, R * (1.0 - math.cos(tc)))], 1)
        p = p * cs + np.cross(np.broadcast_to(ax, p.shape), p) * sn + ax * (p @ ax)[:, None] * (1.0 - cs)
        area = 2.0 * math.pi * R * R * (math.cos(t0) - math.cos(t1)) / naz
        rows.append(np.concatenate([p + np.array(bowl["apex"]), np.full((naz, 1), area)], 1))
    el = torch.as_tensor(np.concatenate(rows), dtype=F64, device=DEV)
    x = (torch.arange(nx, dtype=F64, device=DEV) * dx)[None, :, None]
    y = (torch.arange(ny, dtype=F64, device=DEV) * dx)[:, None, None]
    re = torch.zeros((ny, nx), dtype=F64, device=DEV)
    im = torch.zeros_like(re)
    for s in range(0, el.shape[0], 256):
        c = el[s:s + 256]
        r = torch.sqrt((x - c[:, 0]) ** 2 + (y - c[:, 1]) ** 2 + (z - c[:, 2]) ** 2)
        re += (c[:, 3] * torch.sin(k * r) / r).sum(-1)
        im += (c[:, 3] * torch.cos(k * r) / r).sum(-1)
    return torch.stack([re, im], -1) * (k * bowl["p0"] / (2.0 * math.pi))


def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x * math.sqrt(0.5)))


def _net64(w, x, net):
    """The network on [batch, c_in, nz, ny, nx] doubles; w: the flat blob."""
    W, m, L, H, co, ci = (net[k] for k in ("width", "modes", "n_layers", "hidden", "c_out", "c_in"))
    b, _, nz, ny, nx = x.shape
    pos = 0

    def take(*shape):
        nonlocal pos
        n = int(np.prod(shape))
        pos += n
        return w[pos - n:pos].reshape(shape)
    flat = lambda t: t.reshape(b, t.shape[1], -1)  # noqa: E731
    Wp, bp = take(W, ci), take(W)
    v = Wp @ flat(x) + bp[:, None]
    iz = torch.as_tensor([j if j < m else j - 2 * m + nz for j in range(2 * m)], device=DEV)
    iy = torch.as_tensor([j if j < m else j - 2 * m + ny for j in range(2 * m)], device=DEV)
    for l in range(L):
        R, Wl, bl = torch.view_as_complex(take(2 * m, 2 * m, m, W, W, 2)), take(W, W), take(W)
        vh = torch.fft.rfft(v.reshape(b, W, nz, ny, nx), dim=4)[..., :m]
        vh = torch.fft.fft(vh, dim=3)[:, :, :, iy]
        vh = torch.fft.fft(vh, dim=2)[:, :, iz]
        oh = torch.einsum("zykco,bczyk->bozyk", R, vh)
        full = torch.zeros((b, W, nz, 2 * m, m), dtype=oh.dtype, device=DEV)
        full = torch.fft.ifft(full.index_copy(2, iz, oh), dim=2)
        wide = torch.zeros((b, W, nz, ny, m), dtype=oh.dtype, device=DEV)
        wide = torch.fft.ifft(wide.index_copy(3, iy, full), dim=3)
        s = torch.fft.irfft(wide, n=nx, dim=4).reshape(b, W, -1)
        s = s + Wl @ v + bl[:, None]
        v = _gelu(s) if l < L - 1 else s
    Q1, q1, Q2, q2 = take(H, W), take(H), take(co, H), take(co)
    parts = [Q2 @ _gelu(Q1 @ c + q1[:, None]) + q2[:, None] for c in v.split(2 ** 20, dim=2)]
    return torch.cat(parts, 2).reshape(b, co, nz, ny, nx)


def _features64(a):
    idx = a["index"].long()
    nz, ny, nx = idx.shape
    t = torch.as_tensor(a["table"], dtype=F64, device=DEV)
    w = t[0]
    out = torch.zeros((8, nz, ny, nx), dtype=F64, device=DEV)
    out[0], out[1] = t[:, 1][idx] / w[1] - 1.0, t[:, 0][idx] / w[0] - 1.0
    out[2] = t[:, 3][idx] * w[1] / a["f0"]
    out[3, a["k_src"]], out[4, a["k_src"]] = (a["plane"][..., c].double() / P0 for c in (0, 1))
    for c, n, sh in ((5, nx, (1, 1, -1)), (6, ny, (1, -1, 1)), (7, nz, (-1, 1, 1))):
        out[c] = ((torch.arange(n, dtype=F64, device=DEV) + 0.5) / n).reshape(sh)
    return out


def _amp64(C, S, n):
    return 2.0 * torch.sqrt(C * C + S * S) / n


def exact(case, seed):
    path = case["path"]
    if path == "rs":
        return _rs64(_bowl(case, seed), case["nx"], case["ny"], case["dx"], (PML + 2) * case["dx"],
                     case["f0"])
    if path == "fdtd":
        n, w = case["steps"], case["window"]
        p, peak, C, S = _fdtd64(_acoustic(case, seed), n, n - w + 1, w)
        out = dict(pressure=p, peak=peak)
        if w:
            out["amp"], out["phase"] = _amp64(C, S, w), None   # the phase of a silent voxel is noise
        return out
    if path == "plan":
        a, n, dft, bowl = _plan_case(case, seed)
        a["plane"] = _rs64(bowl, a["nx"], a["ny"], a["dx"], a["k_src"] * a["dx"], a["f0"])
        _, peak, C, S = _fdtd64(a, n, n - dft + 1, dft)
        amp = _amp64(C, S, dft)
        wat = dict(a, index=torch.zeros_like(a["index"]), table=a["table"][:1])
        _, _, C, S = _fdtd64(wat, n, n - dft + 1, dft)
        aw = _amp64(C, S, dft)
        t = torch.as_tensor(a["table"], dtype=F64, device=DEV)
        Ia = amp ** 2 / (2.0 * (t[:, 0] * t[:, 1])[a["index"].long()])
        Iw = aw ** 2 / (2.0 * 1000.0 * 1500.0)
        zm = int(torch.argmax(Iw)) // (a["nx"] * a["ny"])
        el, iw = float(Ia[zm].sum() / Iw[zm].sum()), float(Iw.max())
        sc = math.sqrt(5.0e4 / (el * iw))
        _, Tmax, cem = _bhte64(a["index"], a["table"], a["dx"], sc * amp, 0.1, 400, 800, 0.3)
        return dict(peak=peak, amp=amp, Tmax=Tmax, cem43=cem, EL=el, TS=math.sqrt(el), z_m=zm,
                    Iw_max=iw, p_scale=sc)
    if path == "sweep":
        out = []
        for k, d in enumerate(_sweep_domains(case)):
            p, peak, C, S = _fdtd64(_acoustic(d, seed, k + 100), case["steps"], case["steps"] - 15, 16)
            out.append((p, peak, _amp64(C, S, 16)))
        return out
    if path == "bhte":
        index, table, amp = _heat(case, seed)
        T, Tmax, cem = _bhte64(index, table, case["dx"], amp, 0.1, case["n_on"], case["n_off"], 0.3)
        return dict(T=T, Tmax=Tmax, cem43=cem)
    q = _net_inputs(case, seed)
    w = _weights(seed, NET, path == "train").double()
    with torch.no_grad():
        if path == "fno":
            x = q["x"].double() if "x" in q else _features64(q["a"])
            return _net64(w, x[None], NET)[0]
        if path == "fno16":
            return _net64(w, q["x"].double(), NET)
    w.requires_grad_(True)
    out = _net64(w, q["x"].double(), NET)
    t = q["t"].double()
    b = t.shape[0]
    rel = torch.linalg.vector_norm((out[:, 0] - t).reshape(b, -1), dim=1) / \
        torch.linalg.vector_norm(t.reshape(b, -1), dim=1)
    loss = rel.mean() + EL_WEIGHT * ((out[:, 1].reshape(b, -1).mean(1) - q["el"].double()) ** 2).mean()
    loss.backward()
    return dict(loss=float(loss.detach()), grad=w.grad)
