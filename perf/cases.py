"""What this framework is measured on: time steps of the radiative-transfer
path through its public entry points (native.Grid and the calls it wraps), over
the sizes and options its workloads, tests and benchmark use.

A case describes one context (one box, or a batch of boxes), its medium,
sources and run options.  A pass is what a user's program does with it:

  * kind "evolve": from the stored state (checkpoint), `steps` time steps, then
    the four state fields read back, as a run that writes snapshots does;
  * kind "transport": one transport-only step of a packet-id window, the
    deposits left on the device for the exchange of a split step;
  * kind "exchange": the same, then another process's deposits added on the
    device, the per-cell update, and the state fields read back;
  * kind "noalloc": the allocation-free transport on the caller's buffers.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1101_4127_gb300 import inputs, native

KPC, MYR = inputs.KPC_CM, inputs.MYR_S

# values a case leaves out
DEFAULTS = dict(kind="evolve", nx=64, ny=0, nz=0, boxes=1, precision="mixed", medium="lognormal", sigma=1.0,
                nH=1e-3, cell_pc=6600.0 / 128, he=0.08, bins=8, T_source=1e5, isothermal=False, T0=100.0, thin=False,
                sources=100, ndot=0.0, packets=1_000_000, dt_myr=0.02, steps=1, periodic=False, f_rec=0.0, z=9.0,
                graph=False, per_pass=False)


def listed():
    return [
        # Test 0 of the paper: an isothermal Stroemgren sphere in the FP64 form, stepped and read
        # every step for its front radius; the smallest grid, where launches and latency count
        dict(name="stromgren_32_fp64", nx=32, precision="fp64", medium="uniform", cell_pc=6600.0 / 32, he=0.0, bins=1,
             isothermal=True, T0=1e4, sources=1, ndot=5e48, packets=100_000, dt_myr=0.5, z=-1.0),
        # Test 2 in the FP64 form (H+He, temperature evolving, 8 colours), at half the resolution
        dict(name="hhe_64_fp64", nx=64, precision="fp64", medium="uniform", cell_pc=6600.0 / 64, sources=1, ndot=5e48,
             packets=100_000, dt_myr=0.2, z=-1.0),
        # one small box of many-source runs, stepped alone: little work per step
        dict(name="small_box_32", nx=32, sources=20, packets=100_000),
        # Test 2 in the mixed form at its full size, a few steps between snapshots
        dict(name="hhe_128", nx=128, medium="uniform", sources=1, ndot=5e48, packets=10_000_000, dt_myr=0.2, steps=4,
             z=-1.0),
        # Test 3: a dense H II region around one hot source; stiff cells, many sub-steps each
        dict(name="cloudy_64", nx=64, medium="uniform", nH=0.9, cell_pc=2.0, he=0.1 / 0.9, T_source=6e4, sources=1,
             ndot=6.4e48, packets=6_666_667, dt_myr=0.02, steps=3, z=-1.0),
        # Test 4: 1000 sources in a 128^3 density field, the full 2e8 packets of a step; the largest
        dict(name="lognormal_128", nx=128, sources=1000, packets=200_000_000),
        # the optically thin large field (the benchmark's workload at 256^3): transport of a window
        dict(name="thin_256_transport", kind="transport", nx=256, sigma=1.5, nH=2e-4, cell_pc=27902.0, thin=True,
             sources=2000, packets=64_000_000, dt_myr=0.1),
        # a process of a split step: transport, the deposits of another one added, per-cell update; ragged sizes
        dict(name="exchange_ragged", kind="exchange", nx=97, ny=61, nz=113, thin=True, sources=50, packets=2_000_000,
             dt_myr=0.1),
        # independent boxes of several sizes stepped together, each step one replay of a graph
        dict(name="batch_graph", nx=32, boxes=12, sources=30, packets=6_000_000, graph=True, steps=2),
        # Test 1: the diffuse recombination field, cells re-emitting from the second step on
        dict(name="recombination_64", nx=64, medium="uniform", cell_pc=6600.0 / 64, he=0.0, bins=1, isothermal=True,
             T0=1e4, sources=1, ndot=5e48, packets=1_000_000, dt_myr=25.0, steps=5, f_rec=0.1, z=-1.0),
        # a periodic box with a number of colours that has no kernel of its own
        dict(name="periodic_48", nx=48, bins=5, thin=True, sources=10, packets=500_000, periodic=True,
             dt_myr=0.015),
        # transport inside another program's memory: no allocation, caller's absorbers and deposits
        dict(name="noalloc_64", kind="noalloc", nx=64, thin=True, sources=64, packets=1_024_000),
    ]


def draw(rng):
    """One more case of the ranges above."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    shape = rng.choice(["evolve", "evolve", "evolve", "fp64", "transport", "exchange", "batch", "rec", "periodic", "noalloc"])
    nx = log_int(16, 160)
    c = dict(nx=nx, ny=max(1, int(nx * rng.uniform(0.5, 1.2))), nz=max(1, int(nx * rng.uniform(0.5, 1.2))),
             sources=log_int(1, 1000), thin=rng.random() < 0.4, sigma=round(rng.uniform(0.5, 1.5), 3),
             bins=rng.choice([1, 3, 8, 8, 8, 8, 12]), packets=log_int(2e4, 2e7), dt_myr=round(rng.uniform(0.01, 0.1), 4))
    if shape == "fp64":
        c.update(precision="fp64", nx=log_int(16, 64), ny=0, nz=0, packets=log_int(1e4, 2e5))
    elif shape in ("transport", "exchange", "noalloc"):
        c.update(kind=shape)
        if shape == "noalloc":
            c.update(nx=log_int(16, 96), ny=0, nz=0, packets=log_int(2e4, 2e6))
    elif shape == "batch":
        c.update(boxes=rng.randint(2, 12), nx=rng.choice([16, 32]), ny=0, nz=0, graph=rng.random() < 0.5)
    elif shape == "rec":
        c.update(medium="uniform", he=0.0, bins=1, isothermal=True, T0=1e4, sources=1, ndot=5e48, f_rec=0.1, dt_myr=25.0,
                 thin=False, nx=log_int(16, 96), ny=0, nz=0, steps=rng.randint(2, 5), packets=log_int(2e4, 2e6))
    elif shape == "periodic":
        c.update(periodic=True, nx=log_int(16, 64), ny=0, nz=0, packets=log_int(2e4, 5e5), dt_myr=0.01)
    else:
        c.update(steps=rng.randint(1, 3), isothermal=rng.random() < 0.2, he=rng.choice([0.0, 0.08, 0.08]),
                 per_pass=rng.random() < 0.25)
    return c


# ---------------------------------------------------------------- inputs
def _full(case):
    c = {**DEFAULTS, **case}
    c["ny"], c["nz"] = c["ny"] or c["nx"], c["nz"] or c["nx"]
    return c


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _lognormal(nx, ny, nz, sigma, mean, seed):
    """Seeded lognormal density of log-scatter sigma and power P(k) ~ k^-2.5, float32 [z, y, x]."""
    dev = _device()
    g = torch.Generator(device=dev).manual_seed(seed)
    f = torch.fft.rfftn(torch.randn((nz, ny, nx), generator=g, device=dev, dtype=torch.float64))
    k = [torch.fft.fftfreq(nz, device=dev)[:, None, None], torch.fft.fftfreq(ny, device=dev)[None, :, None],
         torch.fft.rfftfreq(nx, device=dev)[None, None, :]]
    k2 = sum(x.double() ** 2 for x in k)
    k2[0, 0, 0] = 1.0
    amp = k2 ** -0.625
    amp[0, 0, 0] = 0.0
    w = torch.fft.irfftn(f * amp, s=(nz, ny, nx))
    w = (w - w.mean()) / w.std()
    rho = torch.exp(sigma * w)
    return (rho * (mean / rho.mean())).float()


def _spectrum(bins, T):
    if bins == 1:
        return np.array([13.6 if T == 1e5 else 20.0]), np.array([1.0])
    edges = None if bins == 8 else np.geomspace(13.6, 200.0, bins + 1)
    return inputs.blackbody_bins(T, edges)


def _boxes(c, seed):
    """The case's boxes and packets per box and step, as a user's program sets them up."""
    rng = np.random.default_rng(seed)
    E, frac = _spectrum(c["bins"], c["T_source"])
    boxes, packets = [], []
    for b in range(c["boxes"]):
        m = 1 if c["boxes"] == 1 else (2, 3, 4, 6, 8)[(b * 3) % 5] / 2      # batches: sizes nx .. 4 nx
        nx, ny, nz = (max(1, int(c[a] * m)) for a in ("nx", "ny", "nz"))
        n_src = c["sources"] if c["boxes"] == 1 else int(rng.integers(1, c["sources"] + 1))
        n_src = min(n_src, nx * ny * nz)
        if c["medium"] == "uniform":
            nH, pos = None, np.zeros((1, 3)) if c["nH"] < 0.1 else np.array([[nx / 2, ny / 2, nz / 2]])
        else:
            d = _lognormal(nx, ny, nz, c["sigma"], c["nH"], 1000 * (seed + 1) + b)
            lin = torch.topk(d.reshape(-1), n_src).indices.cpu().numpy()
            nH, pos = d.cpu().numpy(), inputs.cell_centres(lin, nx, ny)
        if c["ndot"]:
            ndot = c["ndot"] * rng.uniform(0.8, 1.25, len(pos))
        else:
            ndot = inputs.powerlaw_luminosities(len(pos), 1e46, 1e50, int(rng.integers(1 << 30)))
        boxes.append(inputs.Box(
            n=nx, dims=(nx, ny, nz), box_cm=c["cell_pc"] * 1e-3 * KPC * nx, nH=nH, nH0=c["nH"], he_over_h=c["he"],
            x_HII0=1 - 1e-4 if c["thin"] else 1.2e-3, x_HeII0=1e-4 if c["thin"] and c["he"] else 0.0,
            x_HeIII0=1 - 2e-4 if c["thin"] and c["he"] else 0.0, T0=1e4 if c["thin"] else c["T0"],
            isothermal=int(c["isothermal"]), caseB=0 if c["f_rec"] else 1, z_compton=c["z"],
            seed=int(rng.integers(1 << 62)), src_pos=pos, src_ndot=ndot, bin_eV=E,
            bin_frac=np.tile(frac, (len(pos), 1)), f_rec=c["f_rec"], periodic=int(c["periodic"])))
        share = c["packets"] // c["boxes"]
        packets.append(max(1, share // len(pos)) * len(pos))
    return boxes, packets


class _DeviceArray:
    """A context's device buffer as an array; keeps the context alive."""

    def __init__(self, grid, ptr, cells):
        self.grid = grid
        self.__cuda_array_interface__ = {"shape": (cells, 4), "typestr": "<i8", "data": (ptr, False), "version": 2}


class _State:
    pass


def prepare(case, seed):
    c = _full(case)
    s = _State()
    s.case, s.dt = c, c["dt_myr"] * MYR
    s.boxes, packets = _boxes(c, seed)
    s.packets = packets[0] if c["boxes"] == 1 else packets
    if c["kind"] == "noalloc":
        return _prepare_noalloc(s)
    g = s.grid = native.Grid(s.boxes, native.CRASH_FP64_PLAIN if c["precision"] == "fp64" else native.CRASH_MIXED)
    opts = {}
    if c["graph"]:
        opts["use_graph"] = 1
    if c["per_pass"]:
        opts.update(persistent=0, reg_cap=1)
    if c["kind"] in ("transport", "exchange"):       # this process's half of the packet ids
        per_source = s.packets // s.boxes[0].n_src
        opts.update(chemistry=0, pkt_begin=0, pkt_end=max(1, per_source // 2))
    g.set_options(**opts)
    s.deposits = [torch.as_tensor(_DeviceArray(g, *g.deposits_device(b)), device="cuda") for b in range(c["boxes"])]
    if c["kind"] == "exchange":
        # the other process's deposits: the other half of the packet ids, traced on the same state
        other = native.Grid(s.boxes, native.CRASH_MIXED)
        other.set_options(chemistry=0, pkt_begin=max(1, per_source // 2))
        other.step(s.dt, s.packets)
        s.peer = torch.from_numpy(other.read_deposits()).cuda()
        other.close()
        s.stream = torch.cuda.ExternalStream(g.stream())
    if c["kind"] != "transport":
        g.checkpoint(native.CKPT_SAVE)
        # snapshots go to pinned host memory, as in the benchmark's end-to-end line
        s.fields = [[torch.zeros(b.shape_xyz[::-1], dtype=torch.float64, pin_memory=True) for _ in range(4)]
                    for b in s.boxes]
    return s


def _prepare_noalloc(s):
    b = s.boxes[0]
    cells = int(np.prod(b.shape_xyz))
    nH = torch.from_numpy(b.nH.reshape(-1)).cuda()
    s.absorbers = torch.zeros((cells, 4), dtype=torch.float32, device="cuda")
    s.absorbers[:, 0] = nH * (1.0 - b.x_HII0)
    s.absorbers[:, 1] = nH * b.he_over_h * ((1.0 - b.x_HeII0) - b.x_HeIII0)
    s.absorbers[:, 2] = nH * b.he_over_h * b.x_HeII0
    s.out = torch.zeros((cells, 4), dtype=torch.int64, device="cuda")
    s.desc = native.make_desc(b, native.CRASH_MIXED)
    s.arrays = [np.ascontiguousarray(a, np.float64).reshape(-1) for a in (b.src_pos, b.src_ndot, b.bin_eV, b.bin_frac)]
    return s


# ---------------------------------------------------------------- a pass
def run(s):
    kind = s.case["kind"]
    if kind == "noalloc":
        return _run_noalloc(s)
    g = s.grid
    if kind == "transport":
        g.step(s.dt, s.packets)
        return {"deposits": s.deposits}
    g.checkpoint(native.CKPT_RESTORE)
    if kind == "exchange":
        g.step(s.dt, s.packets)
        with torch.cuda.stream(s.stream):
            s.deposits[0].add_(s.peer)
        g.chemistry(s.dt)
    else:
        for _ in range(s.case["steps"]):
            g.step(s.dt, s.packets)
    for b, out in enumerate(s.fields):
        for f, a in zip((native.F_XHII, native.F_XHEII, native.F_XHEIII, native.F_T), out):
            st = g.L.crash_read_fields_box(g.ctx, b, f, a.data_ptr())
            if st != native.CRASH_OK:
                raise native.CrashError(st, g.L.crash_last_error(g.ctx).decode())
    return {"deposits": s.deposits, "state": s.fields}


def _run_noalloc(s):
    dp = ctypes.POINTER(ctypes.c_double)
    pos, ndot, E, frac = (a.ctypes.data_as(dp) for a in s.arrays)
    s.out.zero_()
    budget = np.zeros(8, np.int64)
    lib = native.lib()
    st = lib.crash_transport_noalloc(
        ctypes.byref(s.desc), s.boxes[0].n_src, pos, ndot, len(s.arrays[2]), E, frac, s.dt, 3, s.packets, 0,
        s.absorbers.data_ptr(), s.out.data_ptr(), budget.ctypes.data_as(ctypes.POINTER(ctypes.c_int64)),
        torch.cuda.current_stream().cuda_stream)
    if st != native.CRASH_OK:
        raise native.CrashError(st, lib.crash_noalloc_last_error().decode())
    return {"deposits": s.out, "budget": budget}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes: each cell's density, state and deposits once per step (read, and written where updated), each packet's
    photons nowhere (they are made and used on the chip).  Flops: per crossing and colour the optical depth, the
    attenuation and the species and heating sums (about 30), and per cell one sub-step of the network (about 400)."""
    c = _full(case)
    scale = 1.0 if c["boxes"] == 1 else sum(((2, 3, 4, 6, 8)[(b * 3) % 5] / 2) ** 3 for b in range(c["boxes"]))
    cells = c["nx"] * c["ny"] * c["nz"] * scale
    side = (c["nx"] * c["ny"] * c["nz"]) ** (1 / 3) * (1.0 if c["boxes"] == 1 else (scale / c["boxes"]) ** (1 / 3))
    path = c["dt_myr"] * 0.3066e6 / c["cell_pc"] * 1.5 if c["periodic"] else 0.9 * side
    if c["bins"] == 1 and not c["thin"]:
        path = min(path, 25.0)                       # one soft colour in a neutral medium: soon absorbed
    steps, packets = c["steps"], c["packets"] * (0.5 if c["kind"] in ("transport", "exchange") else 1.0)
    chem = c["kind"] in ("evolve", "exchange")
    per_cell = (16 + 32) if c["kind"] == "noalloc" else (4 + 24 + 32) + ((8 + 32) if chem else 0)
    return {"bytes": steps * cells * per_cell, "flops": steps * (packets * path * c["bins"] * 30.0 + (cells * 400.0 if chem else 0.0))}


# ---------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    """The state fields after the pass with photons as 64-bit numbers: directions from Philox-4x32-10, the cell walk,
    Eq. 1 of the paper in every cell, and the sub-stepped network.  Deposits are whole numbers and have none."""
    c = _full(case)
    boxes, packets = _boxes(c, seed)
    if c["kind"] not in ("evolve", "exchange") or c["f_rec"] or sum(packets) * c["steps"] > 3_000_000:
        return None
    state = []
    for box, p in zip(boxes, packets):
        med = _Medium(box)
        for step in range(c["steps"]):
            dep, heat = med.transport(step, c["dt_myr"] * MYR, p)
            med.chemistry(dep, heat, c["dt_myr"] * MYR)
        nx, ny, nz = box.shape_xyz
        state.append([f.reshape(nz, ny, nx).cpu().numpy() for f in (med.x, med.y2, med.y3, med.T)])
    return {"deposits": [None] * len(boxes), "state": state}


def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 of int64 tensors holding 32-bit words."""
    m32 = 0xFFFFFFFF

    def mul(a, x):
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        return (hi + (lo >> 16)) >> 16, (lo + ((hi & 0xFFFF) << 16)) & m32

    k0, k1 = seed & m32, seed >> 32
    for _ in range(10):
        ha, la = mul(0xD2511F53, c0)
        hb, lb = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = hb ^ c1 ^ k0, lb, ha ^ c3 ^ k1, la
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c0, c1, c2, c3


def _directions(seed, step, src, pkt):
    """Isotropic unit vectors (Marsaglia 1972), one Philox counter per attempt."""
    d = torch.zeros((len(src), 3), dtype=torch.float64, device=src.device)
    todo = torch.arange(len(src), device=src.device)
    for attempt in range(64):
        if not len(todo):
            break
        s, p = src[todo], pkt[todo]
        w = _philox(p, s, torch.full_like(s, step), torch.full_like(s, attempt), seed)
        v = [2.0 * (((w[2 * i + 1] << 21) | (w[2 * i] >> 11)).double() * 2.0 ** -53) - 1.0 for i in (0, 1)]
        q = v[0] * v[0] + v[1] * v[1]
        ok = (q < 1) & (q != 0)
        r = torch.sqrt((1 - q).clamp(min=0))
        d[todo[ok]] = torch.stack([2 * v[0] * r, 2 * v[1] * r, 1 - 2 * q], 1)[ok]
        todo = todo[~ok]
    return d


class _Medium:
    """One box in 64 bits: absorbers, transport of a step, network and temperature."""

    ETH = (13.6, 24.6, 54.4)
    EV, KB = 1.602176634e-12, 1.380649e-16

    def __init__(self, box):
        dev = _device()
        nx, ny, nz = self.dims = box.shape_xyz
        n = nx * ny * nz
        self.box, self.dl = box, box.box_cm / nx
        nH = np.full(n, box.nH0, np.float32) if box.nH is None else box.nH.reshape(-1)
        self.nH = torch.from_numpy(nH).to(dev).double()
        self.nHe = self.nH * box.he_over_h
        self.x, self.y2, self.y3, self.T = (torch.full_like(self.nH, v) for v in (box.x_HII0, box.x_HeII0, box.x_HeIII0, box.T0))
        e = np.asarray(box.bin_eV, np.float64)
        y = e / 24.6
        sig = [6.30e-18 * (13.6 / e) ** 3, 7.83e-18 * (1.66 * y ** -2.05 - 0.66 * y ** -3.05), 1.58e-18 * (54.4 / e) ** 3]
        above = [e >= t for t in self.ETH]
        self.sigma = torch.tensor(np.array([np.where(a, s, 0.0) for a, s in zip(above, sig)]), device=dev)
        self.excess = torch.tensor(np.array([np.where(a, e - t, 0.0) for a, t in zip(above, self.ETH)]), device=dev)

    def transport(self, step, dt, packets):
        """Absorbed photons [cells, 3] and excess energy [cells] (eV) of a step."""
        b, dev = self.box, self.nH.device
        n = torch.tensor(self.dims, device=dev)
        absorb = torch.stack([self.nH * (1 - self.x), self.nHe * ((1 - self.y2) - self.y3), self.nHe * self.y2], 1)
        dep = torch.zeros((len(self.nH), 3), dtype=torch.float64, device=dev)
        heat = torch.zeros(len(self.nH), dtype=torch.float64, device=dev)
        per = packets // b.n_src
        src = torch.arange(b.n_src, device=dev).repeat_interleave(per)
        d = _directions(b.seed, step, src, torch.arange(per, device=dev).repeat(b.n_src))
        frac = torch.tensor(np.asarray(b.bin_frac)[:, :-1], device=dev)
        frac = torch.cat([frac, 1 - frac.sum(1, keepdim=True)], 1)
        N = (torch.tensor(np.asarray(b.src_ndot), device=dev)[:, None] * dt / per * frac)[src]
        N0 = N.sum(1)
        pos = torch.tensor(np.asarray(b.src_pos, np.float64), device=dev)[src]
        cell = pos.floor().long()
        fwd = d > 0
        t_max = torch.where(d != 0, (cell + fwd - pos) / d, math.inf)
        t_step = torch.where(d != 0, 1 / d.abs(), math.inf)
        sign = torch.where(fwd, 1, torch.where(d < 0, -1, 0))
        now = torch.zeros(len(src), dtype=torch.float64, device=dev)
        limit = 2.99792458e10 * dt / self.dl if b.periodic else math.inf
        while len(N):
            t, axis = t_max.min(1)
            t = t.clamp(max=limit)
            length = (t - now) * self.dl
            at = cell[:, 0] + self.dims[0] * (cell[:, 1] + self.dims[1] * cell[:, 2])
            tau_s = length[:, None, None] * absorb[at][:, :, None] * self.sigma       # [packet, species, colour]
            tau = tau_s.sum(1)
            over = torch.where(tau > 0, -torch.expm1(-tau) / tau, 1.0)
            A = N[:, None, :] * over[:, None, :] * tau_s
            dep.index_add_(0, at, A.sum(2))
            heat.index_add_(0, at, (A * self.excess).sum((1, 2)))
            N = N * torch.exp(-tau)
            pick = torch.nn.functional.one_hot(axis, 3).bool()
            t_max = torch.where(pick, t_max + t_step, t_max)
            cell = cell + torch.where(pick, sign, 0)
            now = t
            if b.periodic:
                cell = torch.remainder(cell, n)
                keep = now < limit
            else:
                keep = ((cell >= 0) & (cell < n)).all(1)
            keep &= N.sum(1) > 1e-18 * N0
            cell, t_max, t_step, sign, now, N, N0 = (v[keep] for v in (cell, t_max, t_step, sign, now, N, N0))
        return dep, heat

    def rates(self, T):
        """Recombination and collisional ionisation coefficients and cooling coefficients at T."""
        lH, l1, l2 = 315614.0 / T, 570670.0 / T, 1263030.0 / T
        sq = 1 / (1 + torch.sqrt(T / 1e5))
        if self.box.caseB:
            def a(l):
                return 2.753e-14 * l ** 1.5 / (1 + (l / 2.740) ** 0.407) ** 2.242

            def cool(l, t):
                return 3.435e-30 * t * l ** 1.970 / (1 + (l / 2.250) ** 0.376) ** 3.720
            a2 = 1.26e-14 * l1 ** 0.750
        else:
            def a(l):
                return 1.269e-13 * l ** 1.503 / (1 + (l / 0.522) ** 0.470) ** 1.923

            def cool(l, t):
                return 1.778e-29 * t * l ** 1.965 / (1 + (l / 0.541) ** 0.502) ** 2.697
            a2 = 3.0e-14 * l1 ** 0.654
        di = 1.90e-3 * T ** -1.5 * torch.exp(-470000.0 / T) * (1 + 0.3 * torch.exp(-94000.0 / T))
        rt = torch.sqrt(T)
        b = [k * rt * torch.exp(-t / T) * sq for k, t in ((5.85e-11, 157809.1), (2.38e-11, 285335.4), (5.68e-12, 631515.0))]
        gff = 1.1 + 0.34 * torch.exp(-(5.5 - torch.log10(T)) ** 2 / 3.0)
        cff = 1.42e-27 * gff * rt
        ion = [t * self.EV * v for t, v in zip(self.ETH, b)]
        c_HI = 7.50e-19 * torch.exp(-118348.0 / T) * sq + ion[0]
        c_HII = cool(lH, T) + cff
        c_HeII = 5.54e-17 * T ** -0.397 * torch.exp(-473638.0 / T) * sq + ion[2] + self.KB * T * a2 + 6.526e-11 * di + cff
        c_HeIII = 8 * cool(l2, 0.25 * T) + 4 * cff
        return a(lH), a2 + di, 2 * a(l2), b, (c_HI, c_HII, ion[1], c_HeII, c_HeIII)

    def chemistry(self, dep, heat, dt, eps=0.1, max_sub=10000):
        """Sub-stepped backward Euler of H and He and the semi-implicit temperature, every cell its own sub-steps."""
        b = self.box
        V = (self.dl * self.dl) * self.dl
        neutral = torch.stack([self.nH * (1 - self.x), self.nHe * ((1 - self.y2) - self.y3), self.nHe * self.y2], 1) * V
        G = torch.where(neutral > 0, dep / (dt * neutral), 0.0)
        absorbed = dep.sum(1)
        e_heat = torch.where(absorbed > 0, heat / absorbed, 0.0) * self.EV
        Tc = 2.725 * (1 + b.z_compton) if b.z_compton >= 0 else 0.0
        comp = 4 * 6.6524587321e-25 * 7.565723e-15 * Tc ** 4 * self.KB / (9.1093837015e-28 * 2.99792458e10)
        at = torch.arange(len(self.nH), device=self.nH.device)
        rem = torch.full_like(self.nH, dt)
        tiny = torch.tensor(1e-3, dtype=torch.float64, device=rem.device)
        helium = b.he_over_h > 0
        nsub = 0
        while len(at):
            nH, nHe, x, y2, y3, T, g, eh, r = (v[at] for v in (self.nH, self.nHe, self.x, self.y2, self.y3, self.T, G, e_heat, rem))
            y1 = (1 - y2) - y3
            aH, a2, a3, bc, cool = self.rates(T)

            def n_e(x, y2, y3):
                return nH * x + nHe * (y2 + 2 * y3)

            def heating(x, y1, y2):
                return eh * (g[:, 0] * nH * (1 - x) + g[:, 1] * nHe * y1 + g[:, 2] * nHe * y2)

            def cooling(ne, x, y1, y2, y3):
                return ne * (nH * (cool[0] * (1 - x) + cool[1] * x) + nHe * (cool[2] * y1 + cool[3] * y2 + cool[4] * y3))

            ne = n_e(x, y2, y3)
            dx = (g[:, 0] + bc[0] * ne) * (1 - x) - aH * ne * x
            d1 = -(g[:, 1] + bc[1] * ne) * y1 + a2 * ne * y2
            d3 = (g[:, 2] + bc[2] * ne) * y2 - a3 * ne * y3
            h = r.clone()
            for v, dv in ([(1 - x, dx), (x, dx)] + ([(y1, d1), (y2, d1 + d3), (y3, d3)] if helium else [])):
                h = torch.minimum(h, eps * torch.maximum(v, tiny) / dv.abs())
            n_tot = nH + nHe + ne
            if not b.isothermal:
                net = heating(x, y1, y2) - cooling(ne, x, y1, y2, y3) - comp * ne * (T - Tc)
                dT = (net / (1.5 * self.KB) - T * (nH * dx + nHe * (-d1 - d3 + 2 * d3))) / n_tot
                h = torch.minimum(h, eps * T / dT.abs())
            last = ~(h < r) | (nsub == max_sub - 1)
            h = torch.where(last, r, h)
            xn, z1, z2, z3, m = x, y1, y2, y3, ne
            for _ in range(4):
                xn = (x + h * (g[:, 0] + bc[0] * m)) / (1 + h * (g[:, 0] + bc[0] * m + aH * m))
                if helium:
                    i1, i2, r2, r3 = h * (g[:, 1] + bc[1] * m), h * (g[:, 2] + bc[2] * m), h * a2 * m, h * a3 * m
                    w = 1 + i1
                    p = 1 + r2 + i2 - i1 * r2 / w
                    q = (y2 + i1 * y1 / w) / p
                    z3 = (y3 + i2 * q) / (1 + r3 - i2 * r3 / p)
                    z2 = q + r3 / p * z3
                    z1 = (y1 + r2 * z2) / w
                m = n_e(xn, z2, z3)
            xn = xn.clamp(0, 1)
            if helium:
                z1, z2, z3 = z1.clamp(min=0), z2.clamp(min=0), z3.clamp(min=0)
                total = z1 + z2 + z3
                z2, z3 = z2 / total, z3 / total
                z1 = (1 - z2) - z3
            m = n_e(xn, z2, z3)
            if not b.isothermal:
                L, k = cooling(m, xn, z1, z2, z3), 1.5 * self.KB
                self.T[at] = (k * n_tot * T + h * (heating(xn, z1, z2) + comp * m * Tc)) / (k * (nH + nHe + m) + h * comp * m + h * L / T)
            self.x[at], self.y2[at], self.y3[at], rem[at] = xn, z2, z3, torch.where(last, 0.0, r - h)
            at = at[~last]
            nsub += 1
