"""The library's work as its users have it done, for timing: windows of hysteresis-loop ensembles at
every coarse-graining level, whole loops with their statistics, the uneven batch, the periodic slab and
the calibration gradient, each through the Python package.

A window (`kind` "window") is what a resumable run does between two checkpoints: the ensemble's state
goes in with its step number, the ensemble advances, the state and the samples taken come out.
"""
import math

import numpy as np
import torch

import paper_1912_00310_gb300 as llg

# magnetite rod of 8 x 24 x 56 cells of a0, the time step of each level b
A0_M, EXCHANGE, MS, K0, T_K, TC_K, DELTA = 0.839e-9, 0.98e-11, 480e3, 10e3, 310.0, 858.0, 0.511
RODS = {1: (8, 24, 56), 2: (4, 12, 28), 4: (2, 6, 14), 8: (1, 3, 7), 22: (1, 1, 1)}
DT = {1: 2e-15, 2: 5e-15, 4: 10e-15, 8: 20e-15, 22: 20e-15}
BLOCK_VOLUME = 8 * 24 * 56 * A0_M ** 3  # b = 22: the whole rod as one prism

LADDER_BS, LADDER_RATES, LADDER_ALPHAS = (1, 2, 4, 8), (1000.0, 100.0, 10.0), (0.05, 0.1, 0.5, 1.0)

# 32-bit operations of the method per cell and Heun step (noise 130, two fields 40, two torques 30,
# predictor and corrector with their normalisations 21)
OPS_PER_CELL_STEP = 221


def _window(name, b, n_real, steps, **kw):
    nx, ny, nz = kw.pop("dims", RODS[b])
    c = dict(kind="window", b=b, nx=nx, ny=ny, nz=nz, n_real=n_real, steps=steps, step0=0, periodic=0, shape=0,
             disp_deg=0.0, rate=1000.0, H=1500.0, sample_dH=1.0, alpha=0.1, mode=1)
    if name:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # the full-resolution rod, 256 realisations in one persistent launch (the benchmark's workload)
        _window("rod_b1_256", 1, 256, 1000),
        # the paper's protocol at full resolution: sinusoid, 5 degree axis dispersion, one rod per SM,
        # resumed in mid-cycle
        _window("rod_b1_protocol", 1, 152, 400, shape=1, disp_deg=5.0, rate=5.0, H=500.0, alpha=0.2, mode=2,
                step0=9_999_800),
        # the protocol at b = 2
        _window("rod_b2_protocol", 2, 256, 2000, shape=1, disp_deg=5.0, rate=2.5, H=500.0, mode=2, step0=15_999_000),
        # a large ensemble of the b = 4 rod
        _window("rod_b4_608", 4, 608, 5000),
        # the protocol's large ensemble at b = 8
        _window("rod_b8_protocol", 8, 4096, 2000, shape=1, disp_deg=5.0, rate=2.5, H=500.0, mode=2, step0=3_999_000),
        # the single-block limit: the rod as one macrospin
        _window("block_b22_4096", 22, 4096, 3000, shape=1, disp_deg=5.0, rate=2.5, H=500.0, mode=2, step0=3_999_000),
        # four realisations of a whole loop into host memory with the loop's statistics: the smallest ensemble
        dict(name="loops_b4_4", kind="loops", b=4, n_real=4, H=100.0, rate=10000.0, sample_dH=1.0, alpha=0.5, mode=1),
        # a rod outside the paper's ladder (odd sizes), equilibrium in a held field
        _window("rod_odd_held", 2, 152, 1500, dims=(5, 11, 23), rate=0.0, H=200.0, sample_dH=100.0),
        # the uneven batch: b x rate x alpha, 64 realisations each, one launch
        dict(name="ladder_batch", kind="batch", b=0, n_real=64, steps=400, H=1500.0, sample_dH=1.0, mode=1),
        # the periodic film that exceeds on-chip memory
        _window("slab_512x512x56", 1, 1, 24, dims=(512, 512, 56), periodic=3, step0=480),
        # a smaller film with odd sides
        _window("slab_odd", 1, 2, 60, dims=(201, 139, 17), periodic=3, step0=470),
        # calibration: loss of a window's mean loop and its gradient in the three scale factors
        dict(name="calibration_b4", kind="calibration", b=4, n_real=64, steps=CALIB_STEPS, method=0,
             H=1500.0, rate=1000.0, sample_dH=1.0, alpha=0.1, mode=1, ckpt_every=512),
    ]


CALIB_STEPS = 2000


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.random()
    if what < 0.1:
        b = rng.choice((4, 8))
        return dict(kind="loops", b=b, n_real=_log_int(rng, 1, 64), H=10.0 * rng.randint(b, 4 * b), rate=10000.0,
                    sample_dH=1.0, alpha=rng.choice((0.5, 1.0)), mode=rng.choice((1, 2)))
    if what < 0.25:
        method = rng.randint(0, 1)
        return dict(kind="calibration", b=rng.choice((4, 8)), n_real=_log_int(rng, 4, 64),
                    steps=100 * rng.randint(6, CALIB_STEPS // 100), method=method,
                    H=1500.0, rate=1000.0, sample_dH=1.0, alpha=0.1, mode=1, ckpt_every=rng.choice((128, 300, 512)))
    if what < 0.3:
        return dict(kind="batch", b=0, n_real=_log_int(rng, 3, 64), steps=_log_int(rng, 20, 400), H=1500.0,
                    sample_dH=1.0, mode=1)
    if what < 0.45:
        dims = (rng.randint(24, 512), rng.randint(24, 512), rng.randint(8, 56))
        return _window(None, 1, 1, _log_int(rng, 4, 24), dims=dims, periodic=3, step0=480)
    protocol = rng.random() < 0.4
    b = rng.choice((1, 1, 2, 4, 8, 22) if protocol else (1, 1, 2, 4, 8, 0))
    if b == 0:  # a rod outside the ladder
        b, dims = 2, (rng.randint(1, 8), rng.randint(2, 16), rng.randint(3, 30))
    else:
        dims = RODS[b]
    cells = math.prod(dims)
    # up to the largest listed case's cell-steps; at most 4096 realisations
    n_real = _log_int(rng, 1, max(4, min(4096, 2_700_000 // cells)))
    steps = max(50, min(_log_int(rng, 100, 3000), int(1.5e9 / (cells * n_real))))
    if protocol:
        per_sample = int(round(1.0 / (2.5e9 * DT[b])))
        return _window(None, b, n_real, steps, dims=dims, shape=1, disp_deg=5.0, rate=2.5, H=500.0, mode=2,
                       step0=rng.randint(1, 400) * per_sample - steps // 2)
    if rng.random() < 0.2:
        return _window(None, b, n_real, steps, dims=dims, rate=0.0, H=float(rng.randint(0, 400)), sample_dH=100.0)
    return _window(None, b, n_real, steps, dims=dims, alpha=rng.choice((0.05, 0.1, 0.5, 1.0)),
                   rate=rng.choice((1000.0, 100.0)), step0=rng.randint(0, 1000) * 10)


# ---------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------

def _grid(c, *, b=None, dims=None, rate=None, alpha=None):
    b = c["b"] if b is None else b
    dims = dims or ((c["nx"], c["ny"], c["nz"]) if "nx" in c else RODS[b])
    rate = c["rate"] if rate is None else rate
    g = llg.Grid(*dims, a0=A0_M, b=b, periodic=c.get("periodic", 0))
    g.set_material(A0=EXCHANGE, Ms=MS, K0=K0, alpha=c.get("alpha") if alpha is None else alpha, T=T_K)
    g.set_scaling(mode=c["mode"], Tc=TC_K, delta=DELTA)
    held = rate == 0.0
    g.set_sweep(H_start=c["H"], H_turn=c["H"] if held else -c["H"], rate=rate, dt=DT[b], sample_dH=c["sample_dH"],
                shape=c.get("shape", 0))
    if held:
        g.set_held_samples(c["steps"] // int(c["sample_dH"]) + 1)
    if b == 22:
        g.set_cell_volume(BLOCK_VOLUME)
    if c.get("disp_deg"):
        g.set_axis_dispersion(math.radians(c["disp_deg"]))
    return g


def _key(seed):
    return (int(seed) * 2654435761 + 12345) & 0x7FFFFFFF


def _initial(c, seed):
    """Unit vectors in a cone about +z (a thermally agitated rod), float32 [n_real][cells][3]."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    shape = (c["n_real"], c["nx"] * c["ny"] * c["nz"])
    cz = 1.0 - (1.0 - math.cos(0.45)) * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
    ph = 2 * math.pi * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
    s = torch.sqrt(torch.clamp(1 - cz * cz, min=0))
    m = torch.stack((s * torch.cos(ph), s * torch.sin(ph), cz), dim=-1)
    return (m / m.norm(dim=-1, keepdim=True)).contiguous()


def _target(n):
    """The loop that a calibration fits."""
    return 0.7 + 0.05 * np.cos(np.arange(n) / 7.0)


def _scales(seed):
    gen = torch.Generator()
    gen.manual_seed(int(seed))
    return 1.0 + 0.1 * (torch.rand(3, generator=gen) - 0.5)


def _ladder(c):
    return [(b, rate, alpha) for b in LADDER_BS for rate in LADDER_RATES for alpha in LADDER_ALPHAS]


def prepare(case, seed):
    c = dict(case)
    key = _key(seed)
    if c["kind"] == "window":
        g = _grid(c)
        g.reset(seed=key, n_real=c["n_real"])
        every = g.sample_every
        S = torch.zeros((c["n_real"], g.n_samples), device="cuda")
        first, last = c["step0"] // every + 1, (c["step0"] + c["steps"]) // every
        return dict(kind="window", c=c, g=g, m0=_initial(c, seed), S=S, taken=S[:, first:last + 1],
                    out=torch.empty((c["n_real"], g.ncells, 3), device="cuda"))
    if c["kind"] == "loops":
        g = _grid(c)
        return dict(kind="loops", c=c, g=g, key=key, S=np.zeros((c["n_real"], g.n_samples), dtype=np.float32))
    if c["kind"] == "batch":
        jobs = [_grid(c, b=b, rate=rate, alpha=alpha) for b, rate, alpha in _ladder(c)]
        S = torch.zeros((len(jobs), c["n_real"], jobs[0].n_samples), device="cuda")
        outs = [torch.empty((c["n_real"], g.ncells, 3), device="cuda") for g in jobs]
        return dict(kind="batch", c=c, jobs=jobs, key=key, S=S, samples=list(S), outs=outs,
                    taken=S[:, :, 1:c["steps"] // min(g.sample_every for g in jobs) + 1])
    g = _grid(c)
    g.set_tuning(llg.TUNE_GRAD_METHOD, c["method"])
    return dict(kind="calibration", c=c, g=g, key=key, scales=_scales(seed).requires_grad_(True),
                target=_target(g.n_samples))


def run(state):
    c = state["c"]
    if state["kind"] == "window":
        g = state["g"]
        g.set_state(state["m0"], c["step0"])
        g.advance(c["steps"], state["S"])
        g.get_state(state["out"])
        return {"m": state["out"], "samples": state["taken"]}
    if state["kind"] == "loops":
        # the statistics are part of the call; they are differences of the samples that come back here
        state["g"].run_loops(state["key"], c["n_real"], state["S"])
        return {"samples": state["S"]}
    if state["kind"] == "batch":
        for j, g in enumerate(state["jobs"]):
            g.reset(seed=state["key"] + j, n_real=c["n_real"])
        llg.run_batch(state["jobs"], c["steps"], state["samples"])
        for g, out in zip(state["jobs"], state["outs"]):
            g.get_state(out)
        return {"m": state["outs"], "samples": state["taken"]}
    s = state["scales"]
    s.grad = None
    loss = llg.loop_loss(s, state["g"], seed=state["key"], n_real=c["n_real"], n_steps=c["steps"],
                         target=state["target"], ckpt_every=c["ckpt_every"], mode=c["mode"], Tc=TC_K, delta=DELTA)
    loss.backward()
    return {"loss": loss.detach(), "grad": s.grad}


def _loop_steps(c):
    return 2 * int(round(2 * c["H"] / (c["rate"] * 1e9 * DT[c["b"]])))


def work(case):
    c = case
    if c["kind"] == "batch":
        cells = sum(math.prod(RODS[b]) for b, _, _ in _ladder(c)) * c["n_real"]
        return {"bytes": 12.0 * cells, "flops": float(OPS_PER_CELL_STEP) * cells * c["steps"]}
    if c["kind"] == "loops":
        cells, steps = math.prod(RODS[c["b"]]) * c["n_real"], _loop_steps(c)
        return {"bytes": 4.0 * c["n_real"] * (4 * c["H"] / c["sample_dH"] + 1),
                "flops": float(OPS_PER_CELL_STEP) * cells * steps}
    if c["kind"] == "calibration":
        cells = math.prod(RODS[c["b"]]) * c["n_real"]
        # the loss and its gradient: the forward step and three times its arithmetic for the derivative
        return {"bytes": 4.0 * 7, "flops": 4.0 * OPS_PER_CELL_STEP * cells * c["steps"]}
    cells = c["nx"] * c["ny"] * c["nz"] * c["n_real"]
    axes = 12.0 if c["disp_deg"] else 0.0
    return {"bytes": (24.0 + axes) * cells, "flops": float(OPS_PER_CELL_STEP) * cells * c["steps"]}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------------

_LOW = 0xFFFFFFFF


def _philox(cell, n_lo, n_hi, tag, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words; the four words."""
    x0, x1, x2, x3 = torch.broadcast_tensors(cell, n_lo, n_hi, tag)
    for _ in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57
        x0, x1, x2, x3 = (((p1 >> 32) & _LOW) ^ x1 ^ k0, p1 & _LOW, ((p0 >> 32) & _LOW) ^ x3 ^ k1, p0 & _LOW)
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    return x0, x1, x2, x3


def _uniform(x):
    return ((x >> 8).double() + 0.5) * 2.0 ** -24


class _Exact:
    """Heun steps of the stochastic LLG equation in 64 bits over tensors [realisation][z][y][x]; every
    coefficient a number or a tensor over the realisations."""

    def __init__(self, dims, periodic, keys, b, dt, H, rate, sample_dH, shape, alpha, mode, disp_deg,
                 scale=(1.0, 1.0, 1.0)):
        dev = "cuda"
        self.dims, self.periodic, self.R = dims, periodic, len(keys)
        self.keys = [torch.tensor(k, dtype=torch.int64, device=dev).reshape(-1, 1) for k in zip(*keys)]
        t = T_K / TC_K
        zeta = t / b + 1 - t if mode else 1.0
        mu0, kb = 4e-7 * math.pi, 1.380649e-23
        g0 = mu0 * 1.76e11
        a = b * A0_M
        volume = BLOCK_VOLUME if b == 22 else a ** 3
        sK, sA, sM = scale
        self.alpha, Ms = alpha * sA, MS * sM
        self.adt = dt * g0 / (1 + self.alpha ** 2)
        self.cex = 2 * zeta * EXCHANGE / (mu0 * Ms * a * a)
        self.can = 2 * zeta ** 3 * K0 * sK / (mu0 * Ms)
        self.sigma = (2 * self.alpha * kb * T_K / (g0 * mu0 * Ms * volume * dt)) ** 0.5
        self.H, self.shape = H, shape
        self.per_step = rate * 1e9 * dt  # Oe (a number or a tensor over the realisations)
        self.cells = torch.arange(math.prod(dims), device=dev, dtype=torch.int64).reshape(1, -1)
        zero = torch.zeros((), dtype=torch.int64, device=dev)
        self.up = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device=dev).reshape(3, 1, 1, 1, 1)
        self.axis = None
        if disp_deg:
            x = _philox(self.cells, zero, zero, zero + 1, *self.keys)
            w = (1 - math.cos(math.radians(disp_deg))) * _uniform(x[0])
            ph, st = 2 * math.pi * _uniform(x[1]), torch.sqrt(w * (2 - w))
            self.axis = self._grid(torch.stack((st * torch.cos(ph), st * torch.sin(ph), 1 - w)))

    def _grid(self, v):
        nx, ny, nz = self.dims
        return v.reshape(v.shape[:-1] + (nz, ny, nx))

    def field(self, n):
        oe = 1000 / (4 * math.pi)
        if self.shape == 1:
            period = int(round(4 * self.H / self.per_step))
            return oe * self.H * math.cos(2 * math.pi * (n % period) / period)
        if not torch.is_tensor(self.per_step) and self.per_step == 0:
            return oe * self.H
        if torch.is_tensor(self.per_step):  # windows from step 0 that do not reach the turn
            return oe * (self.H - n * self.per_step)
        half = int(round(2 * self.H / self.per_step))
        ph = n % (2 * half)
        return oe * (self.H - 2 * self.H * min(ph, 2 * half - ph) / half)

    def normals(self, n, count):
        """Standard normals of steps n .. n + count - 1: [step][component][realisation][z][y][x]."""
        steps = torch.arange(n, n + count, device="cuda", dtype=torch.int64).reshape(-1, 1, 1)
        zero = torch.zeros((), dtype=torch.int64, device="cuda")
        x = _philox(self.cells, steps & _LOW, steps >> 32, zero, *self.keys)
        r0, r2 = torch.sqrt(-2 * torch.log(_uniform(x[0]))), torch.sqrt(-2 * torch.log(_uniform(x[2])))
        p1, p3 = 2 * math.pi * _uniform(x[1]), 2 * math.pi * _uniform(x[3])
        return self._grid(torch.stack((r0 * torch.cos(p1), r0 * torch.sin(p1), r2 * torch.cos(p3)), dim=1))

    def torque(self, m, h, Hz):
        s = 0.0
        for axis, bit in ((-1, 1), (-2, 2), (-3, 4)):
            n = m.shape[axis]
            if self.periodic & bit:
                s = s + torch.roll(m, 1, axis) + torch.roll(m, -1, axis)
            elif n > 1:
                edge = torch.zeros_like(m.narrow(axis, 0, 1))
                w = torch.cat((edge, m, edge), dim=axis)
                s = s + w.narrow(axis, 0, n) + w.narrow(axis, 2, n)
        H = self.cex * s + h
        if self.axis is None:
            H = H + self.can * m * self.up + Hz * self.up
        else:
            H = H + self.can * (m * self.axis).sum(0) * self.axis + Hz * self.up
        A = torch.linalg.cross(m, H, dim=0)
        return A + self.alpha * torch.linalg.cross(m, A, dim=0)

    @staticmethod
    def unit(v):
        return v * torch.rsqrt((v * v).sum(0))

    def step(self, m, xi, n):
        h = self.sigma * xi
        s0 = self.torque(m, h, self.field(n))
        s1 = self.torque(self.unit(m - self.adt * s0), h, self.field(n + 1))
        return self.unit(m - 0.5 * self.adt * (s0 + s1))

    def advance(self, m, step0, steps, every):
        """m: [component][realisation][z][y][x].  The state after the steps, and [(k, mean of m_z)]."""
        block = max(1, min(64, 2_000_000 // (self.R * math.prod(self.dims))))
        taken = []
        for a in range(step0, step0 + steps, block):
            for i, xi in enumerate(self.normals(a, min(block, step0 + steps - a))):
                m = self.step(m, xi, a + i)
                if (a + i + 1) % every == 0:
                    taken.append(((a + i + 1) // every, m[2].mean(dim=(-1, -2, -3))))
        return m, taken

    def start(self, m0=None):
        nx, ny, nz = self.dims
        if m0 is None:
            return self.up.expand(3, self.R, nz, ny, nx).clone()
        return self._grid(m0.double().permute(2, 0, 1).contiguous())

    def state(self, m):
        return m.reshape(3, self.R, -1).permute(1, 2, 0)


def _every(c, b, rate):
    return int(c["sample_dH"]) if rate == 0.0 else int(round(c["sample_dH"] / (rate * 1e9 * DT[b])))


def _of(c, key, n_real, **kw):
    dims = (c["nx"], c["ny"], c["nz"]) if "nx" in c else RODS[c["b"]]
    return _Exact(dims, c.get("periodic", 0), [(key, r) for r in range(n_real)], c["b"], DT[c["b"]], c["H"], c["rate"],
                  c["sample_dH"], c.get("shape", 0), c["alpha"], c["mode"], c.get("disp_deg", 0.0), **kw)


def exact(case, seed):
    c = dict(case)
    key = _key(seed)
    if c["kind"] == "window":
        with torch.no_grad():
            e = _of(c, key, c["n_real"])
            m, taken = e.advance(e.start(_initial(c, seed)), c["step0"], c["steps"], _every(c, c["b"], c["rate"]))
            S = torch.stack([v for _, v in taken], dim=1) if taken else torch.zeros((c["n_real"], 0), dtype=torch.float64)
            return {"m": e.state(m), "samples": S}
    if c["kind"] == "loops":
        with torch.no_grad():
            e = _of(c, key, c["n_real"])
            _, taken = e.advance(e.start(), 0, _loop_steps(c), _every(c, c["b"], c["rate"]))
        S = torch.stack([torch.ones(c["n_real"], dtype=torch.float64, device="cuda")] + [v for _, v in taken], dim=1)
        return {"samples": S.cpu().numpy()}
    if c["kind"] == "batch":
        jobs, R = _ladder(c), c["n_real"]
        ms, S = [None] * len(jobs), None
        with torch.no_grad():
            for b in LADDER_BS:
                at = [j for j, job in enumerate(jobs) if job[0] == b]
                per = lambda v: torch.tensor([x for j in at for x in [v(j)] * R], dtype=torch.float64,  # noqa: E731
                                             device="cuda").reshape(-1, 1, 1, 1)
                e = _Exact(RODS[b], 0, [(key + j, r) for j in at for r in range(R)], b, DT[b], c["H"],
                           per(lambda j: jobs[j][1]), c["sample_dH"], 0, per(lambda j: jobs[j][2]), c["mode"], 0.0)
                every = {j: _every(c, b, jobs[j][1]) for j in at}
                m, taken = e.advance(e.start(), 0, c["steps"], min(every.values()))
                if S is None:
                    least = min(_every(c, job[0], job[1]) for job in jobs)
                    S = torch.zeros((len(jobs), R, c["steps"] // least), dtype=torch.float64, device="cuda")
                for i, j in enumerate(at):
                    ms[j] = e.state(m)[i * R:(i + 1) * R]
                    for k, v in taken:
                        n = k * min(every.values())
                        if n % every[j] == 0:
                            S[j, :, n // every[j] - 1] = v[i * R:(i + 1) * R]
        return {"m": ms, "samples": S}
    scale = _scales(seed).double().cuda().requires_grad_(True)
    e = _of(c, key, c["n_real"], scale=scale.unbind(0))
    every = _every(c, c["b"], c["rate"])
    _, taken = e.advance(e.start(), 0, c["steps"], every)
    mean = torch.stack([v.mean() for _, v in taken])
    goal = torch.tensor(_target(int(4 * c["H"] / c["sample_dH"]) + 1), device="cuda")
    loss = ((mean - goal[1:len(mean) + 1]) ** 2).mean()
    loss.backward()
    return {"loss": loss.detach(), "grad": scale.grad}
