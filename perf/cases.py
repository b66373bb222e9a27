"""What the performance of this library is measured on: the calls a user's program makes,
over the sizes, precisions and options the library is used with.

A simulation's pass is a few time steps and a read of the blob state, as every program
here does it (step, sample, step, sample); its outputs are that blob state and the fluid
velocities, looked at where the library keeps them on the GPU (the library takes its
device memory from an allocator of the program, so the program knows the buffers).  An
FP32 simulation's blob state is handed on in FP32, the accuracy it is computed in.

`exact` states the method once more in plain torch FP64 (arXiv:1212.6427, Sec. III.C).
"""
import ctypes
import math

import numpy as np
import torch

import paper_1212_6427_gb300 as icm

SIDES = sorted(2 ** a * 3 ** b for a in range(10) for b in range(6) if 8 <= 2 ** a * 3 ** b <= 512)


def _sim(name, grid, blobs, kernel, precision, kT, dt, steps, **over):
    """One simulation: a pass is `steps` time steps and one read of the blob state."""
    c = dict(name=name, kind="sim", nx=grid[0], ny=grid[1], nz=grid[2], blobs=blobs, kernel=kernel,
             precision=precision, kT=kT, dt=dt, steps=steps, inertial=True, slip="visc", advection=True,
             force=0.0, trap=0.0, wca=0.0, drift=False, apart=True)
    c.update(over)
    return c


def listed():
    return [
        # a bead in an optical trap, tracked step by step: the temporal accuracy experiment of the
        # paper; the smallest call, all latency and launches
        _sim("trap 16^3 fp64", (16, 16, 16), 1, 4, 64, 0.0, 0.25, 1, trap=0.01),
        # freely diffusing tracers with the thermal drift, sampled every ten steps (300k steps a run)
        _sim("drift 16^3", (16, 16, 16), 400, 3, 32, 1.0, 0.05, 10, inertial=False, drift=True, apart=False),
        # a dense colloid with WCA repulsion: the radial distribution function runs (400k steps)
        _sim("colloid 32^3", (32, 32, 32), 1000, 3, 32, 1e-3, 1.0, 10, wca=1e-3),
        # one neutral bead in a fluctuating fluid, double precision: the bench's plain workload
        _sim("plain 32^3 fp64", (32, 32, 32), 1, 4, 64, 1e-3, 0.05, 10, inertial=False),
        # mobility matrices J (eta L)^-1 P S at 16 positions: the hydrodynamic radius experiment
        dict(name="mobility 32^3 fp64", kind="coupling", side=32, kernel=3, precision=64, pairs=16, stokes=True),
        # the mid-sized suspension of the bench and of the long parity runs, in both precisions
        _sim("bulk 128^3", (128, 128, 128), 2000, 3, 32, 1e-3, 0.02, 10),
        _sim("bulk 128^3 fp64", (128, 128, 128), 2000, 3, 64, 1e-3, 0.02, 2),
        # a box cut to the problem and not to the FFT: sides with factors of three
        _sim("box 144x108x216", (144, 108, 216), 1500, 3, 32, 1e-3, 0.02, 4, slip="full", force=1e-3),
        # an ensemble of replicas stepped as one batch (batched stages, the mode the batch
        # autotuner picks), sides 32 to 96 with 1 to 500 blobs
        dict(name="ensemble of 48", kind="batch", members=48, steps=10, grouped=2),
        # jobs handed to the server, admitted and run together, results collected
        dict(name="served jobs", kind="served", jobs=8, steps=50, per_pump=10),
        # the bench's large workload, driven by forces that the program sets for each sample
        _sim("large 256^3", (256, 256, 256), 20000, 4, 32, 1e-3, 0.01, 4, force=1e-4),
        # the largest box of the tests, a wide channel
        _sim("wide 512x384x256", (512, 384, 256), 3000, 4, 32, 1e-3, 0.01, 2),
    ]


def draw(rng):
    """One more case: most are simulations of any size, shape and option the library takes."""
    what = rng.random()
    if what < 0.08:
        return dict(kind="coupling", side=rng.choice([s for s in SIDES if 16 <= s <= 64]), kernel=rng.choice([3, 4]),
                    precision=rng.choice([32, 64]), pairs=rng.randint(1, 32), stokes=rng.random() < 0.5)
    if what < 0.16:
        return dict(kind="batch", members=rng.randint(2, 48), steps=rng.randint(1, 10),
                    grouped=rng.choice([0, 1, 2, 2, 3]))
    if what < 0.22:
        return dict(kind="served", jobs=rng.randint(1, 8), steps=rng.randint(10, 50), per_pump=rng.choice([1, 5, 10]))
    precision = 64 if rng.random() < 0.3 else 32
    most = 256 ** 3 if precision == 32 else 128 ** 3
    while True:
        base = math.exp(rng.uniform(math.log(10), math.log(320 if precision == 32 else 160)))
        cube = rng.random() < 0.3
        sides = []
        for _ in range(3):
            want = base if cube else base * math.exp(rng.uniform(-0.7, 0.7))
            sides.append(min(SIDES, key=lambda s: abs(math.log(s / want))))
        cells = sides[0] * sides[1] * sides[2]
        if cells <= most:
            break
    room = (sides[0] // 3) * (sides[1] // 3) * (sides[2] // 3) // 2
    blobs = max(0, min(room, 20000, int(math.exp(rng.uniform(0.0, math.log(1.0 + 0.02 * cells))))))
    option = rng.choice(["none", "none", "force", "trap", "wca", "drift"])
    if option == "wca":
        blobs = min(blobs, 2000)
    kT = 0.0 if rng.random() < 0.15 else math.exp(rng.uniform(math.log(1e-4), math.log(1e-2)))
    steps = max(1, min(rng.randint(1, 10), (2 * most) // cells))
    c = _sim("", sides, blobs, rng.choice([3, 4]), precision, kT, rng.choice([0.01, 0.02, 0.05]), steps,
             inertial=rng.random() < 0.75, slip=rng.choice(["visc", "visc", "zero", "full"]),
             advection=rng.random() < 0.85, force=1e-3 if option == "force" else 0.0,
             trap=0.01 if option == "trap" else 0.0, wca=1e-3 if option == "wca" else 0.0,
             drift=option == "drift")
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
DRAGGED = {3: 12.0, 4: 768.0 / 27.0}     # dragged fluid mass of a blob, in rho h^3


def _place(rng, grid, n, apart):
    """n positions: uniform, or two cells apart (jittered sites of a coarse lattice)."""
    box = np.asarray(grid, dtype=np.float64)
    if not apart:
        return rng.uniform(0.0, 1.0, size=(n, 3)) * box
    sites = np.maximum(np.asarray(grid) // 3, 1)
    pick = rng.choice(int(sites.prod()), size=n, replace=False)
    cell = np.stack([pick % sites[0], (pick // sites[0]) % sites[1], pick // (sites[0] * sites[1])], axis=1)
    return ((cell + 0.5) * (box / sites) + rng.uniform(-0.5, 0.5, size=(n, 3))) % box


def _inputs(c, seed):
    """The blobs of a simulation on the host, and its fluid velocities on the GPU (values its
    precision holds): white noise of the equilibrium variance kT / (rho h^3)."""
    rng = np.random.default_rng([seed, 77])
    grid = (c["nx"], c["ny"], c["nz"])
    n = c["blobs"]
    q = _place(rng, grid, n, c["apart"])
    me = rng.uniform(-0.5, 2.0, size=n) if c["inertial"] else np.zeros(n)
    u = rng.standard_normal((n, 3)) * np.sqrt(c["kT"] / (me + DRAGGED[c["kernel"]]))[:, None]
    force = np.zeros((n, 3))
    if c["force"]:
        force = c["force"] * (np.array([1.0, 0.0, 0.0]) + 0.1 * rng.standard_normal((n, 3)))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 2 + 1)
    real = torch.float32 if c["precision"] == 32 else torch.float64
    v = torch.randn((3, c["nz"], c["ny"], c["nx"]), generator=gen, device="cuda", dtype=real)
    v *= math.sqrt(c["kT"]) if c["kT"] > 0 else 0.01
    return dict(q=q, me=me, u=u, force=force, v=v, trap_center=[0.5 * s for s in grid])


def _members(c, seed):
    """The replicas of an ensemble: side in {32, 48, 64, 96}, 1 to 500 blobs, either kernel.  The
    mix of sides is part of the case; the states come from the seed."""
    mix = np.random.default_rng(10_000 + c["members"])
    out = []
    for k in range(c["members"]):
        side = int(mix.choice([32, 48, 64, 96]))
        m = _sim("", (side,) * 3, int(mix.integers(1, 501)), int(mix.choice([3, 4])), 32, 1e-3, 0.05, c["steps"])
        out.append((m, seed * 1000 + k))
    return out


def _jobs(c, seed):
    """The jobs of a server: side in {32, ..., 128}, 1 to 2000 blobs, kT in [1e-4, 1e-2]."""
    mix = np.random.default_rng(30_000 + c["jobs"])
    out = []
    for k in range(c["jobs"]):
        side = int(mix.choice([32, 48, 64, 96, 128]))
        n = min(int(mix.integers(1, 2001)), (side // 3) ** 3 // 2)
        m = _sim("", (side,) * 3, n, int(mix.choice([3, 4])), 32, float(mix.uniform(1e-4, 1e-2)), 0.05, c["steps"])
        out.append((m, seed * 1000 + k))
    return out


def _key(seed):
    return (int(seed) * 0x9E3779B97F4A7C15 + 12345) & 0xFFFFFFFFFFFFFFFF


# ---------------------------------------------------------------------------
# The program's side
# ---------------------------------------------------------------------------
class _Memory:
    """The device memory this program gives to the library: torch's, with the buffers in use
    kept by address."""

    def __init__(self):
        self.held = {}
        make = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
        drop = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p)

        def give(_, size, stream):
            try:
                p = torch.cuda.caching_allocator_alloc(int(size), stream=int(stream or 0))
            except Exception:
                return None
            self.held[p] = int(size)
            return p

        def take(_, p, stream):
            self.held.pop(p, None)
            torch.cuda.caching_allocator_delete(p)

        self.calls = make(give), drop(take)

    def use(self):
        icm.lib().icm_set_default_allocator(self.calls[0], self.calls[1], None)


_memory = None


def _use_memory():
    global _memory
    if _memory is None:
        _memory = _Memory()
    _memory.use()
    return _memory


class _Buffer:
    def __init__(self, p, shape, real):
        self.__cuda_array_interface__ = dict(shape=tuple(shape), typestr="<f4" if real == torch.float32 else "<f8",
                                             data=(p, False), version=2)


class _Simulation:
    def __init__(self, c, seed):
        mem = _use_memory()
        before = set(mem.held)
        x = _inputs(c, seed)
        self.c, self.ncell = c, c["nx"] * c["ny"] * c["nz"]
        self.stream = torch.cuda.Stream()
        flags = {"visc": icm.FLAG_SLIP_VISC, "zero": icm.FLAG_SLIP_ZERO, "full": icm.FLAG_SLIP_FULL}[c["slip"]]
        flags |= 0 if c["advection"] else icm.FLAG_NO_ADVECTION
        flags |= icm.FLAG_THERMAL_DRIFT if c["drift"] else 0
        self.handle = icm.icm_create((c["nx"], c["ny"], c["nz"]), 1.0, 1.0, 1.0, c["kT"], c["dt"], c["kernel"],
                                     _key(seed), c["precision"], flags, ctypes.c_void_p(self.stream.cuda_stream))
        self.force = None
        if c["blobs"]:
            icm.icm_add_blobs(self.handle, x["q"], x["u"], x["me"])
            if c["force"]:
                self.force = x["force"]
            if c["trap"]:
                icm.icm_set_blob_trap(self.handle, c["trap"], x["trap_center"])
            if c["wca"]:
                icm.icm_set_blob_wca(self.handle, c["wca"], 2.0)
        icm.icm_write_state(self.handle, x["q"], x["u"], x["v"].double().cpu().numpy())
        # the buffer that now holds the velocities, among those given out for this simulation
        real, n = x["v"].dtype, x["v"].numel()
        self.fluid = None
        for p in set(mem.held) - before:
            if mem.held[p] >= n * x["v"].element_size():
                t = torch.as_tensor(_Buffer(p, x["v"].shape, real), device="cuda")
                if torch.equal(t, x["v"]):
                    self.fluid = t
        if self.fluid is None:
            raise RuntimeError("the fluid velocities are in none of the buffers given to the library")

    def set_forces(self):
        if self.force is not None:
            icm.icm_set_blob_forces(self.handle, self.force)

    def sample(self):
        pos, vel, _, mom, step, _ = icm.icm_read_state(self.handle, self.ncell)
        if self.c["precision"] == 32:
            pos, vel, mom = pos.astype(np.float32), vel.astype(np.float32), mom.astype(np.float32)
        return pos, vel, mom, step

    def __del__(self):
        if getattr(self, "handle", None) is not None:
            icm.icm_destroy(self.handle)


class _Ensemble:
    def __init__(self, c, seed):
        self.sims = [_Simulation(m, s) for m, s in _members(c, seed)]
        self.steps = c["steps"]
        self.batch = icm.icm_batch_create()
        icm.icm_batch_set(self.batch, [s.handle for s in self.sims])
        icm.icm_batch_set_grouped(self.batch, c["grouped"])

    def __del__(self):
        if getattr(self, "batch", None) is not None:
            icm.icm_batch_destroy(self.batch)


def prepare(case, seed):
    if case["kind"] == "sim":
        return _Simulation(case, seed)
    if case["kind"] == "batch":
        return _Ensemble(case, seed)
    if case["kind"] == "served":
        _use_memory()
        return dict(case=case, jobs=[(m, s, _job_blobs(m, s)) for m, s in _jobs(case, seed)])
    rng = np.random.default_rng([seed, 78])
    q = rng.uniform(0.0, 1.0, size=(case["pairs"], 3)) * case["side"]
    _use_memory()
    state = dict(case=case, q=q, stream=torch.cuda.Stream())
    state["sim"] = _Handle(icm.icm_create((case["side"],) * 3, 1.0, 1.0, 1.0, 0.0, 0.05, case["kernel"], 1,
                                          case["precision"], 0, ctypes.c_void_p(state["stream"].cuda_stream)))
    return state


class _Handle:
    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        icm.icm_destroy(self.handle)


def _job_blobs(m, seed):
    """A job's blobs; its fluid starts at rest."""
    rng = np.random.default_rng([seed, 77])
    n = m["blobs"]
    q = _place(rng, (m["nx"], m["ny"], m["nz"]), n, True)
    me = rng.uniform(-0.5, 2.0, size=n)
    u = rng.standard_normal((n, 3)) * np.sqrt(m["kT"] / (me + DRAGGED[m["kernel"]]))[:, None]
    return dict(q=q, me=me, u=u, force=np.zeros((n, 3)))


def run(state):
    if isinstance(state, _Simulation):
        state.set_forces()
        icm.icm_step(state.handle, state.c["steps"])
        pos, vel, mom, step = state.sample()
        return dict(pos=pos, vel=vel, momentum=mom, step=step, fluid=state.fluid)
    if isinstance(state, _Ensemble):
        icm.icm_batch_step(state.batch, state.steps)
        got = [s.sample() for s in state.sims]
        return dict(pos=np.concatenate([g[0] for g in got]), vel=np.concatenate([g[1] for g in got]),
                    momentum=np.stack([g[2] for g in got]), step=np.array([g[3] for g in got]),
                    fluid=[s.fluid for s in state.sims])
    case = state["case"]
    if case["kind"] == "coupling":
        a, b = (0.0, 1.0) if case["stokes"] else (1.0, 0.0)
        m = icm.icm_op_coupling(state["sim"].handle, state["q"], state["q"], a, b)
        return m if case["precision"] == 64 else m.astype(np.float32)
    server = icm.icm_server_create(100 << 30, 64)
    ids = [icm.icm_server_submit(server, (m["nx"], m["ny"], m["nz"]), 1.0, 1.0, 1.0, m["kT"], m["dt"], m["kernel"],
                                 _key(s), m["precision"], 0, x["q"], x["u"], x["me"], None, m["steps"])
           for m, s, x in state["jobs"]]
    done = 0
    while done < len(ids):
        done += icm.icm_server_pump(server, case["per_pump"])[2]
    got = [icm.icm_server_result(server, i, m["blobs"]) for i, (m, _, _) in zip(ids, state["jobs"])]
    icm.icm_server_destroy(server)
    return dict(state=np.array([g["state"] for g in got]),
                pos=np.concatenate([g["pos"] for g in got]).astype(np.float32),
                vel=np.concatenate([g["vel"] for g in got]).astype(np.float32),
                momentum=np.stack([g["momentum"] for g in got]).astype(np.float32))


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _sim_work(m):
    """Per step: velocities and advective fluxes read and written, the blob state read and
    written; one solve for neutral blobs, three for inertial ones."""
    n = m["nx"] * m["ny"] * m["nz"]
    r = m["precision"] // 8
    solves = 3 if m["inertial"] and m["blobs"] else 1
    fft = 2 * 3 * 2.5 * n * math.log2(n) + 60.0 * n / 2
    stencil = 3 * m["kernel"] ** 3 * 2.0 * m["blobs"]
    return dict(bytes=m["steps"] * (4.0 * 3 * n * r + 13.0 * 8 * m["blobs"]),
                flops=m["steps"] * (solves * (fft + 2 * stencil) + 2 * stencil + (250.0 if m["kT"] else 100.0) * n))


def work(case):
    if case["kind"] == "sim":
        return _sim_work(case)
    if case["kind"] == "coupling":
        n = case["side"] ** 3
        return dict(bytes=case["pairs"] * (6.0 + 9.0) * 8,
                    flops=case["pairs"] * 3 * (2 * 3 * 2.5 * n * math.log2(n) + 60.0 * n / 2))
    parts = [_sim_work(m) for m, _ in (_members(case, 1) if case["kind"] == "batch" else _jobs(case, 1))]
    return dict(bytes=sum(p["bytes"] for p in parts), flops=sum(p["flops"] for p in parts))


# ---------------------------------------------------------------------------
# The same in 64 bits: torch's FFT and plain tensor arithmetic
# ---------------------------------------------------------------------------
def _at(f, axis, s):
    """f[c + s e_axis] on the periodic grid (x is the last dimension)."""
    return torch.roll(f, -s, dims=f.dim() - 1 - axis)


def _words(cell, step, call, key):
    """Philox4x32-10 at counters (cell, step, call, 0)."""
    low = 0xFFFFFFFF
    x = [cell, torch.full_like(cell, step), torch.full_like(cell, call), torch.zeros_like(cell)]
    k0, k1 = key & low, key >> 32
    for _ in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((p1 >> 32) & low) ^ x[1] ^ k0, p1 & low, ((p0 >> 32) & low) ^ x[3] ^ k1, p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return x


def _normals(a, b):
    rad = torch.sqrt(-2.0 * torch.log((a.double() + 0.5) * 2.0 ** -32))
    ang = 2.0 * math.pi * ((b.double() + 0.5) * 2.0 ** -32)
    return rad * torch.cos(ang), rad * torch.sin(ang)


def _peskin(kernel, r):
    a = r.abs()
    if kernel == 3:
        inner = (1 + torch.sqrt((1 - 3 * a * a).clamp(min=0))) / 3
        outer = (5 - 3 * a - torch.sqrt((1 - 3 * (1 - a) ** 2).clamp(min=0))) / 6
        return torch.where(a <= 0.5, inner, torch.where(a <= 1.5, outer, torch.zeros_like(a)))
    inner = (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp(min=0))) / 8
    outer = (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp(min=0))) / 8
    return torch.where(a <= 1, inner, torch.where(a <= 2, outer, torch.zeros_like(a)))


def _peskin_slope(kernel, r):
    a, sign = r.abs(), torch.where(r < 0, -1.0, 1.0).double()
    if kernel == 3:
        t = 1 - a
        inner = -a / torch.sqrt((1 - 3 * a * a).clamp(min=1e-300))
        outer = (-3 - 3 * t / torch.sqrt((1 - 3 * t * t).clamp(min=1e-300))) / 6
        return sign * torch.where(a <= 0.5, inner, torch.where(a <= 1.5, outer, torch.zeros_like(a)))
    inner = (-2 + (2 - 4 * a) / torch.sqrt((1 + 4 * a - 4 * a * a).clamp(min=1e-300))) / 8
    outer = (-2 - (6 - 4 * a) / torch.sqrt((-7 + 12 * a - 4 * a * a).clamp(min=1e-300))) / 8
    return sign * torch.where(a <= 1, inner, torch.where(a <= 2, outer, torch.zeros_like(a)))


class _Exact:
    """The method's step, Sec. III.C in order, h = rho = eta = 1."""

    def __init__(self, c, seed, x):
        self.c = c
        f = lambda y: torch.as_tensor(y, dtype=torch.float64, device="cuda")  # noqa: E731
        self.q, self.u, self.me, self.force, self.v = f(x["q"]), f(x["u"]), f(x["me"]), f(x["force"]), f(x["v"])
        self.center = f(x["trap_center"])
        self.n = (c["nx"], c["ny"], c["nz"])
        self.box = f(self.n)
        self.key, self.level, self.adv = _key(seed), 0, None
        self.g = torch.zeros_like(self.q)
        self.dragged = DRAGGED[c["kernel"]]
        th = [2 * math.pi * torch.arange(s, dtype=torch.float64, device="cuda") / s for s in self.n]
        th[0] = th[0][:self.n[0] // 2 + 1]
        d = [torch.complex(torch.cos(t) - 1, torch.sin(t)) for t in th]
        self.d = d[0][None, None, :], d[1][None, :, None], d[2][:, None, None]
        dd = [4 * torch.sin(t / 2) ** 2 for t in th]
        self.dd = dd[0][None, None, :] + dd[1][None, :, None] + dd[2][:, None, None]

    def stencil(self, q, comp, slope=False):
        """Flat nodes and weights (blob, z, y, x) of one component."""
        w, first, at = [], [], []
        k = self.c["kernel"]
        for ax in range(3):
            s = q[:, ax] - (0.0 if ax == comp else 0.5)
            lo = (torch.floor(s + 0.5) if k == 3 else torch.floor(s)) - 1
            node = lo[:, None] + torch.arange(k, device="cuda", dtype=torch.float64)
            w.append(_peskin_slope(k, s[:, None] - node) if slope and ax == comp else _peskin(k, s[:, None] - node))
            at.append(node.long() % self.n[ax])
        flat = at[0][:, None, None, :] + self.n[0] * (at[1][:, None, :, None] + self.n[1] * at[2][:, :, None, None])
        return flat, w[0][:, None, None, :] * w[1][:, None, :, None] * w[2][:, :, None, None]

    def gather(self, f, q):
        out = torch.zeros_like(q)
        for comp in range(3):
            flat, w = self.stencil(q, comp)
            out[:, comp] = (w * f[comp].reshape(-1)[flat]).sum(dim=(1, 2, 3))
        return out

    def spread(self, amount, q, slope=False):
        out = torch.zeros_like(self.v)
        for comp in range(3):
            flat, w = self.stencil(q, comp, slope)
            a = amount if slope else amount[:, comp]
            out[comp].view(-1).index_add_(0, flat.reshape(-1), (w * a[:, None, None, None]).reshape(-1))
        return out

    def solve(self, r, a, b):
        h = [torch.fft.rfftn(r[k]) for k in range(3)]
        some = self.dd > 0
        ratio = (self.d[0] * h[0] + self.d[1] * h[1] + self.d[2] * h[2]) / torch.where(some, self.dd, 1.0)
        ratio = torch.where(some, ratio, torch.zeros_like(ratio))
        den = a + b * self.dd
        inv = torch.where(den > 0, 1.0 / torch.where(den > 0, den, 1.0), 0.0)
        out = torch.empty_like(r)
        for k in range(3):
            out[k] = torch.fft.irfftn((h[k] - self.d[k].conj() * ratio) * inv, s=r.shape[1:])
        return out

    def advection(self, v):
        out = torch.empty_like(v)
        for a in range(3):
            m = 0.5 * (_at(v[a], a, 1) + v[a])
            t = m * m - _at(m * m, a, -1)
            for b in range(3):
                if b != a:
                    e = 0.25 * (v[a] + _at(v[a], b, -1)) * (v[b] + _at(v[b], a, -1))
                    t = t + _at(e, b, 1) - e
            out[a] = t
        return out

    def noise(self):
        nx, ny, nz = self.n
        cell = torch.arange(nx * ny * nz, device="cuda")
        odd = (cell // (nx * ny)) % 2 == 1
        p = _words(cell, self.level, 0, self.key)
        r = _words(torch.where(odd, cell - nx * ny, cell), self.level, 1, self.key)
        z = [*_normals(p[0], p[1]), *_normals(p[2], p[3]),
             *_normals(torch.where(odd, r[2], r[0]), torch.where(odd, r[3], r[1]))]
        del p, r, cell, odd
        z = [t.reshape(nz, ny, nx) for t in z]
        amp = math.sqrt(self.c["kT"] / self.c["dt"])
        edge = {(0, 1): z[3], (0, 2): z[4], (1, 2): z[5]}
        out = torch.empty_like(self.v)
        for a in range(3):
            t = 2.0 * amp * (z[a] - _at(z[a], a, -1))
            for b in range(3):
                if b != a:
                    e = math.sqrt(2.0) * amp * edge[(min(a, b), max(a, b))]
                    t = t + _at(e, b, 1) - e
            out[a] = t
        return out

    def pair_force(self, q):
        d = q[:, None, :] - q[None, :, :]
        d = d - self.box * torch.round(d / self.box)
        r2 = (d * d).sum(dim=2)
        r2.fill_diagonal_(math.inf)
        s6 = (4.0 / r2) ** 3
        mag = torch.where(r2 < 4.0 * 2.0 ** (1.0 / 3.0), 24.0 * self.c["wca"] * (2.0 * s6 * s6 - s6) / r2, 0.0)
        return (mag[:, :, None] * d).sum(dim=1)

    def step(self):
        c, dt, v, q, me = self.c, self.c["dt"], self.v, self.q, self.me
        jv = self.gather(v, q)
        qh = torch.remainder(q + 0.5 * dt * jv, self.box)
        force = self.force
        if c["trap"] and len(q):
            d = qh - self.center
            force = force - c["trap"] * (d - self.box * torch.round(d / self.box))
        if c["wca"] and len(q) > 1:
            force = force + self.pair_force(qh)
        adv = self.advection(v) if c["advection"] else torch.zeros_like(v)
        r = v / dt - 1.5 * adv + 0.5 * (adv if self.adv is None else self.adv)
        for ax in range(3):
            r = r + 0.5 * (_at(v, ax, 1) - 2.0 * v + _at(v, ax, -1))
        if c["kT"] > 0:
            r = r + self.noise()
        r = r + self.spread(force, qh)
        if c["drift"] and c["kT"] > 0 and len(q):
            r = r + self.spread(c["kT"] * self.dragged / (self.dragged + me), qh, slope=True)
        vt = self.solve(r, 1.0 / dt, 0.5)
        if len(q) and bool((me != 0).any()):
            jvt = self.gather(vt, qh)
            du = torch.zeros_like(q)
            if c["slip"] != "zero":
                du = 0.5 * dt * self.g
            if c["slip"] == "full":
                du = du + self.gather(v, qh) - jv
            dp = me[:, None] * (self.u - jvt - du)
            share = (self.dragged / (self.dragged + me))[:, None]
            jd = self.gather(self.solve(self.spread(share * dp, qh), 1.0, 0.0), qh)
            dv = self.solve(self.spread(dp - me[:, None] * jd, qh), 1.0, 0.5 * dt)
            self.u = jvt + jd + du
            lap = sum(_at(dv, ax, 1) - 2.0 * dv + _at(dv, ax, -1) for ax in range(3))
            self.g = self.gather(lap, qh)
            new = vt + dv
        else:
            new = vt
            self.u = self.gather(new, qh)
            self.g = torch.zeros_like(q)
        self.q = torch.remainder(q + 0.5 * dt * self.gather(new + v, qh), self.box)
        self.v, self.adv = new, adv
        self.level += 1

    def momentum(self):
        return self.v.reshape(3, -1).sum(dim=1) + (self.me[:, None] * self.u).sum(dim=0)


def _exact_run(c, seed, x):
    e = _Exact(c, seed, x)
    for _ in range(c["steps"]):
        e.step()
    return dict(pos=e.q.cpu().numpy(), vel=e.u.cpu().numpy(), momentum=e.momentum().cpu().numpy(), step=e.level,
                fluid=e.v)


def exact(case, seed):
    if case["kind"] == "sim":
        return _exact_run(case, seed, _inputs(case, seed))
    if case["kind"] == "coupling":
        rng = np.random.default_rng([seed, 78])
        q = torch.as_tensor(rng.uniform(0.0, 1.0, size=(case["pairs"], 3)) * case["side"], device="cuda")
        c = _sim("", (case["side"],) * 3, 0, case["kernel"], 64, 0.0, 0.05, 1)
        e = _Exact(c, 0, dict(_inputs(c, 0)))
        out = np.zeros((case["pairs"], 3, 3))
        a, b = (0.0, 1.0) if case["stokes"] else (1.0, 0.0)
        for k in range(case["pairs"]):
            for col in range(3):
                unit = torch.zeros((1, 3), dtype=torch.float64, device="cuda")
                unit[0, col] = 1.0
                out[k, :, col] = e.gather(e.solve(e.spread(unit, q[k:k + 1]), a, b), q[k:k + 1])[0].cpu().numpy()
        return out
    if case["kind"] == "batch":
        got = [_exact_run(m, s, _inputs(m, s)) for m, s in _members(case, seed)]
        return dict(pos=np.concatenate([g["pos"] for g in got]), vel=np.concatenate([g["vel"] for g in got]),
                    momentum=np.stack([g["momentum"] for g in got]), step=np.array([g["step"] for g in got]),
                    fluid=[g["fluid"] for g in got])
    got = []
    for m, s in _jobs(case, seed):
        x = dict(_job_blobs(m, s), v=np.zeros((3, m["nz"], m["ny"], m["nx"])), trap_center=[0.0, 0.0, 0.0])
        got.append(_exact_run(m, s, x))
    return dict(state=np.full(len(got), 2), pos=np.concatenate([g["pos"] for g in got]),
                vel=np.concatenate([g["vel"] for g in got]), momentum=np.stack([g["momentum"] for g in got]))
