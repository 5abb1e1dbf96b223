"""Performance cases of the library: what its users run, through the public entry points.

A case is a dict of plain values.  Its "kind" says which calls one pass makes:

  steps     flb_step(steps) of one box (the simulation itself), the new state left on the device
  sampled   an equipartition / S(q) run: flb_step with automatic statistics samples every few
            steps (stats_every), then flb_mode_stats and flb_structure_factor
  profiles  a decaying or driven flow: flb_step(every), flb_z_profile, again and again
  ensemble  flb_step of a batch of boxes (flb_create_batch) replaying CUDA graphs
  host      host-resident stepping: flb_step_host on a page-locked buffer
  fields    a state set from host arrays, read back as moments and populations

prepare() makes the context (the handle a program keeps) and puts a thermal state into it:
independent Gaussian deviations of variance mu rho0 a_i, which is the stationary state of the
fluctuating equation, plus the velocity field of the flow cases.  Device memory comes from the
library's allocator hook, so the caller owns the memory of the state and a pass can return it
without a copy: flb_state_bytes() bytes per box, planes [q][plane] of the storage type.  A box of
the two-buffer pattern is in its first buffer again after an even number of steps; every case
makes an even number.

Numbers that the library computes in single precision and hands over as doubles (mode moments,
S(q), profiles of a single-precision context) are kept in single precision; the mass, which it
sums in double precision, stays double.
"""
import math

import numpy as np
import torch

from paper_0707_1581_gb300 import flb

DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16dev": torch.float16, "bf16dev": torch.bfloat16,
         "bf16sr": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2, "bf16sr": 2}

# the physics every kind starts from; a case overrides what it needs
BASE = dict(lattice="d3q19", store="f32", pattern="ab", kT=1e-4, gamma_shear=0.3, gamma_bulk=0.2, gamma_ghost=0.0,
            force=0.0, rho_local=False, graph_steps=0, u0=0.0)


def listed():
    return [
        # the smallest call: the FP64 conservation / equipartition check of a 16^3 box
        dict(name="box16_f64", kind="steps", nx=16, ny=16, nz=16, steps=200, store="f64", gamma_shear=0.2),
        # the standard validation run: 64^3 FP32 at the library's defaults, statistics and S(q) every 20 steps
        dict(name="box64_f32_sampled", kind="sampled", nx=64, ny=64, nz=64, steps=100, every=20, gamma_shear=0.5),
        # shear-wave decay on the same box: the viscosity measurement
        dict(name="box64_f32_profiles", kind="profiles", nx=64, ny=64, nz=64, steps=100, every=10, gamma_shear=0.5,
             u0=1e-3),
        # the storage-format comparison: 256^3 in bfloat16 deviations, sampled, in place
        dict(name="box256_bf16dev_sampled", kind="sampled", nx=256, ny=256, nz=256, steps=20, every=20,
             store="bf16dev", pattern="aa", gamma_shear=0.0),
        # the same box with stochastic rounding, two buffers
        dict(name="box256_bf16sr", kind="steps", nx=256, ny=256, nz=256, steps=20, store="bf16sr", gamma_shear=0.0),
        # an odd, ragged box with every option that changes the arithmetic: relaxing kinetic modes, local-density
        # noise, a body force, in place
        dict(name="ragged_f32_options", kind="steps", nx=250, ny=187, nz=93, steps=20, pattern="aa", gamma_ghost=0.1,
             force=1e-5, rho_local=True),
        # the ensemble: 64 replicas of 64^3 and 16 cubes of edges 32 .. 128 in one batch, graphs of 20 steps
        dict(name="ensemble80_f32", kind="ensemble", replicas=64, edge=64, mixed=16, lo=32, hi=128, steps=20,
             graph_steps=20),
        # production flow: 512^3 Kolmogorov forcing, FP32, in place
        dict(name="box512_f32_forced", kind="steps", nx=512, ny=512, nz=512, steps=20, pattern="aa", force=1e-5),
        # the same in FP16 deviations
        dict(name="box512_f16dev_forced", kind="steps", nx=512, ny=512, nz=512, steps=20, store="f16dev",
             pattern="aa", force=1e-5),
        # the two-dimensional lattice at production size
        dict(name="d2q9_8192_f32", kind="steps", lattice="d2q9", nx=8192, ny=8192, nz=1, steps=20),
        # a state that lives on the host (end-to-end leg: upload, step, download)
        dict(name="host256_f32", kind="host", nx=256, ny=256, nz=256, steps=2, pattern="aa", force=1e-5),
        # setting a state and reading the fields back, as analysis and restart programs do
        dict(name="fields128_f32", kind="fields", nx=128, ny=128, nz=128, steps=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(rng, lo, hi, most):
    """Three edges, log-uniform in lo .. hi, mostly ragged, with at most `most` sites."""
    while True:
        e = [_log_int(rng, lo, hi) for _ in range(3)]
        style = rng.randrange(4)
        if style == 0:      # multiples of 4 along x
            e[0] = max(4, e[0] // 4 * 4)
        elif style == 1:    # a cube of a round edge
            c = max(8, e[0] // 8 * 8)
            e = [c, c, c]
        elif style == 2:    # multiples of 32 along x
            e[0] = max(32, e[0] // 32 * 32)
        if e[0] * e[1] * e[2] <= most:
            return e


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "d2q9", "sampled", "sampled", "profiles", "ensemble", "host",
                       "fields"])
    opts = dict(kT=rng.choice([1e-5, 1e-4, 1e-3]), gamma_shear=round(rng.uniform(0.0, 0.8), 3),
                gamma_bulk=round(rng.uniform(0.0, 0.5), 3), pattern=rng.choice(["ab", "aa"]))
    if rng.random() < 0.3:
        opts["gamma_ghost"] = round(rng.uniform(0.0, 0.3), 3)
    if rng.random() < 0.5:
        opts["force"] = 1e-5
    if rng.random() < 0.15:
        opts["rho_local"] = True
    single = rng.choice(["f32", "f32", "f16dev", "bf16dev", "bf16sr"])
    if kind == "steps":
        store = rng.choice(["f64", "f32", "f32", "f16dev", "f16dev", "bf16dev", "bf16sr"])
        hi, most = (96, 128 ** 3) if store == "f64" else (640, 448 ** 3)
        nx, ny, nz = _edges(rng, 8, hi, most)
        return dict(kind="steps", nx=nx, ny=ny, nz=nz, steps=2 * rng.randint(5, 10), store=store,
                    graph_steps=rng.choice([0, 0, 10]), **opts)
    if kind == "d2q9":
        nx, ny = _log_int(rng, 64, 8192), _log_int(rng, 64, 8192)
        if rng.random() < 0.7:
            nx = nx // 4 * 4
        return dict(kind="steps", lattice="d2q9", nx=nx, ny=ny, nz=1, steps=2 * rng.randint(5, 10), store=single,
                    graph_steps=rng.choice([0, 0, 10]), **opts)
    if kind == "sampled":
        nx, ny, nz = _edges(rng, 16, 512, 320 ** 3)
        every = 2 * rng.randint(5, 10)
        return dict(kind="sampled", nx=nx, ny=ny, nz=nz, steps=every * rng.randint(1, 4), every=every, store=single,
                    **opts)
    if kind == "profiles":
        nx, ny, nz = _edges(rng, 8, 320, 192 ** 3)
        every = 2 * rng.randint(1, 10)
        return dict(kind="profiles", nx=nx, ny=ny, nz=nz, steps=every * rng.randint(2, 8), every=every, store=single,
                    u0=1e-3, **opts)
    if kind == "ensemble":
        lo = 8 * rng.randint(2, 6)
        return dict(kind="ensemble", replicas=rng.randint(4, 48), edge=8 * rng.randint(4, 9), mixed=rng.randint(2, 16),
                    lo=lo, hi=lo + 8 * rng.randint(2, 9), steps=20, graph_steps=rng.choice([10, 20]), store=single,
                    kT=opts["kT"], gamma_bulk=opts["gamma_bulk"], pattern=opts["pattern"])
    if kind == "host":
        nx, ny, nz = _edges(rng, 32, 320, 256 ** 3)
        return dict(kind="host", nx=nx, ny=ny, nz=nz, steps=2 * rng.randint(1, 2), store=single, **opts)
    nx, ny, nz = _edges(rng, 16, 200, 128 ** 3)
    return dict(kind="fields", nx=nx, ny=ny, nz=nz, steps=0, store=single, **opts)


# ---------------------------------------------------------------------------------------------
# The boxes of a case
# ---------------------------------------------------------------------------------------------
def _full(case):
    c = dict(BASE)
    c.update(case)
    return c


def _boxes(case, seed):
    """One dict of box parameters per box of the case."""
    c = _full(case)
    keep = ("lattice", "store", "pattern", "kT", "gamma_shear", "gamma_bulk", "gamma_ghost", "force", "rho_local",
            "graph_steps", "u0")
    base = {k: c[k] for k in keep}
    base["seed"] = 1000 + seed
    if c["kind"] != "ensemble":
        return [dict(base, nx=c["nx"], ny=c["ny"], nz=c["nz"], replica=0)]
    n, lo, hi = c["mixed"], c["lo"], c["hi"]
    edges = [c["edge"]] * c["replicas"]
    edges += [lo + 8 * int(round((hi - lo) / 8 * j / max(1, n - 1))) for j in range(n)]
    shear = np.random.default_rng(4).uniform(0.0, 0.8, len(edges))
    return [dict(base, nx=e, ny=e, nz=e, replica=r, gamma_shear=float(g)) for r, (e, g) in enumerate(zip(edges, shear))]


def _sites(b):
    return b["nx"] * b["ny"] * b["nz"]


def _q(b):
    return 9 if b["lattice"] == "d2q9" else 19


def _plane(b):
    return (_sites(b) + 63) // 64 * 64


def _velocities(q):
    """(c [q, 3], a [q]): the lattice's velocities in the library's order, and its weights."""
    if q == 9:
        c = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]
        c = np.array([v + (0,) for v in c])
        return c, np.array([4 / 9, 1 / 9, 1 / 36])[(c ** 2).sum(1)]
    c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
         (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1),
         (1, 0, 1), (-1, 0, -1), (-1, 0, 1), (1, 0, -1)]
    c = np.array(c)
    return c, np.array([1 / 3, 1 / 18, 1 / 36])[(c ** 2).sum(1)]


def _fill(out, b, seed, box):
    """A thermal state (and the shear wave of the flow cases) into out [q, plane], in its storage type."""
    q, n = _q(b), _sites(b)
    c, a = _velocities(q)
    gen = torch.Generator(device=out.device)
    gen.manual_seed(1 + 1009 * int(seed) + box)
    wide = torch.float64 if out.dtype == torch.float64 else torch.float32
    wave = None
    if b["u0"]:
        z = torch.arange(n, device=out.device) // (b["nx"] * b["ny"])
        wave = (3.0 * b["u0"]) * torch.sin(z.to(wide) * (2.0 * math.pi / b["nz"]))
    for i in range(q):
        v = torch.randn(n, generator=gen, device=out.device, dtype=wide) * math.sqrt(3.0 * b["kT"] * a[i])
        if wave is not None and c[i][0]:
            v += float(a[i] * c[i][0]) * wave
        out[i, :n] = v


# ---------------------------------------------------------------------------------------------
# Device memory through the library's hook
# ---------------------------------------------------------------------------------------------
_stream = None
_expected = []      # (bytes, address or None) of the state buffers that the context being made will ask for
_placed = set()     # addresses inside a case's own state memory


def _alloc(nbytes, stream):
    if _expected and _expected[0][0] == nbytes:
        where = _expected.pop(0)[1]
        if where is not None:
            _placed.add(where)
            return where
    return torch.cuda.caching_allocator_alloc(nbytes, torch.cuda.current_device(), stream)


def _free(ptr, stream):
    if ptr in _placed:
        _placed.discard(ptr)
    else:
        torch.cuda.caching_allocator_delete(ptr)


def _offsets(boxes):
    """First element of every box's state in the memory of a case, and its length (both in elements)."""
    at, total = [], 0
    for b in boxes:
        at.append(total)
        total += (_q(b) * _plane(b) * BYTES[b["store"]] + 255) // 256 * 256 // BYTES[b["store"]]
    return at, total


def _context(case, boxes):
    """The context of a case, and its state: the current buffers of all boxes, one after another."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
        flb.flb_set_device_allocator(_alloc, _free)
    every = case["every"] if case["kind"] == "sampled" else 0
    cfgs = [flb.config(b["nx"], b["ny"], b["nz"], kT=b["kT"], gamma_shear=b["gamma_shear"],
                       gamma_bulk=b["gamma_bulk"], gamma_ghost=b["gamma_ghost"], seed=b["seed"],
                       replica=b["replica"], store=b["store"], pattern=b["pattern"], noise_rho_local=b["rho_local"],
                       force_amp=b["force"], graph_steps=b["graph_steps"], lattice=b["lattice"], stats_every=every,
                       stream=_stream) for b in boxes]
    es = BYTES[boxes[0]["store"]]
    at, total = _offsets(boxes)
    with torch.cuda.stream(_stream):
        memory = torch.zeros(total, dtype=DTYPE[boxes[0]["store"]], device="cuda")
    del _expected[:]
    for b, first in zip(boxes, at):
        nbytes = _q(b) * _plane(b) * es
        _expected.append((nbytes, memory.data_ptr() + first * es))
        if b["pattern"] == "ab":
            _expected.append((nbytes, None))
    ctx = flb.flb_create_ex(cfgs[0]) if len(cfgs) == 1 else flb.flb_create_batch(cfgs)
    if _expected:
        raise RuntimeError("the context did not ask for its state buffers in order")
    ctx.memory = memory     # lives as long as the context
    return ctx, memory


class _HostArray:
    """The bytes of a page-locked buffer, which lives as long as an array made from this."""

    def __init__(self, buffer):
        self.buffer = buffer
        self.__array_interface__ = dict(shape=(buffer.nbytes,), typestr="|u1", data=(buffer.ptr, False), version=3)


def _view(memory, boxes, i):
    b, first = boxes[i], _offsets(boxes)[0][i]
    return memory[first:first + _q(b) * _plane(b)].view(_q(b), _plane(b))


# ---------------------------------------------------------------------------------------------
# What the cases need
# ---------------------------------------------------------------------------------------------
def _shells(b):
    return int(math.ceil(math.sqrt(3.0) * max(b["nx"], b["ny"], b["nz"]) / 2.0)) + 2


def prepare(case, seed):
    boxes = _boxes(case, seed)
    state = dict(case=dict(case), boxes=boxes)
    b = boxes[0]
    if case["kind"] == "fields":
        raw = torch.zeros(_q(b), _plane(b), dtype=torch.float64, device="cuda")
        _fill(raw, b, seed, 0)
        a = torch.tensor(_velocities(_q(b))[1], device="cuda")[:, None]
        pops = (raw[:, :_sites(b)] + a).cpu().numpy().reshape(_q(b), b["nz"], b["ny"], b["nx"])
        state["populations"] = np.ascontiguousarray(pops)
    ctx, memory = _context(case, boxes)
    state.update(ctx=ctx, memory=memory)
    with torch.cuda.stream(_stream):
        for i, box in enumerate(boxes):
            _fill(_view(memory, boxes, i), box, seed, i)
        if case["kind"] == "host":
            host = flb.HostBuffer(ctx.flb_state_bytes())
            kind = {8: np.float64, 4: np.float32, 2: np.uint16}[BYTES[b["store"]]]
            ctx.flb_state_download(host.array)
            state.update(host=host, array=np.asarray(_HostArray(host)).view(kind))
    if case["kind"] == "sampled":
        ctx.flb_enable_structure_factor()
    _stream.synchronize()
    return state


def _single(b, x):
    """A result in the type the context computes it in."""
    return x if b["store"] == "f64" else np.asarray(x, dtype=np.float32)


def run(state):
    case, ctx, b = state["case"], state["ctx"], state["boxes"][0]
    kind = case["kind"]
    if kind in ("steps", "ensemble"):
        ctx.flb_step(case["steps"])
        return {"state": state["memory"]}
    if kind == "sampled":
        ctx.flb_stats_reset()
        ctx.flb_step(case["steps"])
        st = ctx.flb_mode_stats()
        S, count = ctx.flb_structure_factor(_shells(b))
        return {"state": state["memory"], "mode_m2": _single(b, st["mode_m2"]), "u2": _single(b, st["u2"]),
                "mass": st["mass_last"], "momentum": _single(b, st["momentum_last"]), "samples": int(st["nsamples"]),
                "nonfinite": int(st["nonfinite"]), "S": _single(b, S), "count": count}
    if kind == "profiles":
        rho, j = [], []
        for _ in range(case["steps"] // case["every"]):
            ctx.flb_step(case["every"])
            r, v = ctx.flb_z_profile()
            rho.append(r)
            j.append(v)
        return {"rho": _single(b, np.stack(rho)), "j": _single(b, np.stack(j)), "state": state["memory"]}
    if kind == "host":
        ctx.flb_step_host(state["host"].array, case["steps"])
        if b["store"] == "f32":
            return {"state": state["array"]}
        return {"state": torch.from_numpy(state["array"].view(np.int16)).view(DTYPE[b["store"]])}
    ctx.flb_set_populations(state["populations"])
    rho, j, Pi = ctx.flb_moments()
    return {"rho": rho, "j": j, "Pi": Pi, "populations": ctx.flb_get_populations()}


def work(case):
    """Every input read once, every output written once; FLOPs of the update: both mode transforms,
    equilibrium, relaxation and noise (320 per site and step on D3Q19, 130 on D2Q9), the Gaussian
    transform counted as 6 per pair."""
    boxes = _boxes(case, 0)
    flops = nbytes = 0.0
    for b in boxes:
        n, q = _sites(b), _q(b)
        nbytes += 2.0 * n * q * BYTES[b["store"]]
        flops += case["steps"] * n * ((320 + 6 * 8) if q == 19 else (130 + 6 * 3))
        if case["kind"] == "sampled":
            flops += case["steps"] // case["every"] * n * (150 + 2.5 * math.log2(max(2, n)))
            nbytes += 16.0 * _shells(b)
        if case["kind"] == "profiles":
            flops += case["steps"] // case["every"] * n * 48.0
            nbytes += case["steps"] // case["every"] * 32.0 * b["nz"]
        if case["kind"] == "fields":
            nbytes = n * 8.0 * (19 + 19 + 10)
            flops = n * 100.0
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------------
# The same in 64 bits, written from the paper with torch: the oracle of the outputs above
# ---------------------------------------------------------------------------------------------
def _basis(q):
    c, a = _velocities(q)
    x, y, z = c.T.astype(float)
    s = x * x + y * y + z * z
    if q == 9:
        e = [1 + 0 * s, x, y, 3 * s - 2, 2 * x * x - s, x * y, (3 * s - 4) * x, (3 * s - 4) * y,
             9 * s * s - 15 * s + 2]
    else:
        e = [1 + 0 * s, x, y, z, s - 1, 3 * x * x - s, y * y - z * z, x * y, y * z, z * x,
             (3 * s - 5) * x, (3 * s - 5) * y, (3 * s - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y,
             (x * x - y * y) * z, 3 * s * s - 6 * s + 1, (2 * s - 3) * (3 * x * x - s), (2 * s - 3) * (y * y - z * z)]
    e = np.array(e)
    return c, a, e, (a * e * e).sum(1)


def _philox(site, step, replica, block, seed):
    """Philox-4x32-10 words of counters (site, step, replica, block), as int64 tensors."""
    mask = 0xFFFFFFFF
    c0, c1, c2, c3 = site, torch.full_like(site, step), torch.full_like(site, replica), torch.full_like(site, block)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57      # wraps modulo 2^64: the bits are those of the product
        c0, c2 = ((p1 >> 32) & mask) ^ c1 ^ k0, ((p0 >> 32) & mask) ^ c3 ^ k1
        c1, c3 = p1 & mask, p0 & mask
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c0, c1, c2, c3


class _Exact:
    """One box in 64 bits: n [q, nz, ny, nx], the canonical deviations at step t."""

    def __init__(self, b, device):
        self.b, self.t, self.device = b, 0, device
        q = _q(b)
        self.c, self.a, e, self.w = _basis(q)
        self.E = torch.tensor(e, device=device)
        self.shape = (b["nz"], b["ny"], b["nx"])
        gs, gb, gk = b["gamma_shear"], b["gamma_bulk"], b["gamma_ghost"]
        first = 3 if q == 9 else 4          # the first relaxing mode
        g = np.ones(q)
        g[first] = gb
        nshear = 2 if q == 9 else 5
        g[first + 1:first + 1 + nshear] = gs
        g[first + 1 + nshear:] = gk
        self.first, self.gamma = first, torch.tensor(g, device=device)
        self.sigma = np.sqrt(3.0 * b["kT"] * self.w * (1.0 - g * g))
        self.back = torch.tensor(self.a[:, None] * e.T / self.w[None, :], device=device)
        u = (torch.arange(65536, device=device, dtype=torch.float64) + 0.5) / 65536.0
        self.R, self.cs = torch.sqrt(-2.0 * torch.log(u)), torch.cos(2.0 * math.pi * u)
        self.sn = torch.sin(2.0 * math.pi * u)
        raw = torch.zeros(q, _plane(b), dtype=DTYPE[b["store"]], device=device)
        self.raw = raw

    def load(self):
        n = self.raw[:, :_sites(self.b)].double().view((_q(self.b),) + self.shape)
        self.n = self._moved(n, 1) if self.b["pattern"] == "ab" else n.clone()

    def store(self):
        """The state after an even number of steps, in the library's layout."""
        n = self._moved(self.n, -1) if self.b["pattern"] == "ab" else self.n
        out = torch.zeros(_q(self.b), _plane(self.b), dtype=torch.float64, device=self.device)
        out[:, :_sites(self.b)] = n.reshape(_q(self.b), -1)
        return out.reshape(-1)

    def _moved(self, n, sign):
        out = torch.empty_like(n)
        for i, (x, y, z) in enumerate(self.c):
            out[i] = torch.roll(n[i], (sign * int(z), sign * int(y), sign * int(x)), (0, 1, 2))
        return out

    def _collide(self, n, z0):
        """Post-collision deviations of planes z0 .. of n [q, planes, ny, nx] (rows y of a D2Q9 box)."""
        b, q = self.b, _q(self.b)
        two = q == 9
        shape = n.shape[1:]
        m = (self.E @ n.reshape(q, -1)).reshape((q,) + tuple(shape))
        F = 0.0
        if b["force"]:
            if two:
                ph = torch.arange(shape[1], device=self.device, dtype=torch.float64)[None, :, None] / b["ny"]
            else:
                ph = torch.arange(z0, z0 + shape[0], device=self.device, dtype=torch.float64)[:, None, None] / b["nz"]
            F = b["force"] * torch.sin(2.0 * math.pi * ph)
        rho = 1.0 + m[0]
        px, py = m[1] + 0.5 * F, m[2]
        ux, uy = px / rho, py / rho
        eq, src = {}, {}
        if two:
            eq[3], eq[4], eq[5] = 3.0 * (px * ux + py * uy), px * ux - py * uy, px * uy
            src[3], src[4], src[5] = 6.0 * ux * F, 2.0 * ux * F, uy * F
        else:
            pz = m[3]
            uz = pz / rho
            xx, yy, zz = px * ux, py * uy, pz * uz
            eq[4], eq[5], eq[6] = xx + yy + zz, 2.0 * xx - yy - zz, yy - zz
            eq[7], eq[8], eq[9] = px * uy, py * uz, pz * ux
            src[4], src[5], src[7], src[9] = 2.0 * ux * F, 4.0 * ux * F, uy * F, uz * F
        scale = torch.sqrt(rho) if b["rho_local"] else 1.0
        cells = shape[0] * shape[1] * shape[2]
        site = torch.arange(cells, device=self.device, dtype=torch.int64) + z0 * shape[1] * shape[2]
        words = []
        for block in range(1 if two else 2):
            words += _philox(site, self.t, b["replica"], block, b["seed"])
        m[1] = m[1] + F
        for k in range(self.first, q):
            g = float(self.gamma[k])
            v = g * m[k]
            if k in eq:
                v = v + (1.0 - g) * eq[k]
            if k in src and b["force"]:
                v = v + 0.5 * (1.0 + g) * src[k]
            if self.sigma[k] > 0.0:
                p = k - self.first
                word = words[p // 2]
                normal = self.R[word & 0xFFFF] * (self.sn if p & 1 else self.cs)[word >> 16]
                v = v + (float(self.sigma[k]) * scale) * normal.view(shape)
            m[k] = v
        return (self.back @ m.reshape(q, -1)).reshape((q,) + tuple(shape))

    def step(self, steps):
        per = max(1, (1 << 24) // max(1, self.shape[1] * self.shape[2]))
        for _ in range(steps):
            for z0 in range(0, self.shape[0], per):
                self.n[:, z0:z0 + per] = self._collide(self.n[:, z0:z0 + per], z0)
            self.n = self._moved(self.n, 1)
            self.t += 1

    def modes(self):
        return torch.stack([torch.tensordot(self.E[k], self.n, 1) for k in range(_q(self.b))])


def _shell_of(b):
    f = []
    for n in (b["nx"], b["ny"], b["nz"]):
        k = np.arange(n)
        f.append(np.where(k <= n // 2, k, k - n) / n)
    fx, fy, fz = f[0][None, None, :], f[1][None, :, None], f[2][:, None, None]
    return np.floor(max(b["nx"], b["ny"], b["nz"]) * np.sqrt((fx * fx + fy * fy) + fz * fz)).astype(np.int64)


def exact(case, seed):
    boxes = _boxes(case, seed)
    kind = case["kind"]
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if sum(_sites(b) for b in boxes) * max(1, case["steps"]) > (3e9 if device == "cuda" else 2e6):
        return None
    b = boxes[0]
    if kind == "ensemble":
        at, total = _offsets(boxes)
        out = torch.zeros(total, dtype=torch.float64, device=device)
        for i, box in enumerate(boxes):
            x = _Exact(box, device)
            _fill(x.raw, box, seed, i)
            x.load()
            x.step(case["steps"])
            out[at[i]:at[i] + x.raw.numel()] = x.store()
        return {"state": out}
    x = _Exact(b, device)
    if kind == "fields":
        x.raw = torch.zeros(_q(b), _plane(b), dtype=torch.float64, device=device)
        _fill(x.raw, b, seed, 0)
        x.n = x.raw[:, :_sites(b)].view((_q(b),) + x.shape)
        pops = x.n + torch.tensor(x.a, device=device)[:, None, None, None]
        c = torch.tensor(x.c, device=device, dtype=torch.float64)
        pairs = [(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (2, 0)]
        j = torch.stack([torch.tensordot(c[:, d], pops, 1) for d in range(3)])
        if b["force"]:
            z = torch.arange(b["nz"], device=device, dtype=torch.float64)[:, None, None] / b["nz"]
            j[0] += 0.5 * b["force"] * torch.sin(2.0 * math.pi * z)
        Pi = torch.stack([torch.tensordot(c[:, d] * c[:, e], pops, 1) for d, e in pairs])
        return {"rho": pops.sum(0), "j": j, "Pi": Pi, "populations": pops}
    _fill(x.raw, b, seed, 0)
    x.load()
    if kind in ("steps", "host"):
        x.step(case["steps"])
        return {"state": x.store()}
    samples = case["steps"] // case["every"]
    n = _sites(b)
    if kind == "profiles":
        rho, js = [], []
        z = torch.arange(b["nz"], device=device, dtype=torch.float64) / b["nz"]
        for _ in range(samples):
            x.step(case["every"])
            m = x.modes()[:4].mean((2, 3))
            m[1] += 0.5 * b["force"] * torch.sin(2.0 * math.pi * z)
            rho.append(1.0 + m[0])
            js.append(m[1:4])
        return {"rho": torch.stack(rho), "j": torch.stack(js), "state": x.store()}
    shell, ns = torch.tensor(_shell_of(b), device=device), _shells(b)
    shell[0, 0, 0] = ns
    count = torch.bincount(shell.reshape(-1), minlength=ns + 1)[:ns]
    m2, u2, S = 0.0, 0.0, 0.0
    for _ in range(samples):
        x.step(case["every"])
        m = x.modes()
        m2 = m2 + (m * m).mean((1, 2, 3)) / samples
        u = m[1:4] / (1.0 + m[0])
        u2 = u2 + (u * u).mean((1, 2, 3)) / samples
        power = torch.fft.fftn(m[0]).abs().square() / n
        S = S + torch.bincount(shell.reshape(-1), weights=power.reshape(-1), minlength=ns + 1)[:ns] / samples
    return {"state": x.store(), "mode_m2": m2, "u2": u2, "mass": float(m[0].sum()) + n, "momentum": m[1:4].sum((1, 2, 3)),
            "samples": samples, "nonfinite": 0, "S": S / count.clamp(min=1), "count": count}
