"""Workloads of the planar photoacoustic operator, as a user's program runs them.

A case names a grid, a library, an entry point and its options; `prepare` makes the plan and
the inputs on the GPU, `run` makes one pass through the public entry points, and `exact` is the
same result in 64 bits from plain torch (its own library, FFTs and loops over depth).

Fields of a case: op (forward, adjoint, pair, gradient, autograd, fista, serve), nx ny nz nt px py,
lib ("kspace": the homogeneous-medium library; "measured": a table without symmetries, complex
spectra), fp64, batch (volumes of one call; requests of "serve"), tensor (split-BF16 contraction),
samp (scan step of the measurement operator), iters, lam.
"""
import math

import torch

from paper_2603_28150_gb300 import Medium, Plan, apply

DEV = "cuda"
L2_BYTES = 126e6
C, DX, DT = 1500.0, 50e-6, 10e-9     # m/s, m (dx = dy = dz), s
CDT = C * DT / DX                    # voxels that sound travels in one sample
POWER_ITERS, MARGIN = 40, 1.1        # step size: 1.1 x the power iteration's estimate
LENGTHS = sorted([16 << k for k in range(7)] + [24 << k for k in range(6)])


def padded(n):
    """The shortest supported transform length that holds a linear convolution (P >= 2n - 1)."""
    return next(p for p in LENGTHS if p >= 2 * n - 1)


def case_of(op, nx, ny, nz, nt, px, py, lib="kspace", fp64=False, batch=1, tensor=False, samp=1,
            iters=0, lam=0.0):
    return dict(op=op, nx=nx, ny=ny, nz=nz, nt=nt, px=px, py=py, lib=lib, fp64=fp64, batch=batch,
                tensor=tensor, samp=samp, iters=iters, lam=lam)


def listed():
    c = case_of
    return [
        # the smallest grid in use: one simulated data set of a 32^2 x 16 volume; latency
        dict(c("forward", 32, 32, 16, 64, 64, 64), name="forward_32"),
        # one gradient of a learned or regularised reconstruction through torch.autograd
        dict(c("autograd", 64, 64, 32, 128, 128, 128), name="autograd_64"),
        # the same grid in double precision: gradient checks, reference reconstructions
        dict(c("gradient", 64, 64, 32, 128, 128, 128, fp64=True), name="gradient_64_fp64"),
        # serving: five requests of the small geometry advance together for 50 iterations
        dict(c("serve", 64, 64, 32, 128, 128, 128, batch=5, iters=50), name="serve_64"),
        # three volumes on a ragged grid, 3 * 2^k transforms, one H and one H* (a Landweber step)
        dict(c("pair", 89, 96, 45, 150, 192, 192, batch=3), name="pair_96_batch3"),
        # the usual reconstruction: 100 iterations on 128^2 x 64 depths x 256 samples
        dict(c("fista", 128, 128, 64, 256, 256, 256, iters=100), name="fista_128"),
        # the same grid with a measured (asymmetric) library: complex spectra for every bin
        dict(c("pair", 128, 128, 64, 256, 256, 256, lib="measured"), name="plain_128"),
        # the wire phantom's voxels, data on every second position, 15 iterations with a prior
        dict(c("fista", 202, 202, 17, 201, 512, 512, samp=2, iters=15, lam=2e-5), name="wire_202"),
        # the in vivo scan grid with a measured library, fewer depths than the full experiment
        dict(c("pair", 384, 326, 12, 40, 768, 768, lib="measured"), name="invivo_384"),
        # one gradient on the largest serving geometry
        dict(c("gradient", 256, 256, 128, 512, 512, 512), name="gradient_256"),
        # sixteen volumes sharing one geometry on the tensor cores
        dict(c("pair", 128, 128, 128, 512, 256, 256, batch=16, tensor=True), name="batch16_128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any entry point, any grid of the range, ragged sizes among them."""
    most = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["forward", "adjoint", "pair", "gradient", "autograd", "fista", "serve"])
        lib = rng.choice(["kspace", "kspace", "kspace", "measured"]) if op != "serve" else "kspace"
        fp64 = op in ("pair", "gradient", "autograd") and rng.random() < 0.15
        tensor = op in ("pair", "serve") and lib == "kspace" and not fp64 and rng.random() < 0.3
        nx = _log_int(rng, 20, 128 if lib == "measured" or fp64 or tensor else 256)
        ny = nx if rng.random() < 0.5 else max(16, int(nx * rng.uniform(0.6, 1.0)))
        nz, nt = _log_int(rng, 6, 128), _log_int(rng, 24, 512)
        px = py = padded(max(nx, ny))
        if lib == "measured":
            py = padded(ny)
            nz, nt = min(nz, 48), min(nt, 160)
        if fp64:
            nz, nt = min(nz, 40), min(nt, 160)
        if tensor:
            nz, nt = 128, 128 * rng.randint(1, 4)
        batch = 1
        if tensor:
            batch = rng.randint(2, 16)
        elif op == "serve":
            batch = rng.randint(1, 8)
        elif op in ("forward", "adjoint", "pair") and rng.random() < 0.4:
            batch = rng.randint(2, 6)
        samp = rng.choice([1, 1, 1, 2, 3]) if not tensor else 1
        iters = rng.choice([5, 10, 15, 25, 50]) if op in ("fista", "serve") else 0
        lam = rng.choice([0.0, 2e-5]) if op in ("fista", "serve") else 0.0
        case = case_of(op, nx, ny, nz, nt, px, py, lib, fp64, batch, tensor, samp, iters, lam)
        vol = batch * max(nz, nt) * (px // 2 + 1) * py * 8.0
        if _cost(case) <= 0.6 * most and vol <= 8e9:
            return case


# ---- inputs --------------------------------------------------------------------------------

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _sources(c, seed, salt):
    """Absorbers along a few random walks and single beads: centres (z, y, x), widths, amplitudes."""
    g = _gen(seed, salt)
    walks, steps, beads = 4, 24, 8
    n = torch.tensor([c["nz"], c["ny"], c["nx"]], dtype=torch.float64, device=DEV)
    start = torch.rand(walks, 1, 3, generator=g, dtype=torch.float64, device=DEV) * (n - 1)
    turn = torch.randn(walks, steps, 3, generator=g, dtype=torch.float64, device=DEV) * 0.3
    way = torch.randn(walks, 1, 3, generator=g, dtype=torch.float64, device=DEV) + turn.cumsum(1)
    path = start + (2.0 * way / way.norm(dim=-1, keepdim=True)).cumsum(1)
    path = torch.minimum(path.clamp_min(0), n - 1).reshape(-1, 3)
    bead = torch.rand(beads, 3, generator=g, dtype=torch.float64, device=DEV) * (n - 1)
    at = torch.cat([path, bead])
    width = 1.0 + 2.0 * torch.rand(at.shape[0], generator=g, dtype=torch.float64, device=DEV)
    amp = 0.5 + 0.5 * torch.rand(at.shape[0], generator=g, dtype=torch.float64, device=DEV)
    return at, width, amp


def _phantom(c, seed, salt):
    """Initial pressure [nz][ny][nx]: Gaussian absorbers on zero."""
    at, w, amp = _sources(c, seed, salt)
    prof = []
    for axis, n in enumerate((c["nz"], c["ny"], c["nx"])):
        r = torch.arange(n, dtype=torch.float64, device=DEV)[None, :] - at[:, axis, None]
        prof.append(torch.exp(-r * r / (2 * w[:, None] ** 2)))
    zy = (amp[:, None, None] * prof[0][:, :, None] * prof[1][:, None, :]).reshape(len(amp), -1)
    return (zy.t() @ prof[2]).reshape(c["nz"], c["ny"], c["nx"])


def _signals(c, seed, salt):
    """Measured time series [nt][my][mx] of such absorbers: the wave of a Gaussian source on the
    scan positions, (r - ct) exp(-(r - ct)^2 / 2w^2) / r, with 5 % noise."""
    at, w, amp = _sources(c, seed, salt)
    s = c["samp"]
    y = torch.arange(0, c["ny"], s, dtype=torch.float64, device=DEV)
    x = torch.arange(0, c["nx"], s, dtype=torch.float64, device=DEV)
    ct = CDT * torch.arange(c["nt"], dtype=torch.float64, device=DEV)[:, None, None]
    d = torch.zeros(c["nt"], len(y), len(x), dtype=torch.float64, device=DEV)
    for j in range(0, len(amp), 4):   # every fourth absorber: enough arrivals in every trace
        dz, dy, dx = at[j, 0] + 1.0, y - at[j, 1], x - at[j, 2]
        r = torch.sqrt(dz * dz + (dy * dy)[:, None] + (dx * dx)[None, :])
        u = r[None] - ct
        d += amp[j] * u * torch.exp(-u * u / (2 * w[j] ** 2)) / r[None]
    noise = torch.randn(d.shape, generator=_gen(seed, salt + 1), dtype=torch.float64, device=DEV)
    return d + 0.05 * d.square().mean().sqrt() * noise


def _stack(make, c, seed, salt, dtype):
    return torch.stack([make(c, seed, salt + 10 * b).to(dtype) for b in range(c["batch"])])


def _measured_depths(c, seed):
    """The measured library a depth at a time: complex spectra [nt][py][px/2+1] of real kernels
    without symmetries, decaying in time and depth, complex64 as such a library is stored."""
    g = _gen(seed, 7)
    fall = torch.exp(-torch.arange(c["nt"], device=DEV, dtype=torch.float32) / c["nt"])
    for z in range(c["nz"]):
        h = torch.randn(c["nt"], c["py"], c["px"], generator=g, device=DEV)
        h *= (fall / ((1.0 + 0.05 * z) * math.sqrt(c["px"] * c["py"])))[:, None, None]
        yield torch.fft.rfft2(h)


def _mz(c):
    need = 2 + c["nz"] + math.ceil(CDT * c["nt"])
    return 1 << (need - 1).bit_length()


def _kspace_rows(c):
    """The homogeneous medium's library in closed form, 64 bits: H[z][t][radius] and the radius of
    every half-spectrum bin [py][px/2+1] (equal spacing, square padded grid)."""
    P, mz = c["px"], _mz(c)
    f = torch.fft.fftfreq(P, 1.0 / P, dtype=torch.float64, device=DEV).abs()
    r2 = (f[:, None] ** 2 + f[None, :P // 2 + 1] ** 2)
    radii, where = torch.unique(r2, return_inverse=True)
    m = torch.arange(mz // 2 + 1, dtype=torch.float64, device=DEV)
    weight = torch.full_like(m, 2.0)
    weight[0] = weight[-1] = 1.0
    z = 1.0 + torch.arange(c["nz"], dtype=torch.float64, device=DEV)
    W = (weight[:, None] / mz) * torch.cos(2 * math.pi * ((m[:, None] * z[None, :]) % mz) / mz)
    t = torch.arange(c["nt"], dtype=torch.float64, device=DEV)
    H = torch.empty(c["nz"], c["nt"], len(radii), dtype=torch.float64, device=DEV)
    step = max(1, int(1.5e8 / (c["nt"] * len(m))))
    for i in range(0, len(radii), step):
        k = torch.sqrt(radii[i:i + step, None] / P ** 2 + (m[None, :] / mz) ** 2)
        turns = (CDT * t[None, :, None] * k[:, None, :]) % 1.0
        H[:, :, i:i + step] = (torch.cos(2 * math.pi * turns) @ W).permute(2, 1, 0)
    return H, where


# ---- a pass --------------------------------------------------------------------------------

def _plan(c, seed):
    kw = dict(max_batch=c["batch"], fp64=c["fp64"], bf16_split=c["tensor"])
    if c["lib"] == "kspace" and not c["fp64"]:
        kw["medium"] = Medium(c=C, dx=DX, dy=DX, dz=DX, dt=DT, mz=_mz(c), z0=1)
    elif c["lib"] == "kspace":   # a double-precision plan takes its library as a table
        H, where = _kspace_rows(c)
        kw["table"] = torch.stack([h[:, where].to(torch.complex128) for h in H])
    else:
        t = torch.empty(c["nz"], c["nt"], c["py"], c["px"] // 2 + 1, dtype=torch.complex64,
                        device=DEV)
        for z, h in enumerate(_measured_depths(c, seed)):
            t[z] = h
        kw["table"] = t.to(torch.complex128) if c["fp64"] else t
    plan = Plan(c["nx"], c["ny"], c["nz"], c["nt"], c["px"], c["py"], **kw)
    if c["samp"] > 1:
        plan.set_sampling(c["samp"], c["samp"])
    return plan


def _start_vector(c, seed):
    return torch.rand(c["nz"], c["ny"], c["nx"], generator=_gen(seed, 3), dtype=torch.float64,
                      device=DEV)


def prepare(case, seed):
    c = case
    dt = torch.float64 if c["fp64"] else torch.float32
    s = {"case": c, "plan": _plan(c, seed)}
    if c["op"] in ("forward", "pair", "gradient", "autograd"):
        s["rho"] = _stack(_phantom, c, seed, 1000, dt)
    if c["op"] != "forward":
        s["y"] = _stack(_signals, c, seed, 2000, dt)
    if c["op"] in ("fista", "serve"):   # the step size, found once per plan
        s["L"] = MARGIN * s["plan"].power_norm(_start_vector(c, seed).to(dt), POWER_ITERS)
    return s


def run(s):
    c, plan = s["case"], s["plan"]
    op = c["op"]
    if op == "forward":
        return plan.forward(s["rho"])
    if op == "adjoint":
        return plan.adjoint(s["y"])
    if op == "pair":
        return plan.forward(s["rho"]), plan.adjoint(s["y"])
    if op == "gradient":
        g, r2 = plan.gradient(s["rho"], s["y"])
        return {"grad": g, "resid2": r2}
    if op == "autograd":
        x = s["rho"].detach().requires_grad_(True)
        loss = 0.5 * (apply(plan, x) - s["y"]).square().sum()
        loss.backward()
        return {"loss": loss.detach(), "grad": x.grad}
    if op == "fista":
        x, rep = plan.fista(s["y"], iters=c["iters"], lam=c["lam"], L=s["L"])
        return {"x": x, "resid2": rep["resid2_last"]}
    for b in range(c["batch"]):
        plan.slot_load(b, s["y"][b], c["lam"], s["L"])
    for _ in range(c["iters"]):
        plan.slots_step(c["batch"])
    return [plan.slot_read(b)[0] for b in range(c["batch"])]


# ---- what a pass cannot do without ---------------------------------------------------------

def _library_bytes(c):
    """The library once: one row per radius where it depends on the radius only, else per bin."""
    if c["lib"] == "kspace":
        h = c["px"] // 2
        rows = len({a * a + b * b for a in range(h + 1) for b in range(a, h + 1)})
        return rows * c["nz"] * c["nt"] * (8.0 if c["fp64"] else 4.0)
    return (c["px"] // 2 + 1) * c["py"] * c["nz"] * c["nt"] * (16.0 if c["fp64"] else 8.0)


def _applications(c):
    return {"forward": 1, "adjoint": 1, "pair": 2, "gradient": 2, "autograd": 2,
            "fista": 2 * c["iters"], "serve": 2 * c["iters"]}[c["op"]]


def work(case):
    """Bytes: the library once per application (once in all where it fits the cache), the volumes
    and data of a call read and written once. Flops: the contraction of every half-spectrum bin and
    the 2D real transforms of every slice."""
    c, n = case, _applications(case)
    e = 8.0 if c["fp64"] else 4.0
    lib = _library_bytes(c)
    obj = c["batch"] * c["nz"] * c["ny"] * c["nx"] * e
    dat = c["batch"] * c["nt"] * -(-c["ny"] // c["samp"]) * -(-c["nx"] // c["samp"]) * e
    io = {"forward": obj + dat, "adjoint": obj + dat, "pair": 2 * (obj + dat)}.get(
        c["op"], 2 * obj + dat)
    bins = (c["px"] // 2 + 1) * c["py"]
    mac = bins * c["nz"] * c["nt"] * (4.0 if c["lib"] == "kspace" else 8.0)
    P2 = float(c["px"] * c["py"])
    fft = (c["nz"] + c["nt"]) * 2.5 * P2 * math.log2(P2)
    return {"bytes": lib * (n if lib > L2_BYTES else 1) + io, "flops": n * c["batch"] * (mac + fft)}


def _cost(c):
    w = work(c)
    return max(w["bytes"] / 6.7e12, w["flops"] / (1.0e12 if c["fp64"] else 4e13))


# ---- the same in 64 bits -------------------------------------------------------------------

class _Exact:
    """H (with the measurement operator) and its transpose, complex128, a depth at a time."""

    def __init__(self, c, seed):
        self.c = c
        if c["lib"] == "kspace":
            self.H, self.where = _kspace_rows(c)
        else:
            self.table = [h for h in _measured_depths(c, seed)]

    def depth(self, z):
        if self.c["lib"] == "kspace":
            return self.H[z][:, self.where]
        return self.table[z].to(torch.complex128)

    def _fft(self, a):
        return torch.fft.rfft2(a, s=(self.c["py"], self.c["px"]))

    def _image(self, F):
        out = [torch.fft.irfft2(f, s=(self.c["py"], self.c["px"]))[..., :self.c["ny"], :self.c["nx"]]
               for f in F.split(max(1, int(4e8 / (F.shape[-1] * F.shape[-2]))))]
        return torch.cat(out)

    def forward(self, rho):
        X = self._fft(rho)
        Y = torch.zeros(self.c["nt"], *X.shape[1:], dtype=torch.complex128, device=DEV)
        for z in range(self.c["nz"]):
            Y += self.depth(z) * X[z]
        s = self.c["samp"]
        return self._image(Y)[:, ::s, ::s].contiguous()

    def adjoint(self, d):
        s = self.c["samp"]
        full = torch.zeros(self.c["nt"], self.c["ny"], self.c["nx"], dtype=torch.float64, device=DEV)
        full[:, ::s, ::s] = d
        D = self._fft(full)
        Z = torch.stack([(self.depth(z).conj() * D).sum(0) for z in range(self.c["nz"])])
        return self._image(Z)

    def step_size(self, seed):
        v = _start_vector(self.c, seed).to(torch.float32).double()
        for _ in range(POWER_ITERS):
            w = self.adjoint(self.forward(v / v.norm()))
            v = w
        return MARGIN * float(v.norm())

    def fista(self, y, L, iters, lam):
        x = torch.zeros(self.c["nz"], self.c["ny"], self.c["nx"], dtype=torch.float64, device=DEV)
        v, t, r2 = x, 1.0, 0.0
        for _ in range(iters):
            r = self.forward(v) - y
            r2 = float(r.square().sum())
            new = (v - self.adjoint(r) / L - lam / L).clamp_min(0)
            tn = (1.0 + math.sqrt(1.0 + 4.0 * t * t)) / 2.0
            v, x, t = new + (t - 1.0) / tn * (new - x), new, tn
        return x, r2


def exact(case, seed):
    c, op, B = case, case["op"], case["batch"]
    slow = _applications(c) * B + (2 * POWER_ITERS if c["iters"] else 0)
    if slow * c["nz"] * c["nt"] * c["px"] * c["py"] > 4e12:   # the loops would take too long
        return None
    A = _Exact(c, seed)
    dt = torch.float64 if c["fp64"] else torch.float32
    if op in ("forward", "pair", "gradient", "autograd"):
        rho = _stack(_phantom, c, seed, 1000, dt).double()
    if op != "forward":
        y = _stack(_signals, c, seed, 2000, dt).double()
    if op == "forward":
        return torch.stack([A.forward(r) for r in rho])
    if op == "adjoint":
        return torch.stack([A.adjoint(d) for d in y])
    if op == "pair":
        return torch.stack([A.forward(r) for r in rho]), torch.stack([A.adjoint(d) for d in y])
    if op in ("gradient", "autograd"):
        r = A.forward(rho[0]) - y[0]
        r2, g = float(r.square().sum()), A.adjoint(r)[None]
        return {"grad": g, "resid2": r2} if op == "gradient" else {
            "loss": torch.tensor(0.5 * r2, dtype=torch.float64, device=DEV), "grad": g}
    L = A.step_size(seed)
    if op == "fista":
        x, r2 = A.fista(y[0], L, c["iters"], c["lam"])
        return {"x": x[None], "resid2": r2}
    return [A.fista(d, L, c["iters"], c["lam"])[0] for d in y]
