"""The work this library is used for, as cases that can be timed and checked.

Every case goes through the public entry points (`pic.Context`, `pic.Batch`, the
C-ABI calls behind them).  A case names the kind of call and its sizes:

  step         a context advances its plasma by `steps` steps, then the program
               reads every field and every particle (in the order of the ids),
               as a run does that writes its state out every so many steps
  batch        the same for many independent boxes stepped together
  adjoint      `steps` steps and the discrete adjoint of the field energy
  diagnostics  the nodal charge density and the energy/charge/div B sums

The workloads are the repository's own recipes (uniform thermal plasmas of 1 to
8 particles per cell at orders 1 to 3, the laser-wakefield moving window, the
ensemble of uneven boxes, the driven plasma of the adjoint) on its sizes and on
grids that no power of two divides.  The precision is part of the case: FP64, or
FP32-mixed, where the library holds and computes the state in 32 bits; its
getters hand that state out widened to 64 bits, and the program keeps it as the
32-bit values it is.

`exact` is a plain PIC step in torch, in 64 bits, written from the method.
"""
import ctypes as ct
import math
import random

import torch

from paper_2101_12149_gb300 import pic

DEV = "cuda"
KEYS = ("x", "y", "z", "ux", "uy", "uz", "w")
SIGMA_U = 0.05  # thermal momentum of the uniform plasmas
FLOPS = {1: 601, 2: 1354, 3: 2491}  # of one particle's gather, push and deposit, by order


def _step(name, n, ppc, order, steps, fp64=False, vay=False, energy=False, ckc=False, passes=0, window=False):
    return {"name": name, "kind": "step", "nx": n[0], "ny": n[1], "nz": n[2], "ppc": ppc, "order": order,
            "fp64": fp64, "steps": steps, "vay": vay, "energy": energy, "ckc": ckc, "passes": passes,
            "window": window}


def _adjoint(name, n, ppc, order, steps, every, fp64):
    return {"name": name, "kind": "adjoint", "nx": n[0], "ny": n[1], "nz": n[2], "ppc": ppc, "order": order,
            "fp64": fp64, "steps": steps, "every": every}


def listed():
    return [
        # the smallest runs: a parameter scan's or a test's box, where launches and latency count
        _step("box16_o3", (16, 16, 16), 2, 3, 20),
        # the small FP64 verification run (50 steps between outputs)
        _step("uniform32_o1_fp64", (32, 32, 32), 2, 1, 50, fp64=True),
        # the weak-scaling study's per-GPU problem: 8 particles per cell, order 3
        _step("uniform256_o3", (256, 256, 256), 8, 3, 6),
        # the same grid at wakefield-like 2 particles per cell and order 1: the memory-bound end
        _step("uniform256_o1", (256, 256, 256), 2, 1, 10),
        # the production order in FP64
        _step("uniform64_o3_fp64", (64, 64, 64), 8, 3, 4, fp64=True),
        # a grid whose extents come from the physics, not from powers of two
        _step("ragged100x75x90_o2", (100, 75, 90), 4, 2, 6),
        # plasma acceleration: laser, moving window, removal and injection
        _step("window64x64x512_o2", (64, 64, 512), 2, 2, 10, window=True),
        # the boosted-frame run's algorithms: Vay, energy-conserving gather, CKC, z filter
        _step("options96x96x128_o3", (96, 96, 128), 4, 3, 6, vay=True, energy=True, ckc=True, passes=2),
        # many uneven boxes stepped together (orders 1 and 3)
        {"name": "batch24", "kind": "batch", "boxes": 24, "mix": 3, "edge": 64, "fp64": False, "steps": 10},
        # differentiation: forward steps, checkpoints and the reverse sweep
        _adjoint("adjoint64_o2", (64, 64, 64), 4, 2, 10, 5, False),
        _adjoint("adjoint32_o2_fp64", (32, 32, 32), 4, 2, 10, 5, True),
        # in-situ diagnostics of a running plasma
        {"name": "diagnostics128_o3", "kind": "diagnostics", "nx": 128, "ny": 128, "nz": 128, "ppc": 8,
         "order": 3, "fp64": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extents(rng, lo, hi):
    """Three extents around one size; a third of the grids have extents that 16 divides, a third 4, the rest any."""
    size = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    unit = rng.choice((16, 4, 1))
    out = []
    for _ in range(3):
        v = size * math.exp(rng.uniform(-0.5, 0.5))
        out.append(int(min(max(int(round(v / unit)) * unit, lo, unit), hi)))
    return out


def draw(rng):
    kind = rng.choice(("step",) * 6 + ("batch", "adjoint", "diagnostics"))
    fp64 = rng.random() < 0.3
    while True:
        if kind == "batch":
            return {"kind": "batch", "boxes": _log_int(rng, 4, 32), "mix": rng.randrange(1 << 20),
                    "edge": rng.choice((32, 48, 64)), "fp64": False, "steps": rng.randint(4, 10)}
        if kind == "adjoint":
            n = _extents(rng, 16, 64)
            c = _adjoint("", n, rng.randint(1, 4), rng.randint(1, 3), rng.randint(4, 10), rng.choice((2, 5)),
                         fp64 and max(n) <= 40)
            if n[0] * n[1] * n[2] * c["ppc"] > 64 ** 3 * 4:
                continue
        elif kind == "diagnostics":
            n = _extents(rng, 16, 160)
            c = {"kind": "diagnostics", "nx": n[0], "ny": n[1], "nz": n[2], "ppc": rng.randint(1, 8),
                 "order": rng.randint(1, 3), "fp64": fp64}
        else:
            window = rng.random() < 0.2
            n = _extents(rng, 12, 64 if fp64 else 224)
            if window:
                n = [min(max(n[0], 24), 96), min(max(n[1], 24), 96), rng.choice((128, 192, 250, 256, 384, 512))]
            c = _step("", n, rng.randint(1, 2) if window else rng.randint(1, 8), rng.randint(1, 3),
                      rng.randint(4, 10), fp64 and not window, vay=rng.random() < 0.3, energy=rng.random() < 0.3,
                      ckc=not window and rng.random() < 0.2, passes=0 if window else rng.choice((0, 0, 0, 1, 2)),
                      window=window)
        c.pop("name", None)
        w = FLOPS[c["order"]] * c["nx"] * c["ny"] * c["nz"] * c["ppc"] * c.get("steps", 1)
        if w <= 2.5e11:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _plasma(g, n, ppc, density=1.0, sigma=SIGMA_U):
    """Uniform thermal plasma, ppc particles at random places of every cell, cell after cell."""
    C = n[0] * n[1] * n[2]
    cell = torch.arange(C, device=DEV).repeat_interleave(ppc)
    out = {"x": cell // (n[1] * n[2]), "y": cell // n[2] % n[1], "z": cell % n[2]}
    for k in "xyz":
        out[k] = out[k].double().add_(_rand(g, C * ppc))
    for k in ("ux", "uy", "uz"):
        out[k] = torch.randn(C * ppc, generator=g, device=DEV, dtype=torch.float64).mul_(sigma)
    out["w"] = torch.full((C * ppc,), density / ppc, device=DEV, dtype=torch.float64)
    return out


def _waves(g, n, amp=0.05):
    """E and B of two smooth waves across the box."""
    ph = _rand(g, 6, 2) * (2 * math.pi)
    ax = [torch.arange(m, device=DEV, dtype=torch.float64) * (2 * math.pi / m) for m in n]
    F = torch.zeros(6, *n, device=DEV, dtype=torch.float64)
    for c in range(6):
        F[c] += amp * torch.sin(ax[0][:, None, None] + ax[1][None, :, None] + ph[c, 0])
        F[c] += amp * torch.cos(2 * ax[2][None, None, :] - ax[0][:, None, None] + ph[c, 1])
    return F


# The wakefield recipe: lengths in cells; the density is a part of the critical one.
LASER = dict(lambda0=24.0, a0=2.0, tau=20.0, z0=60.0, start=100.0, ramp=32.0, n_over_nc=1e-3, speed=1.0)


def _wake_density():
    return LASER["n_over_nc"] * (2 * math.pi / LASER["lambda0"]) ** 2


def _laser(g, n):
    om = 2 * math.pi / LASER["lambda0"]
    e0 = LASER["a0"] * om * (1 + 0.1 * float(_rand(g, 1)))
    w0 = 0.2 * min(n[0], n[1])
    x = torch.arange(n[0], device=DEV, dtype=torch.float64) + 0.5 - 0.5 * n[0]
    y = torch.arange(n[1], device=DEV, dtype=torch.float64) - 0.5 * n[1]
    r = torch.exp(-(x[:, None] ** 2 + y[None, :] ** 2) / w0 ** 2)[:, :, None]
    F = torch.zeros(6, *n, device=DEV, dtype=torch.float64)
    for c, off in ((0, 0.0), (4, 0.5)):
        z = torch.arange(n[2], device=DEV, dtype=torch.float64) + off - LASER["z0"]
        F[c] = e0 * r * (torch.exp(-(z / LASER["tau"]) ** 2) * torch.cos(om * z))[None, None, :]
    return F


def _lattice(i, j, k, ppc, zlab):
    """Cold lattice plasma in the given cells (arrays of one length), the lab z of cell k being k + zlab."""
    m = torch.arange(ppc, device=DEV, dtype=torch.float64)
    off = ((m + 0.5) / ppc)[None, :]
    p = {"x": i[:, None] + off, "y": j[:, None] + off, "z": k[:, None] + off}
    dens = _wake_density() * ((p["z"] + zlab - LASER["start"]) / LASER["ramp"]).clamp(0.0, 1.0)
    p = {a: v.reshape(-1).contiguous() for a, v in p.items()}
    for a in ("ux", "uy", "uz"):
        p[a] = torch.zeros_like(p["x"])
    p["w"] = (dens / ppc).reshape(-1).contiguous()
    return p, p["w"] > 0


def _cells(n):
    c = torch.arange(n[0] * n[1] * n[2], device=DEV)
    return (c // (n[1] * n[2])).double(), (c // n[2] % n[1]).double(), (c % n[2]).double()


def _inputs(case, seed):
    """(fields, particles) a context starts from."""
    n = (case["nx"], case["ny"], case["nz"])
    g = _rng(seed)
    if case.get("window"):
        p, keep = _lattice(*_cells(n), case["ppc"], 0.0)
        return _laser(g, n), {a: v[keep].contiguous() for a, v in p.items()}
    if case["kind"] == "adjoint":
        return None, _plasma(g, n, case["ppc"])
    return _waves(g, n), _plasma(g, n, case["ppc"])


def _drive(case, seed):
    """Amplitude and wavenumber of the adjoint workload's external wave."""
    return 0.05 * (1.0 + random.Random(int(seed)).random()), 2 * math.pi / case["nx"]


def _boxes(case):
    """The boxes of a batch: extents, particles per cell, density, order."""
    r = random.Random(int(case["mix"]))
    edges = [e for e in (16, 24, 32, 48, 64) if e <= case["edge"]]
    return [dict(n=tuple(r.choice(edges) for _ in range(3)), ppc=r.randint(1, 8),
                 density=math.exp(r.uniform(math.log(0.1), math.log(10.0))), order=r.choice((1, 3)))
            for _ in range(case["boxes"])]


def _batch_inputs(case, seed):
    g = _rng(seed)
    return [_plasma(g, b["n"], b["ppc"], b["density"]) for b in _boxes(case)]


def _dtype(case):
    return torch.float64 if case["fp64"] else torch.float32


def _raw(total):
    raw = {k: torch.empty(total, device=DEV, dtype=torch.float64) for k in KEYS}
    raw["id"] = torch.empty(total, device=DEV, dtype=torch.int32)
    return raw


def prepare(case, seed):
    s = {"case": dict(case), "stream": torch.cuda.Stream()}
    prec = pic.FP64 if case["fp64"] else pic.FP32_MIXED
    real = _dtype(case)
    if case["kind"] == "batch":
        boxes, parts = _boxes(case), _batch_inputs(case, seed)
        counts = [p["x"].numel() for p in parts]
        cat = {k: torch.cat([p[k] for p in parts]) for k in KEYS}
        torch.cuda.synchronize()
        b = pic.Batch([x["n"] for x in boxes], [x["order"] for x in boxes], precision=prec, stream=s["stream"])
        b.load_particles(-1.0, 1.0, cat, counts)
        C = [x["n"][0] * x["n"][1] * x["n"][2] for x in boxes]
        s.update(batch=b, counts=counts, cells=C)
        total, C = sum(counts), sum(C)
    else:
        n = (case["nx"], case["ny"], case["nz"])
        F, parts = _inputs(case, seed)
        torch.cuda.synchronize()
        ctx = pic.Context(n, precision=prec, order=case["order"], stream=s["stream"],
                          solver="ckc" if case.get("ckc") else "yee",
                          window_speed=LASER["speed"] if case.get("window") else None)
        if case.get("window"):
            ctx.set_window_plasma(case["ppc"], _wake_density(), LASER["start"], LASER["ramp"])
        if F is not None:
            ctx.set_fields(F)
        ctx.load_particles(-1.0, 1.0, parts)
        if case.get("vay") or case.get("energy"):
            ctx.set_particle_algorithms("vay" if case["vay"] else "boris", "energy" if case["energy"] else "momentum")
        if case.get("passes"):
            ctx.set_gather_filter(case["passes"])
        s["ctx"] = ctx
        C, total = n[0] * n[1] * n[2], ctx.num_particles()
        if case.get("window"):
            total = C * case["ppc"] + 16 * n[0] * n[1] * case["ppc"]
        if case["kind"] == "adjoint":
            ctx.set_external_drive(*_drive(case, seed))
            ctx.reserve_adjoint(case["steps"], case["every"])
            s["du"] = torch.empty(3, total, device=DEV, dtype=torch.float64)
            return s
        if case["kind"] == "diagnostics":
            s["rho"] = torch.empty(n, device=DEV, dtype=torch.float64)
            return s
    # where the state is read to: the getters' 64-bit arrays and the program's own
    s["raw"] = _raw(total)
    s["parts"] = torch.empty(7, total, device=DEV, dtype=real)
    s["field"] = torch.empty(C, device=DEV, dtype=torch.float64)
    s["fields"] = torch.empty(9, C, device=DEV, dtype=real)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _by_id(s, total):
    """The particles just read, in the order of their ids."""
    ids = s["raw"]["id"][:total]
    if s["case"].get("window"):  # ids with gaps: removed particles
        order = torch.argsort(ids)
        return [s["raw"][k][:total][order].to(s["parts"].dtype) for k in KEYS]
    at = ids.long()
    for a, k in enumerate(KEYS):
        s["parts"][a].index_copy_(0, at, s["raw"][k].to(s["parts"].dtype))
    return list(s["parts"])


def run(s):
    case = s["case"]
    with torch.cuda.stream(s["stream"]):
        if case["kind"] == "batch":
            return _run_batch(s)
        ctx = s["ctx"]
        if case["kind"] == "adjoint":
            loss, dA, du = ctx.step_adjoint(case["steps"], case["every"], du=s["du"])
            real = _dtype(case)
            return [torch.tensor([loss, dA], dtype=torch.float64).to(real), du.to(real)]
        if case["kind"] == "diagnostics":
            rho = ctx.charge_density(out=s["rho"])
            d = ctx.diagnostics()
            return [rho, d["field_energy"], d["kinetic_energy"], d["charge"], d["max_div_b"]]
        ctx.step(case["steps"])
        total = ctx.num_particles()
        if total > s["raw"]["id"].numel():  # a moving window can collect plasma
            s["raw"] = _raw(total + total // 4)
        ctx.get_particles(out={k: v[:total] for k, v in s["raw"].items()})
        parts = _by_id(s, total)
        for i in range(9):
            ctx.get_field(i, out=s["field"])
            s["fields"][i].copy_(s["field"])
        return parts + list(s["fields"])


def _run_batch(s):
    b = s["batch"]
    b.step(s["case"]["steps"])
    first = 0
    for box, cnt in enumerate(s["counts"]):
        raw = {k: v[first:first + cnt] for k, v in s["raw"].items()}
        st = b.lib.pic_batch_get_particles(b.h, box, *[ct.c_void_p(raw[k].data_ptr()) for k in KEYS + ("id",)], 1)
        if st != pic.PIC_OK:
            raise RuntimeError(b.lib.pic_last_error().decode())
        raw["id"].add_(first)
        first += cnt
    parts = _by_id(s, first)
    for i in range(9):
        c0 = 0
        for box, C in enumerate(s["cells"]):
            b.get_field(box, i, out=s["field"][c0:c0 + C])
            c0 += C
        s["fields"][i].copy_(s["field"])
    return parts + list(s["fields"])


def work(case):
    """State in and state out once; the arithmetic of every step."""
    real = 8 if case["fp64"] else 4
    if case["kind"] == "batch":
        bytes_ = flops = 0
        for b in _boxes(case):
            C = b["n"][0] * b["n"][1] * b["n"][2]
            bytes_ += C * b["ppc"] * 2 * 8 * real + C * (6 + 9) * real
            flops += case["steps"] * C * (b["ppc"] * FLOPS[b["order"]] + 78)
        return {"bytes": bytes_, "flops": flops}
    C = case["nx"] * case["ny"] * case["nz"]
    N = C * case["ppc"]
    if case["kind"] == "diagnostics":
        return {"bytes": N * 8 * real + C * 6 * real + C * 8, "flops": N * (3 * (case["order"] + 1) ** 3 + 60) + 30 * C}
    if case["kind"] == "adjoint":  # particles and fields in, the gradient out; the reverse step about twice the forward one
        return {"bytes": N * 8 * real + C * 6 * real + N * 3 * real,
                "flops": 3 * case["steps"] * (N * FLOPS[case["order"]] + 78 * C)}
    return {"bytes": N * 2 * 8 * real + C * (6 + 9) * real,
            "flops": case["steps"] * (N * FLOPS[case["order"]] + 78 * C)}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _spline(p, f):
    """First node (relative to the cell) and weights of the order-p B-spline at fraction f."""
    if p == 0:
        return (f >= 0.5).long(), [torch.ones_like(f)]
    if p == 1:
        return torch.zeros_like(f, dtype=torch.long), [1 - f, f]
    if p == 2:
        up = f >= 0.5
        g = f - up.to(f.dtype)
        return up.long() - 1, [0.5 * (0.5 - g) ** 2, 0.75 - g * g, 0.5 * (0.5 + g) ** 2]
    return (torch.full_like(f, -1, dtype=torch.long),
            [(1 - f) ** 3 / 6, (4 - 6 * f ** 2 + 3 * f ** 3) / 6, (1 + 3 * f + 3 * f ** 2 - 3 * f ** 3) / 6, f ** 3 / 6])


def _half(p, f):
    """The same on the lattice shifted by half a cell."""
    hi = f >= 0.5
    first, w = _spline(p, torch.where(hi, f - 0.5, f + 0.5))
    return first - (~hi).long(), w


class _Plain:
    """Fields F (9, nx, ny, nz) and particles of one box, advanced in 64 bits; unit cells, q = -1, m = 1."""

    # the half-cell axes of Ex Ey Ez Bx By Bz
    STAG = ((1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 1, 1), (1, 0, 1), (1, 1, 0))

    def __init__(self, n, order, F, parts, dt, vay=False, energy=False, ckc=False, passes=0, zopen=False, drive=None,
                 chunk=1 << 21):
        self.n, self.p, self.dt = tuple(n), order, dt
        self.vay, self.energy, self.ckc, self.passes, self.zopen = vay, energy, ckc, passes, zopen
        self.drive, self.chunk, self.steps = drive, chunk, 0
        self.F = torch.zeros(9, *self.n, device=DEV, dtype=torch.float64)
        if F is not None:
            self.F[:6] = F
        self.x = torch.stack([parts[k] for k in ("x", "y", "z")])
        self.u = torch.stack([parts[k] for k in ("ux", "uy", "uz")])
        self.w = parts["w"]
        self.keep = None

    def _index(self, a, cell, first, w):
        """Per node of axis a: (element offset, weight), wrapped or zero beyond an open end."""
        st = (self.n[1] * self.n[2], self.n[2], 1)[a]
        out = []
        for r, wr in enumerate(w):
            i = cell + first + r
            if a == 2 and self.zopen:
                wr = torch.where((i >= 0) & (i < self.n[2]), wr, torch.zeros_like(wr))
                i = i.clamp(0, self.n[2] - 1)
            else:
                i = i.remainder(self.n[a])
            out.append((i * st, wr))
        return out

    def _gather(self, F, cell, f):
        node = [self._index(a, cell[a], *_spline(self.p, f[a])) for a in range(3)]
        half = [self._index(a, cell[a], *_half(self.p - int(self.energy), f[a])) for a in range(3)]
        out = []
        for c, stag in enumerate(self.STAG):
            ax, ay, az = [(half if s else node)[a] for a, s in enumerate(stag)]
            flat = F[c].reshape(-1)
            acc = 0.0
            for ix, wx in ax:
                for iy, wy in ay:
                    row = 0.0
                    for iz, wz in az:
                        row = row + wz * flat[ix + iy + iz]
                    acc = acc + wx * wy * row
            out.append(acc)
        return torch.stack(out[:3]), torch.stack(out[3:])

    def _push(self, u, E, B):
        k = -0.5 * self.dt

        def cross(a, b):
            return torch.linalg.cross(a, b, dim=0)

        if self.vay:
            v = u / torch.sqrt(1 + (u * u).sum(0))
            up = u + 2 * k * E + k * cross(v, B)
            tau = k * B
            t2, us = (tau * tau).sum(0), (up * tau).sum(0)
            sig = 1 + (up * up).sum(0) - t2
            t = tau / torch.sqrt(0.5 * (sig + torch.sqrt(sig * sig + 4 * (t2 + us * us))))
            return (up + (up * t).sum(0) * t + cross(up, t)) / (1 + (t * t).sum(0))
        um = u + k * E
        t = k * B / torch.sqrt(1 + (um * um).sum(0))
        s = 2 * t / (1 + (t * t).sum(0))
        return um + cross(um + cross(um, t), s) + k * E

    def _deposit(self, J, cell, f0, f1, w):
        """Esirkepov's current of the straight moves f0 -> f1 (cell units, relative to the old cell)."""
        NW = self.p + 2
        S0, dS, at, ok = [], [], [], []
        for a in range(3):
            fl = f1[a].detach().floor()
            a0, w0 = _spline(self.p, f0[a])
            a1, w1 = _spline(self.p, f1[a] - fl)
            a1 = a1 + fl.long()
            b = torch.minimum(a0, a1)
            z = torch.zeros_like(f0[a])
            s0 = [torch.where(a0 == b, (w0 + [z])[m], ([z] + w0)[m]) for m in range(NW)]
            s1 = [torch.where(a1 == b, (w1 + [z])[m], ([z] + w1)[m]) for m in range(NW)]
            S0.append(s0)
            dS.append([q - r for q, r in zip(s1, s0)])
            st = (self.n[1] * self.n[2], self.n[2], 1)[a]
            i = [cell[a] + b + m for m in range(NW)]
            at.append([v.clamp(0, self.n[2] - 1) if a == 2 and self.zopen else v.remainder(self.n[a]) * st for v in i])
            ok.append([(v >= 0) & (v < self.n[2]) if a == 2 and self.zopen else None for v in i])
        for c in range(3):
            t1, t2 = (c + 1) % 3, (c + 2) % 3
            flat = J[c].view(-1)
            cum, run = [], 0.0
            for m in range(NW - 1):
                run = run + dS[c][m]
                cum.append(run * (w / self.dt))  # -q w / (dt d_t1 d_t2)
            for i in range(NW):
                for j in range(NW):
                    Q = S0[t1][i] * (S0[t2][j] + 0.5 * dS[t2][j]) + dS[t1][i] * (0.5 * S0[t2][j] + dS[t2][j] / 3)
                    base = at[t1][i] + at[t2][j]
                    for m in range(NW - 1):
                        v = cum[m] * Q
                        for good in (ok[c][m], ok[t1][i], ok[t2][j]):
                            if good is not None:
                                v = torch.where(good, v, torch.zeros_like(v))
                        flat.index_add_(0, base + at[c][m], v)

    def _particles(self, F, x, u, w, J):
        """One chunk: gather, push, advance, deposit; the new positions (not wrapped) and momenta."""
        cell = x.detach().floor().long()
        cell = torch.stack([cell[a].clamp(0, self.n[a] - 1) for a in range(3)])
        f0 = x - cell
        E, B = self._gather(F, cell, f0)
        if self.drive is not None:
            amp, k = self.drive
            E = torch.stack([E[0], E[1] + amp * torch.cos(k * x[0] - k * (self.steps * self.dt)), E[2]])
        u = self._push(u, E, B)
        x1 = x + self.dt * u / torch.sqrt(1 + (u * u).sum(0))
        self._deposit(J, cell, f0, x1 - cell, w)
        return x1, u

    def _next(self, f, a):
        g = torch.roll(f, -1, a)
        if a == 2 and self.zopen:
            g = torch.cat([f[:, :, 1:], torch.zeros_like(f[:, :, :1])], 2)
        return g

    def _prev(self, f, a):
        g = torch.roll(f, 1, a)
        if a == 2 and self.zopen:
            g = torch.cat([torch.zeros_like(f[:, :, :1]), f[:, :, :-1]], 2)
        return g

    def _up(self, f, a):
        """Forward difference; with CKC averaged over the two other axes."""
        d = self._next(f, a) - f
        if self.ckc:
            for b in range(3):
                if b != a:
                    d = 0.25 * self._prev(d, b) + 0.5 * d + 0.25 * self._next(d, b)
        return d

    def _b_half(self, E, B):
        h = 0.5 * self.dt
        up = self._up
        return [B[0] - h * (up(E[2], 1) - up(E[1], 2)), B[1] - h * (up(E[0], 2) - up(E[2], 0)),
                B[2] - h * (up(E[1], 0) - up(E[0], 1))]

    def _fields(self, F, J):
        E, B = F[:3], self._b_half(F[:3], F[3:6])

        def dn(f, a):
            return f - self._prev(f, a)

        E = [E[0] + self.dt * (dn(B[2], 1) - dn(B[1], 2) - J[0]), E[1] + self.dt * (dn(B[0], 2) - dn(B[2], 0) - J[1]),
             E[2] + self.dt * (dn(B[1], 0) - dn(B[0], 1) - J[2])]
        return torch.stack(E + self._b_half(E, B) + list(J))

    def _filtered(self, F):
        n = self.passes
        for q in range(n + 1 if n else 0):
            a, b = (0.25, 0.5) if q < n else (-0.25 * n, 1 + 0.5 * n)
            F = a * torch.roll(F, 1, 3) + b * F + a * torch.roll(F, -1, 3)
        return F

    def advance(self):
        Fg = self._filtered(self.F[:6])
        J = torch.zeros(3, *self.n, device=DEV, dtype=torch.float64)
        N = self.w.numel()
        for p in range(0, N, self.chunk):
            q = slice(p, min(p + self.chunk, N))
            self.x[:, q], self.u[:, q] = self._particles(Fg, self.x[:, q].clone(), self.u[:, q].clone(), self.w[q], J)
        self.F = self._fields(self.F, J)
        self.steps += 1
        self._wrap()

    def _wrap(self):
        for a in range(2 if self.zopen else 3):
            v = self.x[a].remainder(self.n[a])
            self.x[a] = torch.where(v >= self.n[a], torch.zeros_like(v), v)

    def state(self):
        return list(self.x) + list(self.u) + [self.w] + [f.reshape(-1) for f in self.F]


class _PlainWindow(_Plain):
    def advance(self):
        super().advance()
        self._drop((self.x[2] >= 0) & (self.x[2] < self.n[2]))
        while LASER["speed"] * self.steps * self.dt >= self.shifts + 1:
            self.F = torch.cat([self.F[..., 1:], torch.zeros_like(self.F[..., :1])], 3)
            self.x[2] -= 1
            self._drop(self.x[2] >= 0)
            self.shifts += 1
            c = torch.arange(self.n[0] * self.n[1], device=DEV)
            i, j = (c // self.n[1]).double(), (c % self.n[1]).double()
            p, keep = _lattice(i, j, torch.full_like(i, self.n[2] - 1.0), self.ppc, float(self.shifts))
            ids = torch.arange(keep.numel(), device=DEV) + self.next_id
            self.next_id += keep.numel()
            self.x = torch.cat([self.x, torch.stack([p[k][keep] for k in ("x", "y", "z")])], 1)
            self.u = torch.cat([self.u, torch.stack([p[k][keep] for k in ("ux", "uy", "uz")])], 1)
            self.w = torch.cat([self.w, p["w"][keep]])
            self.ids = torch.cat([self.ids, ids[keep]])

    def _drop(self, keep):
        self.x, self.u = self.x[:, keep].contiguous(), self.u[:, keep].contiguous()
        self.w, self.ids = self.w[keep], self.ids[keep]


def _exact_adjoint(case, seed, n, dt):
    from torch.utils.checkpoint import checkpoint

    _, parts = _inputs(case, seed)
    amp, k = _drive(case, seed)
    amp = torch.tensor(amp, device=DEV, dtype=torch.float64, requires_grad=True)
    P = _Plain(n, case["order"], None, parts, dt, drive=(amp, k))
    u0 = P.u.clone().requires_grad_(True)

    def step(F, x, u, a, t):
        P.drive, P.steps = (a, k), t
        J = torch.zeros(3, *n, device=DEV, dtype=torch.float64)
        x, u = P._particles(F[:6], x, u, P.w, J)
        F = P._fields(F, J)
        L = torch.tensor(n, device=DEV, dtype=torch.float64)[:, None]
        return F, x - L * (x.detach() / L).floor(), u

    F, x, u = P.F, P.x, u0
    for t in range(case["steps"]):
        F, x, u = checkpoint(step, F, x, u, amp, t, use_reentrant=False)
    loss = 0.5 * (F[:6] ** 2).sum()
    loss.backward()
    return [torch.stack([loss.detach(), amp.grad]).cpu(), u0.grad]


def exact(case, seed):
    if case["kind"] == "batch":
        boxes = _boxes(case)
        dt = 0.99 / math.sqrt(3.0)
        out = []
        for b, parts in zip(boxes, _batch_inputs(case, seed)):
            P = _Plain(b["n"], b["order"], None, parts, dt)
            for _ in range(case["steps"]):
                P.advance()
            out.append(P.state())
        return [torch.cat(v) for v in zip(*out)]
    n = (case["nx"], case["ny"], case["nz"])
    dt = 0.99 if case.get("ckc") else 0.99 / math.sqrt(3.0)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed, n, dt)
    F, parts = _inputs(case, seed)
    if case["kind"] == "diagnostics":
        return _exact_diagnostics(case, n, F, parts)
    make = _PlainWindow if case["window"] else _Plain
    P = make(n, case["order"], F, parts, dt, vay=case["vay"], energy=case["energy"], ckc=case["ckc"],
             passes=case["passes"], zopen=case["window"])
    del F, parts
    if case["window"]:
        P.shifts, P.ppc, P.next_id = 0, case["ppc"], P.w.numel()
        P.ids = torch.arange(P.w.numel(), device=DEV)
    for _ in range(case["steps"]):
        P.advance()
    return P.state()


def _exact_diagnostics(case, n, F, parts):
    rho = torch.zeros(n[0] * n[1] * n[2], device=DEV, dtype=torch.float64)
    P = _Plain(n, case["order"], F, parts, 1.0)
    for p in range(0, P.w.numel(), P.chunk):
        x, w = P.x[:, p:p + P.chunk], P.w[p:p + P.chunk]
        cell = x.floor().long()
        ax, ay, az = [P._index(a, cell[a], *_spline(P.p, x[a] - cell[a])) for a in range(3)]
        for ix, wx in ax:
            for iy, wy in ay:
                for iz, wz in az:
                    rho.index_add_(0, ix + iy + iz, -w * wx * wy * wz)
    g = torch.sqrt(1 + (P.u * P.u).sum(0))
    B = F[3:]
    div = sum(torch.roll(B[a], -1, a) - B[a] for a in range(3))
    return [rho.reshape(n), float(0.5 * (F ** 2).sum()), float((P.w * (P.u * P.u).sum(0) / (g + 1)).sum()),
            float(-P.w.sum()), float(div.abs().max())]
