"""The work that users of this framework have it do, as measurable cases.

Kinds of case, each through the public entry points of ``seisgb``:

- ``step``: one fused time step on caller-owned padded device fields, the call
  of a program that drives its own time loop (``stencil_step``; 16-bit and
  difference-form storage included).  Every pass reads the same u^n and
  overwrites what the previous pass wrote;
- ``layout``: a compact array packed into the padded layout and read back, what
  such a program does around its loop;
- ``shot``: a whole forward shot (``run_shot``), from device or host buffers;
- ``gradient``: misfit and velocity gradient of one shot, one iteration of a
  waveform inversion (``velocity_misfit`` and its backward);
- ``serve``: a batch of shot requests through a running ``Server``.

Grids, layer velocities, wavelet and receiver spacing are those of the tests,
the benchmark and the serving mix, or ragged and unequally spaced ones.  Step
fields are superposed plane waves that decay through the PML, as a propagating
wavefield does there; models are layered with a smooth perturbation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

STORAGE = ("fp32", "fp16", "bf16", "fp32_diff", "bf16_diff")
VMAX = 4650.0  # upper bound of every layered model below (m/s)
R0 = 1e-3      # PML target reflection coefficient
STEP = 32      # the step that a `step` case takes (near the wavelet's peak)
# halves of Fornberg's 8th-order central second-derivative weights
FD8 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _grid(kind, nx, ny, nz, nb, dx=10.0, dy=10.0, dz=10.0, **more):
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "nb": nb, "dx": dx, "dy": dy, "dz": dz,
            **more}


def listed():
    return [
        # the smallest grid in use (64^3 inner + 16-point PML): launch and call latency
        dict(_grid("step", 64, 64, 64, 16, storage="fp32", receivers=0), name="step_fp32_96"),
        # the grid of the inversion and of most served shots
        dict(_grid("step", 224, 224, 224, 16, storage="fp32", receivers=0), name="step_fp32_256"),
        # a survey cut to a licence area: odd extents, unequal spacing, odd PML width, and the
        # receivers sampled at every step of the caller's loop
        dict(_grid("step", 301, 187, 163, 21, 12.5, 10.0, 8.0, storage="fp32", receivers=4),
             name="step_fp32_ragged"),
        # the benchmark's grid: fields far beyond the cache
        dict(_grid("step", 448, 448, 448, 32, storage="fp32", receivers=0), name="step_fp32_512"),
        # the same grid where memory is short: bf16 wavefields
        dict(_grid("step", 448, 448, 448, 32, storage="bf16", receivers=0), name="step_bf16_512"),
        # the largest served grid with scaled fp16 wavefields
        dict(_grid("step", 352, 352, 224, 16, storage="fp16", receivers=0), name="step_fp16_384"),
        # 16-bit wavefields for long runs: difference form
        dict(_grid("step", 224, 224, 224, 16, storage="bf16_diff", receivers=0),
             name="step_bf16_diff_256"),
        # a field brought into the padded layout and a snapshot taken out of it
        dict(_grid("layout", 352, 352, 224, 16), name="layout_384"),
        # the parity case: a short whole shot on the smallest grid, everything on the device
        dict(_grid("shot", 64, 64, 64, 16, storage="fp32", nt=100, host=False, receivers=8),
             name="shot_fp32_96"),
        # a whole shot from pinned host buffers, traces and final wavefield back on the host
        dict(_grid("shot", 160, 160, 224, 16, storage="fp32", nt=120, host=True, receivers=4),
             name="shot_host_192"),
        # one shot's contribution to an inversion iteration, with two checkpoint segments
        dict(_grid("gradient", 96, 96, 96, 16, nt=100, ckpt=50, receivers=4), name="gradient_128"),
        # requests of the serving mix, submitted together
        dict(_grid("serve", 96, 96, 96, 16, nt=100, requests=6), name="serve_mix"),
    ]


def _extents(rng, lo, hi, nb):
    """Inner extents whose computed volume is log-uniform in lo^3 .. hi^3, none
    shorter than half or longer than twice the cube's edge."""
    edge = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    fx, fy = math.exp(rng.uniform(-0.4, 0.4)), math.exp(rng.uniform(-0.4, 0.4))
    f = (fx, fy, 1.0 / (fx * fy))
    ext = [max(24, int(edge * q)) for q in f]
    if rng.random() < 0.4:  # users also like round numbers
        ext = [max(32, e // 16 * 16) for e in ext]
    return [max(8, e - 2 * nb) for e in ext]


def draw(rng):
    # whole shots and gradients stay at 120 steps and fp32 storage: over longer runs, or with
    # 16-bit wavefields, two correct implementations drift apart by their roundings alone
    kind = rng.choice(("step", "step", "step", "step", "layout", "shot", "shot", "gradient", "serve"))
    nb = rng.choice((8, 10, 16, 16, 20, 27, 32))
    h = [10.0, 10.0, 10.0] if rng.random() < 0.5 else [rng.choice((8.0, 10.0, 12.5)) for _ in range(3)]
    if kind == "step":
        if rng.random() < 0.1:
            nb = 0  # zero walls
        storage = rng.choice(("fp32", "fp32", "fp32", "fp16", "bf16", "bf16_diff", "fp32_diff"))
        return _grid("step", *_extents(rng, 90, 490, nb), nb, *h, storage=storage,
                     receivers=rng.choice((0, 4)) if storage.startswith("fp32") else 0)
    if kind == "layout":
        return _grid("layout", *_extents(rng, 90, 480, nb), nb, *h)
    if kind == "shot":
        ext = _extents(rng, 80, 230, nb)
        pts = math.prod(e + 2 * nb for e in ext)
        return _grid("shot", *ext, nb, *h, storage="fp32", nt=min(rng.randrange(40, 121), int(1e9 / pts)),
                     host=rng.random() < 0.4, receivers=rng.choice((4, 8)))
    if kind == "gradient":
        ext = _extents(rng, 64, 140, nb)
        return _grid("gradient", *ext, nb, *h, nt=rng.randrange(40, 101), ckpt=rng.randrange(20, 81),
                     receivers=4)
    ext = _extents(rng, 80, 120, 16)
    return _grid("serve", *ext, 16, *h, nt=rng.randrange(40, 101), requests=rng.randrange(2, 7))


# ---------------------------------------------------------------------------
# inputs (torch and numpy alone: prepare and exact share them)
# ---------------------------------------------------------------------------
def _shape(c):
    return tuple(c[n] + 2 * c["nb"] for n in ("nz", "ny", "nx"))


def _f32(x):
    return float(np.float32(x))


def _dt(c):
    """0.4 of the von Neumann limit for VMAX, as the fp32 number the grid holds."""
    s = sum(1.0 / c[h] ** 2 for h in ("dx", "dy", "dz"))
    return _f32(0.4 * 2.0 / (VMAX * math.sqrt(2048.0 / 315.0 * s)))


def _depth(n, nb, device):
    """Depth in points into the PML of indices -1 .. n + 2 nb (0 in the inner range)."""
    i = torch.arange(-1, n + 2 * nb + 1, device=device, dtype=torch.float64)
    return torch.clamp(torch.maximum(nb - i, i - (nb + n - 1)), min=0.0)


def _axes(c, fn):
    """fn(axis name, torch dimension) for z, y, x, reshaped to broadcast over (Nz, Ny, Nx)."""
    out = []
    for dim, n in enumerate(("nz", "ny", "nx")):
        view = [1, 1, 1]
        view[dim] = -1
        out.append(fn(n).reshape(view))
    return out


def _rng(seed, part):
    return np.random.default_rng([int(seed), part])


def _waves(c, seed, part, count=4, amplitude=1.0):
    """Two snapshots, dt apart, of superposed plane waves (wavelengths of 8 to
    30 points) that decay to zero through the PML: fp32 (Nz, Ny, Nx) each."""
    rng = _rng(seed, part)
    shape, dt = _shape(c), _dt(c)
    env = torch.ones(1, 1, 1, device="cuda")
    if c["nb"] > 0:
        for e in _axes(c, lambda n: (1.0 - _depth(c[n], c["nb"], "cuda")[1:-1] / (c["nb"] + 1)) ** 2):
            env = env * e.float()
    out = [torch.zeros(shape, device="cuda"), torch.zeros(shape, device="cuda")]
    for _ in range(count):
        d = rng.standard_normal(3)
        k = 2.0 * math.pi / rng.uniform(8.0, 30.0) * d / np.linalg.norm(d)
        omega = rng.uniform(1500.0, 3500.0) * float(
            math.sqrt(sum((k[q] / c[h]) ** 2 for q, h in enumerate(("dz", "dy", "dx")))))
        phase, a = rng.uniform(0.0, 2.0 * math.pi), amplitude * rng.uniform(0.3, 1.0)
        args = _axes(c, lambda n: torch.arange(c[n] + 2 * c["nb"], device="cuda", dtype=torch.float32) *
                     float(k[("nz", "ny", "nx").index(n)]))
        arg = args[0] + args[1] + args[2]
        for t in range(2):
            out[t] += a * torch.sin(arg + (phase + t * omega * dt))
    return [(f * env).contiguous() for f in out]  # (earlier, later)


def _velocity(c, seed, part=0):
    """Layered model (8 to 20 layers, 1500 to 4500 m/s) with a smooth perturbation of 3%."""
    rng = _rng(seed, 100 + part)
    nz = _shape(c)[0]
    cuts = np.sort(rng.choice(np.arange(1, nz), size=min(nz - 1, int(rng.integers(7, 20))), replace=False))
    vk = rng.uniform(1500.0, 4500.0, size=len(cuts) + 1)[np.searchsorted(cuts, np.arange(nz), side="right")]
    v = torch.from_numpy(vk.astype(np.float32)).cuda().reshape(-1, 1, 1)
    p = 1.0
    for q in _axes(c, lambda n: torch.cos(torch.arange(c[n] + 2 * c["nb"], device="cuda",
                                                       dtype=torch.float32) *
                                          float(2 * math.pi / rng.uniform(24.0, 80.0)) +
                                          float(rng.uniform(0, 6.28)))):
        p = p * q
    return (v * (1.0 + 0.03 * p)).contiguous()


def _ricker(n, dt, seed):
    fp = _rng(seed, 200).uniform(18.0, 25.0)
    a = (math.pi * fp * (np.arange(n) * dt - 0.6 / fp)) ** 2
    return torch.from_numpy(((1.0 - 2.0 * a) * np.exp(-a) * 1e3).astype(np.float32))


def _source(c, seed):
    """A shot position over the middle of the inner region, a few points deep."""
    rng = _rng(seed, 300)
    at = [c["nb"] + int(rng.integers(c[n] // 4, max(c[n] // 4 + 1, 3 * c[n] // 4))) for n in ("nx", "ny")]
    return at + [c["nb"] + min(4, c["nz"] - 1)]


def _receivers(c, every):
    """Every `every`-th inner point of the top inner plane: int32 rows (i, j, k)."""
    ii = np.arange(c["nb"], c["nb"] + c["nx"], every)
    jj = np.arange(c["nb"], c["nb"] + c["ny"], every)
    J, I = np.meshgrid(jj, ii, indexing="ij")
    return np.stack([I.ravel(), J.ravel(), np.full(I.size, c["nb"])], axis=1).astype(np.int32)


def _pow2_scale(bound):
    """The power of two s with bound / s in [2^13, 2^14)."""
    return 2.0 ** (math.floor(math.log2(bound)) + 1 - 14)


def _injected(c, f):
    """Amplitude that the step adds at the source point."""
    i, j, k = f["source"]
    return abs(float(f["m"][k, j, i]) * float(f["wavelet"][STEP])) / (c["dx"] * c["dy"] * c["dz"])


def _step_inputs(c, seed):
    """The fields one step reads, in their storage types, and its source."""
    shape = _shape(c)
    up, u = _waves(c, seed, 0)
    m = (_velocity(c, seed) * _dt(c)) ** 2
    if c["nb"] > 0:
        phi = _waves(c, seed, 1, count=2, amplitude=1e-4)[0]
        b = c["nb"]
        phi[b:shape[0] - b, b:shape[1] - b, b:shape[2] - b] = 0.0
    else:
        phi = torch.zeros(shape, device="cuda")
    f = {"m": m, "phi": phi, "source": _source(c, seed),
         "wavelet": _ricker(2 * STEP, _dt(c), seed).cuda()}
    if c["storage"] == "fp16":
        top, top_p = float(u.abs().max()), float(up.abs().max())
        s = _pow2_scale(4.0 * max(top, top_p) + _injected(c, f))
        f |= {"u": (u / s).half(), "up": (up / s).half(),  # [STEP & 3] = [0]: u^n, [3]: u^{n-1}
              "scale": torch.tensor([s, s, s, s, top, 0.0, 0.0, top_p], device="cuda")}
    elif c["storage"].endswith("_diff"):
        t = torch.bfloat16 if c["storage"] == "bf16_diff" else torch.float32
        f |= {"u": u.to(t), "d": (u - up).to(t)}
    else:
        t = torch.bfloat16 if c["storage"] == "bf16" else torch.float32
        f |= {"u": u.to(t), "up": up.to(t)}
    return f


def _request(c, seed, q):
    """Request q of a served batch: the case's grid, or one stretched in depth or along a line."""
    r = dict(c)
    if q % 3 == 1:
        r["nz"] = c["nz"] * 3 // 2
    elif q % 3 == 2:
        r["nx"] = c["nx"] * 5 // 4 + 3
    r["nt"] = max(20, c["nt"] - 11 * q)
    return r, int(_rng(seed, 400 + q).integers(1 << 30))


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _seisgb():
    from paper_2009_04619_gb300 import seisgb
    return seisgb


def _make_grid(c):
    s = _seisgb()
    code = {"fp32": s.FP32, "fp16": s.FP16_SCALED, "bf16": s.BF16, "fp32_diff": s.FP32_DIFF,
            "bf16_diff": s.BF16_DIFF}[c.get("storage", "fp32")]
    return s.make_grid(c["nx"], c["ny"], c["nz"], c["nb"], c["dx"], c["dy"], c["dz"], _dt(c), VMAX, R0, code)


def _padded(g, compact):
    """(padded buffer, view of its computed points) holding a compact field."""
    L = _seisgb().layout(g)
    buf = torch.zeros(int(L.elems), dtype=compact.dtype, device="cuda")
    view = buf.as_strided((L.Nz, L.Ny, L.Nx), (L.stride_z, L.stride_y, 1), L.origin)
    view.copy_(compact)
    return buf, view


class _Serving:
    """A running server, stopped with the state that holds it."""

    def __init__(self):
        self.server = _seisgb().Server(16 << 30, max_slots=8, steps_per_graph=16)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    c = case
    g = _make_grid(c)
    s = {"kind": c["kind"], "grid": g}
    if c["kind"] == "step":
        f = _step_inputs(c, seed)
        names = ("u", "up", "d", "m", "phi")
        s |= {n: _padded(g, f[n]) for n in names if n in f}
        if "d" in s:  # difference form: u^{n+1} goes to a buffer of its own
            s["up"] = _padded(g, torch.zeros_like(f["u"]))
        s |= {"scale": f.get("scale"), "source": (*f["source"], f["wavelet"]), "rec": None}
        if c["receivers"]:
            ijk = _receivers(c, c["receivers"])
            s["rec"] = (ijk, torch.zeros(len(ijk), device="cuda"))
    elif c["kind"] == "layout":
        s["field"] = _waves(c, seed, 0)[0]
        s["padded"] = torch.empty(int(_seisgb().layout(g).elems), device="cuda")
        s["back"] = torch.empty_like(s["field"])
    elif c["kind"] == "shot":
        v, w = _velocity(c, seed), _ricker(c["nt"], _dt(c), seed)
        ijk = _receivers(c, c["receivers"])
        tr, fin = torch.zeros(c["nt"], len(ijk)), torch.zeros(_shape(c))
        if c["host"]:
            s |= {"v": v.cpu().pin_memory(), "w": w.pin_memory(), "tr": tr.pin_memory(),
                  "fin": fin.pin_memory()}
        else:
            s |= {"v": v, "w": w.cuda(), "tr": tr.cuda(), "fin": fin.cuda()}
        s |= {"nt": c["nt"], "src": _source(c, seed), "rec": ijk}
    elif c["kind"] == "gradient":
        ijk = _receivers(c, c["receivers"])
        s |= {"v": _velocity(c, seed).requires_grad_(True), "w": _ricker(c["nt"], _dt(c), seed).cuda(),
              "nt": c["nt"], "src": _source(c, seed), "rec": ijk, "ckpt": c["ckpt"],
              "obs": _observed(c, seed, len(ijk)).cuda()}
    else:
        s["serving"], s["requests"] = _Serving(), []
        for q in range(c["requests"]):
            r, rs = _request(c, seed, q)
            s["requests"].append((_make_grid(r), _velocity(r, rs).cpu().numpy(),
                                  _ricker(r["nt"], _dt(r), rs).numpy(), r["nt"], _source(r, rs),
                                  _receivers(r, 8)))
    return s


def _observed(c, seed, nrec):
    """Recorded traces of an inversion: a wavelet arriving later along the line, with noise."""
    rng = _rng(seed, 500)
    t = np.arange(c["nt"])[:, None] - (20.0 + 0.2 * c["nt"] * rng.random((1, nrec)))
    a = (t / 12.0) ** 2
    return torch.from_numpy(((1.0 - 2.0 * a) * np.exp(-a) * 1e-3 +
                             1e-5 * rng.standard_normal((c["nt"], nrec))).astype(np.float32))


def run(state):
    s, lib = state, _seisgb()
    if s["kind"] == "step":
        g = s["grid"]
        if "d" in s:
            lib.stencil_step_diff(g, s["u"][0], s["up"][0], s["d"][0], s["m"][0], s["phi"][0], STEP,
                                  s["source"], s["rec"])
        else:
            lib.stencil_step(g, s["u"][0], s["up"][0], s["m"][0], s["phi"][0], STEP, s["source"],
                             s["rec"], scale_state=s["scale"])
        out = {"u": s["up"][1], "phi": s["phi"][1]}
        if "d" in s:
            out["d"] = s["d"][1]
        if s["scale"] is not None:
            out["scale"] = s["scale"]
        if s["rec"] is not None:
            out["traces"] = s["rec"][1]
        return out
    if s["kind"] == "layout":
        lib.pack(s["grid"], s["field"], s["padded"])
        lib.unpack(s["grid"], s["padded"], s["back"])
        return {"padded": s["padded"], "back": s["back"]}
    if s["kind"] == "shot":
        lib.run_shot(s["grid"], s["v"], s["w"], s["nt"], s["src"], s["rec"], s["tr"], s["fin"])
        return {"traces": s["tr"], "final": s["fin"]}
    if s["kind"] == "gradient":
        from paper_2009_04619_gb300.autograd import velocity_misfit
        v = s["v"]
        v.grad = None
        J = velocity_misfit(v, s["grid"], s["w"], s["nt"], s["src"], s["rec"], s["obs"], s["ckpt"])
        J.backward()
        return {"misfit": J.detach().to(v.dtype), "grad": v.grad}  # in the model's type, as an optimiser takes them
    srv, tickets = s["serving"].server, []
    for r in s["requests"]:
        tickets.append(srv.submit(*r))
    out = []
    for t, r in zip(tickets, s["requests"]):
        out.append(srv.poll(t, r[3], len(r[5]), timeout_us=60_000_000)[2])
    return out


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _points(c):
    """(computed points, PML points)"""
    n = math.prod(_shape(c))
    return n, n - c["nx"] * c["ny"] * c["nz"]


def _step_bytes(c, storage):
    """One step: both wavefields and m read, u^{n+1} written (difference form: d read and written,
    u read and written); phi read and written in the PML."""
    w = 4 if storage.startswith("fp32") else 2
    n, p = _points(c)
    return n * (4 + (4 if storage.endswith("_diff") else 3) * w) + 8 * p


STEP_FLOPS = 41  # 12 symmetric sums, 13 multiply-adds of the 25-point star, 3 of the update


def work(case):
    c = case
    n, p = _points(c)
    flops = STEP_FLOPS * n + 16 * p
    if c["kind"] == "step":
        nrec = len(_receivers(c, c["receivers"])) if c["receivers"] else 0
        return {"bytes": _step_bytes(c, c["storage"]) + 16 * nrec, "flops": flops}
    if c["kind"] == "layout":
        return {"bytes": 16 * n, "flops": 0}
    nrec = len(_receivers(c, c.get("receivers", 8)))
    if c["kind"] == "shot":
        return {"bytes": c["nt"] * (_step_bytes(c, c["storage"]) + 4 * nrec) + 8 * n, "flops": c["nt"] * flops}
    if c["kind"] == "gradient":
        # forward, recomputation (also writes the acceleration), adjoint (reads two multipliers,
        # m, the acceleration and the running sum, writes multiplier and sum)
        per = _step_bytes(c, "fp32") + (20 * n + 8 * p) + (28 * n + 8 * p)
        return {"bytes": c["nt"] * per + 8 * n, "flops": 3 * c["nt"] * flops}
    total = {"bytes": 0, "flops": 0}
    for q in range(c["requests"]):
        r, _ = _request(c, 0, q)
        w = work(dict(r, kind="shot", storage="fp32", receivers=8))
        total = {k: total[k] + w[k] for k in total}
    return total


# ---------------------------------------------------------------------------
# what run() computes, in 64 bits
# ---------------------------------------------------------------------------
class _Exact:
    """The scheme in fp64: leapfrog with the 25-point star, single-stretch PML
    outside the inner box, zero beyond the computed domain."""

    def __init__(self, c):
        self.c = c
        h = {"nz": _f32(c["dz"]), "ny": _f32(c["dy"]), "nx": _f32(c["dx"])}
        self.h, dt, nb = h, _dt(c), c["nb"]
        self.vol = math.prod(h.values())
        self.e = self.grad = self.pml = None
        if nb > 0:
            d = {n: _depth(c[n], nb, "cuda") for n in h}
            top = {n: -3.0 * _f32(VMAX) * math.log(_f32(R0)) / (2.0 * nb * h[n]) for n in h}
            ez, ey, ex = _axes(c, lambda n: top[n] * dt / nb ** 2 * d[n][1:-1] ** 2)
            self.e = ex + ey + ez
            self.grad = _axes(c, lambda n: dt * top[n] / (4.0 * nb ** 2 * h[n] ** 2) *
                              (d[n][2:] ** 2 - d[n][:-2] ** 2))
            self.pml = self.e > 0

    def step(self, u, up, phi, m, source, w):
        """(u^{n+1}, phi^{n+1}) from u^n, u^{n-1}, phi^n; w: the source sample."""
        P = torch.nn.functional.pad(u, (4, 4, 4, 4, 4, 4))
        N = u.shape

        def at(dim, q):
            s = [slice(4, 4 + n) for n in N]
            s[dim] = slice(4 + q, 4 + q + N[dim])
            return P[tuple(s)]

        L = (FD8[0] * sum(1.0 / v ** 2 for v in self.h.values())) * u
        for dim, n in enumerate(("nz", "ny", "nx")):
            for q in range(1, 5):
                L = L + (FD8[q] / self.h[n] ** 2) * (at(dim, q) + at(dim, -q))
        new = 2.0 * u - up + m * L
        if self.e is not None:
            e = self.e
            damped = ((2.0 - e * e) * u - (1.0 - e) * up + m * (L + phi)) / (1.0 + e)
            new = torch.where(self.pml, damped, new)
            G = sum(k * (at(dim, 1) - at(dim, -1)) for dim, k in enumerate(self.grad))
            phi = torch.where(self.pml, (phi - G) / (1.0 + e), phi)
        if w is not None:
            i, j, k = source
            f = torch.zeros_like(new)
            f[k, j, i] = w / self.vol
            new = new + m * f
        return new, phi


def _exact_shot(c, v, wavelet, source, ijk, nt):
    """(traces, u^{nt}) of a shot in fp64."""
    X = _Exact(c)
    m = (v.double() * _dt(c)) ** 2
    u, up, phi = (torch.zeros(_shape(c), dtype=torch.float64, device="cuda") for _ in range(3))
    at = torch.from_numpy(ijk.astype(np.int64)).cuda()
    tr = torch.empty(nt, len(ijk), dtype=torch.float64, device="cuda")
    for n in range(nt):
        new, phi = X.step(u, up, phi, m, source, float(wavelet[n]))
        u, up = new, u
        tr[n] = u[at[:, 2], at[:, 1], at[:, 0]]
    return tr, u


def _exact_gradient(c, v, wavelet, source, ijk, obs):
    """(misfit, dJ/dv): each step differentiated in turn, last to first."""
    X, nt = _Exact(c), c["nt"]
    at = torch.from_numpy(ijk.astype(np.int64)).cuda()
    at = (at[:, 2], at[:, 1], at[:, 0])
    v64 = v.detach().double().requires_grad_(True)
    m = ((v64 * _dt(c)) ** 2)
    m0 = m.detach().requires_grad_(True)
    zero = torch.zeros(_shape(c), dtype=torch.float64, device="cuda")
    us, phis, res, J = [zero, zero], [zero], [], 0.0
    with torch.no_grad():
        for n in range(nt):
            new, phi = X.step(us[-1], us[-2], phis[-1], m0, source, float(wavelet[n]))
            us.append(new)
            phis.append(phi)
            res.append(new[at] - obs[n].double())
            J = J + 0.5 * (res[-1] ** 2).sum()
    gu, gup, gphi, gm = zero, zero, zero, zero
    for n in range(nt - 1, -1, -1):
        a = [t.detach().requires_grad_(True) for t in (us[n + 1], us[n], phis[n])]
        new, phi = X.step(*a, m0, source, float(wavelet[n]))
        r = torch.zeros_like(zero)
        r[at] = res[n]
        du, dup, dphi, dm = torch.autograd.grad((new, phi), (*a, m0), (gu + r, gphi), allow_unused=True)
        gu, gup = du + gup, dup
        gphi = zero if dphi is None else dphi
        gm = gm + dm
    (gv,) = torch.autograd.grad(m, v64, gm)
    return J, gv


def exact(case, seed):
    c = case
    if c["kind"] == "step":
        f = _step_inputs(c, seed)
        s = f["scale"].double() if "scale" in f else None
        u = f["u"].double() * (s[0] if s is not None else 1.0)
        up = u - f["d"].double() if "d" in f else f["up"].double() * (s[3] if s is not None else 1.0)
        w = float(f["wavelet"][STEP])
        X = _Exact(c)
        m = f["m"].double()
        new, phi = X.step(u, up, f["phi"].double(), m, f["source"], w)
        out = {"u": new, "phi": phi}
        if "d" in f:
            out["d"] = new - u
        if s is not None:
            nxt = _pow2_scale(4.0 * max(float(s[4]), float(s[7])) + _injected(c, f))
            out["u"] = new / nxt  # stored values
            state = s.clone()
            state[1], state[5], state[6] = nxt, new.abs().max(), 0.0
            out["scale"] = state
        if c["receivers"]:
            at = torch.from_numpy(_receivers(c, c["receivers"]).astype(np.int64)).cuda()
            out["traces"] = new[at[:, 2], at[:, 1], at[:, 0]]
        return out
    if c["kind"] == "layout":
        field = _waves(c, seed, 0)[0]
        Nz, Ny, Nx = _shape(c)
        pitch = (8 + Nx + 4 + 31) // 32 * 32
        P = torch.zeros(Nz + 8, Ny + 8, pitch, device="cuda")
        P[4:4 + Nz, 4:4 + Ny, 8:8 + Nx] = field
        return {"padded": P.reshape(-1), "back": field}
    if c["kind"] == "shot":
        tr, fin = _exact_shot(c, _velocity(c, seed), _ricker(c["nt"], _dt(c), seed), _source(c, seed),
                              _receivers(c, c["receivers"]), c["nt"])
        return {"traces": tr, "final": fin}
    if c["kind"] == "gradient":
        ijk = _receivers(c, c["receivers"])
        J, gv = _exact_gradient(c, _velocity(c, seed), _ricker(c["nt"], _dt(c), seed), _source(c, seed),
                                ijk, _observed(c, seed, len(ijk)).cuda())
        return {"misfit": J, "grad": gv}
    out = []
    for q in range(c["requests"]):
        r, rs = _request(c, seed, q)
        out.append(_exact_shot(r, _velocity(r, rs), _ricker(r["nt"], _dt(r), rs), _source(r, rs),
                               _receivers(r, 8), r["nt"])[0])
    return out
