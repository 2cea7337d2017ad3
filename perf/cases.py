"""The workloads this framework is timed on: FDTD design gradients through its public calls.

A case is one problem a user's program runs again and again: one forward time
loop with the compressed boundary tape, and (but for the field simulation) one
time-reversed backward loop.  The handle, its workspace and the permittivity
on the device are what such a program keeps; a pass is the call or calls it
makes per design.  Time loops are shortened to a few hundred steps (the cost
per step does not depend on their number) with a broadband pulse and monitors
close enough that the gradient is not zero.

`exact` restates the method (Yee leapfrog, convolutional PML, quantised tape,
time-reversed interior with the adjoint alongside) in plain 64-bit torch.
"""
import math

import numpy as np
import torch
import torch.nn.functional as Fn

from paper_2603_24027_gb300 import _capi as A
from paper_2603_24027_gb300 import fdtd
from paper_2603_24027_gb300 import inputs as I

SIO2, SI = 2.085, 12.25
LARGEST = 600 * 600 * 300 * 160          # cell updates of the largest case (forward loop)


def _case(call, nx, ny, nz, pml, steps, tape, k, interp, **kw):
    return dict(call=call, nx=nx, ny=ny, nz=nz, pml=pml, steps=steps, tape=tape, k=k,
                interp=interp, **kw)


def listed():
    def c(name, *a, **kw):
        return dict(_case(*a, **kw), name=name)
    return [
        # smallest call: a point dipole in a 48^3 box with the uncompressed tape, the size of
        # gradient checks and unit cells; launches and latency count
        c("dipole48", "grad", 48, 48, 48, 8, 400, "f32", 1, "linear", device="dipole"),
        # the precision study's grid: many short gradients in BF16
        c("sweep100", "grad", 100, 100, 50, 12, 500, "bf16", 4, "linear", device="strip"),
        # odd small grid with the 8 x 8 block-transform tape and cubic restoring
        c("block131", "grad", 131, 97, 61, 10, 400, "bdct", 8, "cubic", device="strip"),
        # one iteration of the coupler optimisation: two flux detectors, an unscaled 8-bit tape
        # at k = 16, through the autograd function
        c("coupler150", "autograd", 150, 110, 70, 12, 400, "e4m3b11fnuz", 16, "linear",
          device="coupler"),
        # a batch of independent uneven cubes in one group call
        c("cubes20", "group", 128, 128, 128, 8, 200, "bf16", 4, "linear", device="cubes", count=20),
        # the mid-size device (200 x 200 x 100) with the scaled 8-bit tape
        c("waveguide200", "grad", 200, 200, 100, 12, 400, "e4m3", 8, "linear", device="strip"),
        # the same grid with bit-exact reversal (increments on a fixed grid), uncompressed tape
        c("exact200", "grad", 200, 200, 100, 12, 160, "f32", 1, "linear", device="strip", exact_q=22),
        # plain simulation, no gradient: odd ragged grid, objective and final fields
        c("fields233", "forward", 233, 181, 117, 11, 300, "bf16", 8, "linear", device="strip"),
        # host buffers in and out, pinned: what a caller without device arrays pays
        c("host301", "host", 301, 203, 151, 12, 160, "e4m3", 8, "linear", device="strip"),
        # an odd grid well beyond the L2 cache, FP16 tape with cubic restoring
        c("grating411", "grad", 411, 389, 203, 14, 120, "f16", 4, "cubic", device="strip"),
        # the largest single-device problem: 108 M cells, scaled 8-bit tape every 8th step
        c("waveguide600", "grad", 600, 600, 300, 16, 160, "e4m3", 8, "linear", device="strip"),
    ]


def draw(rng):
    """A problem of the same ranges: 14 thousand to 108 million cells, any aspect up to 4:1."""
    call = rng.choice(["grad", "grad", "grad", "grad", "autograd", "forward", "host", "group"])
    tape, k = rng.choice([("f32", 1), ("bf16", 1), ("bf16", 4), ("f16", 4), ("e4m3", 8),
                          ("e4m3", 8), ("e4m3b11fnuz", 16), ("bdct", 8)])
    interp = rng.choice(["linear", "linear", "cubic"])
    if call == "group":
        big = rng.randint(32, 144)
        steps = rng.randint(80, 200)
        return _case(call, big, big, big, rng.randint(6, 9), steps, "bf16", 4, "linear",
                     device="cubes", count=rng.randint(2, 20))
    cells = math.exp(rng.uniform(math.log(14e3), math.log(108e6)))
    if call == "autograd":
        cells = min(max(cells, 3e5), 6e6)
    ax, ay = math.exp(rng.uniform(0.0, 0.9)), math.exp(rng.uniform(0.0, 0.7))
    nz = (cells / (ax * ay)) ** (1.0 / 3.0)
    nx, ny, nz = int(nz * ax), int(nz * ay), int(nz)
    pml = min(rng.randint(6, 16), (min(nx, ny, nz) - 12) // 2)
    if call == "autograd":
        nx, ny, nz = max(nx, 110), max(ny, 90), max(nz, 60)
        pml = 12
    steps = rng.randint(100, 500)
    steps = max(60, min(steps, int(0.9 * LARGEST / (nx * ny * nz))))
    if tape == "f32" or (tape == "bf16" and k == 1):    # the tape of every step fits beside the state
        steps = min(steps, 200)
    kw = {}
    if call == "grad" and rng.random() < 0.15:
        kw["exact_q"] = rng.randint(20, 24)
        tape, k = "f32", 1
        steps = min(steps, 200)
    device = "coupler" if call == "autograd" else ("dipole" if cells < 2e5 else "strip")
    return _case(call, nx, ny, nz, pml, steps, tape, k, interp, device=device, **kw)


# ------------------------------------------------------------------ inputs --

def _smooth_random(shape, sigma, seed):
    """Unit-variance Gaussian-filtered noise through a sigmoid, in [0, 1] (device, float32)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(shape, generator=gen, device="cuda")
    r = int(math.ceil(3.0 * sigma))
    t = torch.arange(-r, r + 1, dtype=torch.float32, device="cuda")
    w = torch.exp(-0.5 * (t / sigma) ** 2)
    w = w / w.sum()
    for ax in range(3):
        v = a.movedim(ax, -1)
        s = v.shape
        v = Fn.pad(v.reshape(-1, 1, s[-1]), (r, r), mode="replicate")
        a = Fn.conv1d(v, w.view(1, 1, -1)).reshape(s).movedim(-1, ax).contiguous()
    a = (a - a.mean()) / (a.std() + 1e-12)
    return torch.sigmoid(a)


def _problem(case, seed):
    """(Workload, eps on the device) of a single-design case."""
    nx, ny, nz, P, N = case["nx"], case["ny"], case["nz"], case["pml"], case["steps"]
    dx = 20e-9 if nx < 500 else 10e-9
    dt = 0.99 * dx / (299792458.0 * math.sqrt(3.0))
    kw = dict(nx=nx, ny=ny, nz=nz, dx=dx, dt=dt, n_steps=N, pml_thickness=P, eps=None,
              rel_bandwidth=1.0, t0_over_tau=1.2)
    if case["device"] == "dipole":
        # random permittivity in the middle, Ez dipole below it, |E|^2 on a plane above
        eps = torch.ones((nz, ny, nx), device="cuda")
        lo = [max(P, n // 3) for n in (nx, ny, nz)]
        hi = [min(n - P, l + max(2, n // 3)) for n, l in zip((nx, ny, nz), lo)]
        gen = torch.Generator(device="cuda").manual_seed(seed)
        eps[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = 1.0 + (SI - 1.0) * torch.rand(
            (hi[2] - lo[2], hi[1] - lo[1], hi[0] - lo[0]), generator=gen, device="cuda")
        w = I.Workload(name="dipole", design_lo=tuple(lo), design_hi=tuple(hi),
                       src_kind=I.SRC_POINT, src_component=2,
                       src_pos=(nx // 2, ny // 2, P + 1), det_kind=I.OBJ_E2_PLANE, det_axis=2,
                       det_index=nz - P - 2, det_lo=(P, P), det_hi=(nx - P, ny - P), **kw)
        return w, eps
    eps = torch.full((nz, ny, nx), SIO2, device="cuda")
    h = max(2, int(round(220e-9 / dx)))
    h = min(h, nz - 2 * P - 2)
    z0 = (nz - h) // 2
    if case["device"] == "coupler":
        # normally incident sheet above a patterned square that feeds a strip along +x; the
        # flux through the strip and the flux above the square
        dev = min(ny - 2 * P - 8, nx - 2 * P - 40, 80)
        wy = max(6, dev // 4)
        x0, y0 = P + 6, (ny - dev) // 2
        yw = (ny - wy) // 2
        eps[z0:z0 + h, yw:yw + wy, x0 + dev:] = SI
        rho = _smooth_random((1, dev, dev), 3.0, seed)
        eps[z0:z0 + h, y0:y0 + dev, x0:x0 + dev] = SIO2 + (SI - SIO2) * rho
        w = I.Workload(name="coupler", design_lo=(x0, y0, z0), design_hi=(x0 + dev, y0 + dev, z0 + h),
                       src_kind=I.SRC_PLANE_UNIFORM, src_component=1, src_axis=2,
                       src_pos=(nx // 2, ny // 2, min(z0 + h + 14, nz - P - 2)),
                       det_kind=I.OBJ_POYNTING_PLANE, det_axis=0,
                       det_index=min(x0 + dev + 8, nx - P - 4),
                       det_lo=(max(P, yw - 6), max(P, z0 - 6)),
                       det_hi=(min(ny - P, yw + wy + 6), min(nz - P, z0 + h + 6)),
                       det2_kind=I.OBJ_POYNTING_PLANE, det2_axis=2,
                       det2_index=min(z0 + h + 8, nz - P - 4),
                       det2_lo=(x0, y0), det2_hi=(x0 + dev, y0 + dev), **kw)
        return w, eps
    # strip waveguide along x with a random smoothed design box; a Gaussian-profile sheet at the
    # low end and the flux through a plane: at the far end where the pulse arrives in time, else
    # just behind the sheet (the wave the device throws back crosses it too)
    wy = max(4, min(ny - 2 * P - 2, int(round(500e-9 / dx))))
    y0 = (ny - wy) // 2
    eps[z0:z0 + h, y0:y0 + wy, :] = SI
    far = (nx - 2 * P) * 5 < N
    lox = P + 8
    hix = max(lox + 2, min(nx - P - 8, nx - P - (nx - 2 * P) // 5))
    dy = max(2, int((ny - 2 * P) * 0.7))
    loy = P + (ny - 2 * P - dy) // 2
    box = (h, dy, hix - lox)
    eps[z0:z0 + h, loy:loy + dy, lox:hix] = SIO2 + (SI - SIO2) * _smooth_random(box, 60e-9 / dx, seed)
    w = I.Workload(name="strip", design_lo=(lox, loy, z0), design_hi=(hix, loy + dy, z0 + h),
                   src_kind=I.SRC_PLANE_GAUSS, src_component=1, src_axis=0,
                   src_pos=(P + 4, ny // 2, nz // 2), src_sigma_uv=(160e-9 / dx, 80e-9 / dx),
                   det_kind=I.OBJ_POYNTING_PLANE, det_axis=0,
                   det_index=nx - P - 4 if far else P + 6,
                   det_lo=(P, P), det_hi=(ny - P, nz - P), **kw)
    return w, eps


def _members(case, seed):
    """The single-design cases of a group: cubes of uneven size and step count."""
    rng = np.random.default_rng(1000 + case["count"])     # the sizes belong to the case
    big, P, N = case["nx"], case["pml"], case["steps"]
    sizes = [max(2 * P + 12, int(big * s)) for s in (0.25, 0.375, 0.5, 0.75, 1.0)]
    out = []
    for s in range(case["count"]):
        n = int(sizes[rng.integers(len(sizes))])
        out.append((_case("grad", n, n, n, P, int(rng.integers(N // 2, N + 1)), case["tape"],
                          case["k"], case["interp"], device="dipole"), seed * 1000 + s))
    return out


def _rec(case):
    return A.record_cfg(case["tape"], case["k"], case["interp"])


def _simulation(case, w):
    sim = fdtd.Simulation(w, device="cuda")
    if case.get("exact_q"):
        sim.set_option(A.OPT_EXACT_REVERSAL, case["exact_q"])
    sim.ensure_workspace(_rec(case))
    return sim


def prepare(case, seed):
    st = dict(call=case["call"], rec=_rec(case))
    if case["call"] == "group":
        pairs = [(c, _problem(c, s)) for c, s in _members(case, seed)]
        st["sims"] = [_simulation(c, w) for c, (w, _) in pairs]
        st["eps"] = [eps for _, (_, eps) in pairs]
        return st
    w, eps = _problem(case, seed)
    st["sim"] = _simulation(case, w)
    if case["call"] == "host":
        st["eps"] = eps.cpu().pin_memory()
        st["grad"] = torch.empty(w.design_shape, dtype=torch.float32, pin_memory=True)
    elif case["call"] == "autograd":
        st["eps"] = eps
        st["design"] = eps[w.design_slice()].clone().requires_grad_(True)
    else:
        st["eps"] = eps
    return st


def run(st):
    call, rec = st["call"], st["rec"]
    if call == "grad":
        L = st["sim"].forward(st["eps"], rec)
        return {"L": L, "grad": st["sim"].backward(1.0)}
    if call == "forward":
        L = st["sim"].forward(st["eps"], rec)
        return {"L": L, "fields": st["sim"].read_fields()}
    if call == "host":
        L, g = st["sim"].value_and_grad_host(st["eps"], rec, 1.0, st["grad"])
        return {"L": L, "grad": g}
    if call == "autograd":
        st["design"].grad = None
        LM = fdtd.objectives(st["design"], st["eps"], st["sim"], rec)
        (LM[0] - 0.5 * LM[1]).backward()
        return {"LM": LM.detach(), "grad": st["design"].grad}
    Ls = fdtd.group_forward(st["sims"], st["eps"], rec)
    return {"L": Ls, "grad": fdtd.group_backward(st["sims"])}


# -------------------------------------------------------------------- work --

def _design_cells(case):
    h = max(2, int(round(220e-9 / (20e-9 if case["nx"] < 500 else 10e-9))))
    P = case["pml"]
    if case["device"] == "dipole":
        return (case["nx"] // 3) * (case["ny"] // 3) * (case["nz"] // 3)
    if case["device"] == "coupler":
        return 80 * 80 * h
    return int((case["nx"] - 2 * P) * 0.8 * (case["ny"] - 2 * P) * 0.7) * min(h, case["nz"] - 2 * P - 2)


def work(case):
    """Permittivity read once, gradient (or fields) written once, the tape written once and read
    once; the additions and multiplications of the updates: 30 a cell and forward step, 30 more
    an interior cell and reverse step for the reversed fields, 36 a cell for the adjoint, 20 a
    cell, CPML axis and step for the auxiliaries."""
    if case["call"] == "group":
        parts = [work(c) for c, _ in _members(case, 0)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    n, P, N = (case["nx"], case["ny"], case["nz"]), case["pml"], case["steps"]
    cells = n[0] * n[1] * n[2]
    m = [d - 2 * P for d in n]
    inner = m[0] * m[1] * m[2]
    axes = sum(2 * P * cells // d for d in n)
    face = 4 * (m[0] * m[1] + m[1] * m[2] + m[0] * m[2])
    width = {"f32": 4.0, "bf16": 2.0, "f16": 2.0, "bdct": 14.0 / 64.0}.get(case["tape"], 1.0)
    tape = int(face * width * ((N + case["k"] - 1) // case["k"]))
    if case["call"] == "forward":
        return {"bytes": 4 * cells + tape + 24 * cells, "flops": N * (30 * cells + 20 * axes)}
    return {"bytes": 4 * cells + 2 * tape + 4 * _design_cells(case),
            "flops": N * (66 * cells + 30 * inner + 40 * axes)}


# ------------------------------------------------------------------- exact --

def _profiles(w, S):
    """Per axis, (b, a, 1/kappa) of the E (integer) and H (half-integer) positions in the two slabs."""
    out = []
    w0 = 2.0 * math.pi * S * w.dx / w.lambda0
    P = w.pml_thickness
    for ax, n in enumerate((w.nx, w.ny, w.nz)):
        sides = []
        for off in (0.0, 0.5):
            per = []
            for cells in (range(0, P), range(n - P, n)):
                co = []
                for i in cells:
                    x = i + off
                    lo, hi = float(P), n - P - 0.5
                    d = (lo - x if x < lo else max(0.0, x - hi)) / P
                    if d <= 0.0:
                        co.append((0.0, 0.0, 1.0))
                        continue
                    g = d ** w.pml_order
                    sig = w.pml_sigma_factor * (w.pml_order + 1.0) * S * g
                    kap = 1.0 + (w.pml_kappa_max - 1.0) * g
                    alp = w.pml_alpha_factor * w0 * (1.0 - d)
                    b = math.exp(-(sig / kap + alp))
                    co.append((b, sig * (b - 1.0) / (kap * (sig + kap * alp)), 1.0 / kap))
                t = torch.tensor(co, dtype=torch.float64, device="cuda").T
                shape = [1, 1, 1]
                shape[2 - ax] = P
                per.append([v.reshape(shape) for v in t])
            sides.append(per)
        out.append(sides)
    return out


# curl terms: (component, axis, sign, differentiated component)
_T = ((0, 1, 1, 2), (0, 2, -1, 1), (1, 2, 1, 0), (1, 0, -1, 2), (2, 0, 1, 1), (2, 1, -1, 0))


def _fdiff(f, ax):
    d = 2 - ax
    o = -f
    o.narrow(d, 0, f.shape[d] - 1).add_(f.narrow(d, 1, f.shape[d] - 1))
    return o


def _bdiff(f, ax):
    d = 2 - ax
    o = f.clone()
    o.narrow(d, 1, f.shape[d] - 1).sub_(f.narrow(d, 0, f.shape[d] - 1))
    return o


def _knot_weights(N, k, interp, n, field):
    """{sample: weight} of the tape at step n; field 0 = Ht, 1 = E."""
    r = (N - 1) % k
    t, slot = [], []
    if field == 0:
        t.append(-1.0); slot.append(-1)
    elif r > 0:
        t.append(0.0); slot.append(-1)
    for j in range((N - 1 - r) // k + 1):
        t.append(float(r + j * k)); slot.append(j)
    if float(n) in t:
        j = t.index(float(n))
        return {slot[j]: 1.0} if slot[j] >= 0 else {}
    b = next(i for i, v in enumerate(t) if v > n)
    a = b - 1
    hh = t[b] - t[a]
    s = (n - t[a]) / hh
    acc = {}

    def add(j, v):
        acc[j] = acc.get(j, 0.0) + v
    if interp == "linear":
        add(a, 1.0 - s); add(b, s)
    else:
        def slope(j):
            if len(t) == 2:
                h = t[1] - t[0]
                return ((0, -1.0 / h), (1, 1.0 / h))
            c = min(max(j, 1), len(t) - 2)
            p, q, u, x = t[c - 1], t[c], t[c + 1], t[j]
            return ((c - 1, ((x - q) + (x - u)) / ((p - q) * (p - u))),
                    (c, ((x - p) + (x - u)) / ((q - p) * (q - u))),
                    (c + 1, ((x - p) + (x - q)) / ((u - p) * (u - q))))
        add(a, (1 + 2 * s) * (1 - s) ** 2)
        add(b, s * s * (3 - 2 * s))
        for j, wgt in slope(a):
            add(j, s * (1 - s) ** 2 * hh * wgt)
        for j, wgt in slope(b):
            add(j, -s * s * (1 - s) * hh * wgt)
    return {slot[j]: v for j, v in acc.items() if slot[j] >= 0}


def _round8(x, M, bias, fmax):
    """Nearest value (ties to even, saturating) with M mantissa bits and the given exponent bias."""
    a = x.abs().clamp(max=fmax)
    m, e = torch.frexp(a)
    step = torch.ldexp(torch.ones_like(a), (e - 1).clamp(min=1 - bias) - M)
    return torch.sign(x) * torch.round(a / step) * step


def _quantise(planes, tape):
    """One face sample (two planes [v][u]) as it comes back from the tape."""
    if tape == "f32":
        return [p.float().double() for p in planes]
    if tape == "bf16":
        return [p.float().bfloat16().double() for p in planes]
    if tape == "bdct":
        return [_block_codec(p.float().double()) for p in planes]
    if tape in ("f16", "e4m3"):
        fmax = 65504.0 if tape == "f16" else 448.0
        amax = torch.stack([p.float().abs().max() for p in planes]).max()
        s = torch.where(amax > 0, (amax / fmax).clamp(min=2.0 ** -126), torch.ones_like(amax))
        q = [(p.float() / s).clamp(-fmax, fmax) for p in planes]
        q = [v.half().double() if tape == "f16" else _round8(v.double(), 3, 7, fmax) for v in q]
        return [v * s.double() for v in q]
    M, bias, fmax = {"e4m3b11fnuz": (3, 11, 30.0)}[tape]
    return [_round8(p.float().double(), M, bias, fmax) for p in planes]


def _block_codec(p, K=10):
    i = torch.arange(8, dtype=torch.float64, device=p.device)
    D = torch.cos(math.pi * (2 * i[None] + 1) * i[:, None] / 16) * 0.5
    D[0] *= math.sqrt(0.5)
    order = sorted(((u, v) for v in range(8) for u in range(8)), key=lambda t: (t[0] + t[1], t[1]))
    nv, nu = p.shape
    q = Fn.pad(p[None, None], (0, -nu % 8, 0, -nv % 8), mode="replicate")[0, 0]
    b = q.reshape(q.shape[0] // 8, 8, q.shape[1] // 8, 8).permute(0, 2, 1, 3)     # [bv, bu, y, x]
    C = D @ b @ D.T                                                               # [.., v, u]
    keep = torch.zeros(8, 8, dtype=torch.float64, device=p.device)
    for u, v in order[:K]:
        keep[v, u] = 1.0
    C = C * keep
    m = C.abs().amax((2, 3), keepdim=True)
    s = torch.where(m > 0, (m / 127.0).clamp(min=2.0 ** -126), torch.ones_like(m))
    b = D.T @ (torch.round(C / s) * s) @ D
    return b.permute(0, 2, 1, 3).reshape(q.shape)[:nv, :nu]


def _plane(w, det):
    """Index of a detector plane's cells in [z][y][x]."""
    ax, idx, lo, hi = det
    sl = [None, None, None]
    sl[2 - ax] = idx
    rest = [a for a in range(3) if a != ax]
    for a, l, h in zip(rest, lo, hi):
        sl[2 - a] = slice(l, h)
    return tuple(sl)


def _flux(E, H, kind, ax, sl):
    if kind == I.OBJ_E2_PLANE:
        return sum((e[sl] ** 2).sum() for e in E)
    b, c = (ax + 1) % 3, (ax + 2) % 3
    return (E[b][sl] * H[c][sl] - E[c][sl] * H[b][sl]).sum()


def _add_seed(E, H, kind, ax, sl, seed, lE, lH):
    if kind == I.OBJ_E2_PLANE:
        for e, l in zip(E, lE):
            l[sl] += 2.0 * seed * e[sl]
        return
    b, c = (ax + 1) % 3, (ax + 2) % 3
    lE[b][sl] += seed * H[c][sl]
    lE[c][sl] -= seed * H[b][sl]
    lH[c][sl] += seed * E[b][sl]
    lH[b][sl] -= seed * E[c][sl]


def _method(case, w, eps, seeds):
    """(L, M, fields, gradient) of the method in 64 bits; gradient None for seeds None."""
    f64 = dict(dtype=torch.float64, device="cuda")
    S = 299792458.0 * w.dt / w.dx
    cb = S / eps.double()
    pr = _profiles(w, S)
    P, N, n = w.pml_thickness, w.n_steps, (w.nx, w.ny, w.nz)
    E = [torch.zeros(w.shape, **f64) for _ in range(3)]
    H = [torch.zeros(w.shape, **f64) for _ in range(3)]

    def aux():
        return [[torch.zeros(1, **f64), torch.zeros(1, **f64)] for _ in range(6)]
    psE, psH = aux(), aux()

    def slabs(v, ax):
        return v.narrow(2 - ax, 0, P), v.narrow(2 - ax, n[ax] - P, P)
    # source weights and waveform
    w0 = 2.0 * math.pi * S * w.dx / w.lambda0
    tau = 2.0 * math.sqrt(2.0 * math.log(2.0)) / (w.rel_bandwidth * w0)

    def wave(i):
        t = (i + 0.5) - w.t0_over_tau * tau
        return w.amplitude * math.exp(-(t / tau) ** 2) * math.sin(w0 * t)
    if w.src_kind == I.SRC_POINT:
        x, y, z = w.src_pos
        ssl, sw = (slice(z, z + 1), slice(y, y + 1), slice(x, x + 1)), torch.ones(1, 1, 1, **f64)
    else:
        a = w.src_axis
        rest = [c for c in range(3) if c != a]
        ssl = [None] * 3
        ssl[2 - a] = slice(w.src_pos[a], w.src_pos[a] + 1)
        shape = [n[2], n[1], n[0]]
        sw = torch.ones(1, 1, 1, **f64)
        for c, sg in zip(rest, w.src_sigma_uv):
            ssl[2 - c] = slice(P, n[c] - P)
            r = (torch.arange(P, n[c] - P, **f64) - w.src_pos[c]) / sg
            g = torch.exp(-0.5 * r * r) if w.src_kind == I.SRC_PLANE_GAUSS else torch.ones_like(r)
            shape = [1, 1, 1]
            shape[2 - c] = -1
            sw = sw * g.reshape(shape)
        ssl = tuple(ssl)
    dets = [(w.det_kind, w.det_axis, _plane(w, (w.det_axis, w.det_index, w.det_lo, w.det_hi)))]
    if w.det2_kind:
        dets.append((w.det2_kind, w.det2_axis,
                     _plane(w, (w.det2_axis, w.det2_index, w.det2_lo, w.det2_hi))))
    # interface layers: Ht on the low faces at P - 1, E on the high faces at n - P
    faces = []
    for ax in range(3):
        for high in (0, 1):
            sl = [slice(P, n[2] - P), slice(P, n[1] - P), slice(P, n[0] - P)]
            sl[2 - ax] = n[ax] - P if high else P - 1
            faces.append((high, tuple(sl), [c for c in range(3) if c != ax]))
    k = case["k"]
    r = (N - 1) % k
    tape = []
    obj = [torch.zeros((), **f64) for _ in dets]
    for i in range(N):
        for t, (c, ax, sg, d) in enumerate(_T):
            v = _fdiff(E[d], ax)
            for s, (vs, (b, a, kv)) in enumerate(zip(slabs(v, ax), pr[ax][1])):
                psH[t][s] = b * psH[t][s] + a * vs
                vs.mul_(kv).add_(psH[t][s])
            H[c].add_(v, alpha=-S * sg)
        if seeds is not None and i >= r and (i - r) % k == 0:
            tape.append([_quantise([(E if hi else H)[c][sl] for c in cs], case["tape"])
                         for hi, sl, cs in faces])
        cur = [None] * 3
        for t, (c, ax, sg, d) in enumerate(_T):
            v = _bdiff(H[d], ax)
            for s, (vs, (b, a, kv)) in enumerate(zip(slabs(v, ax), pr[ax][0])):
                psE[t][s] = b * psE[t][s] + a * vs
                vs.mul_(kv).add_(psE[t][s])
            cur[c] = v.mul_(sg) if cur[c] is None else cur[c].add_(v, alpha=sg)
        cur[w.src_component][ssl] -= sw * wave(i)
        for c in range(3):
            E[c].addcmul_(cb, cur[c])
        for t, (kind, ax, sl) in enumerate(dets):
            obj[t] += _flux(E, H, kind, ax, sl)
    del cur, psE, psH, v, vs
    LM = [float(o) for o in obj]
    if seeds is None:
        return LM, torch.stack(E + H), None
    lE = [torch.zeros(w.shape, **f64) for _ in range(3)]
    lH = [torch.zeros(w.shape, **f64) for _ in range(3)]
    lpE, lpH = aux(), aux()
    ds = w.design_slice()
    acc = torch.zeros(w.design_shape, **f64)
    # the interior and its one-cell neighbours; the differences are taken on that box
    box = tuple(slice(P - 1, m - P + 1) for m in (n[2], n[1], n[0]))
    inn = (slice(1, -1),) * 3
    dsb = tuple(slice(s.start - P, s.stop - P) for s in ds)
    ssb = tuple(slice(s.start - P, s.stop - P) for s in ssl)
    core = (slice(P, n[2] - P), slice(P, n[1] - P), slice(P, n[0] - P))
    for i in range(N - 1, -1, -1):
        for field in (0, 1):
            wts = _knot_weights(N, k, case["interp"], i, field)
            for f, (hi, sl, cs) in enumerate(faces):
                if hi != field:
                    continue
                for m, c in enumerate(cs):
                    v = sum(wt * tape[j][f][m] for j, wt in wts.items())
                    (E if hi else H)[c][sl] = v
        for (kind, ax, sl), sd in zip(dets, seeds):
            _add_seed(E, H, kind, ax, sl, sd, lE, lH)
        cur = [None] * 3
        for c, ax, sg, d in _T:
            v = _bdiff(H[d][box], ax)[inn]
            cur[c] = v.mul_(sg) if cur[c] is None else cur[c].add_(v, alpha=sg)
        cur[w.src_component][ssb] -= sw * wave(i)
        for c in range(3):
            acc += lE[c][ds] * cur[c][dsb]
            E[c][core].addcmul_(cb[core], cur[c], value=-1.0)
        for c, ax, sg, d in _T:
            v = _fdiff(E[d][box], ax)[inn]
            H[c][core].add_(v, alpha=S * sg)
        del cur
        for t, (c, ax, sg, d) in enumerate(_T):
            v = cb * lE[c]
            v.mul_(sg)
            for s, (vs, (b, a, kv)) in enumerate(zip(slabs(v, ax), pr[ax][0])):
                mu = lpE[t][s] + vs
                lpE[t][s] = b * mu
                vs.mul_(kv).add_(a * mu)
            lH[d].sub_(_fdiff(v, ax))
        for t, (c, ax, sg, d) in enumerate(_T):
            v = lH[c] * (-S * sg)
            for s, (vs, (b, a, kv)) in enumerate(zip(slabs(v, ax), pr[ax][1])):
                mu = lpH[t][s] + vs
                lpH[t][s] = b * mu
                vs.mul_(kv).add_(a * mu)
            lE[d].sub_(_bdiff(v, ax))
    return LM, None, acc * (-(cb[ds] ** 2) / S)


def exact(case, seed):
    if case["call"] == "group":
        parts = [exact(c, s) for c, s in _members(case, seed)]
        return {"L": [p["L"] for p in parts], "grad": [p["grad"] for p in parts]}
    # 64-bit torch takes about 60 ns a thousand cells and forward step, three times that in reverse
    if case["nx"] * case["ny"] * case["nz"] * case["steps"] > 6e9:
        return None
    w, eps = _problem(case, seed)
    if case["call"] == "forward":
        LM, fields, _ = _method(case, w, eps, None)
        return {"L": LM[0], "fields": fields}
    if case["call"] == "autograd":
        LM, _, g = _method(case, w, eps, (1.0, -0.5))
        return {"LM": torch.tensor(LM, dtype=torch.float64, device="cuda"), "grad": g}
    LM, _, g = _method(case, w, eps, (1.0,))
    return {"L": LM[0], "grad": g.cpu() if case["call"] == "host" else g}
