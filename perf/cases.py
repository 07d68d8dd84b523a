"""Performance cases of the PSATD push: what a user's program has the library do.

A case is a flat dict.  Its geometry is either a Cartesian split of a domain
(``split`` = "global", "local" or "hybrid": ``sx * sy * sz`` boxes of
``nx * ny * nz`` cells each, guards included, ``gx/gy/gz`` guard cells per face
and axis) or a batch of self-periodic boxes (``split`` = "independent":
``boxes`` boxes drawn from ``box_seed``).  ``mode`` says which entry points a
pass calls:

  push     Plan.push of ``steps`` steps (laser propagation, stand-alone runs)
  pic      Plan.guard_exchange of fields and sources, then a one-step push: the
           field part of a particle-in-cell step, whose current is new each step
  cycle    the same step with the particles on their own grid: Coupling.to_fft
           of the current, a one-step push, Coupling.from_fft of the fields
  filter   Plan.forward_fft of one component, a filter on the spectrum,
           Plan.inverse_fft (spectral diagnostics and filtering)
  host     Plan.push_host_global: whole-domain arrays in page-locked host memory

Sizes are the repository's own configurations (the 32^3 plane waves, the 128^3
sources box, 96^3 local boxes, 192^3 local boxes and 384 x 256 x 256 hybrid
groups with 64 guards, the uneven batch of boxes from {48, 60, 80, 96, 120}),
cut in the number of boxes where a full batch only repeats them, and the ragged
sizes of its tests (even 5-smooth lengths such as 50, 72, 90, 100).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1812_07357_gb300 import inputs as I
from paper_1812_07357_gb300.solver import Coupling, Plan

E_B = ("Ex", "Ey", "Ez", "Bx", "By", "Bz")
SRC = ("rho", "Jx", "Jy", "Jz")
# Yee positions in cells, (x, y, z)
YEE = {"Ex": (.5, 0, 0), "Ey": (0, .5, 0), "Ez": (0, 0, .5), "Bx": (0, .5, .5), "By": (.5, 0, .5),
       "Bz": (.5, .5, 0), "Jx": (.5, 0, 0), "Jy": (0, .5, 0), "Jz": (0, 0, .5), "rho": (0, 0, 0)}
UNEVEN_SIZES = (48, 60, 80, 96, 120)
UNEVEN_GUARDS = (8, 24, 40)
UNEVEN_ORDERS = (8, 16, 32, 0)


def _case(name, split, n, s, g, p, prec, **kw):
    c = dict(name=name, mode="push", split=split, nx=n[0], ny=n[1], nz=n[2], sx=s[0], sy=s[1], sz=s[2], gx=g[0],
             gy=g[1], gz=g[2], p=p, prec=prec, sources="vacuum", j_constant=False, nodal=False, steps=1, dt=0.9,
             dx=1.0, dy=1.0, dz=1.0, pml=0, boxes=0, box_seed=0)
    c.update(kw)
    return c


def listed():
    one, none = (1, 1, 1), (0, 0, 0)
    return [
        # the smallest stand-alone run: 32^3 plane waves, infinite order, FP64, its 64 steps as one push
        _case("waves_32_f64", "global", (32, 32, 32), one, none, 0, 64, steps=64, dt=0.5),
        # the smallest call that PIC codes repeat: one step of a 64^3 box, the particles on 8 sub-domains of 32^3
        _case("pic_cycle_64_f32", "global", (64, 64, 64), one, none, 16, 32, mode="cycle", sources="rho"),
        # the 128^3 box with a constant current, advanced by continuity
        _case("sources_128_f32", "global", (128, 128, 128), one, none, 16, 32, sources="rho", j_constant=True,
              steps=16),
        # the same box as a PIC step in FP64: a new current each step
        _case("pic_128_f64", "global", (128, 128, 128), one, none, 16, 64, mode="pic", sources="rho"),
        # 'local' decomposition of the laser run: sub-domains of 64^3 with 16 guards (96^3 boxes), FP32 vacuum
        _case("local_96_f32", "local", (96, 96, 96), (8, 4, 4), (16, 16, 16), 32, 32, steps=4),
        # 'local' decomposition at high order: sub-domains of 64^3 with 64 guards (192^3 boxes)
        _case("local_192_f32", "local", (192, 192, 192), (4, 2, 2), (64, 64, 64), 64, 32, steps=2),
        # 'hybrid' decomposition: groups of 256^3 with 64 guards on the x faces (384 x 256 x 256 boxes)
        _case("hybrid_384_f32", "hybrid", (384, 256, 256), (2, 1, 1), (64, 0, 0), 64, 32, steps=2),
        # uneven batch of self-periodic sub-domains with a constant current
        _case("uneven_40_f32", "independent", none, none, none, 0, 32, sources="rho", j_constant=True, steps=4,
              boxes=40, box_seed=5),
        # open domain with absorbing layers, local decomposition into 96^3 boxes
        _case("pml_96_f32", "local", (96, 96, 96), (2, 2, 2), (16, 16, 16), 16, 32, steps=2, pml=12),
        # ragged FP64 sub-domains of a PIC step: lengths of no power of two, unequal cells, J form
        _case("ragged_f64", "local", (100, 90, 72), (2, 2, 2), (8, 8, 8), 8, 64, mode="pic", sources="J", dx=1.0,
              dy=0.8, dz=1.25, dt=0.5),
        # spectral filter of one component over a ragged FP32 domain
        _case("filter_240_f32", "global", (240, 200, 180), one, none, 16, 32, mode="filter"),
        # fields in host memory: one step of a 256 x 256 x 128 domain in 96^3 boxes
        _case("host_96_f32", "local", (96, 96, 96), (4, 4, 2), (16, 16, 16), 32, 32, mode="host"),
    ]


# ---- drawn cases -----------------------------------------------------------

def _lengths(lo, hi, step=2):
    out = []
    for v in range(lo, hi + 1):
        m = v
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        if m == 1 and v % step == 0:
            out.append(v)
    return out


def _near(rng, lo, hi):
    """An admissible box length, spread over the logarithm of [lo, hi]."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_lengths(lo, hi), key=lambda v: (abs(math.log(v / t)), v))


def draw(rng: random.Random):
    kind = rng.choice(("single", "single", "local", "local", "hybrid", "independent", "pml", "cycle", "filter",
                       "host"))
    prec = rng.choice((32, 32, 64))
    if kind in ("host", "independent"):
        prec = 32
    # padded cells of a pass: up to the listed cases of the precision (FP64 and layers at a tenth)
    cap = math.exp(rng.uniform(math.log(1 << 15), math.log(24e6 if prec == 32 else 3e6)))
    order = rng.choice((0, 4, 8, 16, 32, 64))
    sources = rng.choice(("vacuum", "J", "rho"))
    h = dict(dx=1.0, dy=rng.choice((1.0, 0.8, 1.25)), dz=rng.choice((1.0, 0.8, 1.25)), dt=rng.choice((0.4, 0.7, 0.9)))
    if kind == "independent":
        c = _case("", "independent", (0, 0, 0), (0, 0, 0), (0, 0, 0), 0, prec, sources="rho", j_constant=True,
                  boxes=rng.randint(3, 30), box_seed=rng.randrange(1 << 30), steps=rng.choice((1, 2, 4)), dt=h["dt"])
    else:
        if kind == "pml":
            cap = min(cap, 5e6 if prec == 32 else 1e6)
        hi = max(24, min(320, int(1.9 * cap ** (1 / 3))))
        n = [_near(rng, 16, hi) for _ in range(3)]
        while n[0] * n[1] * n[2] > cap and max(n) > 16:
            i = n.index(max(n))
            n[i] = _lengths(16, n[i] - 1)[-1]
        s, g, split = [1, 1, 1], [0, 0, 0], "global"
        if kind in ("local", "host", "pml"):
            split = "local"
            ng = rng.choice((2, 4, 5, 8, 16))
            g = [min(ng, (v - 8) // 2) for v in n]
            s = [2, 2, 2] if kind == "pml" else [rng.randint(1, 4) for _ in range(3)]
            while s[0] * s[1] * s[2] * n[0] * n[1] * n[2] > 2 * cap and max(s) > 1:
                s[s.index(max(s))] -= 1
        if kind == "hybrid":
            split = "hybrid"
            s[0] = rng.choice((2, 3, 4))
            g[0] = min(rng.choice((4, 8, 16, 32)), (n[0] - 8) // 2)
            while s[0] > 2 and s[0] * n[0] * n[1] * n[2] > 2 * cap:
                s[0] -= 1
        c = _case("", split, n, s, g, order, prec, sources=sources, **h)
        if kind == "pml":
            c.update(sources="vacuum", pml=rng.choice((2, 4, 6)), steps=rng.choice((1, 2, 3)))
        elif kind == "cycle":
            c.update(mode="cycle", sources=rng.choice(("J", "rho")))
        elif kind == "filter":
            c.update(mode="filter", sources="vacuum")
        elif kind == "host":
            c.update(mode="host", sources="vacuum")
        else:
            c.update(nodal=rng.random() < 0.15)
            if sources != "vacuum" and rng.random() < 0.5:
                c.update(mode="pic")
            else:
                c.update(steps=rng.choice((1, 2, 4, 8)), j_constant=sources != "vacuum" and rng.random() < 0.5)
    # no more work than the listed cases of the precision
    while c["steps"] > 1 and work(c)["bytes"] > (8e9 if prec == 32 and not c["pml"] else 8e8):
        c["steps"] //= 2
    del c["name"]
    return c


# ---- geometry ----------------------------------------------------------------

def _geometry(case):
    """[(n, guards, origin of the interior, order)] of every box, x fastest, and the domain size."""
    if case["split"] == "independent":
        r = np.random.default_rng(case["box_seed"])
        out = []
        for _ in range(case["boxes"]):
            n = tuple(int(v) for v in r.choice(UNEVEN_SIZES, size=3))
            g = int(r.choice([v for v in UNEVEN_GUARDS if min(n) - 2 * v >= 16]))
            out.append((n, (g, g, g), (0, 0, 0), int(r.choice(UNEVEN_ORDERS))))
        return out, None
    n, g = (case["nx"], case["ny"], case["nz"]), (case["gx"], case["gy"], case["gz"])
    s = (case["sx"], case["sy"], case["sz"])
    m = tuple(n[d] - 2 * g[d] for d in range(3))
    out = [(n, g, (i * m[0], j * m[1], k * m[2]), case["p"])
           for k in range(s[2]) for j in range(s[1]) for i in range(s[0])]
    return out, tuple(s[d] * m[d] for d in range(3))


def _periodic(case):
    return 0 if case["pml"] else 1


def _offsets(sizes, align):
    off, total = [], 0
    for v in sizes:
        off.append(total)
        total += -(-v // align) * align
    return off, total


def _layout(case):
    geo, dom = _geometry(case)
    boxes = [I.Box(n, g, g, o, p) for n, g, o, p in geo]
    per = (_periodic(case),) * 3
    return I.Layout(case["split"], dom or (0, 0, 0), per, boxes)


def _index(n, g, o, N, periodic):
    """Global index of every cell of one axis of a box, clamped, and whether it lies in the domain."""
    i = torch.arange(n, device="cuda") + (o - g)
    if periodic:
        return i % N, None
    return i.clamp(0, N - 1), (i >= 0) & (i < N)


def _scatter(case, doms):
    """Padded boxes of every domain array: doms is [ncomp, Nz, Ny, Nx], or a list of them, one per
    independent box; returns [ncomp, elements]."""
    geo, dom = _geometry(case)
    off, total = _offsets([n[0] * n[1] * n[2] for n, _, _, _ in geo], 64)
    first = doms if dom else doms[0]
    out = torch.zeros(first.shape[0], total, dtype=first.dtype, device="cuda")
    per = _periodic(case)
    for b, (n, g, o, _) in enumerate(geo):
        src = doms if dom else doms[b]
        N = dom or tuple(n[d] - 2 * g[d] for d in range(3))
        (ix, mx), (iy, my), (iz, mz) = (_index(n[d], g[d], o[d], N[d], per) for d in range(3))
        v = src[:, iz[:, None, None], iy[None, :, None], ix[None, None, :]]
        if mx is not None:
            v = v * (mz[:, None, None] & my[None, :, None] & mx[None, None, :])
        out[:, off[b]:off[b] + n[0] * n[1] * n[2]] = v.reshape(v.shape[0], -1)
    return out


# ---- inputs --------------------------------------------------------------------

def _noise(n, comps, gen):
    """Filtered noise of unit variance: normal deviates times a Gaussian of a quarter of Nyquist."""
    k = [torch.fft.fftfreq(n[2], device="cuda"), torch.fft.fftfreq(n[1], device="cuda"),
         torch.fft.rfftfreq(n[0], device="cuda")]
    f = [torch.exp(-0.5 * (a / 0.125) ** 2) for a in k]
    filt = f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    out = torch.empty(len(comps), n[2], n[1], n[0], device="cuda")
    for c in range(len(comps)):
        a = torch.randn(n[2], n[1], n[0], device="cuda", generator=gen)
        a = torch.fft.irfftn(torch.fft.rfftn(a) * filt, s=(n[2], n[1], n[0]))
        out[c] = a / a.std()
    return out


def _laser(n, h):
    """A pulse along +x in the middle of the domain: E_y and B_z at their Yee positions."""
    L = [n[d] * h[d] for d in range(3)]
    lam = max(8.0, min(16.0, L[0] / 8))
    out = []
    for comp in ("Ey", "Bz"):
        x, y, z = ((torch.arange(n[d], device="cuda") + YEE[comp][d]) * h[d] - L[d] / 2 for d in range(3))
        fx = torch.exp(-(x / (1.25 * lam)) ** 2) * torch.cos(2 * math.pi / lam * x)
        fy, fz = torch.exp(-(y / (L[1] / 6)) ** 2), torch.exp(-(z / (L[2] / 6)) ** 2)
        out.append(fz[:, None, None] * fy[None, :, None] * fx[None, None, :])
    return out


def _components(case):
    if case["mode"] == "filter":
        return ("Ey",)
    return E_B + {"vacuum": (), "J": SRC[1:], "rho": SRC}[case["sources"]]


def _domain_inputs(case, seed):
    """Initial data on the domain (or on every independent box's interior), rounded to the precision:
    a laser pulse over filtered noise in the fields, filtered noise in the current and the charge."""
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * (seed + 1))
    comps = _components(case)
    geo, dom = _geometry(case)
    h = (case["dx"], case["dy"], case["dz"])
    out = []
    for N in [dom] if dom else [tuple(n[d] - 2 * g[d] for d in range(3)) for n, g, _, _ in geo]:
        a = _noise(N, comps, gen) * 0.1
        ey, bz = _laser(N, h)
        a[comps.index("Ey")] += ey
        if "Bz" in comps:
            a[comps.index("Bz")] += bz
        if case["pml"]:   # the fields vanish inside the layers
            for d in range(3):
                i = torch.arange(N[d], device="cuda") + 0.5
                edge = torch.minimum(i, N[d] - i) - case["pml"] - 1
                w = torch.sin((edge / (0.2 * N[d])).clamp(0, 1) * (math.pi / 2)) ** 2
                a *= w.reshape([-1 if e == 2 - d else 1 for e in range(3)])
        out.append(a if case["prec"] == 32 else a.double())
    return out[0] if dom else out


def _pml_args(case):
    if not case["pml"]:
        return None
    w = case["pml"]
    return dict(width=(w, w, w), sigma_max=(2.5 / w * 6,) * 3, order=3)


def _g1_layout(case):
    """The particles' grid: sub-domains of half the domain with 4 guards, as they come."""
    N = (case["nx"], case["ny"], case["nz"])
    boxes = []
    for k in range(2):
        for j in range(2):
            for i in range(2):
                o = tuple((0, N[d] // 2)[(i, j, k)[d]] for d in range(3))
                m = tuple((N[d] // 2, N[d] - N[d] // 2)[(i, j, k)[d]] for d in range(3))
                boxes.append(I.Box(tuple(v + 8 for v in m), (4, 4, 4), (4, 4, 4), o, 0))
    return I.Layout("local", N, (1, 1, 1), boxes)


def _g1_scatter(case, dom):
    """Domain arrays [ncomp, ...] on the particles' grid, laid out as Coupling lays its buffers out."""
    g1 = _g1_layout(case)
    off, _ = _offsets([b.cells for b in g1.boxes], 64)
    total = off[-1] + g1.boxes[-1].cells + 64
    out = torch.zeros(dom.shape[0], total + (-total) % 64, dtype=dom.dtype, device="cuda")
    for b, q in enumerate(g1.boxes):
        iz, iy, ix = (_index(q.n[d], 4, q.origin[d], (case["nx"], case["ny"], case["nz"])[d], True)[0]
                      for d in (2, 1, 0))
        v = dom[:, iz[:, None, None], iy[None, :, None], ix[None, None, :]]
        out[:, off[b]:off[b] + q.cells] = v.reshape(v.shape[0], -1)
    return out, total


def _named(comps, rows, elems=None):
    return {c: rows[i] if elems is None else rows[i, :elems] for i, c in enumerate(comps)}


class _PlanMemory:
    """A plan-owned buffer that keeps its plan alive for as long as a tensor refers to it."""

    def __init__(self, plan, view):
        self.plan = plan
        self.__cuda_array_interface__ = view.__cuda_array_interface__


def prepare(case, seed):
    comps = _components(case)
    dom = _domain_inputs(case, seed)
    plan = Plan(_layout(case), (case["dx"], case["dy"], case["dz"]), case["dt"], precision=case["prec"],
                sources=case["sources"], j_constant=case["j_constant"], nodal=case["nodal"], pml=_pml_args(case))
    st = dict(case=case, plan=plan)
    if case["mode"] == "host":
        st["host_in"] = {c: dom[i].reshape(-1).cpu().pin_memory() for i, c in enumerate(comps)}
        st["host_out"] = {c: torch.empty_like(v).pin_memory() for c, v in st["host_in"].items()}
        return st
    rows = _scatter(case, dom)
    named = _named(comps, rows)
    if case["mode"] == "filter":
        # a smooth low-pass filter over the box's spectrum, as a diagnostics program keeps it
        n = (case["nx"], case["ny"], case["nz"])
        st["field"] = named["Ey"]
        st["filter"] = torch.zeros(plan.spec_elems, dtype=plan.dtype, device="cuda")
        f = _lowpass(n).to(plan.dtype).reshape(-1)
        st["filter"][:f.numel()] = f
        return st
    st["fields"] = {c: named[c] for c in E_B}
    st["src"] = {c: named[c] for c in comps if c not in E_B} or None
    if case["mode"] == "cycle":
        st["coupling"] = Coupling(plan, _g1_layout(case))
        j = [i for i, c in enumerate(comps) if c in SRC[1:]]
        g1, total = _g1_scatter(case, dom[j])
        st["g1_j"] = _named(SRC[1:], g1, total)
        g1f = torch.zeros(6, g1.shape[1], dtype=plan.dtype, device="cuda")
        st["g1_f"] = _named(E_B, g1f, total)
        for c in SRC[1:]:
            st["src"][c].zero_()
    if case["pml"]:
        st["parts"] = {c: torch.as_tensor(_PlanMemory(plan, v), device="cuda") for c, v in plan.pml_parts().items()}
    return st


def _lowpass(n):
    k = [torch.fft.fftfreq(n[2], device="cuda", dtype=torch.float64),
         torch.fft.fftfreq(n[1], device="cuda", dtype=torch.float64),
         torch.fft.rfftfreq(n[0], device="cuda", dtype=torch.float64)]
    f = [torch.cos(math.pi * a) ** 2 for a in k]
    return f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]


def run(state):
    case, plan = state["case"], state["plan"]
    mode = case["mode"]
    if mode == "host":
        plan.push_host_global(state["host_in"], state["host_out"], nsteps=case["steps"])
        return state["host_out"]
    if mode == "filter":
        spec = plan.forward_fft(state["field"])
        return {"spectrum": spec, "field": plan.inverse_fft(spec * state["filter"])}
    fields, src = state["fields"], state["src"]
    out = dict(fields)
    if mode == "pic":
        plan.guard_exchange(fields, src)
        plan.push(fields, src, 1)
    elif mode == "cycle":
        state["coupling"].to_fft(state["g1_j"], src)
        plan.push(fields, src, 1)
        state["coupling"].from_fft(fields, state["g1_f"])
        out.update({"g1_" + k: v for k, v in state["g1_f"].items()})
    else:
        plan.push(fields, src, case["steps"])
    if case["sources"] == "rho":
        out["rho"] = src["rho"]
    if case["pml"]:
        out.update(state["parts"])
    return out


# ---- work of one pass ----------------------------------------------------------

def work(case):
    """Bytes: every padded cell of every input read once and of every output written once, in every step
    where the fields exceed the 126 MB of L2 (a step's transforms need the whole of the step before), else
    once per pass; host arrays once.  Operations: 2.5 N log2 N per real transform and about 60 per mode and
    output slot for the update."""
    geo, dom = _geometry(case)
    cells = sum(n[0] * n[1] * n[2] for n, _, _, _ in geo)
    logs = sum(n[0] * n[1] * n[2] * math.log2(n[0] * n[1] * n[2]) for n, _, _, _ in geo)
    size = case["prec"] // 8
    if case["mode"] == "filter":   # real field in, spectrum out; spectrum in, real field out
        return {"bytes": cells * size * 4, "flops": 5.0 * logs + 2.0 * cells}
    fin = {"vacuum": 6, "J": 9, "rho": 10}[case["sources"]]
    fout = 7 if case["sources"] == "rho" else 6
    if case["pml"]:
        fin, fout = 12, 12
    steps = case["steps"]
    byts = (fin + fout) * cells * size * (steps if fin * cells * size > 126e6 else 1)
    if case["mode"] == "host":
        byts = 12 * dom[0] * dom[1] * dom[2] * size
    if case["mode"] == "cycle":
        byts += (3 + 6) * sum(b.cells for b in _g1_layout(case).boxes) * size
    flops = (2.5 * (fin + fout) * logs + 60.0 * fout * cells / 2) * steps
    return {"bytes": byts, "flops": flops}


# ---- the same in 64 bits with plain torch ----------------------------------------

def _modified_k(m, n, h, p, nodal):
    """Order-p modified wavenumber (p = 0: the wavenumber itself) of the indices m and its true one."""
    m = torch.where(2 * m > n, m - n, m).double()
    k = 2 * math.pi * m / (n * h)
    if p == 0:
        K = k.clone()
        if nodal:
            K[2 * m.abs() == n] = 0.0
        return K, k
    K = torch.zeros_like(k)
    q = p // 2
    for l in range(1, q + 1):
        x = lambda j: float(j * j if nodal else (2 * j - 1) ** 2)
        w = 1.0
        for j in range(1, q + 1):
            if j != l:
                w *= x(j) / (x(j) - x(l))
        if nodal:
            K += w * torch.sin(l * k * h) / (l * h)
        else:
            K += w * 2 * torch.sin((2 * l - 1) * k * h / 2) / ((2 * l - 1) * h)
    return K, k


class _Modes:
    """Everything the update of one box shape needs, c = eps0 = 1."""

    def __init__(self, case, n, p):
        h, dt = (case["dx"], case["dy"], case["dz"]), case["dt"]
        ar = [torch.arange(v, device="cuda") for v in (n[0] // 2 + 1, n[1], n[2])]
        kk = [_modified_k(ar[d], n[d], h[d], p, case["nodal"]) for d in range(3)]
        view = ((1, 1, -1), (1, -1, 1), (-1, 1, 1))
        self.K = [kk[d][0].reshape(view[d]) for d in range(3)]
        self.half = [torch.exp(0.5j * kk[d][1] * h[d]).reshape(view[d]) for d in range(3)]
        self.nodal = case["nodal"]
        K2 = self.K[0] ** 2 + self.K[1] ** 2 + self.K[2] ** 2
        th = torch.sqrt(K2) * dt
        small = th < 0.1
        t = torch.where(small, torch.ones_like(th), th)
        t2 = th * th
        self.C = torch.cos(th)
        self.S = dt * torch.where(small, 1 - t2 / 6 * (1 - t2 / 20 * (1 - t2 / 42 * (1 - t2 / 72))),
                                  torch.sin(t) / t)
        s = torch.where(small, 1 - t2 / 24 * (1 - t2 / 80 * (1 - t2 / 168)), torch.sin(t / 2) / (t / 2))
        self.X1 = dt * dt / 2 * s * s
        self.X3 = dt ** 3 * torch.where(
            small, -1 / 6 + t2 / 120 * (1 - t2 / 42 * (1 - t2 / 72 * (1 - t2 / 110))), (torch.sin(t) / t - 1) / (t * t))
        self.dt = dt

    def phase(self, comp):
        if self.nodal:
            return None
        ph = None
        for d in range(3):
            if YEE[comp][d]:
                ph = self.half[d] if ph is None else ph * self.half[d]
        return ph


def _cross(K, a):
    return [K[1] * a[2] - K[2] * a[1], K[2] * a[0] - K[0] * a[2], K[0] * a[1] - K[1] * a[0]]


def _dot(K, a):
    return K[0] * a[0] + K[1] * a[1] + K[2] * a[2]


def _step64(case, M, box):
    """One step of one padded box: {component: real array} -> new fields (and rho, and increments)."""
    f = {}
    for c, a in box.items():
        v, ph = torch.fft.rfftn(a), M.phase(c)
        f[c] = v if ph is None else v * ph.conj()
    K, C, S, X1, X3 = M.K, M.C, M.S, M.X1, M.X3
    E, B = [f[c] for c in E_B[:3]], [f[c] for c in E_B[3:]]
    kb, ke = _cross(K, B), _cross(K, E)
    kdb, kde = _dot(K, B), _dot(K, E)
    new = {}
    for a in range(3):
        new[E_B[3 + a]] = C * B[a] + X1 * K[a] * kdb - 1j * S * ke[a]
        new[E_B[a]] = C * E[a] + 1j * S * kb[a]
    if "Jx" in f:
        J = [f[c] for c in SRC[1:]]
        kj, kdj = _cross(K, J), _dot(K, J)
        for a in range(3):
            new[E_B[3 + a]] = new[E_B[3 + a]] + 1j * X1 * kj[a]
            new[E_B[a]] = new[E_B[a]] - S * J[a]
    if case["sources"] == "rho":
        rho1 = f["rho"] - 1j * M.dt * kdj
        g = 1j * (X3 / M.dt * rho1 - (X1 + X3 / M.dt) * f["rho"])
        for a in range(3):
            new[E_B[a]] = new[E_B[a]] + K[a] * g
        new["rho"] = rho1
    else:
        for a in range(3):
            new[E_B[a]] = new[E_B[a]] + X1 * K[a] * kde
            if "Jx" in f:
                new[E_B[a]] = new[E_B[a]] + X3 * K[a] * kdj
    if case["pml"]:
        IE = [S * E[a] - X3 * K[a] * kde + 1j * X1 * kb[a] for a in range(3)]
        IB = [S * B[a] - X3 * K[a] * kdb - 1j * X1 * ke[a] for a in range(3)]
        # the stored part of component a is its derivative along axis a + 1 of component a + 2
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            new["d" + E_B[a]] = 1j * K[b] * IB[c]
            new["d" + E_B[3 + a]] = -1j * K[b] * IE[c]
    out = {}
    shape = next(iter(box.values())).shape
    for c, v in new.items():
        ph = M.phase(c.removeprefix("d"))
        out[c] = torch.fft.irfftn(v if ph is None else v * ph, s=shape)
    return out


def _damping(case, dom, axis, offset):
    a = _pml_args(case)
    w, sig, m = a["width"][axis], a["sigma_max"][axis], a["order"]
    pos = torch.arange(dom[axis], device="cuda", dtype=torch.float64) + offset
    xi = torch.maximum(w - pos, pos - (dom[axis] - w)).clamp(0, w) / w
    return torch.exp(-sig * xi ** m * case["dt"]).reshape([-1 if e == 2 - axis else 1 for e in range(3)])


PARTS = ("Exy", "Eyz", "Ezx", "Bxy", "Byz", "Bzx")


def exact(case, seed):
    comps = _components(case)
    geo, dom = _geometry(case)
    src = _domain_inputs(case, seed)
    if case["mode"] == "filter":
        n = geo[0][0]
        spec = torch.fft.rfftn(src[0].double())
        low = _lowpass(n).to(torch.float32 if case["prec"] == 32 else torch.float64)   # as the program holds it
        field = torch.fft.irfftn(spec * low, s=(n[2], n[1], n[0]))
        flat = torch.zeros(spec.numel() + 64, dtype=spec.dtype, device="cuda")
        flat[:spec.numel()] = spec.reshape(-1)
        _, total = _offsets([n[0] * n[1] * n[2]], 64)
        real = torch.zeros(total, dtype=torch.float64, device="cuda")
        real[:field.numel()] = field.reshape(-1)
        return {"spectrum": flat, "field": real}
    doms = [src.double()] if dom else [a.double() for a in src]
    kept = E_B + (("rho",) if case["sources"] == "rho" else ())
    ik = [comps.index(c) for c in kept]
    modes = {}
    steps = 1 if case["mode"] in ("pic", "cycle") else case["steps"]
    parts = torch.zeros(6, *doms[0].shape[1:], dtype=torch.float64, device="cuda") if case["pml"] else None
    per = _periodic(case)
    for _ in range(steps):
        new = [a.clone() for a in doms]
        for b, (n, g, o, p) in enumerate(geo):
            which = 0 if dom else b
            N = dom or tuple(n[d] - 2 * g[d] for d in range(3))
            (ix, mx), (iy, my), (iz, mz) = (_index(n[d], g[d], o[d], N[d], per) for d in range(3))
            pad = doms[which][:, iz[:, None, None], iy[None, :, None], ix[None, None, :]]
            if mx is not None:
                pad = pad * (mz[:, None, None] & my[None, :, None] & mx[None, None, :])
            if (n, p) not in modes:
                modes[n, p] = _Modes(case, n, p)
            res = _step64(case, modes[n, p], dict(zip(comps, pad)))
            inner = tuple(slice(g[d], n[d] - g[d]) for d in (2, 1, 0))
            at = tuple(slice(o[d], o[d] + n[d] - 2 * g[d]) for d in (2, 1, 0))
            for i, c in zip(ik, kept):
                new[which][i][at] = res[c][inner]
            if case["pml"]:
                for q, c in enumerate(E_B):
                    parts[q][at] += res["d" + c][inner]
            del pad, res
        if case["pml"]:
            for q, c in enumerate(E_B):
                a = q % 3
                d1, d2 = (_damping(case, dom, (a + e) % 3, YEE[c][(a + e) % 3]) for e in (1, 2))
                other = new[0][q] - parts[q]
                parts[q] *= d1
                new[0][q] = parts[q] + d2 * other
        doms = new
    rows = _scatter(case, doms[0] if dom else doms)
    if case["mode"] == "host":
        return {c: doms[0][i].reshape(-1).cpu() for i, c in enumerate(comps)}
    out = {c: rows[i] for i, c in zip(ik, kept)}
    if case["mode"] == "cycle":
        g1, total = _g1_scatter(case, doms[0][:6])
        out.update({"g1_" + c: g1[i, :total] for i, c in enumerate(E_B)})
    if case["pml"]:
        prow = _interior_only(case, parts)
        out.update({c: prow[q] for q, c in enumerate(PARTS)})
    return out


def _interior_only(case, dom):
    """Domain arrays in the box layout, the guard cells zero."""
    geo, _ = _geometry(case)
    off, total = _offsets([n[0] * n[1] * n[2] for n, _, _, _ in geo], 64)
    out = torch.zeros(dom.shape[0], total, dtype=dom.dtype, device="cuda")
    for b, (n, g, o, _) in enumerate(geo):
        v = torch.zeros(dom.shape[0], n[2], n[1], n[0], dtype=dom.dtype, device="cuda")
        inner = (slice(None),) + tuple(slice(g[d], n[d] - g[d]) for d in (2, 1, 0))
        v[inner] = dom[(slice(None),) + tuple(slice(o[d], o[d] + n[d] - 2 * g[d]) for d in (2, 1, 0))]
        out[:, off[b]:off[b] + v[0].numel()] = v.reshape(dom.shape[0], -1)
    return out
