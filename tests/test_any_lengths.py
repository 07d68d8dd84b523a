"""The generic kernels' two-pass lines at every length they take, and their fused
z pass at the edges of its tiles, against the FP64 oracle.

FFT bound: an FFT of n points done in factors has a relative L2 error of at most
a few unit roundoffs per factor-of-two level; 3 u log2(n0 n1 n2) covers the three
axes (u = 6e-8 in FP32, 1.1e-16 in FP64).  Pushes are held to the bounds of every
other parity test (_parity.TOL)."""
import math

import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_1812_07357_gb300 import inputs as I
from _parity import assert_fields

pytestmark = pytest.mark.gpu

U = {32: 2.0 ** -24, 64: 2.0 ** -53}


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_07357_gb300 import build
    build.build()


def _smooth(lo, hi, step):
    out = []
    for n in range(lo, hi + 1, step):
        m = n
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        if m == 1:
            out.append(n)
    return out


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_every_length(prec, axis):
    """Forward and inverse transform with one axis at every length: n0/2 from 2
    to 512 (odd ones too), n1 and n2 from 4 to 512; the other axes 6 and 10, so
    that the last tile of rows and columns is partial."""
    from paper_1812_07357_gb300.solver import Plan
    lengths = [2 * v for v in _smooth(2, 512, 1)] if axis == 0 else _smooth(4, 512, 2)
    boxes = []
    for n in lengths:
        dims = [6, 10, 6]
        dims[axis] = n
        boxes.append(I.Box(tuple(dims), (0, 0, 0), (0, 0, 0), (0, 0, 0), 0))
    lay = I.Layout("independent", (0, 0, 0), (1, 1, 1), boxes)
    rng = np.random.default_rng(31 + axis)
    arrs = I.round_to([rng.standard_normal(b.shape) for b in boxes], np.float32 if prec == 32 else np.float64)
    plan = Plan(lay, (1.0,) * 3, 0.5, precision=prec)
    spec = plan.forward_fft(plan.pack(arrs))
    got = plan.unpack_spectrum(spec)
    back = plan.unpack(plan.inverse_fft(spec))
    plan.sync()
    plan.close()
    for b, a, g, r in zip(boxes, arrs, got, back):
        ref = O.fft3(a)[:, :, : b.n[0] // 2 + 1]
        tol = 3 * U[prec] * math.log2(b.cells)
        assert np.linalg.norm(g - ref) <= tol * np.linalg.norm(ref), b.n
        assert np.linalg.norm(r - a) <= 2 * tol * np.linalg.norm(a), b.n


# z lengths of one and two prime-factor passes, of twiddled ones, of radices above 16 and the longest; column
# counts below, at and past a tile
SHAPES = [(4, 4, 4), (6, 4, 18), (30, 10, 16), (16, 6, 54), (10, 4, 270), (6, 4, 512), (50, 18, 72)]


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("form", ["vacuum", "J", "rho"])
def test_push_at_tile_edges(prec, form):
    from paper_1812_07357_gb300.solver import Plan
    # x guards of both parities: an even pair of guards stores pairs of cells, an odd one single cells
    boxes = [I.Box(n, (1 + i % 2, 1, 1), (1 + i % 2, 0, 1), (0, 0, 0), p)
             for i, (n, p) in enumerate(zip(SHAPES, (0, 2, 8, 16, 4, 0, 8)))]
    lay = I.Layout("independent", (0, 0, 0), (1, 1, 1), boxes)
    rng = np.random.default_rng(41)
    dt = np.float32 if prec == 32 else np.float64
    draw = lambda: I.round_to(I.scatter_self([rng.standard_normal(b.interior[::-1]) for b in boxes], lay), dt)
    fields = {k: draw() for k in O.COMPS}
    names = {"vacuum": (), "J": ("Jx", "Jy", "Jz"), "rho": ("Jx", "Jy", "Jz", "rho")}[form]
    src = {k: draw() for k in names}
    plan = Plan(lay, (1.0, 0.8, 1.25), 0.6, precision=prec, sources=form, generic=True)
    assert (plan.fast_boxes, plan.pencil_boxes) == (0, 0)
    df, ds = plan.pack_fields(fields), plan.pack_fields(src)
    plan.push(df, ds or None, 2)
    plan.sync()
    got = plan.unpack_fields(df)
    if form == "rho":
        got["rho"] = plan.unpack(ds["rho"])
    plan.close()
    ref = O.push(lay, fields, src, 2, (1.0, 0.8, 1.25), 0.6, form=form)
    assert_fields(lay, got, ref, O.COMPS + (("rho",) if form == "rho" else ()), prec)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("n", [(12, 10, 6), (10, 8, 270), (18, 6, 50)])
def test_layers_at_tile_edges(prec, n):
    from paper_1812_07357_gb300.solver import Plan
    lay = I.global_layout(n, 4)
    rng = np.random.default_rng(43)
    fields = {k: I.round_to([rng.standard_normal(lay.boxes[0].shape)], np.float32 if prec == 32 else np.float64)
              for k in O.COMPS}
    pml = dict(width=(2, 2, 2), sigma_max=(0.5, 0.4, 0.3), order=2)
    plan = Plan(lay, (1.0,) * 3, 0.7, precision=prec, sources="vacuum", pml=pml)
    df = plan.pack_fields(fields)
    plan.push(df, None, 2)
    plan.sync()
    got = plan.unpack_fields(df)
    parts = {k: plan.unpack(v) for k, v in plan.pml_parts().items()}
    plan.close()
    ref = O.push(lay, fields, {}, 2, (1.0,) * 3, 0.7, pml=pml)
    assert_fields(lay, got, ref, O.COMPS, prec)
    for k in O.SPLIT:
        err = np.linalg.norm(parts[k][0] - ref[k][0])
        assert err <= {64: 1e-12, 32: 2e-5}[prec] * np.linalg.norm(ref[k][0]), k


@pytest.mark.parametrize("n1", [48, 60])
def test_layers_on_register_planes(n1):
    """FP32 boxes of a register plane shape: x and y on the plane kernels, z on
    the generic pass (lengths with and without a register z kernel), layers on
    the faces of an open domain, the exchange after the damping."""
    from paper_1812_07357_gb300.solver import Plan
    lay = I.local_layout((80, 2 * n1 - 24, 36), (2, 2, 2), (4, 6, 3), 8, periodic=(0, 0, 1))
    rng = np.random.default_rng(47)
    fields = {}
    for k in O.COMPS:
        g = rng.standard_normal(lay.global_n[::-1])
        fields[k] = I.round_to(I.scatter_global(g, lay), np.float32)
    pml = dict(width=(4, 3, 2), sigma_max=(0.5, 0.4, 0.3), order=2)
    plan = Plan(lay, (1.0,) * 3, 0.7, precision=32, sources="vacuum", pml=pml)
    assert plan.fast_boxes == 8 and not plan.deferred_exchange
    df = plan.pack_fields(fields)
    plan.push(df, None, 3)
    plan.sync()
    got = plan.unpack_fields(df)
    parts = {k: plan.unpack(v) for k, v in plan.pml_parts().items()}
    plan.close()
    ref = O.push(lay, fields, {}, 3, (1.0,) * 3, 0.7, pml=pml)
    assert_fields(lay, got, ref, O.COMPS, 32)
    for k in O.COMPS:   # guards stored after the damping
        for g, r in zip(got[k], ref[k]):
            assert np.abs(g - r).max() <= 2e-4 * np.abs(r).max(), k
    for k in O.SPLIT:
        num = sum(np.linalg.norm((a - b)[3:-3, 6:-6, 4:-4]) ** 2 for a, b in zip(parts[k], ref[k])) ** 0.5
        den = sum(np.linalg.norm(b[3:-3, 6:-6, 4:-4]) ** 2 for b in ref[k]) ** 0.5
        assert num <= 2e-5 * den, k


@pytest.mark.parametrize("form,j_constant", [("vacuum", False), ("J", True), ("rho", False)])
def test_register_planes_with_any_z_length(form, j_constant):
    """Register plane shapes whose z length has no register z kernel: the generic
    z pass between the plane kernels, with the deferred exchange."""
    from paper_1812_07357_gb300.solver import Plan
    boxes = [I.Box(n, (4, 4, 2), (4, 4, 2), (0, 0, 0), p)
             for n, p in zip([(48, 48, 50), (96, 60, 18), (60, 48, 162)], (8, 0, 16))]
    lay = I.Layout("independent", (0, 0, 0), (1, 1, 1), boxes)
    rng = np.random.default_rng(53)
    draw = lambda: I.round_to(I.scatter_self([rng.standard_normal(b.interior[::-1]) for b in boxes], lay), np.float32)
    fields = {k: draw() for k in O.COMPS}
    src = {k: draw() for k in {"vacuum": (), "J": ("Jx", "Jy", "Jz"), "rho": ("Jx", "Jy", "Jz", "rho")}[form]}
    plan = Plan(lay, (1.0, 0.8, 1.25), 0.6, precision=32, sources=form, j_constant=j_constant)
    assert plan.fast_boxes == 3 and plan.deferred_exchange
    df, ds = plan.pack_fields(fields), plan.pack_fields(src)
    plan.push(df, ds or None, 3)
    plan.sync()
    got = plan.unpack_fields(df)
    if form == "rho":
        got["rho"] = plan.unpack(ds["rho"])
    plan.close()
    ref = O.push(lay, fields, src, 3, (1.0, 0.8, 1.25), 0.6, form=form)
    assert_fields(lay, got, ref, O.COMPS + (("rho",) if form == "rho" else ()), 32)
