"""Order of the launches of a pass over boxes of several plane shapes and z
lengths.  The later launches of such a pass run beside the earlier ones, and a
CUDA graph carries only the edge from the pass's last launch into the next
pass, so the end of each launch has to imply the end of the one before it:
every kernel that lets its successor start early either waits before it reads
(grid_order) or has a block that does nothing but wait (grid_join)."""
import os
import re

import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_1812_07357_gb300 import inputs as I

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_07357_gb300", "csrc")


def _kernels():
    """(file, name, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        txt = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?\b([kg]_\w+)\s*\([^{;]*\)\s*\{", txt):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(txt[i], 0)
                i += 1
            yield f, m.group(1), txt[m.end():i - 1]


def test_kernels_that_release_their_successor_wait():
    ks = list(_kernels())
    released = [k for k in ks if "grid_release()" in k[2]]
    assert len(released) >= 7
    for f, name, body in released:
        assert re.search(r"if \((extra|MANY && grid_extra\(P\.order(, 2)?\))\) return grid_join\(\);", body), (f, name)
    # a kernel launched with an order has the device side of it
    launched = {n for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))
                for n in re.findall(r"launch_ordered\([^;]*?\b(k_\w+)", open(os.path.join(CSRC, f)).read())}
    known = {k[1] for k in ks if "grid_release()" in k[2] or "grid_order(" in k[2]}
    assert launched and launched <= known, launched - known


@pytest.fixture(scope="module")
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_07357_gb300 import build
    build.build()


# In every pass a long launch (boxes of 96^3) and after it a short one: plane
# shapes in the order 96 x 96, 48 x 48, 96 x 48, z lengths 48, 96, 120.
_MANY = [(96, 96, 96)] * 8 + [(48, 48, 120), (96, 48, 48)]


def _case(form):
    lay = I.Layout("independent", (0, 0, 0), (1, 1, 1),
                   [I.Box(n, (8,) * 3, (8,) * 3, (0, 0, 0), 8) for n in _MANY])
    rng = np.random.default_rng(17)
    names = O.COMPS + (("Jx", "Jy", "Jz") if form != "vacuum" else ()) + (("rho",) if form == "rho" else ())
    data = {k: I.scatter_self([rng.standard_normal(b.interior[::-1]) for b in lay.boxes], lay) for k in names}
    return lay, {k: data[k] for k in O.COMPS}, {k: v for k, v in data.items() if k not in O.COMPS}


@pytest.mark.gpu
@pytest.mark.parametrize("form,j_constant", [("vacuum", False), ("rho", True)])
def test_replayed_direct_captured_and_ordered_launches_agree(built, form, j_constant):
    import torch
    from paper_1812_07357_gb300 import _abi as A
    from paper_1812_07357_gb300.solver import Plan
    lay, fields, src = _case(form)
    s = torch.cuda.Stream()

    def run(how):
        plan = Plan(lay, (1.0,) * 3, 0.9, precision=32, sources=form, j_constant=j_constant, stream=s,
                    no_graph=how == "direct")
        if how == "ordered":   # per-kernel timing: every launch ordinary
            A.psatd_plan_set_timing(plan.handle, True)
        with torch.cuda.stream(s):
            df, ds = plan.pack_fields(fields), plan.pack_fields(src) if src else None
            if how == "captured":
                plan.push({k: v.clone() for k, v in df.items()},
                          {k: v.clone() for k, v in ds.items()} if ds else None, 1)
                plan.sync()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    plan.push(df, ds, 4)
            for _ in range(3):
                if how == "captured":
                    g.replay()
                else:
                    plan.push(df, ds, 4)
        plan.sync()
        torch.cuda.synchronize()
        out = dict(df, **({"rho": ds["rho"]} if form == "rho" else {}))
        out = {k: v.cpu().numpy() for k, v in out.items()}
        plan.close()
        return out

    want = run("ordered")
    assert all(np.isfinite(v).all() for v in want.values())
    for how in ("replayed", "direct", "captured"):
        got = run(how)
        for k in want:
            assert np.array_equal(got[k], want[k]), (how, k)


@pytest.mark.gpu
@pytest.mark.parametrize("nsteps", [1, 3])
def test_chained_launches_in_a_callers_capture(built, nsteps):
    """A plan on the line kernels, whose launches wait for one another: one push
    captured by the caller and replayed equals the same pushes launched directly."""
    import torch
    from paper_1812_07357_gb300.solver import Plan
    lay = I.local_layout((40, 32, 24), (2, 1, 1), (5, 4, 3), 4)
    rng = np.random.default_rng(19)
    fields = {k: I.scatter_global(rng.standard_normal((24, 32, 40)), lay) for k in O.COMPS}
    s = torch.cuda.Stream()
    plan = Plan(lay, (1.0,) * 3, 0.6, precision=32, sources="vacuum", stream=s, no_graph=True)
    assert plan.fast_boxes == 0
    with torch.cuda.stream(s):
        want, got = plan.pack_fields(fields), plan.pack_fields(fields)
        for _ in range(3):
            plan.push(want, None, nsteps)
        plan.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            plan.push(got, None, nsteps)
        for _ in range(3):
            g.replay()
    plan.sync()
    torch.cuda.synchronize()
    for k in O.COMPS:
        assert torch.equal(want[k], got[k]), k
    plan.close()
