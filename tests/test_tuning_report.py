"""Knobs that a plan keeps and reports without a kernel that uses them: the
value given at creation comes back, and the autotuner spends no trial on it."""
import pytest

from paper_1812_07357_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_07357_gb300 import build
    build.build()


@pytest.mark.parametrize("n,family", [((64, 64, 64), True), ((20, 18, 12), False)])
@pytest.mark.parametrize("tuning,want", [(None, 64), ({"pencil_rows_kb": 32}, 32)])
def test_pencil_plans_report_their_rows_knob(n, family, tuning, want):
    from paper_1812_07357_gb300.solver import Plan
    plan = Plan(I.global_layout(n, 8), (1.0,) * 3, 0.5, precision=32, sources="vacuum", tuning=tuning)
    assert plan.pencil_boxes == int(family)
    assert plan.tuning().get("pencil_rows_kb") == (want if family else None)
    plan.close()


def test_autotuner_measures_no_unused_knob():
    # the families' times decide which knobs search() tries, so the measurement itself is asked
    from paper_1812_07357_gb300 import autotune as T
    measure = T.gpu_measure(I.global_layout((64, 64, 64), 8), (1.0,) * 3, 0.5, precision=64)
    _, used = measure("pencil", {"pencil_rows_kb": 32})
    assert "z_tile" in used and "pencil_rows_kb" not in used


@pytest.mark.parametrize("n,form,follows", [((128, 128, 128), "rho", False), ((96, 96, 192), "J", False),
                                            ((128, 128, 160), "rho", True)])
def test_z_tile_of_long_z_lines_with_sources(n, form, follows):
    """FP32 boxes on the register planes with sources: z lengths 128 and 192 keep
    their own tiles whatever z_tile and pencil_reg_z say, so neither is reported; other
    lengths follow them.  No result depends on it."""
    import torch
    from paper_1812_07357_gb300.solver import Plan
    out = []
    for tuning in (None, {"z_tile": 1}, {"z_tile": 3}):
        plan = Plan(I.global_layout(n, 8), (1.0,) * 3, 0.5, precision=32, sources=form, tuning=tuning)
        assert plan.fast_boxes == 1
        assert ("z_tile" in plan.tuning()) == follows
        assert ("pencil_reg_z" in plan.tuning()) == follows
        g = torch.Generator(device="cuda").manual_seed(3)
        f = {k: torch.randn(plan.field_elems, device="cuda", generator=g)
             for k in ("Ex", "Ey", "Ez", "Bx", "By", "Bz", "Jx", "Jy", "Jz", "rho")}
        s = {k: f[k] for k in ("Jx", "Jy", "Jz")}
        s["rho"] = f["rho"] if form == "rho" else None
        plan.push(f, s, 2)
        plan.sync()
        out.append(torch.cat([f[k] for k in ("Ex", "By")]))
        plan.close()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
