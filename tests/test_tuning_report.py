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
