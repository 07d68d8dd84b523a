"""FP64 x rows of radices above 16 (x lengths 250, 324, 500, 1000, 1024: half
lengths 5 x 25, 9 x 18, 10 x 25, 20 x 25, 16 x 32) run in blocks with fewer
threads than pass 1 has sub-transforms, alone and in one launch with shorter
lengths.  Against the FP64 oracle, FP64 bound."""
import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_1812_07357_gb300 import inputs as I
from _parity import assert_fields

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_07357_gb300 import build
    build.build()


@pytest.mark.parametrize("xs", [(250,), (324,), (500,), (1000,), (1024,), (250, 16, 90), (500, 96, 1000)])
def test_rows_of_wide_radices_match_the_oracle(xs):
    from paper_1812_07357_gb300.solver import Plan
    # nine interior rows a plane: the second tile of 8 is partial
    lay = I.Layout("independent", (0, 0, 0), (1, 1, 1),
                   [I.Box((x, 12, 10), (3, 2, 1), (2, 1, 3), (0, 0, 0), 4) for x in xs])
    rng = np.random.default_rng(sum(xs))
    fields = {k: I.scatter_self([rng.standard_normal(b.interior[::-1]) for b in lay.boxes], lay) for k in O.COMPS}
    plan = Plan(lay, (1.0,) * 3, 0.6, precision=64, sources="vacuum")
    df = plan.pack_fields(fields)
    plan.push(df, None, 3)
    plan.sync()
    got = plan.unpack_fields(df)
    f0 = plan.pack(fields["Ex"])
    back = plan.unpack(plan.inverse_fft(plan.forward_fft(f0)))
    plan.close()
    assert_fields(lay, got, O.push(lay, fields, {}, 3, (1.0,) * 3, 0.6), O.COMPS, 64)
    for a, b in zip(back, fields["Ex"]):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
