"""Absorbing layers with PSATD_J_CONSTANT: the form has no current, so the flag
changes nothing -- every slot (B among them) is transformed in every step."""
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


@pytest.mark.parametrize("n,prec", [((40, 18, 20), 64), ((40, 18, 20), 32), ((96, 96, 12), 32)])
@pytest.mark.parametrize("nsteps", [1, 3])
def test_layers_ignore_the_constant_current_flag(n, prec, nsteps):
    from paper_1812_07357_gb300.solver import Plan
    lay = I.global_layout(n, 8)
    pml = dict(width=(8, 4, 0), sigma_max=(0.4, 0.3, 0.0), order=2)
    rng = np.random.default_rng(41)
    inside = np.zeros(lay.boxes[0].shape)
    inside[:, 4:-4, 8:-8] = 1.0                    # the fields vanish in the layers
    fields = {k: [rng.standard_normal(inside.shape) * inside] for k in O.COMPS}
    if prec == 32:
        fields = {k: I.round_to(v, np.float32) for k, v in fields.items()}
    got = []
    for flag in (False, True):
        plan = Plan(lay, (1.0,) * 3, 0.7, precision=prec, sources="vacuum", pml=pml, j_constant=flag)
        df = plan.pack_fields(fields)
        plan.push(df, None, nsteps)
        plan.sync()
        out = plan.unpack_fields(df)
        out.update({k: plan.unpack(v) for k, v in plan.pml_parts().items()})
        got.append(out)
        plan.close()
    for k in got[0]:
        assert np.array_equal(got[0][k][0], got[1][k][0]), k
    ref = O.push(lay, fields, {}, nsteps, (1.0,) * 3, 0.7, pml=pml)
    assert_fields(lay, got[1], ref, O.COMPS, prec)
