"""Sizes that psatd_push_box_static takes: the boxes nearest the limit of its
static scratch on either side, and one that fits exactly against the
plan-based push.  The byte count of a size is checked before any GPU call, and
no step is run here but in the GPU test."""
import numpy as np
import pytest

from paper_1812_07357_gb300 import _abi as A
from paper_1812_07357_gb300 import build as B

COMPS = ("Ex", "Ey", "Ez", "Bx", "By", "Bz")


def _refused(n, p):
    """Whether the box is refused for its size (any other status, such as no
    device, comes after that check)."""
    B.build()
    f = A.psatd_fields()
    f.E[:] = f.B[:] = [4096] * 3      # never read: zero steps
    try:
        A.psatd_push_box_static(n, p, (1.0,) * 3, 0.5, 1.0, f, 0)
    except A.PsatdError as e:
        if e.status == A.PSATD_ERR_UNSUPPORTED_SIZE:
            assert str(A.PSATD_STATIC_SCRATCH_BYTES) in str(e)
            return True
    return False


# bytes that the limit leaves, with the job lists it was set for: 1152 and 384
# (162 x 270 x 50 with 1 and 128 weights), some 37000 for the next two; missing
# bytes of the first four refused: 2432, 6400, 24064, 24832
@pytest.mark.parametrize("n", [(162, 270, 50), (162, 54, 250), (162, 250, 54), (128, 128, 128)])
@pytest.mark.parametrize("p", [0, 256])
def test_boxes_up_to_the_limit_are_taken(n, p):
    assert not _refused(n, p)


@pytest.mark.parametrize("n", [(162, 50, 270), (32, 256, 256), (150, 270, 54), (270, 270, 30), (144, 144, 144)])
@pytest.mark.parametrize("p", [0, 256])
def test_boxes_beyond_the_limit_are_refused(n, p):
    assert _refused(n, p)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(162, 270, 50), (8, 4, 4)])
def test_static_push_equals_plan_push(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_07357_gb300 import inputs as I
    from paper_1812_07357_gb300.solver import Plan
    B.build()
    rng = np.random.default_rng(43)
    f = {k: rng.standard_normal((n[2], n[1], n[0])).astype(np.float32) for k in COMPS}
    plan = Plan(I.global_layout(n, 16), (1.0, 0.9, 1.1), 0.7, precision=32, sources="vacuum")
    ref = plan.pack_fields({k: [v] for k, v in f.items()})
    got = {k: torch.from_numpy(v.ravel().copy()).cuda() for k, v in f.items()}
    for _ in range(2):
        plan.push(ref, None, 2)
        A.psatd_push_box_static(n, 16, (1.0, 0.9, 1.1), 0.7, 1.0, Plan.fields_struct(got), 2,
                                plan.stream.cuda_stream)
    torch.cuda.synchronize()
    # FP32 rounding of two FFT orders over 4 steps, the bound of every FP32 parity test
    for k in COMPS:
        r = ref[k][:got[k].numel()].double()
        assert float((got[k].double() - r).norm() / r.norm()) <= 2e-5, k
    plan.close()
