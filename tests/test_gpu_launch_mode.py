"""sv_get_launch names the mode that a single next step runs in."""
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec, N, persistent", [
    ("FP64", 4864, True), ("FP64", 4865, True), ("FP64", 20000, True), ("FP64", 1 << 20, False),
    ("FP32", 4864, True), ("FP32", 4865, False), ("FP32", 100000, False)])
def test_auto_mode_of_a_single_step(prec, N, persistent):
    """Double takes the resident loop for any run on a grid that it holds, float
    beyond 4864 cells for runs of two steps and more."""
    sv = need_gpu()
    torch = pytest.importorskip("torch")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes of a 152-SM device")
    with sv.Solver(sv.Params(precision=getattr(sv, prec)), (N,), (1.0,)) as s:
        assert s.launch == (sv.LAUNCH_PERSISTENT if persistent else sv.LAUNCH_PER_STEP)
        s.set_launch(sv.LAUNCH_PER_STEP)
        assert s.launch == sv.LAUNCH_PER_STEP
