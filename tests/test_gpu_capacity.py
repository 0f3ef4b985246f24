"""What a session takes of the device memory: how many fit a budget follows from it."""
import pytest

from paper_1711_07999_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


@pytest.mark.parametrize("mib,size", [
    (38, dict(V=50000, width=640, height=480)), (128, dict(V=200000, width=1280, height=720)),
    (40, dict(V=55474, width=512, height=424, shape_solver=1)), (110, dict(V=200000, width=640, height=480, shape_solver=1)),
    (4, dict(V=5000, width=160, height=120)), (10, dict(V=9000, width=320, height=240))])
def test_device_bytes_of_a_session(mib, size):
    """The budgets a session of these sizes was admitted to since its buffers were laid out (pages of 2 MiB)."""
    with trk.Session(synth.make_model(2, session=0, **size), evicted=True) as s:
        assert s.info()["device_bytes"] <= mib << 20
