"""A batch on the default stream (NULL): reading a member's result, checkpointing and tracking it on follow its frame."""
import numpy as np
import pytest

from paper_1711_07999_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


def test_a_read_follows_a_batch_on_the_default_stream():
    m = synth.make_model(2, V=20000, width=320)
    with trk.Session(m) as s:
        depth = synth.add_noise(s.render_depth(synth.gt_theta(m, 0.1), synth.gt_offsets(m, 0.1)), 2, np.random.default_rng(1))
        s.set_pose(synth.gt_theta(m, 0.0))
        want = [s.track_frame(depth) for _ in range(3)]
        blob = s.export_state()
    d = torch.from_numpy(depth).cuda()
    torch.cuda.synchronize()
    with trk.Session(m) as s, trk.Batch([s]) as b:
        for _ in range(5):
            s.set_pose(synth.gt_theta(m, 0.0))
            for k in range(3):  # (0.7 ms of frame on the GPU: a read that does not wait is far too early)
                b.track_device([d.data_ptr()], 0)
                if k == 1:
                    continue  # two frames in a row
                got = s.read_result()
                for key in ("theta", "offsets", "energy"):
                    assert np.array_equal(got[key], want[k][key]), (k, key)
        s.set_pose(synth.gt_theta(m, 0.0))
        for _ in range(3):
            b.track_device([d.data_ptr()], 0)
        state = 8 * (s.L + 1) + 16 * s.V  # theta, lambda, Phi; before them a header that counts the session's own frames
        assert s.export_state()[-state:] == blob[-state:]
