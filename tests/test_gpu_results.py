"""The ways a frame's results are fetched (in the frame's graph, after it, copied by the server's per-session dispatch),
with and without offsets, with and without shape iterations: the same bits each way."""
import numpy as np
import pytest

from paper_1711_07999_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


@pytest.mark.parametrize("mode", [trk.MODE_TRACK, trk.MODE_SHAPE_MATCH, trk.MODE_SMOOTH_BIND])
def test_every_way_to_fetch_results_gives_the_same(mode):
    m = synth.make_model(1, V=1501, width=96, mode=mode)
    rng = np.random.default_rng(4)
    with trk.Session(m) as s:
        frames = [synth.add_noise(s.render_depth(synth.gt_theta(m, f / 30.0), synth.gt_offsets(m, f / 30.0)), 1, rng)
                  for f in range(5)]

    def device(s, f, want):
        d = torch.from_numpy(f).cuda()
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        s.track_frame_device(d.data_ptr(), st.cuda_stream)
        out = s.read_result(want_offsets=want)  # (waits for the frame on its stream)
        assert st.query()
        return out

    def served(s, f, want):
        return sv.wait(s, sv.submit(s, f), want_offsets=want)

    got = {}
    for way in ("host", "mixed", "device", "served"):
        with trk.Session(m) as s, trk.Server(1 << 40, dispatch=trk.SERVER_DISPATCH_SESSION) as sv:
            s.set_pose(synth.start_theta(m))
            if way == "served":
                sv.attach(s)
            outs = []
            for k, f in enumerate(frames):
                want = way != "mixed" or k % 2 == 1
                outs.append((s.track_frame if way in ("host", "mixed") else
                             lambda x, want_offsets: (device if way == "device" else served)(s, x, want_offsets))(
                                 f, want_offsets=want))
                assert np.array_equal(outs[-1]["theta"], s.read("THETA"))
                if want:
                    assert np.array_equal(outs[-1]["offsets"], s.read("PHI")[:, :3])
                else:
                    assert outs[-1]["offsets"] is None
            if way == "served":
                sv.detach(s)
        got[way] = outs
    for way, outs in got.items():
        for a, b in zip(outs, got["host"]):
            for key in ("theta", "energy", "n_assoc_px", "n_assoc_verts"):
                assert np.array_equal(a[key], b[key], equal_nan=True), (way, key)
            if a["offsets"] is not None:
                assert np.array_equal(a["offsets"], b["offsets"]), way
