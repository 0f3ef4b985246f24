"""The association's tail on queues of many pixels per warp: an image with every pixel valid over a mesh far coarser than
the pixels, so that nearly all of them search on past the nearest buckets."""
import numpy as np
import pytest

import oracle
from tests import helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


def _scene(window):
    """320 x 240 pixels over 23 x 17 vertices 14 pixels apart: eight lanes a pixel up to a window of 31, a warp beyond."""
    V, T = H.grid_patch(23, 17, -1.2, 1.2, -0.9, 0.9, 2.0)
    rng = np.random.default_rng(11)
    V[:, :2] += rng.normal(size=(len(V), 2)) * 1e-3
    m = H.make_model([-1], [1], [[0, 0, 1]], [[0, 0, 0]], V, T, [[0, 0, 0, 0]] * len(V), [[1, 0, 0, 0]] * len(V),
                     W=320, H=240, fx=262.0, fy=262.0, cutoff=0.5, window_half=window)
    depth = (2.0 + rng.normal(size=(240, 320)) * 1e-3).astype(np.float32)
    return m, depth


@pytest.mark.parametrize("window", [3, 8, 31, 32])
def test_a_long_queue_matches_the_oracle(window):
    m, depth = _scene(window)
    o = oracle.Oracle(m)
    ref = o.pass_at(np.zeros(1), np.zeros((o.V, 3)), depth, with_ties=True)
    with trk.Session(m) as s:
        s.set_pose(np.zeros(1))
        s.set_depth(depth)
        for st in ("skin", "raster", "visibility", "associate"):
            s.step(st)
        corr = s.read("CORR").reshape(ref["corr"].shape)
    diff = corr != ref["corr"]
    assert (ref["corr"] >= 0).sum() > (10000 if window < 8 else 60000)
    assert not (diff & ~(ref["tie"] > 0)).any(), np.argwhere(diff & ~(ref["tie"] > 0))[:5]


@pytest.mark.parametrize("windows", [(0, 3, 0), (0, 0, 0), (31, 32, 31)])
def test_a_batch_of_different_windows_equals_each_alone(windows):
    """A session without rings (window 0) beside one that has them takes its units whole; windows up to 31 and beyond."""
    scenes = [_scene(w) for w in windows]
    alone = []
    for m, depth in scenes:
        with trk.Session(m) as s:
            s.set_pose(np.zeros(1))
            out = s.track_frame(depth)
            alone.append((out["theta"], out["offsets"], out["energy"], s.read("CORR")))
    sess = [trk.Session(m) for m, _ in scenes]
    for rows in (240, 40):  # more units than the grid has warps (7,200), and fewer
        part = []
        for (m, depth), s in zip(scenes, sess):
            d = depth.copy()
            d[rows:] = 0
            part.append(d)
            s.set_pose(np.zeros(1))
        if rows < 240:
            alone = []
            for (m, _), d in zip(scenes, part):
                with trk.Session(m) as s:
                    s.set_pose(np.zeros(1))
                    out = s.track_frame(d)
                    alone.append((out["theta"], out["offsets"], out["energy"], s.read("CORR")))
        dev = [torch.from_numpy(d).cuda() for d in part]
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        with trk.Batch(sess) as b:
            b.track_device([d.data_ptr() for d in dev], st.cuda_stream)
            for s, want in zip(sess, alone):
                r = s.read_result()
                for x, y in zip((r["theta"], r["offsets"], r["energy"], s.read("CORR")), want):
                    assert np.array_equal(x, y)
    for s in sess:
        s.close()
