"""The LM solve of a batch whose candidates are more than two CTAs per SM (51 sessions of six), which runs with fewer
threads and less shared memory: the same bits as each session alone, for link counts at the block edges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402
from tests.test_gpu_chains import _tree_scene  # noqa: E402


def test_a_crowded_solve_equals_each_session_alone():
    links = [1, 2, 7, 8, 9, 31, 32, 33, 40, 55, 63, 64, 65, 72, 79]
    scenes = [_tree_scene(L, 300 + L) for L in links]
    alone = []
    for m, th, depth in scenes:
        with trk.Session(m) as s:
            s.set_pose(th)
            out = s.track_frame(depth)
            alone.append((out["theta"], out["offsets"], out["energy"], s.read("LM_SOLVER"), s.read("LAMBDA")))
    n = 51
    sess = [trk.Session(scenes[k % len(links)][0]) for k in range(n)]
    dev = [torch.from_numpy(d).cuda() for _, _, d in scenes]
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for count in (50, 51):
        for k, s in enumerate(sess):
            s.set_pose(scenes[k % len(links)][1])
        with trk.Batch(sess[:count]) as b:
            b.track_device([dev[k % len(links)].data_ptr() for k in range(count)], st.cuda_stream)
            for k in range(count):
                r = sess[k].read_result()
                got = (r["theta"], r["offsets"], r["energy"], sess[k].read("LM_SOLVER"), sess[k].read("LAMBDA"))
                for x, y in zip(got, alone[k % len(links)]):
                    assert np.array_equal(x, y), (count, links[k % len(links)])
    for s in sess:
        s.close()
