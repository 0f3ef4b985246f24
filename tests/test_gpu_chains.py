"""The kernels whose work is a chain (forward kinematics, the LM solve) and the association's alternative paths, at the
sizes where they change: block and row-set edges of the solve, rotated link offsets and links without
vertices, a list of units longer than the grid's warps, a batch's searches over rows of occupancy bits, vertex
counts around a block of the result kernel."""
import numpy as np
import pytest

import oracle
from paper_1711_07999_gb300 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


def _tree_scene(L, seed):
    """A patch at 2 m whose vertices hang on random links of a random tree with prismatic joints, every other
    offset rotated (a general dual quaternion), the last link without vertices (its parameter is frozen)."""
    rng = np.random.default_rng(seed)
    parent, jtype, axis, offs = H.random_tree(rng, L=L)
    offs = [offs[0]] + [0.3 * t for t in offs[1:]]
    V, T = H.grid_patch(24, 18, -0.5, 0.5, -0.35, 0.35, 2.0)
    use = max(1, L - 1)
    k = min(4, use)
    idx = np.zeros((len(V), 4), np.uint8)
    w = np.zeros((len(V), 4), np.float32)
    for i in range(len(V)):
        idx[i, :k] = rng.choice(use, k, replace=False)
        w[i, :k] = rng.uniform(0.2, 1.0, k)
    w = (w / w.sum(1, keepdims=True)).astype(np.float32)
    m = H.make_model(parent, jtype, axis, offs, V, T, idx, w, W=96, H=72, fx=100.0, fy=100.0)
    for j in range(0, L, 2):
        q = np.array([1.0, *rng.uniform(-0.3, 0.3, 3)])
        q /= np.linalg.norm(q)
        t = np.array(offs[j]) / 2
        dual = [-(t @ q[1:]), *(t * q[0] + np.cross(t, q[1:]))]  # (0, t / 2) q
        m["skeleton"]["offset_dq"][j] = [*q, *dual]
    th = rng.normal(size=L) * 0.03
    depth = np.full((72, 96), 2.01, np.float32) + rng.normal(size=(72, 96)).astype(np.float32) * 0.002
    return m, th, depth


@pytest.mark.parametrize("L", [1, 2, 7, 8, 9, 31, 32, 33, 40, 63, 64, 65, 72, 79])
def test_kinematics_and_lm_step_at_the_block_edges(L):
    """Positions: a chain of up to L products of a few FP32 ulps at ~2 m (5e-6 m).  The LM step solves the GPU's own
    FP64 system to a scaled residual of 1e-10, so it is the FP64 solution to 1e-6 rad, as in the other tests."""
    m, th, depth = _tree_scene(L, 100 + L)
    o = oracle.Oracle(m)
    with trk.Session(m) as s:
        s.set_pose(th)
        s.set_depth(depth)
        for st in ("skin", "raster", "visibility", "associate", "normal_equations"):
            s.step(st)
        zero = np.zeros((o.V, 3))
        v, _ = o.skin(th, zero)
        assert np.abs(s.read("VERTS")[:, :3] - v).max() < 5e-6
        A, corr, lam0 = s.read("NORMAL_EQ"), s.read("CORR"), s.read("LAMBDA")[0]
        assert np.array_equal(A, A.T)
        s.step("lm")
        trials, th_gpu = s.read("LM_TRIALS"), s.read("THETA")
        n, ok = o.normals(v)
        acc, cnt = o.accumulate(v, depth, corr)
        _, inA, _ = o.residuals(th, n, ok, acc, cnt)
        assert inA.sum() > 50
        o.set_state(th, None)
        a_ref, th_ref, lam_ref, _ = o.lm_step(A[:L, :L], A[:L, L], trials[6], v, n, acc, cnt, inA, th, lam0)
        assert int(trials[7]) == a_ref
        assert np.abs(th_gpu - th_ref).max() < 1e-6
        assert s.read("LAMBDA")[0] == pytest.approx(lam_ref, rel=1e-12)
        if L > 1 and L - 1 not in m["skeleton"]["parent"]:
            assert th_gpu[-1] == th[-1]  # nothing observes the last link: its value stays


def test_association_of_a_full_image_matches_the_oracle():
    """Every pixel of a 640x480 image valid: more units than warps (a lane per pixel, own bucket first), with vertices
    four times denser than the pixels at the left and sparser than them at the right."""
    nx, ny = 500, 200
    xs = np.concatenate([np.linspace(-1.22, -1.05, 200), np.linspace(-1.04, 1.22, 300)])
    V, T = H.grid_patch(nx, ny, 0, 1, -0.92, 0.92, 2.0)
    V[:, 0] = xs[(V[:, 0] * (nx - 1) + 0.5).astype(int)]
    rng = np.random.default_rng(5)
    V[:, 2] += rng.normal(size=len(V)) * 2e-5
    m = H.make_model([-1], [1], [[0, 0, 1]], [[0, 0, 0]], V, T, [[0, 0, 0, 0]] * len(V), [[1, 0, 0, 0]] * len(V),
                     W=640, H=480, fx=525.0, fy=525.0, cutoff=0.02, window_half=6)
    o = oracle.Oracle(m)
    depth = (2.0 + rng.normal(size=(480, 640)) * 1e-3).astype(np.float32)
    ref = o.pass_at(np.zeros(1), np.zeros((o.V, 3)), depth, with_ties=True)
    with trk.Session(m) as s:
        s.set_pose(np.zeros(1))
        s.set_depth(depth)
        for st in ("skin", "raster", "visibility", "associate"):
            s.step(st)
        corr = s.read("CORR").reshape(ref["corr"].shape)
    diff = corr != ref["corr"]
    assert (ref["corr"] >= 0).sum() > 200000
    assert not (diff & ~(ref["tie"] > 0)).any(), np.argwhere(diff & ~(ref["tie"] > 0))[:5]


@pytest.mark.parametrize("window,cutoff", [(1, 0.05), (2, 0.1), (7, 0.15), (31, 0.5), (32, 0.5), (45, 0.7)])
def test_a_batchs_row_search_equals_the_ring_search_alone(window, cutoff):
    """A coarse mesh in a large image: searches of many rings.  Alone the tail scans rings of buckets, in a batch rows of
    occupancy bits (windows beyond 63 columns in pieces); the maps and results are the same bits."""
    ms = [synth.make_model(1, session=k, V=500 + 211 * k, width=333, height=251, window_half=window, cutoff=cutoff)
          for k in range(2)]
    frames, alone = [], []
    for k, m in enumerate(ms):
        with trk.Session(m) as s:
            rng = np.random.default_rng(k)
            z = s.render_depth(synth.gt_theta(m, 0.0), synth.gt_offsets(m, 0.0))
            z = np.where(z > 0, z + rng.normal(size=z.shape) * 0.02, 0).astype(np.float32)
            z[rng.random(z.shape) < 0.002] = 2.6  # lone pixels in the empty part of the image
            frames.append(z)
            s.set_pose(synth.start_theta(m))
            out = s.track_frame(z)
            alone.append((out, s.read("CORR")))
    sess = [trk.Session(m) for m in ms]
    dev = [torch.from_numpy(f).cuda() for f in frames]
    torch.cuda.synchronize()
    for s, m in zip(sess, ms):
        s.set_pose(synth.start_theta(m))
    st = torch.cuda.Stream()
    with trk.Batch(sess) as b:
        b.track_device([d.data_ptr() for d in dev], st.cuda_stream)
        for s, (ref, corr) in zip(sess, alone):
            got = s.read_result()
            assert np.array_equal(s.read("CORR"), corr)
            for key in ("theta", "offsets", "energy"):
                assert np.array_equal(got[key], ref[key]), key
    for s in sess:
        s.close()


@pytest.mark.parametrize("side", [(3, 5), (5, 51), (16, 16), (257, 1), (33, 31)])
def test_result_offsets_are_the_sessions(side):
    nx, ny = side
    if ny == 1:  # a strip of triangles over two rows, cut to an odd vertex count
        V, T = H.grid_patch(129, 2, -0.4, 0.4, -0.1, 0.1, 2.0)
        V = V[:257]
        T = T[(T < 257).all(1)]
    else:
        V, T = H.grid_patch(nx, ny, -0.4, 0.4, -0.3, 0.3, 2.0)
    m = H.make_model([-1], [1], [[0, 0, 1]], [[0, 0, 0]], V, T, [[0, 0, 0, 0]] * len(V), [[1, 0, 0, 0]] * len(V),
                     W=64, H=48, fx=60.0, fy=60.0)
    with trk.Session(m) as s:
        s.set_pose(np.zeros(1))
        out = s.track_frame(np.full((48, 64), 2.005, np.float32))
        assert np.array_equal(out["offsets"], s.read("PHI")[:, :3])
        assert np.array_equal(out["theta"], s.read("THETA"))
        assert np.array_equal(out["energy"], s.read("ENERGY"))
        assert np.abs(out["offsets"]).max() > 0


def test_batches_around_the_in_block_queue_prefix():
    """Up to 256 sessions a batch's tail forms the queues' prefix in its blocks, beyond that a kernel of its own does: 256
    and 257 tiny sessions, whose pixels lie far from their few vertices so that most are queued, equal each alone."""
    V, T = H.grid_patch(5, 4, -0.3, 0.3, -0.2, 0.2, 2.0)
    m = H.make_model([-1], [1], [[0, 0, 1]], [[0, 0, 0]], V, T, [[0, 0, 0, 0]] * len(V), [[1, 0, 0, 0]] * len(V),
                     W=24, H=18, fx=24.0, fy=24.0, window_half=6, cutoff=0.3, pose_iters=2, shape_iters=1)
    n = 257
    depth = [torch.full((18, 24), 1.95 + 0.0004 * k, dtype=torch.float32, device="cuda") for k in range(n)]
    sess = [trk.Session(m) for _ in range(n)]
    alone = []
    for s, d in zip(sess, depth):
        s.set_pose(np.zeros(1))
        out = s.track_frame(d.cpu().numpy())
        alone.append((out["theta"], out["offsets"], out["energy"], s.read("CORR")))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for count in (256, 257):
        for s in sess:
            s.set_pose(np.zeros(1))
        with trk.Batch(sess[:count]) as b:
            b.track_device([d.data_ptr() for d in depth[:count]], st.cuda_stream)
            for k in range(count):
                got = sess[k].read_result()
                for x, y in zip((got["theta"], got["offsets"], got["energy"], sess[k].read("CORR")), alone[k]):
                    assert np.array_equal(x, y), (count, k)
    assert (alone[0][3] >= 0).sum() > 50
    for s in sess:
        s.close()
