"""The standalone [J r]^T [J r] contraction (trk_jtj_rows) against an FP64 product of the same rows.

Tolerance: each entry is a sum of FP32 products formed and summed per CTA in FP32, so its error is a
few 1e-7 of the sum of the magnitudes of its terms; checked at 1e-5 of sqrt(diag_i diag_j)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


def _ref(J):
    J64 = J.astype(np.float64)
    return J64.T @ J64


def _run(J, nc, ld):
    n = J.shape[0]
    dev = torch.zeros((max(n, 1), ld), dtype=torch.float32, device="cuda")
    if n:
        dev[:n, :nc] = torch.from_numpy(J)
    out = torch.full((nc, nc), np.nan, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    trk.jtj_rows(dev.data_ptr(), n, nc, ld, out.data_ptr(), st.cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("n,nc,ld", [(50010, 56, 56), (1, 1, 1), (257, 80, 96), (100003, 33, 40), (300, 17, 17)])
def test_matches_fp64_product(n, nc, ld):
    rng = np.random.default_rng(n + nc)
    J = (rng.normal(size=(n, nc)) * rng.uniform(0.01, 1.0, nc)).astype(np.float32)
    got = _run(J, nc, ld)
    ref = _ref(J)
    scale = np.sqrt(np.outer(np.diag(ref), np.diag(ref))) + 1e-30
    assert (np.abs(got - ref) / scale).max() < 1e-5
    assert np.array_equal(got, got.T)


def test_zero_rows_give_zeros():
    got = _run(np.zeros((0, 8), np.float32), 8, 8)
    assert np.all(got == 0)


def test_invalid_arguments_are_rejected():
    with pytest.raises(trk.TrkError) as e:
        trk.jtj_rows(0, 10, 8, 8, 0, 0)
    assert e.value.status == trk.TRK_ERR_INVALID_ARG
    dev = torch.zeros((4, 90), device="cuda")
    out = torch.zeros((90, 90), dtype=torch.float64, device="cuda")
    with pytest.raises(trk.TrkError):
        trk.jtj_rows(dev.data_ptr(), 4, 90, 90, out.data_ptr(), 0)


@pytest.mark.parametrize("n,nc,ld,offset", [
    (1, 80, 80, 0), (15, 32, 32, 0), (16, 33, 36, 0), (17, 64, 64, 0), (256, 65, 68, 0), (257, 4, 4, 0),
    (4097, 8, 9, 0), (38913, 40, 44, 0), (5000, 73, 76, 1), (5000, 73, 73, 0)])
def test_tile_and_alignment_edges(n, nc, ld, offset):
    """Column counts at the edges of the tile shapes (32 / 33, 64 / 65, 80), row counts at the edges of a
    16-row stage and of the grid, rows that allow 16-byte copies and rows that do not (odd ld, a base off by
    one float), NaN in the columns past nc, which must not count; the allocation-free call gives the same
    bits up to 38,912 rows.  Bound: a sum of n products in FP32, one chain per CTA of at most max(256, n / 152)
    rows: gamma = (rows + 1) 2^-24 of the sum of magnitudes."""
    rng = np.random.default_rng(7 * n + nc)
    J = (rng.normal(size=(n, nc)) * rng.uniform(0.01, 1.0, nc)).astype(np.float32)
    full = np.full((n, ld), np.nan, np.float32)
    full[:, :nc] = J
    buf = torch.empty(n * ld + 4, dtype=torch.float32, device="cuda")
    rows = buf[offset:offset + n * ld]
    rows.copy_(torch.from_numpy(full.ravel()))
    out = torch.empty((nc, nc), dtype=torch.float64, device="cuda")
    trk.jtj_rows(rows.data_ptr(), n, nc, ld, out.data_ptr())
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    X = J.astype(np.float64)
    bound = (max(256, n // 152 + 1) + 1) * 2.0 ** -24 * (np.abs(X).T @ np.abs(X))
    assert (np.abs(got - X.T @ X) <= bound + 1e-300).all()
    assert (got == got.T).all()
    if n <= 152 * 256:
        trk.jtj_rows_noalloc(rows.data_ptr(), n, nc, ld, out.data_ptr())
        torch.cuda.synchronize()
        assert (out.cpu().numpy() == got).all()
