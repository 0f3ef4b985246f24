"""The row contraction at the edges of its row widths and of their stages (16, 32, 48 and 80 columns; 64, 32 and 16 rows),
and the FP64 sums of its partials where they are neither normal numbers nor zero.

The rows hold small whole numbers (times a power of two), so every product and sum is exact: the result is the exact
product, to the bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1711_07999_gb300 import trk  # noqa: E402


def _contract(J, ld, offset, call):
    n, nc = J.shape
    full = np.full((n, ld), np.nan, np.float32)
    full[:, :nc] = J
    buf = torch.empty(n * ld + 4, dtype=torch.float32, device="cuda")
    rows = buf[offset:offset + n * ld]
    rows.copy_(torch.from_numpy(full.ravel()))
    out = torch.empty((nc, nc), dtype=torch.float64, device="cuda")
    call(rows.data_ptr(), n, nc, ld, out.data_ptr())
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("nc", [1, 3, 4, 5, 15, 16, 17, 20, 31, 32, 33, 47, 48, 49, 64, 80])
@pytest.mark.parametrize("n", [1, 15, 17, 63, 64, 65, 255, 257, 3001])
def test_exact_at_the_edges_of_widths_and_stages(n, nc):
    J = np.random.default_rng(100 * n + nc).integers(-9, 10, (n, nc)).astype(np.float32)
    want = J.astype(np.float64).T @ J
    for ld, offset in (((nc + 3) // 4 * 4, 0), (nc | 1, 0), ((nc + 3) // 4 * 4 + 4, 1)):
        for call in (trk.jtj_rows, trk.jtj_rows_noalloc):
            assert np.array_equal(_contract(J, ld, offset, call), want), (ld, offset)


@pytest.mark.parametrize("n", [200, 600, 12000])  # one, three and 47 partials
@pytest.mark.parametrize("nc", [5, 40, 73])
def test_partials_that_are_subnormal_infinite_or_nan(n, nc):
    rng = np.random.default_rng(n + nc)
    J = rng.integers(-3, 4, (n, nc)).astype(np.float32) * np.float32(2.0 ** -71)  # products: multiples of 2^-142
    J[:, 1] *= np.float32(2.0 ** 71)
    want = J.astype(np.float64).T @ J
    assert np.abs(want[0, 0]) < 2.0 ** -126 or n > 1000
    got = _contract(J, (nc + 3) // 4 * 4, 0, trk.jtj_rows)
    assert np.array_equal(got, want)
    J = rng.integers(1, 4, (n, nc)).astype(np.float32)
    J[n // 2, 2] = np.inf
    J[n - 1, 3] = -np.inf
    J[0, 4] = np.nan
    want = J.astype(np.float64).T @ J
    got = _contract(J, (nc + 3) // 4 * 4, 0, trk.jtj_rows)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    want[np.isnan(want)] = got[np.isnan(got)] = 0
    assert np.array_equal(got, want)
