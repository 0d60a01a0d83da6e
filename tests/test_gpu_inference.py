"""The column statistics of the network's rows at the edges of their tiles."""
import numpy as np
import pytest

from paper_2411_05799_gb300 import npx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(autouse=True)
def _own_stream():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        yield
    s.synchronize()


@pytest.mark.parametrize("rows,cols", [(1, 1), (7, 3), (2047, 36), (2048, 37), (4097, 72), (999, 73), (1000, 144),
                                       (5000, 145), (3001, 271)])
def test_column_moments(rows, cols):
    """FP64 sums: n terms in any order stay within n 2^-53 sum |term| of the exact sum (here against
    numpy's, itself within a few 2^-53); they add to what is there and repeat bit for bit."""
    g = torch.Generator("cuda").manual_seed(rows)
    X = torch.randn(rows, cols, device="cuda", generator=g) * 10.0 ** (torch.arange(cols, device="cuda") % 5 - 2) + 1.0
    st = torch.cuda.current_stream().cuda_stream
    got = []
    for _ in range(2):
        s = torch.full((2, cols), 0.5, dtype=torch.float64, device="cuda")
        npx.column_moments(X.data_ptr(), rows, cols, s[0].data_ptr(), s[1].data_ptr(), st)
        torch.cuda.synchronize()
        got.append(s.cpu().numpy())
    np.testing.assert_array_equal(got[0], got[1])
    h = X.cpu().numpy().astype(np.float64)
    for k, v in enumerate((h, h * h)):
        exact = np.array([np.sum(v[:, c].astype(np.longdouble)) for c in range(cols)], dtype=np.float64)
        bound = (rows + 2) * 2.0 ** -53 * (np.abs(v).sum(0) + 0.5) * 1.01
        assert (np.abs(got[0][k] - 0.5 - exact) <= bound).all()


def test_column_moments_of_infinities_and_nan():
    X = torch.ones(3000, 5, device="cuda")
    X[5, 1], X[2999, 2], X[7, 3], X[8, 3] = float("inf"), float("nan"), float("inf"), float("-inf")
    s = torch.zeros(2, 5, dtype=torch.float64, device="cuda")
    npx.column_moments(X.data_ptr(), 3000, 5, s[0].data_ptr(), s[1].data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    a, q = s.cpu().numpy()
    assert a[0] == 3000 and a[1] == np.inf and np.isnan(a[2]) and np.isnan(a[3]) and a[4] == 3000
    assert q[1] == np.inf and np.isnan(q[2]) and q[3] == np.inf
