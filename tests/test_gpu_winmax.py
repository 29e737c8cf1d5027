"""Window peaks of series in memory: windows split over thread-block clusters, odd starts and
ragged last windows.  Samples are small integers, so |z|^2 and every tie are exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("W", [1, 255, 4097, 8192, 16383, 32769, 65536, 100001, 1 << 18])
def test_split_windows(dtype, W):
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n, count = 1 << 18, 3
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    rng = np.random.default_rng(W)
    z = rng.integers(-40, 41, (count, n)) + 1j * rng.integers(-40, 41, (count, n))
    z[1, :] = 3.0          # every sample ties: the first index of each window wins
    t = torch.tensor(z, dtype=rf.cdtype, device="cuda")
    P, A = rf.winmax(t, W)
    m = np.abs(z.real) ** 2 + np.abs(z.imag) ** 2
    for w in range(-(-n // W)):
        seg = m[:, w * W:(w + 1) * W]
        assert np.array_equal(P[:, w].cpu().numpy(), seg.max(axis=1).astype(np.float32))
        assert np.array_equal(A[:, w].cpu().numpy(), w * W + seg.argmax(axis=1))
        if W < 256 and w > 40:   # enough of the short ones
            break


def test_nan_never_wins():
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n, W = 1 << 17, 1 << 16
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, "f32")
    z = torch.zeros((1, n), dtype=rf.cdtype, device="cuda")
    z[0, : W] = float("nan")
    z[0, W + 77] = 2.0
    z[0, W + 40000] = float("nan")
    P, A = rf.winmax(z, W)
    assert P[0].tolist() == [-1.0, 4.0] and A[0].tolist() == [0, W + 77]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("W", [1, 2, 31, 32, 33, 64, 257, 1000, 1023, 1024, 1025, 2049])
def test_short_windows(dtype, W):
    """A warp per window up to 1024 samples, a block beyond: odd starts, ragged last windows, ties, windows
    of NaN and infinity."""
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n, count = 1 << 14, 2
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    rng = np.random.default_rng(W)
    z = rng.integers(-3, 4, (count, n)) + 1j * rng.integers(-3, 4, (count, n))
    z[0, rng.integers(0, n, 300)] = np.nan
    z[1, : 3 * W] = np.nan
    z[1, rng.integers(3 * W, n, 9)] = np.inf
    P, A = rf.winmax(torch.tensor(z, dtype=rf.cdtype, device="cuda"), W)
    nw = -(-n // W)
    with np.errstate(invalid="ignore"):
        m = np.abs(z.real) ** 2 + np.abs(z.imag) ** 2
    m = np.pad(np.where(np.isnan(m), -1.0, m), ((0, 0), (0, nw * W - n)), constant_values=-2.0).reshape(count, nw, W)
    best = m.max(-1)
    assert np.array_equal(P.cpu().numpy(), best.astype(np.float32))
    assert np.array_equal(A.cpu().numpy(), np.where(best < 0, 0, m.argmax(-1) + W * np.arange(nw)))
