"""Window peaks of overlap-save blocks whose magnitudes share the transform's shared memory (seven eighths of
1024 and 2048 points as outputs) and of their neighbours in size, over several blocks per launch unit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("B", [512, 1024, 2048, 4096])
def test_peaks_of_eighth_partitions(B, real):
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n = 1 << 16
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, "f32")
    rng = np.random.default_rng(B)
    z = torch.tensor(rng.standard_normal(n) + 1j * rng.standard_normal(n), dtype=rf.cdtype, device="cuda")
    lens, lag0 = [1, B // 8, B // 8 + 1, 900, 0], [0, -5, n - 1, -40000, 7]
    taps = rng.standard_normal(sum(lens)) + (0 if real else 1j * rng.standard_normal(sum(lens)))
    kern = rf.kernels_import(lag0, lens, taps, real=real)
    kern.prepare(B, B // 8)
    y = rf.reconstruct(z, kern, "direct")
    m = (y.real.double() ** 2 + y.imag.double() ** 2)
    tol = 4e-6 * m.amax(1, keepdim=True)              # of each row's largest |z|^2
    for W in (100, 1000, 4096, n):
        P, A = rf.reconstruct_winmax(z, kern, W, "os")
        nw = -(-n // W)
        pad = torch.cat([m, m.new_full((m.shape[0], nw * W - n), -1.0)], 1).view(m.shape[0], nw, W)
        assert ((P.double() - pad.amax(-1)).abs() <= tol).all(), W
        assert (A // W == torch.arange(nw, device="cuda")).all()
        assert ((m.gather(1, A.long()) - pad.amax(-1)).abs() <= 2 * tol).all(), W
