"""Truncation of built kernels over ranges of lags: the shortest circular arc, its first lag and
ties, against a direct search on the library's own untruncated kernels (threshold 0 keeps the
whole grid from its first signed lag)."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


def _arc(keep):
    """Shortest arc covering keep, ties to the smallest signed start: (m0, L)."""
    n = keep.size
    at = np.flatnonzero(keep)
    if not at.size:
        return 0, 0
    gap = np.diff(np.concatenate([at, [at[0] + n]])) - 1
    start = np.concatenate([at[1:], at[:1]])
    signed = np.where(start <= n // 2, start, start - n)
    best = min((-g, s) for g, s in zip(gap, signed))
    return best[1], n + best[0]


@pytest.mark.parametrize("n_build", [16, 32, 64, 1024, 8192, 1 << 15])
@pytest.mark.parametrize("real", [False, True])
def test_arcs(n_build, real):
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n = 1 << 15
    rf = RatioFilter(n, 1024.0, 40.0, 459.0, 2, "f64")
    ip = torch.ones(n // 2 + 1, dtype=torch.float64, device="cuda")
    ref = workload.Template(2.8, 2.8)
    nb = [workload.Template(2.8 + d, 2.8 - d / 2) for d in (0.0, 0.004, 0.02, -0.01, 0.1)]
    full = rf.build_ratio_kernels(ref, nb, ip, 0.0, n_build=n_build, real=real)
    assert (full.length == n_build).all()
    taps = full.taps().cpu().numpy().reshape(len(nb), n_build)
    for thr in (1e-6, 1e-3, 0.05, 0.5, 1.0):
        k = rf.build_ratio_kernels(ref, nb, ip, thr, n_build=n_build, real=real)
        for j in range(len(nb)):
            rho = np.roll(taps[j], int(full.lag0[j]))   # lag m at index m mod n
            m2 = rho.real ** 2 + rho.imag ** 2
            m0, L = _arc(m2 >= thr * thr * m2.max())
            assert (k.lag0[j], k.length[j]) == (m0, L), (n_build, thr, j)


@pytest.mark.parametrize("n_build", [4096, 1 << 14, 0, -1])
@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("analytic", [False, True])
def test_fp32_grids_keep_the_fp64_spans(n_build, real, analytic):
    """Kernels of an FP32 grid (transforms in FP32 pairs): spans equal to those of the FP64 grid, every
    tap within one FP32 rounding (2^-24 of it) plus the pairs' error (2^-43 of the largest tap)."""
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n = 1 << 17
    grids = [RatioFilter(n, 2048.0, 20.0, 971.0, 7, d) for d in ("f32", "f64")]
    ip = torch.ones(n // 2 + 1, dtype=torch.float64, device="cuda")
    ref = workload.Template(1.6, 1.5)
    rng = np.random.default_rng(3)
    nb = [ref] + [workload.Template(1.6 + a, 1.5 + b) for a, b in rng.uniform(-0.02, 0.02, (6, 2))]
    for thr in (1e-2, 3e-5, 1e-6, 1e-7, 1e-9) if not analytic else (1e-4, 1e-6):
        k32, k64 = (g.build_ratio_kernels(ref, nb, ip, thr, n_build=n_build, real=real, analytic=analytic)
                    for g in grids)
        assert np.array_equal(k32.lag0, k64.lag0) and np.array_equal(k32.length, k64.length), thr
        a, b = k32.taps().to(k64.taps().dtype).cpu().numpy(), k64.taps().cpu().numpy()
        a, b = a.view(np.float64), b.view(np.float64)
        assert (np.abs(a - b) <= 2.0 ** -24 * np.abs(b) + 2.0 ** -43 * np.abs(b).max()).all(), thr
