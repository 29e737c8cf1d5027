"""Kept spans of kernels built on FP32 grids (transforms in FP32 pairs) against those of the FP64 grid,
which are the definition's: |rho|^2 >= thr^2 max|rho|^2 decided in FP64."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


def _grids(n):
    from paper_2511_12894_gb300 import RatioFilter
    return [RatioFilter(n, 2048.0, 20.0, 971.0, 7, d) for d in ("f32", "f64")]


def _bank(count, seed):
    rng = np.random.default_rng(seed)
    return workload.Template(1.6, 1.5), [workload.Template(1.6 + a, 1.5 + b)
                                         for a, b in rng.uniform(-0.01, 0.01, (count, 2))]


@pytest.mark.parametrize("thr", [1e-7, 1e-6, 1e-5, 3e-5, 1e-2])
def test_spans_of_many_kernels(thr):
    """The lags left out before |rho|^2 is formed are judged by the whole value, h + l: at 1e-7 of the
    row's largest the low parts are a large share of it."""
    torch = pytest.importorskip("torch")
    n = 1 << 15
    r32, r64 = _grids(n)
    ip = torch.ones(n // 2 + 1, dtype=torch.float64, device="cuda")
    ref, nb = _bank(1500, 11)
    k32, k64 = (r.build_ratio_kernels(ref, nb, ip, thr) for r in (r32, r64))
    off = np.flatnonzero((k32.lag0 != k64.lag0) | (k32.length != k64.length))
    assert not off.size, (thr, off.size, off[:5])


def _edge(k64, j, thr):
    """Two neighbouring thresholds that keep and drop the smaller end of kernel j's span at thr."""
    t = k64.taps().cpu().numpy()[k64.offset[j]:k64.offset[j + 1]]
    m2 = t.real ** 2 + t.imag ** 2 if np.iscomplexobj(t) else t ** 2
    a, end = float(m2.max()), float(min(m2[0], m2[-1]))
    lo = np.sqrt(end / a)
    for _ in range(64):      # a few last places at most
        if lo * lo * a > end:
            lo = np.nextafter(lo, 0.0)
        elif np.nextafter(lo, 2.0) ** 2 * a <= end:
            lo = np.nextafter(lo, 2.0)
    assert lo * lo * a <= end < np.nextafter(lo, 2.0) ** 2 * a
    return float(lo), float(np.nextafter(lo, 2.0))


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("n_build", [0, -1])
@pytest.mark.parametrize("thr", [3e-5, 1e-3, 0.1])
def test_a_lag_at_the_cut(thr, n_build, real):
    """A threshold at the very value of a span's last or first lag: kept, and with the next larger threshold
    dropped, as in FP64; the taps are those of FP64 too."""
    torch = pytest.importorskip("torch")
    n = 1 << 16
    r32, r64 = _grids(n)
    ip = torch.ones(n // 2 + 1, dtype=torch.float64, device="cuda")
    ref, nb = _bank(5, 3)
    build = lambda r, t: r.build_ratio_kernels(ref, nb, ip, t, n_build=n_build, real=real)
    k64 = build(r64, thr)
    for j in range(len(nb)):
        lengths = []
        for t in _edge(k64, j, thr):
            a, b = build(r32, t), build(r64, t)
            assert np.array_equal(a.lag0, b.lag0) and np.array_equal(a.length, b.length), (j, t)
            x, y = a.taps().to(b.taps().dtype).cpu().numpy(), b.taps().cpu().numpy()
            x, y = x.view(np.float64), y.view(np.float64)
            assert (np.abs(x - y) <= 2.0 ** -24 * np.abs(y) + 2.0 ** -43 * np.abs(y).max()).all()
            lengths.append((int(b.lag0[j]), int(b.length[j])))
        assert lengths[0] != lengths[1], j


def test_each_kernel_is_judged_by_itself():
    """Neighbours far from the reference (a phase difference of many turns, a late coalescence) beside
    near ones, and phases of many whole turns: every kernel equals the one built alone and the FP64
    grid's."""
    torch = pytest.importorskip("torch")
    n = 1 << 16
    r32, r64 = _grids(n)
    ip = torch.ones(n // 2 + 1, dtype=torch.float64, device="cuda")
    ref = workload.Template(1.6, 1.5)
    nb = [workload.Template(1.601, 1.5), workload.Template(0.2, 0.2), workload.Template(1.6, 1.501, phic=4e7),
          workload.Template(1.6, 1.5, tc=3.0), workload.Template(1.6, 0.01), workload.Template(1.599, 1.502)]
    for thr in (3e-5, 1e-2):
        both, wide = (r.build_ratio_kernels(ref, nb, ip, thr) for r in (r32, r64))
        t, w = both.taps().cpu().numpy(), wide.taps().cpu().numpy()
        assert np.array_equal(both.lag0, wide.lag0) and np.array_equal(both.length, wide.length)
        for j, x in enumerate(nb):
            one = r32.build_ratio_kernels(ref, [x], ip, thr)
            a = t[both.offset[j]:both.offset[j + 1]]
            assert np.array_equal(one.taps().cpu().numpy(), a), j
            b = w[wide.offset[j]:wide.offset[j + 1]]
            assert np.abs(a - b).max() <= 2.0 ** -23 * np.abs(b).max(), j


@pytest.mark.parametrize("relative", [True, False])
def test_analytic_spans_on_both_grids(relative):
    """Analytic truncation: spans of the FP64 grid, at amplitudes far below the largest tap too."""
    torch = pytest.importorskip("torch")
    n = 1 << 16
    r32, r64 = _grids(n)
    ip = torch.ones(n // 2 + 1, dtype=torch.float64, device="cuda")
    ref, nb = _bank(40, 8)
    for thr in (1e-2, 1e-4, 1e-6, 1e-8) if relative else (1.0, 1e-3, 1e-5):
        for real in (False, True):
            a, b = (r.build_ratio_kernels(ref, nb, ip, thr, relative=relative, analytic=True, real=real)
                    for r in (r32, r64))
            assert np.array_equal(a.lag0, b.lag0) and np.array_equal(a.length, b.length), (thr, real)
