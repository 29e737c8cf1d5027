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
