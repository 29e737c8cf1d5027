"""Rows of the reference matched filter: each equals the call with that reference alone, whatever shares
the call, and its phase is good to the grid's rounding at any size."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


def _inputs(torch, n, dtype="f32", fs=2048.0, f_low=20.0):
    from paper_2511_12894_gb300 import RatioFilter
    rf = RatioFilter(n, fs, f_low, 971.0, 7, dtype)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).to(rf.rdtype)
    ip = 0.5 + 1.5 * torch.rand(n // 2 + 1, dtype=torch.float64, device="cuda", generator=g)
    return rf, x, ip


def _mixed(count, seed):
    """Coalescence times of 0 and others, light bodies (a large phase) and heavy ones."""
    rng = np.random.default_rng(seed)
    return [workload.Template(0.02 if r % 5 == 3 else float(rng.uniform(1.0, 3.0)), 0.03 if r % 5 == 3 else 1.2,
                              tc=0.0 if r % 3 else float(rng.uniform(0.0, 0.1)), phic=0.3) for r in range(count)]


@pytest.mark.parametrize("n,nref", [(1 << 9, 3), (1 << 13, 9), (1 << 18, 8), (1 << 20, 11)])
def test_rows_of_mixed_references(n, nref):
    torch = pytest.importorskip("torch")
    rf, x, ip = _inputs(torch, n)
    refs = _mixed(nref, nref)
    z, sg = rf.mf_reference(x, ip, refs)
    for r, t in enumerate(refs):
        z1, s1 = rf.mf_reference(x, ip, [t])
        assert torch.equal(z[r], z1[0]) and torch.equal(sg[r], s1[0]), r


@pytest.mark.parametrize("m", [2.0, 0.3, 0.03, 0.003])
def test_phase_of_light_bodies(m):
    """One bin of data passes one bin of the template: |angle| of the result against the FP64 grid's, to
    four roundings of an angle in FP32 (the filter's, the transforms') and no more for larger phases."""
    torch = pytest.importorskip("torch")
    n, fs = 1 << 16, 2048.0
    r32, _, ip = _inputs(torch, n, "f32", fs, 5.0)
    r64, _, _ = _inputs(torch, n, "f64", fs, 5.0)
    t = workload.Template(m, m)
    worst = 0.0
    for k in (161, 200, 331, 1999):                    # bins from 5 Hz on
        x = torch.cos(2.0 * np.pi * k / n * torch.arange(n, dtype=torch.float64, device="cuda"))
        z = [r.mf_reference(x.to(r.rdtype), ip, [t])[0][0, :16].cpu().numpy().astype(np.complex128)
             for r in (r32, r64)]
        worst = max(worst, np.abs(np.angle(z[0] * np.conj(z[1]))).max())
    assert worst <= 4 * np.pi * 2.0 ** -24, worst
