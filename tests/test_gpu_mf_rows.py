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


@pytest.mark.parametrize("log2n,nref", [(9, 3), (13, 5), (14, 5), (14, 25), (16, 3)])
def test_output_over_the_inputs_keeps_the_bits(log2n, nref):
    """Rows of an output that overlaps the data or the filters are those of a separate output."""
    torch = pytest.importorskip("torch")
    n = 1 << log2n
    rf, x, ip = _inputs(torch, n)
    g = torch.Generator(device="cuda")
    g.manual_seed(nref)
    filt = torch.view_as_complex(torch.randn((nref, n // 2 + 1, 2), device="cuda", generator=g))
    want = rf.mf_filtered(x, filt)
    buf = torch.zeros(nref * n * 2, device="cuda")
    out = torch.view_as_complex(buf.view(-1, 2)).view(nref, n)
    for at in (0, n, 2 * n):
        buf[at:at + n] = x
        assert torch.equal(rf.mf_filtered(buf[at:at + n], filt, z_out=out), want)
    flat = torch.zeros(nref * n, dtype=torch.complex64, device="cuda")
    flat[: filt.numel()] = filt.flatten()
    assert torch.equal(rf.mf_filtered(x, flat[: filt.numel()].view(nref, -1), z_out=flat.view(nref, n)), want)
    refs = _mixed(nref, 6)
    want, _ = rf.mf_reference(x, ip, refs)
    buf[n:2 * n] = x
    assert torch.equal(rf.mf_reference(buf[n:2 * n], ip, refs, z_out=out)[0], want)


@pytest.mark.parametrize("log2n", [14, 15, 16])
def test_rows_within_each_form(log2n):
    """2^14 to 2^16 samples: calls of few references agree bit for bit, and so do calls of many; between
    the two forms rows differ by rounding."""
    torch = pytest.importorskip("torch")
    n = 1 << log2n
    few = torch.cuda.get_device_properties(0).multi_processor_count // 8
    rf, x, _ = _inputs(torch, n)
    g = torch.Generator(device="cuda")
    g.manual_seed(log2n)
    filt = torch.view_as_complex(torch.randn((2 * few + 3, n // 2 + 1, 2), device="cuda", generator=g))
    call = lambda count: rf.mf_filtered(x, filt[:count].contiguous())
    many, more = call(few + 1), call(2 * few + 3)
    assert torch.equal(many, more[: few + 1])
    one, full = call(1), call(few)
    assert torch.equal(one[0], full[0]) and torch.equal(call(few // 2), full[: few // 2])
    assert (full - many[:few]).abs().max().item() <= 1e-6 * many.abs().max().item()
