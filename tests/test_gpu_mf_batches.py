"""Reference templates generated in batches: every row equals the call with that reference alone,
at the edges of a batch, and the matched filter of its stored filter."""
import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("n,nref", [(1 << 9, 1), (1 << 12, 8), (1 << 12, 9), (1 << 13, 17), (1 << 20, 5),
                                    (1 << 22, 2)])
def test_rows_equal_single_calls(dtype, n, nref):
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    if dtype == "f64" and n > 1 << 20:
        pytest.skip("the FP64 passes are the same code at every batch of one")
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    rng = np.random.default_rng(nref)
    x = torch.tensor(rng.standard_normal(n), dtype=rf.rdtype, device="cuda")
    ip = torch.tensor(rng.uniform(0.5, 2.0, n // 2 + 1), device="cuda")
    refs = [workload.Template(float(m), 1.2, tc=float(t), phic=0.3)
            for m, t in zip(rng.uniform(1.2, 2.4, nref), rng.uniform(0.0, 0.1, nref))]
    z, sg = rf.mf_reference(x, ip, refs)
    for r, t in enumerate(refs):
        z1, s1 = rf.mf_reference(x, ip, [t])
        assert torch.equal(z[r], z1[0]) and torch.equal(sg[r], s1[0])
    filt, sf = rf.reference_filters(ip, refs)
    zf = rf.mf_filtered(x, filt)
    assert torch.equal(sf, sg)
    tol = 1e-12 if dtype == "f64" else 2e-6
    assert (zf - z).abs().max().item() <= tol * z.abs().max().item()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("log2n", list(range(8, 19)) + [20])
def test_every_size_against_a_64_bit_transform(dtype, log2n):
    """One-block, four-step (every line length) and radix-pass transforms of the stored-filter
    matched filter; an odd number of references."""
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n, nref = 1 << log2n, 3
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    g = torch.Generator(device="cuda")
    g.manual_seed(log2n)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).to(rf.rdtype)
    f = torch.randn((nref, n // 2 + 1, 2), dtype=torch.float64, device="cuda", generator=g)
    filt = torch.view_as_complex(f).to(rf.cdtype)
    z = rf.mf_filtered(x, filt)
    full = torch.zeros((nref, n), dtype=torch.complex128, device="cuda")
    full[:, : n // 2 + 1] = torch.fft.rfft(x.double()) * filt.to(torch.complex128)
    want = torch.fft.ifft(full) * n
    tol = 1e-12 if dtype == "f64" else 2e-6
    assert (z - want).abs().max().item() <= tol * want.abs().max().item()


@pytest.mark.parametrize("log2n", [14, 15, 16])
@pytest.mark.parametrize("nref", [1, 19, 20, 40])
def test_clusters_and_the_forms_beyond_them(log2n, nref):
    """Few references run on clusters, more on the other forms: rows agree with a 64-bit transform on
    both sides of the line."""
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter, launch_count
    n = 1 << log2n
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, "f32")
    g = torch.Generator(device="cuda")
    g.manual_seed(nref)
    x = torch.randn(n, device="cuda", generator=g)
    filt = torch.view_as_complex(torch.randn((nref, n // 2 + 1, 2), device="cuda", generator=g))
    a = launch_count()
    z = rf.mf_filtered(x, filt)
    if nref * 8 <= torch.cuda.get_device_properties(0).multi_processor_count:
        assert launch_count() - a == 1
    full = torch.zeros((nref, n), dtype=torch.complex128, device="cuda")
    full[:, : n // 2 + 1] = torch.fft.rfft(x.double()) * filt.to(torch.complex128)
    want = torch.fft.ifft(full) * n
    assert (z - want).abs().max().item() <= 2e-6 * want.abs().max().item()


def test_output_over_the_inputs():
    """An output that overlaps the data or the filters gives the same rows."""
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n, nref = 1 << 14, 5
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, "f32")
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    x = torch.randn(n, device="cuda", generator=g)
    filt = torch.view_as_complex(torch.randn((nref, n // 2 + 1, 2), device="cuda", generator=g))
    want = rf.mf_filtered(x, filt)
    buf = torch.zeros(nref * n * 2, device="cuda")
    for at in (0, 2 * n):                             # the data inside the output rows
        buf[at:at + n] = x
        z = rf.mf_filtered(buf[at:at + n], filt, z_out=torch.view_as_complex(buf.view(-1, 2)).view(nref, n))
        assert (z - want).abs().max().item() <= 4e-6 * want.abs().max().item()
    flat = torch.zeros(nref * n, dtype=torch.complex64, device="cuda")
    flat[: filt.numel()] = filt.flatten()             # the filters inside the output rows
    z = rf.mf_filtered(x, flat[: filt.numel()].view(nref, -1), z_out=flat.view(nref, n))
    assert (z - want).abs().max().item() <= 4e-6 * want.abs().max().item()
