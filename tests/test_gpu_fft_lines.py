"""Stored-filter matched filters at the edges of the transforms' rules: FP64 sizes of both forms up to
the largest grid, and launches of the inverse with a ragged last one."""
import pytest

pytestmark = pytest.mark.gpu


def _run(torch, n, nref, dtype, rows):
    """Rows of a call against the call with that row alone and a 64-bit transform."""
    from paper_2511_12894_gb300 import RatioFilter
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    g = torch.Generator(device="cuda")
    g.manual_seed(nref)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).to(rf.rdtype)
    filt = torch.view_as_complex(torch.randn((nref, n // 2 + 1, 2), device="cuda", generator=g).to(rf.rdtype))
    z = rf.mf_filtered(x, filt)
    X = torch.fft.rfft(x.double())
    tol = 1e-12 if dtype == "f64" else 2e-6
    for r in rows:
        assert torch.equal(rf.mf_filtered(x, filt[r:r + 1])[0], z[r]), r
        full = torch.zeros(n, dtype=torch.complex128, device="cuda")
        full[: n // 2 + 1] = X * filt[r].to(torch.complex128)
        want = torch.fft.ifft(full) * n
        assert (z[r] - want).abs().max().item() <= tol * want.abs().max().item(), r
    rf.close()


@pytest.mark.parametrize("log2n", [18, 19, 20, 21, 22, 24])
def test_fp64_sizes(log2n):
    """Four-step data transforms up to 2^21 samples and inverses up to 2^18, radix passes beyond."""
    torch = pytest.importorskip("torch")
    _run(torch, 1 << log2n, 2, "f64", (0, 1))


@pytest.mark.parametrize("log2n,nref,rows", [(20, 35, (0, 31, 32, 34)), (23, 5, (3, 4)), (24, 3, (1, 2))])
def test_ragged_last_launch(log2n, nref, rows):
    """The inverses of 2^25 values share a launch pair (32 rows of 2^20, 4 of 2^23, 2 of 2^24): calls of a
    few more rows end with a short launch."""
    torch = pytest.importorskip("torch")
    _run(torch, 1 << log2n, nref, "f32", rows)
