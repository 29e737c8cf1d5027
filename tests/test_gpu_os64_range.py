"""FP64 overlap-save (AUTO on FP64 grids) on series whose samples are not finite, or loud beside quiet:
as the direct sum, a sample reaches the outputs of the kernel's own length and no others, and quiet
outputs keep their own 1e-12."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N, W = 1 << 15, 256


def _case(torch, real, lens=(200, 1500, 900)):
    from paper_2511_12894_gb300 import RatioFilter, launch_count
    rf = RatioFilter(N, 1024.0, 40.0, 459.0, 2, "f64")
    rng = np.random.default_rng(4)
    z = torch.tensor(rng.standard_normal(N) + 1j * rng.standard_normal(N), device="cuda")
    taps = rng.standard_normal(sum(lens)) + (0 if real else 1j * rng.standard_normal(sum(lens)))
    kern = rf.kernels_import([-300, 17, 9000], list(lens), taps, real=real)
    rf.reconstruct(z, kern)                           # prepares
    a = launch_count()
    rf.reconstruct(z, kern)
    assert launch_count() - a == 2, "the overlap-save form should have been chosen"
    return rf, z, kern


def _both(torch, rf, z, kern):
    zd, zo = rf.reconstruct(z, kern, "direct"), rf.reconstruct(z, kern)
    Pd, Ad = rf.reconstruct_winmax(z, kern, W, "direct")
    Po, Ao = rf.reconstruct_winmax(z, kern, W)
    return zd, zo, Pd, Ad, Po, Ao


def _reached(torch, kern, at):
    """The outputs that hold a sample of `at`: i = at + m0 + l (mod N), 0 <= l < L (Eq. 8)."""
    mask = torch.zeros((kern.k, N), dtype=torch.bool, device="cuda")
    for j in range(kern.k):
        for a in at:
            mask[j, (a + int(kern.lag0[j]) + torch.arange(int(kern.length[j]), device="cuda")) % N] = True
    return mask


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 1e300])
def test_samples_that_are_not_finite(real, bad):
    """Checked against the definition: the direct sum pads its kernels with zero taps, over which such a
    sample reaches a little further."""
    torch = pytest.importorskip("torch")
    rf, z, kern = _case(torch, real)
    at = [5, 6, 20000]
    z[at] = complex(bad, 1.0)
    zd, zo, Pd, Ad, Po, Ao = _both(torch, rf, z, kern)
    hit = _reached(torch, kern, at)
    finite = torch.view_as_real(zo).isfinite()
    assert torch.equal(finite[..., 0], ~hit if not np.isfinite(bad) else torch.ones_like(hit))
    assert torch.equal(finite[..., 1], ~hit if not np.isfinite(bad) and not real else torch.ones_like(hit))
    same = torch.view_as_real(zd).isfinite().all(-1) & ~hit
    assert same.float().mean().item() > 0.5
    assert (zo - zd)[same].abs().max().item() <= 1e-11
    m2 = zo.real ** 2 + zo.imag ** 2
    m2 = torch.where(m2.isnan(), -torch.ones_like(m2), m2).view(kern.k, -1, W)
    best = m2.amax(-1)
    assert torch.equal(Ao, torch.where(best < 0, 0, m2.argmax(-1) + W * torch.arange(N // W, device="cuda")).int())
    assert torch.allclose(Po.double(), best, rtol=1e-6, atol=0.0)


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("loud", [1e5, 1e12])
def test_quiet_samples_beside_loud_ones(real, loud):
    torch = pytest.importorskip("torch")
    rf, z, kern = _case(torch, real)
    z[7000:7100] *= loud
    zd, zo, _, _, _, _ = _both(torch, rf, z, kern)
    # every run of 64 outputs to 1e-11 of its own largest value
    err = (zo - zd).abs().view(3, -1, 64).amax(-1)
    assert (err <= 1e-11 * zd.abs().view(3, -1, 64).amax(-1)).all()


@pytest.mark.parametrize("real", [False, True])
def test_silence(real):
    """Outputs that see only zeros are zero, and their windows' first sample is the peak."""
    torch = pytest.importorskip("torch")
    rf, z, kern = _case(torch, real)
    z[12000:18000] = 0
    zd, zo, Pd, Ad, Po, Ao = _both(torch, rf, z, kern)
    assert torch.equal(zo == 0, zd == 0) and bool((zd == 0).any())
    assert torch.equal(Ao, Ad) and torch.allclose(Po, Pd, rtol=1e-6, atol=0.0)
