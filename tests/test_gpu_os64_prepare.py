"""Preparation of FP64 kernel sets for the overlap-save form of AUTO."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _set(torch, n, lens, seed=0):
    from paper_2511_12894_gb300 import RatioFilter
    rf = RatioFilter(n, 1024.0, 40.0, 459.0, 2, "f64")
    rng = np.random.default_rng(seed)
    z = torch.tensor(rng.standard_normal(n) + 1j * rng.standard_normal(n), device="cuda")
    taps = rng.standard_normal(sum(lens)) + 1j * rng.standard_normal(sum(lens))
    return rf, z, rf.kernels_import(np.zeros(len(lens), np.int32), lens, taps)


def _launches(call):
    from paper_2511_12894_gb300 import launch_count
    a = launch_count()
    call()
    return launch_count() - a


def test_a_shortage_of_memory_passes():
    """A first call without room for the spectra (67 MB, with 32 MB left) runs the direct sum; once there is room,
    the next one prepares."""
    torch = pytest.importorskip("torch")
    n = 1 << 15
    rf, z, kern = _set(torch, n, [n] * 64)
    call = lambda: rf.reconstruct_winmax(z, kern, n, max_out=mo, arg_out=ao)
    mo = torch.empty((64, 1), dtype=torch.float32, device="cuda")
    ao = torch.empty((64, 1), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (32 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert _launches(call) == 1
        torch.cuda.synchronize()
        want, arg = mo.clone(), ao.clone()
    finally:
        del hog
        torch.cuda.empty_cache()
    call()
    assert _launches(call) == 3
    assert torch.equal(ao, arg) and torch.allclose(mo, want, rtol=1e-6, atol=0.0)


def test_prepared_ahead_of_the_first_call():
    """A set prepared by the caller: its first AUTO call neither prepares nor synchronises, so it can be captured in
    the overlap-save form; other layouts are refused as before."""
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RFError
    n, W = 1 << 14, 512
    rf, z, kern = _set(torch, n, [900, 901, 902, 903])
    with pytest.raises(RFError):
        kern.prepare(4096, 1024)
    kern.prepare()
    want, arg = rf.reconstruct_winmax(z, kern, W, "direct")
    mo, ao = torch.empty_like(want), torch.empty_like(arg)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        used = _launches(lambda: rf.reconstruct_winmax(z, kern, W, max_out=mo, arg_out=ao))
    assert used == 3
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(ao, arg) and torch.allclose(mo, want, rtol=1e-6, atol=0.0)
    rf2, z2, short = _set(torch, n, [1, 2, 3])
    short.prepare()                                   # the direct sum is cheaper: nothing to prepare
    assert _launches(lambda: rf2.reconstruct(z2, short)) == 1
