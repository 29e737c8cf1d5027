"""FP64 overlap-save (AUTO on FP64 grids) against the FP64 direct sum: lengths around the partition
sizes, negative and wrapping first lags, real-form taps, windows from a few samples to the segment,
the series form, independent streams and stream capture.  Both sums are FP64: 1e-12 of max|z|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return pytest.importorskip("torch")


def _case(torch, n, lens, real=False, seed=0):
    from paper_2511_12894_gb300 import RatioFilter
    rf = RatioFilter(n, 1024.0, 40.0, 459.0, 2, "f64")
    rng = np.random.default_rng(seed)
    z = torch.tensor(rng.standard_normal(n) + 1j * rng.standard_normal(n), device="cuda")
    lag0 = rng.integers(-n // 2, n // 2, len(lens))
    total = int(sum(lens))
    taps = rng.standard_normal(total) if real else rng.standard_normal(total) + 1j * rng.standard_normal(total)
    return rf, z, rf.kernels_import(lag0, lens, taps, real=real)


def _route(rf_call):
    from paper_2511_12894_gb300 import launch_count
    a = launch_count()
    out = rf_call()
    return out, launch_count() - a


@pytest.mark.parametrize("real", [False, True])
@pytest.mark.parametrize("n,lens", [(1 << 10, [700, 1024, 333]), (1 << 12, [1, 511, 512, 513, 4096]),
                                    (1 << 13, [1023, 1024, 1025, 2049, 0]), (1 << 15, [930, 12000, 40])])
def test_matches_the_direct_sum(torch, n, lens, real):
    rf, z, kern = _case(torch, n, lens, real, seed=n)
    zd = rf.reconstruct(z, kern, "direct")
    zo = rf.reconstruct(z, kern)                      # prepares
    zo, used = _route(lambda: rf.reconstruct(z, kern))
    assert used == 2, "the overlap-save form should have been chosen"
    scale = zd.abs().max().item()
    assert (zo - zd).abs().max().item() <= 1e-12 * scale
    for W in (5, 100, 1000, 1024, n // 2 + 3, n):
        Pd, Ad = rf.reconstruct_winmax(z, kern, W, "direct")
        (Po, Ao), used = _route(lambda: rf.reconstruct_winmax(z, kern, W))
        assert used == 3
        assert torch.equal(Ao, Ad)
        assert (Po - Pd).abs().max().item() <= 1e-6 * Pd.abs().max().item()   # FP32 outputs


def test_batched_groups_and_short_kernels(torch):
    n = 1 << 14
    rf, z, kern = _case(torch, n, [800, 900, 1000])
    z2 = torch.flip(z, [0]).contiguous()
    P, A = rf.reconstruct_batched([z, z2], [kern, kern], 1024)
    for g, zg in enumerate((z, z2)):
        Pd, Ad = rf.reconstruct_winmax(zg, kern, 1024, "direct")
        assert torch.equal(A[3 * g:3 * g + 3], Ad)
        assert torch.allclose(P[3 * g:3 * g + 3], Pd, rtol=1e-6, atol=0)
    rf2, zs, short = _case(torch, n, [1, 2, 3])
    _, used = _route(lambda: rf2.reconstruct(zs, short))
    assert used == 1, "a few taps: the direct sum"


def test_streams_are_independent_and_capture_works(torch):
    n, W = 1 << 14, 512
    rf, z, kern = _case(torch, n, [900, 901, 902, 903])
    z2 = torch.flip(z, [0]).contiguous()
    # capture before the set is prepared: the direct sum, no allocation
    out = torch.empty((4, n), dtype=torch.complex128, device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        rf.reconstruct(z, kern, out=out)
    g.replay()
    torch.cuda.synchronize()
    want = rf.reconstruct(z, kern, "direct")
    assert torch.equal(out, want)
    # prepared now: captured and on two streams at once
    want1, want2 = rf.reconstruct_winmax(z, kern, W), rf.reconstruct_winmax(z2, kern, W)
    torch.cuda.synchronize()
    mo = torch.empty_like(want1[0])
    ao = torch.empty_like(want1[1])
    g2 = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g2):
        rf.reconstruct_winmax(z, kern, W, max_out=mo, arg_out=ao)
    g2.replay()
    torch.cuda.synchronize()
    assert torch.equal(mo, want1[0]) and torch.equal(ao, want1[1])
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    o1 = [torch.empty_like(t) for t in want1]
    o2 = [torch.empty_like(t) for t in want2]
    torch.cuda.synchronize()
    for _ in range(10):
        rf.reconstruct_winmax(z, kern, W, max_out=o1[0], arg_out=o1[1], stream=s1)
        rf.reconstruct_winmax(z2, kern, W, max_out=o2[0], arg_out=o2[1], stream=s2)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(o1, want1))
    assert all(torch.equal(a, b) for a, b in zip(o2, want2))


def test_first_calls_of_several_threads(torch):
    """One kernel set, a context per thread: the first calls at once, one of them while another
    stream is captured."""
    import threading
    from paper_2511_12894_gb300 import RatioFilter
    n, W = 1 << 14, 512
    rf, z, kern = _case(torch, n, [900, 901, 902, 903])
    want, wanta = rf.reconstruct_winmax(z, kern, W, "direct")
    rfs = [RatioFilter(n, 1024.0, 40.0, 459.0, 2, "f64") for _ in range(4)]
    outs = [(torch.empty_like(want), torch.empty_like(wanta)) for _ in rfs]
    streams = [torch.cuda.Stream() for _ in rfs]
    start = threading.Barrier(len(rfs))
    errors = []

    def work(r, s, o):
        try:
            start.wait()
            r.reconstruct_winmax(z, kern, W, max_out=o[0], arg_out=o[1], stream=s)
        except Exception as e:
            errors.append(e)

    buf = torch.zeros(16, device="cuda")
    threads = [threading.Thread(target=work, args=a) for a in zip(rfs, streams, outs)]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="global"):
        buf.add_(1.0)
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        buf.add_(1.0)
    assert not errors
    g.replay()
    torch.cuda.synchronize()
    assert buf.min().item() == buf.max().item() == 2.0
    for p, a in outs:
        assert torch.equal(a, wanta)
        assert (p - want).abs().max().item() <= 1e-6 * want.max().item()   # FP32 outputs
