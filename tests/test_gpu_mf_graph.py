"""A captured matched filter stays valid when a later call needs a larger temporary."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2n,few,many,dtype", [(17, 1, 7, "f32"), (22, 1, 8, "f32"), (14, 1, 5, "f64")])
def test_graph_replayed_after_a_larger_call(log2n, few, many, dtype):
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    n = 1 << log2n
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    g = torch.Generator(device="cuda")
    g.manual_seed(log2n)
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).to(rf.rdtype)
    filt = torch.view_as_complex(torch.randn((many, n // 2 + 1, 2), device="cuda", generator=g).to(rf.rdtype))
    one = filt[:few].contiguous()
    z = torch.empty((few, n), dtype=rf.cdtype, device="cuda")
    want = rf.mf_filtered(x, one)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        rf.mf_filtered(x, one, z_out=z)
    rf.mf_filtered(x, filt)
    held = torch.full((16, n), 7.0, dtype=rf.cdtype, device="cuda")   # whatever was given back is reused
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(z, want) and bool((held == 7.0).all())
