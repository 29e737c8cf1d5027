"""Device memory of a context: the header's figures, from which callers size what they keep free."""
import os
import re

import pytest

pytestmark = pytest.mark.gpu

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include", "rf.h")


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_context_bytes(dtype):
    torch = pytest.importorskip("torch")
    from paper_2511_12894_gb300 import RatioFilter
    text = " ".join(open(HEADER).read().split("rf_status rf_create(")[0].rsplit("/*", 1)[1].replace("*", " ").split())
    kind = "RF_" + dtype.upper()
    per_n = int(re.search(r"(\d+) n bytes for " + kind, text).group(1))
    batch = int(re.search(r"(\d+) MB \(" + kind + r"\)", text).group(1)) << 20
    n = 1 << 22
    RatioFilter(1 << 12, 2048.0, 20.0, 971.0, 7, dtype).close()   # the library's own first-use memory
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    rf = RatioFilter(n, 2048.0, 20.0, 971.0, 7, dtype)
    used = before - torch.cuda.mem_get_info()[0]
    rf.close()
    assert 0.98 * per_n * n <= used <= per_n * n + batch + (32 << 20), (used / n, per_n)
