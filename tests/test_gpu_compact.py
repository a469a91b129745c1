"""The compaction against a boolean mask: tile edges, ragged ends, tiles of every
size class (one tile per block up to the largest), all live, none live."""
import numpy as np
import pytest

from paper_1807_04733_gb300 import pic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("live", [0.0, 0.5, 0.97, 1.0])
@pytest.mark.parametrize("n", [1, 31, 2047, 2048, 2049, 300_001, 2_490_369, 7_000_003, 30_000_001])
def test_compact_equals_mask(n, live):
    g = torch.Generator(device="cuda").manual_seed(n)
    z = torch.rand(n + 3, device="cuda", generator=g)
    mu = torch.rand(n + 3, device="cuda", generator=g)
    i = torch.arange(n + 3, device="cuda", dtype=torch.int32)
    p = torch.randint(1, 256, (n + 3,), device="cuda", generator=g, dtype=torch.int32) | (5 << 13)
    p[torch.rand(n + 3, device="cuda", generator=g) >= live] &= ~0xFF
    out = [torch.zeros_like(x) for x in (z, mu, i, p)]
    k = pic.pic_compact_static(z.data_ptr(), mu.data_ptr(), i.data_ptr(), p.data_ptr(), n,
                               *[x.data_ptr() for x in out], torch.cuda.current_stream().cuda_stream)
    m = (p[:n] & 0xFF) != 0
    assert k == int(m.sum())
    for a, b in zip((z, mu, i, p), out):
        assert torch.equal(a[:n][m], b[:k])
        assert not b[k:].any()                    # nothing written past the live slots
