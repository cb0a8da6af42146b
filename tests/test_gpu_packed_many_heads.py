"""Packed sequences with more heads than a grid's second dimension holds: every head's
rows are computed and every head's spare rows filled, the same bits as a few heads at
a time."""
import pytest
import torch

from paper_2609_13141_gb300 import sas

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("H", [65535, 65536, 65539])
def test_more_heads_than_grid_y(H):
    N, d, topk, some = 68, 64, 1, 4
    g = torch.Generator(device=DEV).manual_seed(H)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    Q, K, V = (rnd(H, N, d).bfloat16() for _ in range(3))
    S = rnd(H, N, -(-N // 64))
    cu = torch.tensor([0, 66], dtype=torch.int32, device=DEV)
    layer = sas.SasLayer(1, H, N, d, topk, max_seqs=1)
    poison = torch.full((H * N * d * 2,), 255, dtype=torch.uint8, device=DEV)   # O's block, as a caller may find it
    del poison
    got = layer.attention_varlen(cu, Q, K, V, S, sel_fill=-7)
    torch.cuda.synchronize()
    assert sas.sas_get_device_status(layer.h) == 0
    layer.close()
    few = sas.SasLayer(1, some, N, d, topk, max_seqs=1)
    for h0 in (0, H // 2, H - some):
        part = [t[h0:h0 + some].contiguous() for t in (Q, K, V, S)]
        want = few.attention_varlen(cu, *part, sel_fill=-7)
        for a, b in zip(got, want):
            assert torch.equal(a[h0:h0 + some].view(torch.int16 if a.element_size() == 2 else torch.int32),
                               b.view(torch.int16 if b.element_size() == 2 else torch.int32))
    few.close()
    O, LSE, si, sl = got
    for t, fill in ((O, 0), (LSE, 0), (si, -7), (sl, 0)):
        assert bool((t[:, 66:] == fill).all())
