"""What the bits of a result may depend on.  An MLP row: the sizes of the call, not the
other rows' values or the row's place in its tile.  A decode output: neither the other
sequences' tokens and lengths nor how many there are.  Repeated calls give the same bits."""
import pytest
import torch

from paper_2609_13141_gb300 import sas, synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("T,D,F", [(64, 1024, 4096), (200, 2560, 9728), (777, 768, 3072)])
def test_mlp_rows_do_not_see_each_other(T, D, F):
    X, W1, W2, _, _ = (None if t is None else t.to(DEV) for t in synth.mlp(T, D, F, seed=T))
    layer = sas.SasLayer(1, 1, 64, 64, 0)
    Y = layer.mlp(X, W1, W2)
    perm = torch.randperm(T, generator=torch.Generator().manual_seed(1)).to(DEV)
    assert torch.equal(layer.mlp(X[perm].contiguous(), W1, W2), Y[perm])
    Z = X.clone()
    Z[1:] = 0
    assert torch.equal(layer.mlp(Z, W1, W2)[0], Y[0])
    for _ in range(10):
        assert torch.equal(layer.mlp(X, W1, W2), Y)
    layer.close()


@pytest.mark.parametrize("B,Hq,Hkv,topk", [(1, 32, 8, 32), (8, 32, 8, 32), (40, 16, 8, 16)])
def test_decode_sequences_do_not_see_each_other(B, Hq, Hkv, topk):
    d, n, max_blocks = 128, 64 * 70 + 5, 72
    pages = max_blocks * 2
    g = torch.Generator(device=DEV).manual_seed(B)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEV).bfloat16()  # noqa: E731
    K, V, q = rnd(pages, Hkv, 64, d), rnd(pages, Hkv, 64, d), rnd(B, Hq, d)
    Wq, Wk = (w.to(DEV) for w in synth.decode_selector_weights(Hkv, Hq // Hkv, d, d, seed=2))
    # sequence 0 has pages of its own; the others share the rest
    table = torch.randint(max_blocks, pages, (B, max_blocks), generator=g, device=DEV, dtype=torch.int32)
    table[0] = torch.arange(max_blocks, device=DEV)
    dec = sas.SasDecoder(B, Hq, Hkv, d, topk, max_blocks, pages, d_sel=d)

    def step(lens, q):
        lens = torch.tensor(lens, dtype=torch.int32, device=DEV)
        ks = torch.zeros(B, Hkv, max_blocks, d, device=DEV, dtype=torch.bfloat16)
        dec.summarize(K, table, lens, Wk, ks)
        out = dec.step(q, K, V, table, lens, None, None, Wq, Wk, ks)
        torch.cuda.synchronize()
        return [t.clone() for t in out]

    a = step([n] * B, q)
    q2 = q.clone()
    q2[1:] = rnd(B, Hq, d)[1:]
    b = step([n] + [1 + 113 * k % (64 * max_blocks) for k in range(1, B)], q2)
    for x, y in zip(a, b):
        assert torch.equal(x[0], y[0])
    for _ in range(5):
        assert all(torch.equal(x, y) for x, y in zip(step([n] * B, q), a))
    assert sas.sas_decode_get_device_status(dec.h) == 0
    dec.close()


@pytest.mark.parametrize("Hq,Hkv,topk,d,dense", [
    (32, 8, 32, 128, False), (8, 8, 64, 128, False), (64, 8, 48, 128, False), (16, 8, 7, 128, False),
    (4, 1, 33, 128, False), (32, 8, 32, 64, False), (32, 8, 0, 128, True),
])
def test_decode_output_is_the_same_in_any_batch(Hq, Hkv, topk, d, dense):
    # 1 to 1024 groups: clusters of up to 16 CTAs down to single ones; sequences that fill
    # their lists and short ones
    lens = [64 * 70 + 5, 64 * 40 + 64, 64 * 5 + 1, 17]
    max_blocks, Bmax = 72, 128
    pages = max_blocks * len(lens)
    g = torch.Generator(device=DEV).manual_seed(topk)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEV).bfloat16()  # noqa: E731
    K, V, q = rnd(pages, Hkv, 64, d), rnd(pages, Hkv, 64, d), rnd(len(lens), Hq, d)
    Wq, Wk = (w.to(DEV) for w in synth.decode_selector_weights(Hkv, Hq // Hkv, d, d, seed=3))
    table = torch.arange(pages, device=DEV, dtype=torch.int32).view(len(lens), max_blocks)
    first = None
    for B in (4, 8, 20, 40, Bmax):
        rep = [t.repeat(B // 4, *([1] * (t.dim() - 1))).contiguous() for t in (q, table)]
        n = torch.tensor(lens * (B // 4), dtype=torch.int32, device=DEV)
        dec = sas.SasDecoder(B, Hq, Hkv, d, topk, max_blocks, pages, d_sel=0 if dense else d, dense=dense)
        if dense:
            out = dec.step(rep[0], K, V, rep[1], n)
        else:
            ks = torch.zeros(B, Hkv, max_blocks, d, device=DEV, dtype=torch.bfloat16)
            dec.summarize(K, rep[1], n, Wk, ks)
            out = dec.step(rep[0], K, V, rep[1], n, None, None, Wq, Wk, ks)
        torch.cuda.synchronize()
        assert sas.sas_decode_get_device_status(dec.h) == 0
        dec.close()
        out = [t for t in out if t is not None]
        if first is None:
            first = out
        for x, y in zip(out, first):
            assert torch.equal(x[:4], y[:4]) and torch.equal(x[-4:], y[:4])
