"""Packed outputs: rows past the last sequence are filled after the kernels, in memory
that held NaN before.  Every output must equal, bit for bit, the one the kernels leave
in tensors filled beforehand: no row or entry may be left as it was."""
import pytest
import torch

from paper_2609_13141_gb300 import sas, synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _poison(*like):
    """Freed blocks of the sizes the next outputs ask for, full of NaN (all ones)."""
    keep = [torch.full((t.numel() * t.element_size(),), 255, dtype=torch.uint8, device=DEV) for t in like]
    torch.cuda.synchronize()
    del keep


def _same(a, b):
    return torch.equal(a.contiguous().view(torch.uint8), b.contiguous().view(torch.uint8))


@pytest.mark.parametrize("lens,N,H,Hkv,topk,mode,learned", [
    ((300, 65, 1, 0, 64), 430, 2, 2, 3, sas.SAS_MODE_TRAIN_SOFT, False),     # no spare row
    ((300, 65, 1, 0, 64), 431, 4, 2, 3, sas.SAS_MODE_TRAIN_SOFT, False),     # one
    ((700, 129), 4000, 4, 1, 5, sas.SAS_MODE_TRAIN_SOFT, False),             # most of them
    ((700, 129), 1001, 4, 2, 4, sas.SAS_MODE_INFER_HARD, True),
    ((130, 50), 300, 2, 2, 0, sas.SAS_MODE_TRAIN_SOFT, False),               # nothing kept
    ((), 300, 2, 1, 2, sas.SAS_MODE_TRAIN_SOFT, False),                      # bad offsets: all rows are spare
])
def test_equal_to_prefilled_outputs(lens, N, H, Hkv, topk, mode, learned):
    d, C = 128, -(-N // 64)
    g = torch.Generator(device=DEV).manual_seed(N)
    rnd = lambda h, w: torch.randn(h, N, w, generator=g, device=DEV)  # noqa: E731
    Q, dO = rnd(H, d).bfloat16(), rnd(H, d).bfloat16()
    K, V, S = rnd(Hkv, d).bfloat16(), rnd(Hkv, d).bfloat16(), rnd(Hkv, C)
    sel = sas.SAS_SEL_MEANPOOL_PROJ if learned else sas.SAS_SEL_SCORES_GIVEN
    Wq = Wk = None
    if learned:
        Wq, Wk = (w.to(DEV) for w in synth.decode_selector_weights(Hkv, H // Hkv, d, d, seed=1, exact=True))
        S = None
    offs = [0]
    for n in lens:
        offs.append(offs[-1] + n)
    cu = torch.tensor(offs if lens else [0, 200, 100], dtype=torch.int32, device=DEV)
    layer = sas.SasLayer(1, H, N, d, topk, mode=mode, selector=sel, d_sel=d if learned else 0, Hkv=Hkv, max_seqs=8)
    k = max(topk, 1)
    O = torch.zeros_like(Q)
    L = torch.zeros(H, N, device=DEV)
    si = torch.full((Hkv, N, k), -7, device=DEV, dtype=torch.int32)
    sl = torch.zeros(Hkv, N, k, device=DEV)
    sas.sas_attention_fwd_varlen(layer.h, cu, Q, K, V, S, O, L, si, sl, Wq=Wq, Wk=Wk)
    _poison(O, L, si, sl)
    got = layer.attention_varlen(cu, Q, K, V, S, sel_fill=-7, Wq=Wq, Wk=Wk)
    torch.cuda.synchronize()
    for a, b in zip(got, (O, L, si, sl)):
        assert _same(a, b)
    assert sas.sas_get_device_status(layer.h) == (0 if lens else sas.SAS_ERR_INVALID_ARG)
    if lens and not learned:
        zero = [torch.zeros_like(t) for t in (Q, K, V)] + [torch.zeros(Hkv, N, k, device=DEV), torch.zeros_like(S)]
        sas.sas_attention_bwd(layer.h, Q, K, V, O, L, dO, *zero[:3], S, si, sl, zero[3], zero[4])
        last = int(cu[-1])
        zero = [torch.cat([t[:, :last], torch.zeros_like(t[:, last:])], 1) for t in zero]
        _poison(*zero)
        got = layer.attention_bwd_varlen(Q, K, V, O, L, dO, scores=S, sel_idx=si, sel_logg=sl, want_ds=True)
        torch.cuda.synchronize()
        for a, b in zip(got, zero):
            assert _same(a, b)
    layer.close()


def test_tails_refuse_bad_tensors():
    layer = sas.SasLayer(1, 2, 256, 128, 2, max_seqs=2)
    x = torch.zeros(2, 256, 2, device=DEV)
    for tails in ([], [(x, 2, 6, 0)], [(x, 0, 8, 0)], [(x, 2, 8, 0)] * 9):
        with pytest.raises(sas.SasError):
            sas.sas_fill_varlen_tails(layer.h, tails)
    layer.close()
    layer = sas.SasLayer(1, 2, 256, 128, 2)
    with pytest.raises(sas.SasError):
        sas.sas_fill_varlen_tails(layer.h, [(x, 2, 8, 0)])
    layer.close()
