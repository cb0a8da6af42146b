"""Pass 2 of the backward over the 64-row halves that attend a key pair: tiles
whose two query blocks keep different blocks, the same ones, or none; short
histories (every half kept), a last tile of one query block; against the oracle with the backward's tolerance."""
import pytest
import torch

from oracle import backward_oracle as BO
from paper_2609_13141_gb300 import sas, synth
from tests import parity as P

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _scores(N, C, pattern, seed):
    """Block-coherent scores: 'apart' sends even query blocks to even key blocks and odd ones to odd ones
    (one half of a tile per key block), 'same' gives both the same blocks, 'first' everyone block 0."""
    s = synth.scores(1, 1, N, C, seed=seed, regime="R1")[0, 0]
    q, m = torch.arange(N)[:, None] // 64, torch.arange(C)[None]
    if pattern == "apart":
        s = s + 10.0 * ((q + m) % 2 == 0)
    elif pattern == "same":
        s = s - 0.5 * m
    else:
        s = s + 20.0 * (m == 0)
    return s.to(torch.float32)


@pytest.mark.parametrize("pattern", ["apart", "same", "first"])
@pytest.mark.parametrize("N,topk", [(1000, 2), (832, 3), (129, 1), (64, 2), (513, 0)])
def test_halves_against_oracle(pattern, N, topk):
    d, C = 128, -(-N // 64)
    Q, K, V = synth.qkv(1, 1, N, d, seed=N)
    S = _scores(N, C, pattern, N + topk)[None, None].contiguous()
    dO = synth.normal((1, 1, N, d), N + 1).to(torch.bfloat16)
    layer = sas.SasLayer(1, 1, N, d, topk)
    dev = [t.to(DEV) for t in (Q, K, V, S, dO)]
    O, LSE, si, sl = layer.attention(*dev[:3], scores=dev[3])
    dQ, dK, dV, dl, ds = layer.attention_bwd(*dev[:3], O, LSE, dev[4], scores=dev[3], sel_idx=si, sel_logg=sl,
                                             want_ds=True)
    torch.cuda.synchronize()
    assert sas.sas_get_device_status(layer.h) == 0
    layer.close()
    f = P.f64
    q, k, v, s, do = (f(t[0, 0]) for t in (Q, K, V, S, dO))
    ref = BO.sas_attention_bwd_head(q, k, v, s, do, 64, topk)
    extra = P.grad_extra(q, k, v, s, do, f(O[0, 0].cpu()), 64, topk, sas.SAS_MODE_TRAIN_SOFT)
    for name, got in (("dQ", dQ), ("dK", dK), ("dV", dV)):
        P.compare_o(f(got[0, 0].cpu()), ref[name], name, extra[name])
