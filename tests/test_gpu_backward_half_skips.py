"""Pass 2 of the backward leaves out the 64-row halves of a query tile no row of which
attends a key pair.  Scores that send even query blocks to even blocks and odd ones to
odd ones make such halves; that there are some is read off the kept lists.  All five
gradients against the oracle: several heads, the outer gate position (its own marks of
attending rows), and packed sequences (their own map from tiles to slots)."""
import numpy as np
import pytest
import torch

from oracle import backward_oracle as BO
from paper_2609_13141_gb300 import sas, synth
from tests import parity as P
from tests.test_gpu_backward import _delta_bound
from tests.test_gpu_backward_varlen import _check, _packed, _run

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _apart(N, C, seed):
    """Scores [N, C]: even query blocks keep block pairs 4j, odd ones pairs 4j + 2."""
    s = synth.scores(1, 1, N, C, seed=seed, regime="R1")[0, 0]
    q, m = torch.arange(N)[:, None] // 64, torch.arange(C)[None] // 2
    return (s + 10.0 * ((q + m) % 2 == 0)).to(torch.float32)


def _half_skips(kept, n):
    """(tile, key pair) products of one head with exactly one half that attends the pair."""
    found = 0
    for t in range(-(-n // 128)):
        pairs = []
        for r0 in (128 * t, 128 * t + 64):
            k = kept[r0:min(r0 + 64, n)]
            pairs.append({int(m) // 2 for m in k[k >= 0].ravel()} - {t})
        found += len(pairs[0] ^ pairs[1])
    return found


@pytest.mark.parametrize("pos", [sas.SAS_GATE_INNER, sas.SAS_GATE_OUTER])
@pytest.mark.parametrize("B,H,N,topk", [(1, 3, 1000, 2), (2, 2, 832, 3)])
def test_heads_and_gate_positions(pos, B, H, N, topk):
    d, C = 128, -(-N // 64)
    Q, K, V = synth.qkv(B, H, N, d, seed=N + topk)
    S = torch.stack([_apart(N, C, 7 * k + N) for k in range(B * H)]).view(B, H, N, C).contiguous()
    dO = synth.normal((B, H, N, d), N + 1).to(torch.bfloat16)
    layer = sas.SasLayer(B, H, N, d, topk, gate_pos=pos)
    dev = [t.to(DEV) for t in (Q, K, V, S, dO)]
    O, LSE, si, sl = layer.attention(*dev[:3], scores=dev[3])
    dQ, dK, dV, dl, ds = layer.attention_bwd(*dev[:3], O, LSE, dev[4], scores=dev[3], sel_idx=si, sel_logg=sl,
                                             want_ds=True)
    torch.cuda.synchronize()
    assert sas.sas_get_device_status(layer.h) == 0
    layer.close()
    f = P.f64
    for b in range(B):
        for h in range(H):
            assert _half_skips(si[b, h].cpu().numpy(), N) > 0
            q, k, v, s, do = (f(t[b, h]) for t in (Q, K, V, S, dO))
            ref = BO.sas_attention_bwd_head(q, k, v, s, do, 64, topk, pos=pos)
            extra = P.grad_extra(q, k, v, s, do, f(O[b, h].cpu()), 64, topk, sas.SAS_MODE_TRAIN_SOFT, pos=pos)
            for name, got in (("dQ", dQ), ("dK", dK), ("dV", dV)):
                P.compare_o(f(got[b, h].cpu()), ref[name], f"{name}[{b},{h}]", extra[name])
            tol = _delta_bound(O[b, h].cpu(), dO[b, h])[:, None]
            assert np.all(np.abs(dl[b, h].cpu().numpy() - ref["dlogg"]) <= tol), "dlogg"
            assert np.all(np.abs(ds[b, h].cpu().numpy() - ref["ds"]) <= 2 * tol), "ds"


@pytest.mark.parametrize("lens,cap", [([1000, 1, 64, 700, 129], 2000), ([513, 832], 1345)])
def test_packed_heads(lens, cap):
    H, topk = 2, 3
    Q, K, V, S, dO, cu = _packed(lens, cap, H, H, max(lens), seed=cap)
    for h in range(H):
        for a, b in zip(cu[:-1].tolist(), cu[1:].tolist()):
            S[h, a:b] = _apart(b - a, S.shape[-1], cap + h)
    g = _run(lens, cap, H, H, topk, sas.SAS_MODE_TRAIN_SOFT, max(lens), Q, K, V, S, dO, cu)
    assert g["status"] == 0
    _check(g, Q, K, V, S, dO, cu.numpy(), topk, sas.SAS_MODE_TRAIN_SOFT)
    layer = sas.SasLayer(1, H, cap, 128, topk, max_seqs=len(lens), max_seqlen=max(lens))
    _, _, si, _ = layer.attention_varlen(cu.to(DEV), *(t.to(DEV).contiguous() for t in (Q, K, V, S)))
    si = si.cpu().numpy()
    layer.close()
    at = cu.tolist()
    assert _half_skips(si[0, at[0]:at[1]], lens[0]) > 0
