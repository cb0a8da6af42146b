"""The score gradient's row kernel: 16-byte words and single words, rows held in
registers (up to 128 and 384 blocks) and longer ones, ds from the returned dlogg
in 64 bits: ds_m = dlogg_m - g_m sum dlogg over the history, 0 past it."""
import pytest
import torch

from paper_2609_13141_gb300 import sas

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _inputs(N, K, shift):
    g = torch.Generator(device=DEV).manual_seed(N + K)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    C, H, d = -(-N // 64), 1, 128
    Q, Kk, V, dO = (rnd(1, H, N, d).bfloat16() for _ in range(4))
    flat = torch.zeros(H * N * C + 4, device=DEV)
    S = flat[shift:shift + H * N * C].view(1, H, N, C)   # shift words off a 16-byte boundary
    S.copy_(rnd(1, H, N, C))
    return Q, Kk, V, dO, S


def _run(N, K, shift):
    Q, Kk, V, dO, S = _inputs(N, K, shift)
    layer = sas.SasLayer(1, 1, N, 128, K)
    O, LSE, si, sl = layer.attention(Q, Kk, V, scores=S)
    out = layer.attention_bwd(Q, Kk, V, O, LSE, dO, scores=S, sel_idx=si, sel_logg=sl, want_ds=True)
    torch.cuda.synchronize()
    layer.close()
    return S, si, out[3], out[4]


# 1, 4, 5, 128, 129, 132, 384, 385, 388 blocks
@pytest.mark.parametrize("N", [60, 250, 319, 8192, 8250, 8400, 24576, 24600, 24800])
def test_against_dlogg(N):
    K = 6
    S, si, dlogg, ds = _run(N, K, 0)
    C = S.shape[-1]
    step = max(1, N // 200)
    rows = torch.tensor(sorted(set(range(0, N, step)) | set(range(max(0, N - 130), N))), device=DEV)
    hist = torch.arange(C, device=DEV)[None] < (rows // 64)[:, None]
    s = S[0, 0, rows].double().masked_fill(~hist, -float("inf"))
    idx, dl = si[0, 0, rows].long(), dlogg[0, 0, rows].double()
    dl = torch.where(idx >= 0, dl, 0.0)
    kept = torch.zeros(len(rows), C + 1, device=DEV, dtype=torch.float64)
    kept.scatter_(1, torch.where(idx >= 0, idx, C), dl)
    kept = kept[:, :C]
    gate = torch.where(hist, torch.softmax(s, -1), 0.0).nan_to_num(0.0)
    want = torch.where(hist, kept - gate * dl.sum(-1, keepdim=True), 0.0)
    got = ds[0, 0, rows].double()
    # fp32 sum, log-normaliser and exponential: below 1e-5 of the terms' sizes
    tol = 1e-5 * (kept.abs() + gate * dl.abs().sum(-1, keepdim=True)) + 1e-30
    assert torch.all((got - want).abs() <= tol)
    assert torch.all(got[~hist] == 0)


@pytest.mark.parametrize("N", [250, 8192, 24576, 24800])
def test_unaligned_scores_give_the_same_bits(N):
    a, b = _run(N, 5, 0), _run(N, 5, 1)
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2]) and torch.equal(a[3], b[3])
