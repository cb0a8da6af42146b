"""Selection from given scores, eight lanes per row: both sides of the shortest and
longest rows it takes (64 and 704 blocks with K <= 32, 1280 above), 32-block groups,
score distributions its bracketing has to survive (ties, two values, heavy tails,
one huge score, tiny and denormal spreads, sorted rows), GQA segment unions, full*
noise.  Kept sets must equal a stable sort's (score descending, lower block
first) on every checked row, log-gates s - logsumexp(s) within the fp32 bound."""
import pytest
import torch

from paper_2609_13141_gb300 import sas, synth
from tests import parity as P

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _scores(kind, H, N, C, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    z = torch.randn(H, N, C, generator=g, device=DEV)
    if kind == "ties":
        return (z * 1.5).round()
    if kind == "two":
        return (z > 1.2).float() - 3.0
    if kind == "cauchy":
        return (z / (torch.randn(H, N, C, generator=g, device=DEV).abs() + 1e-3)).clamp(-1e30, 1e30)
    if kind == "spike":
        return z + 1e6 * (torch.arange(C, device=DEV) == 3)
    if kind == "tiny":
        return 1.0 + z * 1e-7
    if kind == "denormal":
        return z * 1e-42
    if kind == "sorted":
        return torch.arange(C, device=DEV, dtype=torch.float32).expand(H, N, C) * 0.01 + z * 1e-3
    return z


def _check(S, si, sl, rows, K):
    """Rows of one group against a stable sort."""
    for i in rows:
        C = i // 64
        s = S[i, :C]
        k = min(K, C)
        want = torch.sort(s, descending=True, stable=True).indices[:k].sort().values
        got = si[i]
        assert torch.equal(got[:k].long(), want), f"row {i}"
        assert torch.all(got[k:] == -1) and torch.all(sl[i, k:] == 0)
        if k:
            lg = s.double()[want] - torch.logsumexp(s.double(), 0)
            # absolute, plus the fp32 rounding of s - LSE at the row's magnitude
            tol = P.LOGG_MAX_ABS + 2.0 ** -22 * float(s.abs().max())
            assert float((sl[i, :k].double() - lg).abs().max()) <= tol, f"row {i}"


def _run(kind, H, Hkv, N, K, seed=0, noise=False):
    C, d = -(-N // 64), 64
    S = _scores(kind, Hkv, N, C, seed)[None].contiguous()
    z = lambda h: torch.zeros(1, h, N, d, device=DEV, dtype=torch.bfloat16)  # noqa: E731
    layer = sas.SasLayer(1, H, N, d, K, Hkv=Hkv)
    if noise:
        e = torch.randn(1, Hkv, N, C, generator=torch.Generator(device=DEV).manual_seed(seed + 1), device=DEV) * 0.5
        _, _, si, sl = layer.attention_noisy(z(H), z(Hkv), z(Hkv), e, scores=S)
        S = S + e
    else:
        _, _, si, sl = layer.attention(z(H), z(Hkv), z(Hkv), scores=S)
    torch.cuda.synchronize()
    assert sas.sas_get_device_status(layer.h) == 0
    unions = sas.sas_get_tile_union_counts(layer.h, Hkv * -(-N // 128))
    tiles, blocks = sas.sas_get_attention_work(layer.h)
    layer.close()
    rows = sorted({r for m in (0, 1, K, K + 1, 2, 4, 8, 12, 16, 24, 40, C) for r in
                   (64 * m * (1 if m <= K + 1 or m == C else 32) + o for o in (-1, 0, 65)) if 0 <= r < N} |
                  set(range(0, N, max(1, N // 60))) | {N - 1})
    for h in range(Hkv):
        _check(S[0, h], si[0, h], sl[0, h], rows, K)
        # the tile unions: kept blocks below the tile's first diagonal block
        for t in sorted({0, 1, (N - 1) // 256, (N - 1) // 128}):
            kept = si[0, h, 128 * t:128 * (t + 1)]
            assert unions[h * -(-N // 128) + t] == int(torch.unique(kept[(kept >= 0) & (kept < 2 * t)]).numel())
    if H > Hkv:   # head-packed tiles: each segment's union and its one diagonal block
        R = 128 // (H // Hkv)
        want = 0
        for h in range(Hkv):
            for i in range(0, N, R):
                kept = si[0, h, i:i + R]
                want += int(torch.unique(kept[kept >= 0]).numel()) + 1
        assert blocks == want


@pytest.mark.parametrize("kind", ["normal", "ties", "two", "cauchy", "spike", "tiny", "denormal", "sorted"])
@pytest.mark.parametrize("N,K", [(6500, 32), (5000, 7), (4300, 64)])
def test_distributions(kind, N, K):
    _run(kind, 2, 2, N, K, seed=N + K)


@pytest.mark.parametrize("N", [64 * 64 - 64, 64 * 64 - 63, 64 * 257, 64 * 512 + 1, 64 * 704, 64 * 704 + 1, 64 * 1280,
                               64 * 1280 + 1])
@pytest.mark.parametrize("kind,K", [("normal", 32), ("ties", 33)])
def test_row_lengths(N, kind, K):
    _run(kind, 1, 1, N, K, seed=K)


@pytest.mark.parametrize("H,Hkv,N", [(4, 1, 5001), (16, 2, 4500), (32, 2, 4099), (4, 1, 3001)])
def test_segment_unions(H, Hkv, N):
    _run("normal", H, Hkv, N, 5, seed=N)


def test_noise():
    _run("normal", 2, 2, 3000, 9, seed=4, noise=True)


@pytest.mark.parametrize("act", ["softmax", "sigmoid", "logit"])
@pytest.mark.parametrize("kind", ["masked", "lowest", "posinf", "nan", "all_masked"])
def test_special_values(kind, act):
    """Infinities, the lowest float and NaN: sets as replace-the-worst defines them (a
    NaN stays if it is among the first K blocks and never enters later)."""
    H, N, K, d = 1, 5000, 9, 64
    C = -(-N // 64)
    S = _scores("normal", H, N, C, 3)[None].contiguous()
    u = torch.rand(S.shape, generator=torch.Generator(device=DEV).manual_seed(8), device=DEV)
    hit = u < (0.9 if kind in ("masked", "lowest") else 0.08)
    S[hit] = {"masked": -float("inf"), "lowest": torch.finfo(torch.float32).min, "posinf": float("inf"),
              "nan": float("nan"), "all_masked": 0.0}[kind]
    if kind == "all_masked":
        S[:, :, ::3] = -float("inf")
    z = torch.zeros(1, H, N, d, device=DEV, dtype=torch.bfloat16)
    code = {"softmax": sas.SAS_GATE_SOFTMAX, "sigmoid": sas.SAS_GATE_SIGMOID, "logit": sas.SAS_GATE_LOGIT}
    layer = sas.SasLayer(1, H, N, d, K, gate_act=code[act])
    _, _, si, sl = layer.attention(z, z, z, scores=S)
    torch.cuda.synchronize()
    layer.close()
    for i in range(0, N, 37):
        n = i // 64
        k = min(K, n)
        s = S[0, 0, i, :n]
        key = torch.where(s.isnan(), torch.where(torch.arange(n, device=DEV) < K, float("inf"), -float("inf")), s)
        want = torch.sort(key, descending=True, stable=True).indices[:k].sort().values
        assert torch.equal(si[0, 0, i, :k].long(), want), f"row {i}"
        if k == 0:
            continue
        x = s[want].double()
        lg = {"softmax": x - torch.logsumexp(s.double(), 0), "logit": x,
              "sigmoid": torch.nn.functional.logsigmoid(x)}[act]
        fin = lg.isfinite()
        got = sl[0, 0, i, :k].double()
        assert float((got - lg)[fin].abs().max() if fin.any() else 0.0) <= P.LOGG_MAX_ABS, f"row {i}"


@pytest.mark.parametrize("N", [64 * 5120, 64 * 5120 + 1])
def test_segment_lists_of_long_histories(N):
    """Learned selection, head-packed tiles: the segment lists' sets hold a byte per
    block up to 5120 blocks, a bit beyond.  Each list is its tokens' distinct blocks."""
    H, Hkv, K, d = 2, 1, 2, 64
    g = torch.Generator(device=DEV).manual_seed(N)
    Q, Kk, V = (torch.randn(1, h, N, d, generator=g, device=DEV).bfloat16() for h in (H, Hkv, Hkv))
    Wq, Wk = (w.to(DEV) for w in synth.decode_selector_weights(Hkv, H // Hkv, d, d, seed=1, exact=True))
    layer = sas.SasLayer(1, H, N, d, K, Hkv=Hkv, selector=sas.SAS_SEL_MEANPOOL_PROJ, d_sel=d)
    _, _, si, _ = layer.attention(Q, Kk, V, Wq=Wq, Wk=Wk)
    torch.cuda.synchronize()
    _, blocks = sas.sas_get_attention_work(layer.h)
    layer.close()
    seg = torch.arange(N, device=DEV)[:, None].expand(N, K) // 64   # 64 tokens of two heads fill a tile
    kept = si[0, 0].long()
    pairs = torch.unique((seg * (1 << 20) + kept)[kept >= 0])
    assert blocks == int(pairs.numel()) + -(-N // 64)
