"""The calls this library is used for, with their sizes: what a speed comparison of two builds runs.

A case is one call (or one layer's calls) of the public entry points on the
shapes of the benchmark's workloads: SAS attention layers of diffusion
transformers (learned selector, one KV head per query head), Qwen3-4B-shaped
GQA layers (prefill with given scores, packed sequences, training), the
attention backward, the GELU MLP, and the decode step over a paged cache.
listed() gives the named ones, draw() others of the same ranges, prepare()
what a program holds before the call, run() one pass, work() the bytes and
FLOPs no implementation can do without, exact() the results in 64 bits.

Inputs are drawn on the GPU from the case's seed alone: keys, values and
gradients N(0, 1), weights N(0, 0.02), queries of the learned selector
correlated within a 64-token block (q = (mu[block] + 0.3 eps) / sqrt(1.09)),
given scores either block-coherent (u[block] + 0.05 eps) or independent.
"""
import math

import torch

from paper_2609_13141_gb300 import sas

BLOCK = 64
BF = torch.bfloat16

# Fields every case carries, with the values most cases share.
DEFAULTS = dict(B=1, H=24, Hkv=24, N=0, d=128, K=32, learned=False, coherent=True, hard=False, lens="", D=0, F=0,
                bias=False)


def _case(kind, **kw):
    unknown = set(kw) - set(DEFAULTS) - {"name"}
    assert not unknown, unknown
    return dict(DEFAULTS, kind=kind, **kw)


def listed():
    return [
        # The smallest layer of the benchmark, attention and MLP: a unit of a small model or a short prompt,
        # where the launches and the host path are what a user waits for.
        _case("layer", name="layer_256", H=4, Hkv=4, N=256, d=64, learned=True, D=256, F=1024),
        # Attention of an image diffusion transformer (4096 patches + 512 text tokens, two images).
        _case("attention", name="attention_image", B=2, N=4608, learned=True),
        # Attention of a video diffusion transformer, the benchmark's default: 21 x 45 x 80 patches + 512 text
        # tokens, a last block of 16 tokens.
        _case("attention", name="attention_video", N=76112, learned=True),
        # Inference form of a d = 64 layer on an odd length with independent given scores: neighbouring tokens
        # keep different blocks.
        _case("attention", name="attention_d64_odd", B=2, H=12, Hkv=12, N=6001, d=64, K=16, coherent=False, hard=True),
        # Prefill of a Qwen3-4B-shaped GQA layer at its full context, scores given per KV group.
        _case("attention", name="gqa_prefill_32k", H=32, Hkv=8, N=32768),
        # The same layer over a ragged batch of packed prompts, the selector learned.
        _case("packed", name="gqa_packed_prompts", H=32, Hkv=8, learned=True,
              lens="8192,4999,3000,1777,640,257,64,31,1"),
        # Attention backward of a training step: the high-resolution layer, score gradient included.
        _case("backward", name="backward_hires", N=16896),
        # Attention backward of a GQA layer on a training batch packed from sequences of geometric lengths.
        _case("packed_backward", name="gqa_packed_backward", H=32, Hkv=8,
              lens="8192,4096,2048,1024,512,256,128,64,32,16,16"),
        # The MLP of the image layer.
        _case("mlp", name="mlp_image", N=9216, D=3072, F=12288),
        # The MLP of the GQA layer on one short prompt: few rows, so few output tiles.
        _case("mlp", name="mlp_prompt_777", N=777, D=2560, F=9728, bias=True),
        # One decode step of one sequence at a short context: latency.
        _case("decode", name="decode_1x8k", H=32, Hkv=8, lens="8200"),
        # One decode step of a batch at long, unequal contexts.
        _case("decode", name="decode_8x64k", H=32, Hkv=8, lens="65536,65000,61441,57344,50001,65536,33333,64000"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_lens(rng, total):
    lens = []
    while sum(lens) < total and len(lens) < 24:
        lens.append(min(total - sum(lens), _log_int(rng, 1, total)))
    return ",".join(map(str, lens))


def draw(rng):
    kind = rng.choice(["layer", "attention", "attention", "gqa", "packed", "backward", "packed_backward", "mlp", "mlp",
                       "decode", "decode"])
    K = rng.choice([16, 32, 32, 32, 48, 64])
    if kind == "layer":
        H, d = rng.choice([(4, 64), (8, 64), (8, 128), (24, 128)])
        return _case("layer", H=H, Hkv=H, d=d, N=_log_int(rng, 65, 4608), K=K, learned=True, D=H * d, F=4 * H * d)
    if kind == "attention":
        B, H, d = rng.choice([(1, 24, 128), (2, 24, 128), (1, 12, 64), (2, 8, 128)])
        return _case("attention", B=B, H=H, Hkv=H, d=d, N=_log_int(rng, 500, 40000 // B), K=K,
                     learned=rng.random() < 0.7, coherent=rng.random() < 0.7, hard=rng.random() < 0.3)
    if kind == "gqa":
        H, Hkv = rng.choice([(32, 8), (16, 8), (32, 4), (28, 4)])
        return _case("attention", H=H, Hkv=Hkv, N=_log_int(rng, 1000, 32768), K=K, learned=rng.random() < 0.4,
                     coherent=rng.random() < 0.7)
    if kind == "packed":
        H, Hkv = rng.choice([(32, 8), (16, 8), (24, 24)])
        return _case("packed", H=H, Hkv=Hkv, K=K, learned=rng.random() < 0.6,
                     lens=_draw_lens(rng, _log_int(rng, 1000, 30000)))
    if kind == "backward":
        B, H, Hkv = rng.choice([(1, 24, 24), (2, 24, 24), (1, 32, 8), (1, 8, 8)])
        return _case("backward", B=B, H=H, Hkv=Hkv, N=_log_int(rng, 300, 12000 // B), K=min(K, 48),
                     coherent=rng.random() < 0.7, hard=rng.random() < 0.2)
    if kind == "packed_backward":
        H, Hkv = rng.choice([(32, 8), (16, 8), (8, 8)])
        return _case("packed_backward", H=H, Hkv=Hkv, K=min(K, 48), lens=_draw_lens(rng, _log_int(rng, 500, 14000)))
    if kind == "mlp":
        D, F = rng.choice([(3072, 12288), (2560, 9728), (1024, 4096), (1536, 6144), (1600, 6400)])
        return _case("mlp", N=_log_int(rng, 1, 16384), D=D, F=F, bias=rng.random() < 0.5)
    B = rng.choice([1, 1, 2, 4, 8, 12])
    lens = [_log_int(rng, 64, 262144 // B) for _ in range(B)]
    H, Hkv = rng.choice([(32, 8), (32, 8), (16, 8), (32, 4)])
    return _case("decode", H=H, Hkv=Hkv, K=min(K, 64), lens=",".join(map(str, lens)))


# ------------------------------------------------------------------ inputs

def _lens(c):
    return [int(x) for x in c["lens"].split(",")] if c["lens"] else []


def _tokens(c):
    """Rows of the token axis: a packed case's sequences back to back."""
    return sum(_lens(c)) if c["kind"].startswith("packed") else c["N"]


def _normal(g, *shape, std=1.0):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32).mul_(std)


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _mlp_inputs(c, g):
    T, D, F = c["B"] * c["N"], c["D"], c["F"]
    x = dict(X=_normal(g, T, D).to(BF), W1=_normal(g, F, D, std=0.02).to(BF), W2=_normal(g, D, F, std=0.02).to(BF))
    x["b1"] = _normal(g, F, std=0.02).to(BF) if c["bias"] else None
    x["b2"] = _normal(g, D, std=0.02).to(BF) if c["bias"] else None
    return x


def _attention_inputs(c, g):
    B, H, Hkv, N, d = c["B"], c["H"], c["Hkv"], _tokens(c), c["d"]
    x = dict(K=_normal(g, B, Hkv, N, d).to(BF), V=_normal(g, B, Hkv, N, d).to(BF))
    nb, blk = -(-N // BLOCK), torch.arange(N, device="cuda") // BLOCK
    if c["learned"]:
        mu = _normal(g, B, H, nb, d)
        q = _normal(g, B, H, N, d).mul_(0.3)
        x["Q"] = q.add_(mu[:, :, blk]).div_(math.sqrt(1.09)).to(BF)
        x["Wq"] = _normal(g, Hkv, d, H // Hkv * d, std=0.02).to(BF)
        x["Wk"] = _normal(g, Hkv, d, d, std=0.02).to(BF)
        x["S"] = None
    else:
        x["Q"] = _normal(g, B, H, N, d).to(BF)
        C = -(-max(_lens(c) or [N]) // BLOCK)
        if c["coherent"]:
            u = _normal(g, B, Hkv, nb, C)
            x["S"] = _normal(g, B, Hkv, N, C, std=0.05).add_(u[:, :, blk])
        else:
            x["S"] = _normal(g, B, Hkv, N, C)
        x["Wq"] = x["Wk"] = None
    return x


def _decode_inputs(c, g):
    lens, H, Hkv, d = _lens(c), c["H"], c["Hkv"], c["d"]
    B, max_blocks = len(lens), -(-max(lens) // BLOCK) + 8
    need = [-(-n // BLOCK) for n in lens]
    P = sum(need) + 3
    perm = torch.randperm(P, generator=g, device="cuda").to(torch.int32)
    table = torch.full((B, max_blocks), -1, device="cuda", dtype=torch.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = perm[at:at + n]
        at += n
    mu = _normal(g, P, Hkv, 1, d)
    Kc = _normal(g, P, Hkv, BLOCK, d, std=0.5).add_(mu).div_(math.sqrt(1.25)).to(BF)
    return dict(Kc=Kc, Vc=_normal(g, P, Hkv, BLOCK, d).to(BF), table=table, pages=P, max_blocks=max_blocks,
                lens=torch.tensor(lens, dtype=torch.int32, device="cuda"), q=_normal(g, B, H, d).to(BF),
                kn=_normal(g, B, Hkv, d).to(BF), vn=_normal(g, B, Hkv, d).to(BF),
                Wq=_normal(g, Hkv, d, H // Hkv * d, std=0.02).to(BF), Wk=_normal(g, Hkv, d, d, std=0.02).to(BF))


# ------------------------------------------------- the method in plain torch

def _plain(c, x, dt, back=None):
    """Selection, gated block-sparse attention and (back = {dO, O, LSE}) its backward in dtype dt, one query block
    of every KV group at a time over the blocks some row of it keeps.  The bf16 storage points of the selector
    (projected queries and summaries) are part of the method and kept.  Returns a dict of dt tensors."""
    B, H, Hkv, N, d, K = c["B"], c["H"], c["Hkv"], _tokens(c), c["d"], c["K"]
    G, M = H // Hkv, B * Hkv
    scale = 1.0 / math.sqrt(d)
    dev = x["Q"].device
    Q = x["Q"].reshape(M, G, N, d)
    Kx, Vx = x["K"].reshape(M, N, d), x["V"].reshape(M, N, d)
    Sx = None if x["S"] is None else x["S"].reshape(M, N, -1)
    new = lambda *s: torch.zeros(*s, device=dev, dtype=dt)  # noqa: E731
    O, LSE = new(M, G, N, d), new(M, G, N)
    sel_i = torch.full((M, N, K), -1, device=dev, dtype=torch.int32)
    sel_g = new(M, N, K)
    if back is not None:
        dO, Og = back["dO"].reshape(M, G, N, d), back["O"].reshape(M, G, N, d)
        Lg = back["LSE"].reshape(M, G, N)
        dQ, dK, dV = new(M, G, N, d), new(M, N, d), new(M, N, d)
        dlg, ds = new(M, N, K), new(M, N, Sx.shape[-1])
    at, spans = 0, []
    for n in (_lens(c) if c["kind"].startswith("packed") else [N]):
        spans.append((at, n))
        at += n
    for s0, n in spans:
        F, nb = n // BLOCK, -(-n // BLOCK)
        pad = torch.zeros(M, nb * BLOCK - n, d, device=dev, dtype=BF)
        kb = torch.cat([Kx[:, s0:s0 + n], pad], 1).view(M, nb, BLOCK, d)
        vb = torch.cat([Vx[:, s0:s0 + n], pad], 1).view(M, nb, BLOCK, d)
        if Sx is None:
            mean = kb[:, :F].to(dt).mean(2)
            Wk = x["Wk"].to(dt).repeat(B, 1, 1)
            Kt = (mean @ Wk.transpose(1, 2)).to(BF).to(dt)
            Wq = x["Wq"].to(dt).repeat(B, 1, 1)
        if back is not None:
            gk, gv = new(M * nb, BLOCK, d), new(M * nb, BLOCK, d)
        for cb in range(nb):
            r0 = s0 + cb * BLOCK
            R = min(BLOCK, n - cb * BLOCK)
            rows = slice(r0, r0 + R)
            q = Q[:, :, rows].to(dt)
            kk = min(K, cb)
            if kk:
                if Sx is None:
                    qt = (q.transpose(1, 2).reshape(M, R, G * d) @ Wq.transpose(1, 2)).to(BF).to(dt)
                    s = qt @ Kt[:, :cb].transpose(1, 2) / math.sqrt(d)
                else:
                    s = Sx[:, rows, :cb].to(dt)
                lg = s - torch.logsumexp(s, -1, keepdim=True)
                idx = torch.topk(s, kk, dim=-1).indices.sort(-1).values
                kept_lg = lg.gather(-1, idx)
                sel_i[:, rows, :kk] = idx.to(torch.int32)
                sel_g[:, rows, :kk] = kept_lg
                keep = torch.zeros(M, R, cb, device=dev, dtype=torch.bool).scatter_(-1, idx, True)
                some = keep.any(1)
                U = int(some.sum(-1).max())
                union = torch.argsort((~some).to(torch.int8), dim=-1, stable=True)[:, :U]
                pick = union[:, None].expand(M, R, U)
                bias = torch.zeros_like(lg) if c["hard"] else lg
                bias = bias.masked_fill(~keep, -math.inf).gather(-1, pick)
            else:
                U, union, bias = 0, torch.zeros(M, 0, device=dev, dtype=torch.int64), new(M, R, 0)
            blocks = torch.cat([union, torch.full((M, 1), cb, device=dev)], 1)
            take = blocks[:, :, None, None].expand(M, U + 1, BLOCK, d)
            ks = kb.gather(1, take).view(M, (U + 1) * BLOCK, d).to(dt)
            vs = vb.gather(1, take).view(M, (U + 1) * BLOCK, d).to(dt)
            causal = torch.arange(BLOCK, device=dev)[None] <= torch.arange(R, device=dev)[:, None]
            own = new(R, BLOCK).masked_fill(~causal, -math.inf)
            mask = torch.cat([bias.repeat_interleave(BLOCK, -1), own.expand(M, R, BLOCK)], -1)
            z = (q.reshape(M, G * R, d) @ ks.transpose(1, 2)).view(M, G, R, -1) * scale + mask[:, None]
            if back is None:
                lse = torch.logsumexp(z, -1)
                p = torch.exp(z - lse[..., None])
                O[:, :, rows] = (p.view(M, G * R, -1) @ vs).view(M, G, R, d)
                LSE[:, :, rows] = lse
                continue
            p = torch.exp(z - Lg[:, :, rows, None].to(dt))
            do = dO[:, :, rows].to(dt)
            delta = (do * Og[:, :, rows].to(dt)).sum(-1, keepdim=True)
            do = do.reshape(M, G * R, d)
            dz = p * ((do @ vs.transpose(1, 2)).view(M, G, R, -1) - delta)
            dz2, p2 = dz.view(M, G * R, -1), p.view(M, G * R, -1)
            dQ[:, :, rows] = (dz2 @ ks).view(M, G, R, d) * scale
            flat = (blocks + torch.arange(M, device=dev)[:, None] * nb).view(-1)
            gk.index_add_(0, flat, (dz2.transpose(1, 2) @ q.reshape(M, G * R, d)).view(-1, BLOCK, d) * scale)
            gv.index_add_(0, flat, (p2.transpose(1, 2) @ do).view(-1, BLOCK, d))
            if kk and not c["hard"]:
                per = dz.sum(1)[..., :U * BLOCK].reshape(M, R, U, BLOCK).sum(-1)
                every = new(M, R, cb).scatter_(-1, pick, per).masked_fill(~keep, 0.0)
                dlg[:, rows, :kk] = every.gather(-1, idx)
                ds[:, rows, :cb] = every - torch.exp(lg) * every.sum(-1, keepdim=True)
        if back is not None:
            dK[:, s0:s0 + n] = gk.view(M, nb * BLOCK, d)[:, :n]
            dV[:, s0:s0 + n] = gv.view(M, nb * BLOCK, d)[:, :n]
    lead = () if c["kind"].startswith("packed") else (B,)
    shape = lambda t, heads: t.reshape(*lead, heads, *t.shape[-2:])  # noqa: E731
    rows_ = lambda t: t.reshape(*lead, H, N)  # noqa: E731
    if back is None:
        return dict(O=O.reshape(*lead, H, N, d), LSE=rows_(LSE), sel_i=shape(sel_i, Hkv), sel_g=shape(sel_g, Hkv))
    return dict(dQ=dQ.reshape(*lead, H, N, d), dK=shape(dK, Hkv), dV=shape(dV, Hkv), dlogg=shape(dlg, Hkv),
                dscores=shape(ds, Hkv))


def _backward_inputs(c, g):
    """What the forward left for the backward: its inputs, O, LSE and the incoming gradient, all from the seed."""
    x = _attention_inputs(c, g)
    f = _plain(c, x, torch.float32)
    lead = () if c["kind"].startswith("packed") else (c["B"],)
    x["O"], x["LSE"] = f["O"].to(BF), f["LSE"].contiguous()
    x["dO"] = _normal(g, *lead, c["H"], _tokens(c), c["d"]).to(BF)
    return x


def _plain_mlp(x, dt):
    f = torch.nn.functional
    b1, b2 = (None if x[b] is None else x[b].to(dt) for b in ("b1", "b2"))
    h = f.gelu(f.linear(x["X"].to(dt), x["W1"].to(dt), b1)).to(BF).to(dt)
    return f.linear(h, x["W2"].to(dt), b2)


def _plain_decode(c, x, dt):
    """One decode step of every sequence in dtype dt: (O, LSE)."""
    H, Hkv, d, K = c["H"], c["Hkv"], c["d"], c["K"]
    G = H // Hkv
    Os, Ls = [], []
    for b, n in enumerate(_lens(c)):
        C = (n - 1) // BLOCK
        pages = x["table"][b, :C + 1].long()
        ks, vs = x["Kc"][pages].clone(), x["Vc"][pages].clone()       # [C + 1, Hkv, 64, d]
        ks[C, :, (n - 1) % BLOCK], vs[C, :, (n - 1) % BLOCK] = x["kn"][b], x["vn"][b]
        q = x["q"][b].view(Hkv, G, d).to(dt)
        qt = torch.einsum("hsk,hk->hs", x["Wq"].to(dt), q.reshape(Hkv, G * d)).to(BF).to(dt)
        kk = min(K, C)
        Kt = torch.einsum("hsd,chd->hcs", x["Wk"].to(dt), ks[:C].to(dt).mean(2)).to(BF).to(dt)
        s = torch.einsum("hs,hcs->hc", qt, Kt) / math.sqrt(d)
        idx = torch.cat([torch.topk(s, kk, -1).indices, torch.full((Hkv, 1), C, device=s.device)], -1)
        hk = torch.arange(Hkv, device=s.device)[:, None]
        kg = ks.transpose(0, 1)[hk, idx].reshape(Hkv, -1, d).to(dt)
        vg = vs.transpose(0, 1)[hk, idx].reshape(Hkv, -1, d).to(dt)
        z = torch.einsum("hgd,hkd->hgk", q, kg) / math.sqrt(d)
        z[..., kk * BLOCK + (n - 1) % BLOCK + 1:] = -math.inf
        lse = torch.logsumexp(z, -1)
        Os.append((torch.exp(z - lse[..., None]) @ vg).reshape(H, d))
        Ls.append(lse.reshape(H))
    return torch.stack(Os), torch.stack(Ls)


# ------------------------------------------------------------------ the calls

def _layer(c):
    packed = c["kind"].startswith("packed")
    lens = _lens(c)
    return sas.SasLayer(c["B"], c["H"], _tokens(c), c["d"], c["K"],
                        mode=sas.SAS_MODE_INFER_HARD if c["hard"] else sas.SAS_MODE_TRAIN_SOFT,
                        selector=sas.SAS_SEL_MEANPOOL_PROJ if c["learned"] else sas.SAS_SEL_SCORES_GIVEN, d_sel=c["d"],
                        Hkv=c["Hkv"], max_seqs=len(lens) if packed else 0, max_seqlen=max(lens) if packed else 0)


def _attend(c, s):
    x = s["x"]
    if c["kind"].startswith("packed"):
        return s["layer"].attention_varlen(s["cu"], x["Q"], x["K"], x["V"], x["S"], Wq=x["Wq"], Wk=x["Wk"])
    return s["layer"].attention(x["Q"], x["K"], x["V"], x["S"], x["Wq"], x["Wk"])


def _drop_batch(c, x):
    """Packed calls take [H, N, d] tensors."""
    if c["kind"].startswith("packed"):
        for k in ("Q", "K", "V", "S"):
            if x[k] is not None and x[k].dim() == 4:
                x[k] = x[k][0]


def prepare(case, seed):
    c, g = case, _rng(seed)
    s = dict(case=c)
    if c["kind"] == "decode":
        x = _decode_inputs(c, g)
        B, H, Hkv, d, K = len(_lens(c)), c["H"], c["Hkv"], c["d"], c["K"]
        dec = sas.SasDecoder(B, H, Hkv, d, K, x["max_blocks"], x["pages"], d_sel=d)
        Ksum = torch.zeros(B, Hkv, x["max_blocks"], d, device="cuda", dtype=BF)
        dec.summarize(x["Kc"], x["table"], x["lens"] - 1, x["Wk"], Ksum)
        out = (torch.empty(B, H, d, device="cuda", dtype=BF), torch.empty(B, H, device="cuda"),
               torch.empty(B, Hkv, K, device="cuda", dtype=torch.int32))
        # the serving loop replays one captured step while lengths, pages and tokens change in place
        step = lambda: dec.step(x["q"], x["Kc"], x["Vc"], x["table"], x["lens"], x["kn"], x["vn"],  # noqa: E731
                                x["Wq"], x["Wk"], Ksum, out=out)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            step()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            step()
        s.update(x=x, dec=dec, Ksum=Ksum, out=out, graph=graph)
        return s
    if c["kind"] == "mlp":
        # the handle's attention shape is not used
        s.update(x=_mlp_inputs(c, g), layer=sas.SasLayer(1, 1, 64, 128, 0))
        return s
    if c["kind"].endswith("backward"):
        s["x"] = _backward_inputs(c, g)
        s["layer"] = _layer(c)
    else:
        s["x"] = _attention_inputs(c, g)
        s["layer"] = _layer(c)
        if c["kind"] == "layer":
            s["mlp"] = _mlp_inputs(c, g)
    _drop_batch(c, s["x"])
    if c["kind"].startswith("packed"):
        at = [0]
        for n in _lens(c):
            at.append(at[-1] + n)
        s["cu"] = torch.tensor(at, dtype=torch.int32, device="cuda")
    if c["kind"].endswith("backward"):
        # the training step's forward: its kept lists and the handle's block lists; O and LSE stay those of the
        # plain forward above, so that they depend on the seed alone
        s["sel"] = _attend(c, s)[2:]
    return s


def run(state):
    c = state["case"]
    if c["kind"] == "decode":
        state["graph"].replay()
        return list(state["out"])
    x = state.get("x")
    if c["kind"] == "mlp":
        return state["layer"].mlp(x["X"], x["W1"], x["W2"], x["b1"], x["b2"])
    if c["kind"].endswith("backward"):
        layer = state["layer"]
        back = layer.attention_bwd_varlen if c["kind"].startswith("packed") else layer.attention_bwd
        idx, lg = state["sel"]
        return list(back(x["Q"], x["K"], x["V"], x["O"], x["LSE"], x["dO"], scores=x["S"], sel_idx=idx, sel_logg=lg,
                         want_ds=True))
    out = list(_attend(c, state))
    if c["kind"] == "layer":
        m = state["mlp"]
        out.append(state["layer"].mlp(m["X"], m["W1"], m["W2"], m["b1"], m["b2"]))
    return out


# ------------------------------------------------------------------ the work

def _pairs(n, K):
    """Attended (row, key) pairs of one head over n tokens."""
    own = kept = 0
    for cb in range(-(-n // BLOCK)):
        R = min(BLOCK, n - cb * BLOCK)
        own += R * (R + 1) // 2
        kept += R * BLOCK * min(K, cb)
    return own + kept


def _scored(n):
    """(row, historical block) pairs of one group over n tokens."""
    return sum(min(BLOCK, n - cb * BLOCK) * cb for cb in range(-(-n // BLOCK)))


def work(case):
    c = case
    B, H, Hkv, d, K = c["B"], c["H"], c["Hkv"], c["d"], c["K"]
    if c["kind"] == "decode":
        nbytes = flops = 0
        for n in _lens(c):
            C = (n - 1) // BLOCK
            keys = min(K, C) * BLOCK + (n - 1) % BLOCK + 1
            nbytes += Hkv * (C * d * 2 + keys * d * 4) + H * d * 4 + Hkv * (d * 4 + K * 4) + H * 4
            flops += Hkv * 2 * C * d + H * 4 * keys * d + Hkv * 2 * d * (H // Hkv) * d
        return dict(bytes=nbytes + Hkv * d * H // Hkv * d * 2, flops=flops)
    nbytes = flops = 0
    if c["kind"] in ("mlp", "layer"):
        T, D, F = B * c["N"], c["D"], c["F"]
        nbytes += 2 * (2 * T * D + 2 * D * F)
        flops += 4 * T * D * F
    if c["kind"] == "mlp":
        return dict(bytes=nbytes, flops=flops)
    N = _tokens(c)
    lens = _lens(c) if c["kind"].startswith("packed") else [N] * B
    pairs, scored = sum(_pairs(n, K) for n in lens), sum(_scored(n) for n in lens)
    kept = B * Hkv * N * K * 8                                    # kept lists: index and log-gate
    qo, kv = B * H * N * d * 2, B * Hkv * N * d * 2
    if c["kind"].endswith("backward"):
        # Q, O, dO, dQ; K, V, dK, dV; LSE; lists and d(log g); the scores read and their gradient written
        nbytes += 4 * qo + 4 * kv + B * H * N * 4 + kept + B * Hkv * N * K * 4
        nbytes += Hkv * (4 * scored + 4 * B * N * (-(-max(lens) // BLOCK)))
        return dict(bytes=nbytes, flops=H * 10 * d * pairs)
    nbytes += 2 * qo + 2 * kv + B * H * N * 4 + kept
    flops += H * 4 * d * pairs
    if c["learned"]:
        flops += Hkv * (2 * d * scored + 2 * d * (H // Hkv) * d * N * B + 2 * d * d * (N * B // BLOCK))
        nbytes += Hkv * d * d * 2 * (H // Hkv + 1)
    else:
        nbytes += Hkv * 4 * scored
    return dict(bytes=nbytes, flops=flops)


def exact(case, seed):
    c, g, dt = case, _rng(seed), torch.float64
    if c["kind"] == "decode":
        return list(_plain_decode(c, _decode_inputs(c, g), dt)) + [None]
    if c["kind"] == "mlp":
        return _plain_mlp(_mlp_inputs(c, g), dt)
    if c["kind"].endswith("backward"):
        x = _backward_inputs(c, g)
        r = _plain(c, x, dt, back=x)
        return [r["dQ"], r["dK"], r["dV"], r["dlogg"], r["dscores"]]
    x = _attention_inputs(c, g)
    r = _plain(c, x, dt)
    # kept sets: integers, and where two scores nearly tie the selector's own rounding decides
    out = [r["O"], r["LSE"], None, None if c["learned"] else r["sel_g"]]
    if c["kind"] == "layer":
        out.append(_plain_mlp(_mlp_inputs(c, g), dt))
    return out
