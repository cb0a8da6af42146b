"""Kept lists of the decode step when candidates are missing, as after a summary load
whose bounded wait gave up: the list holds the blocks that were scored and nothing
else, sel_idx is -1 past them, and the attention reads no table entry for a block
that the sequence does not have."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2609_13141_gb300 import _build, sas
from tests import parity as P

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    sas.lib()
    so = str(tmp_path_factory.mktemp("native") / "decode_lists.so")
    cmd = [_build._nvcc(), *_build.CFLAGS, "-shared", "-o", so, os.path.join(HERE, "native", "decode_lists.cu"),
           _build.LIB_PATH, "-Xlinker", "-rpath=" + os.path.dirname(_build.LIB_PATH)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("radix", [0, 1])
@pytest.mark.parametrize("M,K,filled", [
    (8, 4, 8), (8, 4, 4), (8, 4, 3), (8, 4, 0), (64, 64, 63), (256, 64, 64), (256, 64, 17), (255, 1, 0),
])
def test_missing_candidates_shorten_the_list(shim, radix, M, K, filled):
    g = torch.Generator().manual_seed(M + K + filled)
    key = torch.randint(1, 50, (M,), generator=g, dtype=torch.int32)   # ties among them
    drop = torch.randperm(M, generator=g)[: M - filled]
    key[drop] = 0
    blk = torch.arange(M, dtype=torch.int32) * 3
    blk[drop] = -1
    order = torch.argsort(key, descending=True, stable=True)
    want = sorted(blk[i].item() for i in order[:K] if key[i] > 0)
    dk, db = key.to(DEV), blk.to(DEV)
    lst = torch.full((64,), 7777, dtype=torch.int32, device=DEV)
    n = torch.full((1,), 7777, dtype=torch.int32, device=DEV)
    sel = torch.full((K,), 7777, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    assert shim.decode_lists_select(_p(dk), _p(db), M, K, radix, _p(lst), _p(n), _p(sel)) == 0
    assert n.item() == len(want)
    assert lst[:len(want)].tolist() == want
    assert sel.tolist() == want + [-1] * (K - len(want))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("entries", [[2, -1, 5, 1 << 20], [-1, -1, -1, -1], [-(2 ** 31), 2 ** 31 - 1, 0, 3]])
def test_attention_skips_blocks_the_sequence_does_not_have(shim, d, entries):
    G, max_blocks, pages, n, K = 4, 8, 8, 64 * 6 + 9, 4   # own block 6: blocks 0 .. 5 are its history
    g = torch.Generator(device=DEV).manual_seed(d)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEV).bfloat16()  # noqa: E731
    q, Kc, Vc = rnd(1, G, d), rnd(pages, 1, 64, d), rnd(pages, 1, 64, d)
    table = torch.arange(max_blocks, dtype=torch.int32, device=DEV)[None].contiguous()
    i32 = lambda v: torch.tensor(v, dtype=torch.int32, device=DEV)  # noqa: E731
    lst, ln, lens, status = i32(entries + [0] * 60), i32([len(entries)]), i32([n]), i32([0] * 4)
    O, LSE = torch.empty(1, G, d, device=DEV, dtype=torch.bfloat16), torch.empty(1, G, device=DEV)
    part, cnt = torch.empty(1 << 16, device=DEV), i32([0, 0])
    torch.cuda.synchronize()
    assert shim.decode_lists_attend(_p(q), _p(Kc), _p(Vc), _p(table), _p(lens), max_blocks, pages, G, d, K, _p(lst),
                                    _p(ln), _p(O), _p(LSE), _p(part), part.numel(), _p(cnt), _p(status)) == 0
    assert status[0].item() == 0
    have = [6] + [m for m in entries if 0 <= m < 6]
    keys = torch.cat([Kc[m, 0, :9 if j == 0 else 64] for j, m in enumerate(have)]).double()
    vals = torch.cat([Vc[m, 0, :9 if j == 0 else 64] for j, m in enumerate(have)]).double()
    z = q[0].double() @ keys.T / d ** 0.5
    P.compare_o(P.f64(O[0].cpu()), (torch.softmax(z, -1) @ vals).cpu().numpy(), "O")
    assert (torch.logsumexp(z, -1) - LSE[0].double()).abs().max().item() <= P.LSE_MAX_ABS
