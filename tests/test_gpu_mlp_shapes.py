"""The MLP at the sizes where the tile width and the split of K change: few
rows (tiles that do not fill the chip, K shared by a cluster), remainders of
the 128-row tiles, widths that divide by 64 only, and the allocation-free entry
point on the same shapes.  Tolerance as in test_gpu_mlp."""
import pytest
import torch

from paper_2609_13141_gb300 import sas, synth
from tests.test_gpu_mlp import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,D,F", [
    (1, 1600, 6400), (2, 1024, 4096), (127, 512, 2048), (128, 1600, 6400), (129, 1024, 4096),
    (77, 576, 2880),            # 576 = 9 x 64, 2880 = 45 x 64: 64-wide tiles, K blocks that do not split evenly
    (300, 2560, 1216), (777, 640, 2432),
])
def test_mlp_few_rows(T, D, F):
    _run(T, D, F, bias=T % 2 == 1, seed=T)


def test_mlp_noalloc_takes_the_same_path():
    T, D, F = 130, 1024, 4096
    X, W1, W2, b1, b2 = (t.cuda() for t in synth.mlp(T, D, F, seed=5, bias=True))
    layer = sas.SasLayer(1, 1, 64, 64, 0)
    Y0 = layer.mlp(X, W1, W2, b1, b2)
    Y = torch.empty_like(Y0)
    sas.sas_mlp_fwd_noalloc(X, W1, W2, Y, b1, b2)
    torch.cuda.synchronize()
    assert sas.sas_mlp_noalloc_get_device_status() == 0
    assert torch.equal(Y, Y0)
    layer.close()


def test_mlp_repeated_calls_overlapping_their_setup():
    # the down-projection starts ahead of the up-projection's end, and the next
    # call's up-projection overwrites the hidden activation the last one read
    T, D, F = 64, 1024, 4096
    X, W1, W2, _, _ = (None if t is None else t.cuda() for t in synth.mlp(T, D, F, seed=6))
    X2 = (X.float() * 0.5).to(torch.bfloat16)
    layer = sas.SasLayer(1, 1, 64, 64, 0)
    a, b = layer.mlp(X, W1, W2), layer.mlp(X2, W1, W2)
    torch.cuda.synchronize()
    for _ in range(50):
        y, z = layer.mlp(X, W1, W2), layer.mlp(X2, W1, W2)
    assert torch.equal(y, a) and torch.equal(z, b)
    layer.close()
