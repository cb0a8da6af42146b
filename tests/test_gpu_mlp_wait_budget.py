"""The second product of the MLP is launched ahead of the first one's end; the time the
first one takes does not count against the second one's bounded waits.

64 rows of D = 32768, F = 512: the first product is a single wave of 64 K blocks a CTA
(at least 300 SM cycles each, so 19000 in all) on part of the SMs, so the second one's
CTAs are resident on the others from its start.  A budget of 14000 cycles is longer than
any wait within a product (a K block's loads; the second product's 8 K blocks) and
shorter than the first product."""
import pytest
import torch

from paper_2609_13141_gb300 import sas, synth

pytestmark = pytest.mark.gpu


def test_first_product_is_not_on_the_second_ones_budget():
    T, D, F = 64, 32768, 512
    X, W1, W2, _, _ = (None if t is None else t.cuda() for t in synth.mlp(T, D, F, seed=1))
    layer = sas.SasLayer(1, 1, 64, 64, 0)
    ref = layer.mlp(X, W1, W2)
    torch.cuda.synchronize()
    assert sas.sas_get_device_status(layer.h) == sas.SAS_OK
    sas.sas_set_wait_limit(layer.h, 14000)
    for _ in range(20):
        y = layer.mlp(X, W1, W2)
        torch.cuda.synchronize()
        assert sas.sas_get_device_status(layer.h) == sas.SAS_OK
        assert torch.equal(y, ref)
    layer.close()
