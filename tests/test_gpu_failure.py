"""Failure detection and recovery on the device, without a GPU fault: a wait that runs out ends with a recorded status, and
clearing the status gives back a layer that works."""
import numpy as np
import pytest

from oracle import layout_spec as spec
from synth import make_layer, make_x
from tests.gpu_util import check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 5, 16])
def test_clearing_the_status_restores_the_whole_scratch(batch):
    """A recorded failure may leave the exchange buffer and the accumulate words incomplete (planted here from the host): after
    a clear the next call must be right."""
    import torch
    import paper_2602_05367_b200 as rabit
    K, M, N = 2, 300, 4352
    L = make_layer(M, N, K, key=(120,))
    layer = rabit.rabit_pack(L.planes, L.g, L.h)
    hd = spec.read_header(layer.dev_buf[:256].cpu().numpy())
    words = layer.dev_buf[hd["off_acc"]:hd["total_bytes"]].view(torch.int64)
    words.fill_((3 << 55) + 12345)                                           # three arrivals and a sum
    layer.dev_buf[hd["off_partial"]:hd["off_flags"]].zero_()                 # "published" partial sums
    status = hd["off_flags"] + 4 * (hd["n_rt"] * K + 320)
    layer.dev_buf[status:status + 4].view(torch.int32).fill_(1)
    assert layer.status() == -5                                              # seen, not cleared
    assert layer.status(clear=True) == -5
    assert layer.status() == 0
    for variant in (0, 2):                                                   # accumulate words, exchange buffer
        layer.set_variant(variant)
        x = make_x(batch, N, key=(120, batch))
        y = rabit.rabit_linear(layer, torch.from_numpy(x).cuda())
        check_against_oracle(L, x, y.cpu().numpy())
    assert layer.status() == 0
    layer.free()
