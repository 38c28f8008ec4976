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


@pytest.mark.parametrize("shapes,batch,variant,stages", [
    ([(2, 2560, 8192)], 12, 3, (0, 2)),                     # ranges of (row tile, slice) pairs
    ([(1, 2560, 8192)], 12, 3, (1,)),                       # four accumulators for one path
    ([(2, 3000, 8192)], 48, 3, (0, 3)),                     # the contraction over clusters
    ([(3, 2500, 8192)], 200, 3, (2, 20)),                   # path after path, over clusters
    ([(2, 20000, 1024)], 300, 3, (3,)),                     # several passes of 16-column groups a CTA
    ([(2, 20153, 992)], 46, 3, (5,)),                       # contiguous ranges of 16-column groups
    ([(3, 1000, 2048)], 100, 4, (1,)),                      # dequantised tiles
    ([(2, 700, 8192), (2, 2500, 4352)], 16, 0, (0, 1)),     # several layers in one launch
    ([(3, 6400, 6400)], 4, 2, (8, 11)),                     # integer tensor-core GEMV: 12.7 stages of 16 tiles a CTA
])
def test_withheld_copy_ends_as_a_recorded_time_out(shapes, batch, variant, stages):
    """The producer of the GEMM (or of the integer tensor-core GEMV) waits for a barrier that nothing signals: every role gives up, the launch ends, the status of every
    layer of the call says so, and after a clear the same layers compute the right result.  (Only the checked build has the
    switch, tests/test_gpu_checked_build.py runs this under it; the ordinary library refuses the call.)"""
    import time
    import torch
    import paper_2602_05367_b200 as rabit
    from paper_2602_05367_b200 import binding
    lib = binding.raw_lib()
    inputs = [make_layer(M, N, K, key=(121, K, M, N)) for K, M, N in shapes]
    layers = [rabit.rabit_pack(L.planes, L.g, L.h) for L in inputs]
    if lib.rabit_selftest_withhold(layers[0].handle, 0) != 0:
        assert "RABIT_CHECKED" in rabit.last_error()
        return
    xn = [make_x(batch, N, key=(121, N, batch)) for _, _, N in shapes]
    xs = [torch.from_numpy(x).cuda() for x in xn]
    ys = [torch.zeros((batch, M), dtype=torch.float16, device="cuda") for _, M, _ in shapes]

    def call():
        if len(layers) > 1:
            rabit.rabit_linear_group(layers, xs, ys)
        else:
            layers[0].set_variant(variant)
            rabit.rabit_linear(layers[0], xs[0], ys[0])
        torch.cuda.synchronize()

    for stage in stages:
        for layer in layers:
            assert lib.rabit_selftest_withhold(layer.handle, stage) == 0
        t0 = time.time()
        call()
        assert time.time() - t0 < 20.0
        for layer in layers:
            assert layer.status() == -5
            assert layer.status(clear=True) == -5
            assert lib.rabit_selftest_withhold(layer.handle, -1) == 0
        call()
        for L, x, y, layer in zip(inputs, xn, ys, layers):
            assert layer.status() == 0
            rows = np.unique(np.concatenate([np.arange(0, L.M, 61), [L.M - 1]]))
            check_against_oracle(L, x, y.cpu().numpy(), tight=variant != 4, rows=rows)
    for layer in layers:
        layer.free()
