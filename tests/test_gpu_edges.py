"""Sizes at which a kernel's work split, a remainder or a dispatch boundary can go wrong, against the float64 CPU oracle (or, for
images and host buffers, the host packer and the device-buffer call, bit by bit)."""
import numpy as np
import pytest

from synth import make_layer, make_x
from tests.gpu_util import run_layer, check_against_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,M,N,batch", [
    # up to 16 columns: contiguous ranges of (row tile, slice) pairs that meet in the accumulate words
    (1, 33, 96, 9), (2, 129, 32, 16), (3, 700, 8192, 16), (2, 2500, 96, 12), (2, 1000, 4352, 1),
    (1, 1000, 8256, 16),                     # the last slice is a single step: one accumulator instead of two
    (1, 1000, 8224, 10),                     # and that step a single column tile
    # the contraction over clusters of 3, 5, 7 and 8 CTAs
    (3, 5000, 832, 24), (2, 3200, 2080, 33), (1, 2600, 2048, 40), (2, 160, 4096, 17),
    # three paths one after the other on one accumulator, the contraction whole and over a cluster; one column more and it is not
    (3, 13000, 2080, 208), (3, 2500, 8192, 200), (3, 13000, 2080, 209),
    # several 16-column groups per pass, ranges of groups, boxes of one and more steps
    (2, 3000, 160, 200), (2, 20000, 128, 300), (1, 300, 4096, 65),
])
def test_gemm_work_splits(K, M, N, batch):
    L = make_layer(M, N, K, key=(110, K, M, N))
    x = make_x(batch, N, key=(110, M, N, batch))
    y = run_layer(L, x, 3)
    check_against_oracle(L, x, y)
    assert np.array_equal(y.view(np.uint16), run_layer(L, x, 3).view(np.uint16))


@pytest.mark.parametrize("K,M,N,batch", [
    (2, 128, 32, 8), (1, 1, 96, 3), (2, 11008, 1024, 3), (3, 12000, 512, 8), (1, 5000, 3200, 5), (2, 20000, 2048, 4), (3, 260, 20000, 7),
])
def test_f16_gemv_work_splits(K, M, N, batch):
    """One group of 16 warps per CTA and two of 8, ranges inside a row tile, of one, and across several."""
    L = make_layer(M, N, K, key=(111, K, M, N))
    x = make_x(batch, N, key=(111, M, N, batch))
    y = run_layer(L, x, 6)
    check_against_oracle(L, x, y)
    assert np.array_equal(y.view(np.uint16), run_layer(L, x, 6).view(np.uint16))


@pytest.mark.parametrize("K", [1, 2, 3])
@pytest.mark.parametrize("batch", [3, 8, 9, 16])
@pytest.mark.parametrize("shapes", [
    [(128, 32), (129, 96)],
    [(300, 640), (300, 672), (1000, 4352)],                         # an odd number of column tiles beside an even one
    [(100, 256), (2500, 256), (33, 8192), (5000, 288), (7, 32)],    # more layers than one launch of the GEMM takes
])
def test_groups_of_three_to_sixteen_rows(K, batch, shapes):
    import torch
    import paper_2602_05367_b200 as rabit
    inputs = [make_layer(M, N, K, key=(112, K, M, N)) for M, N in shapes]
    layers = [rabit.rabit_pack(L.planes, L.g, L.h) for L in inputs]
    xs = [make_x(batch, N, key=(112, N, batch)) for M, N in shapes]
    dev = {N: torch.from_numpy(x).cuda() for (M, N), x in zip(shapes, xs)}        # layers of equal width share their input
    ys = [torch.full((batch, M), float("nan"), dtype=torch.float16, device="cuda") for M, N in shapes]
    for _ in range(2):                                                            # the second call finds the scratch as the first left it
        rabit.rabit_linear_group(layers, [dev[N] for M, N in shapes], ys)
    torch.cuda.synchronize()
    for L, layer, x, y in zip(inputs, layers, xs, ys):
        assert layer.status() == 0
        check_against_oracle(L, x, y.cpu().numpy())
        layer.free()


@pytest.mark.parametrize("K,M,N", [(1, 1, 32), (2, 129, 96), (3, 300, 672), (2, 1000, 1184)])
def test_packing_on_the_device_gives_the_host_packer_s_image(K, M, N):
    import paper_2602_05367_b200 as rabit
    L = make_layer(M, N, K, key=(113, K, M, N))
    layer = rabit.rabit_pack(L.planes, L.g, L.h)
    assert np.array_equal(layer.dev_buf.cpu().numpy(), rabit.pack_host(L.planes, L.g, L.h))
    layer.free()


@pytest.mark.parametrize("N,batch,offset", [(32, 1, 0), (8192, 16, 0), (8192, 17, 0), (4096, 2, 4)])
def test_page_locked_inputs_up_to_and_beyond_what_a_kernel_fetches(N, batch, offset):
    """256 KB is the most that a kernel fetches; an input that does not start on a 16-byte boundary is copied."""
    import torch
    import paper_2602_05367_b200 as rabit
    M = 96
    L = make_layer(M, N, 2, key=(114, N))
    layer = rabit.rabit_pack(L.planes, L.g, L.h)
    x = torch.from_numpy(make_x(batch, N, key=(114, N, batch)))
    host = torch.zeros(offset + batch * N, dtype=torch.float16).pin_memory()[offset:].view(batch, N)
    host.copy_(x)
    y_host = torch.zeros((batch, M), dtype=torch.float16).pin_memory()
    rabit.rabit_linear_host(layer, host, y_host)
    want = rabit.rabit_linear(layer, x.cuda())
    torch.cuda.synchronize()
    assert np.array_equal(y_host.numpy().view(np.uint16), want.cpu().numpy().view(np.uint16))
    layer.free()


@pytest.mark.parametrize("K,M,N", [(1, 1, 32), (3, 129, 96), (2, 300, 672)])
def test_packing_and_host_calls_write_nothing_outside_their_buffers(K, M, N):
    """The kernels that the checked build leaves out (packing, derivation, fetching of inputs): image, stage and outputs lie between
    guard bands that have to come back untouched."""
    import ctypes
    import torch
    import paper_2602_05367_b200 as rabit
    from paper_2602_05367_b200 import binding
    lib, vp, band = binding.raw_lib(), ctypes.c_void_p, 4096
    L = make_layer(M, N, K, key=(115, K, M, N))
    g16, h16 = L.g.view(np.uint16), L.h.view(np.uint16)
    nbytes = rabit.packed_bytes(K, M, N)
    stream = vp(torch.cuda.current_stream().cuda_stream)

    def guarded(n, dtype, device):
        raw = torch.full((band + n + band,), 0xA5, dtype=torch.uint8, device=device)
        if device == "cpu":
            raw = raw.pin_memory()
        return raw, raw[band:band + n].view(dtype), lambda: bool((raw[:band] == 0xA5).all()) and bool((raw[band + n:] == 0xA5).all())

    W = torch.randn((M, N), device="cuda")
    for derive in (False, True):
        raw, image, intact = guarded(nbytes, torch.uint8, "cuda")
        assert image.data_ptr() % 256 == 0
        out = vp()
        if derive:
            rc = lib.rabit_derive_pack(vp(W.data_ptr()), g16.ctypes.data, h16.ctypes.data, K, M, N, vp(image.data_ptr()), nbytes, stream, ctypes.byref(out))
        else:
            rc = lib.rabit_pack(L.planes.ctypes.data, g16.ctypes.data, h16.ctypes.data, K, M, N, vp(image.data_ptr()), nbytes, stream, ctypes.byref(out))
        assert rc == 0, rabit.last_error()
        for batch in (1, 5):
            need = lib.rabit_stage_bytes(out, batch)
            stage_raw, stage, stage_intact = guarded(need, torch.uint8, "cuda")
            x = torch.from_numpy(make_x(batch, N, key=(115, batch))).pin_memory()
            y_raw, y, y_intact = guarded(batch * M * 2, torch.float16, "cpu")
            assert lib.rabit_linear_host(out, vp(x.data_ptr()), vp(y.data_ptr()), batch, vp(stage.data_ptr()), need, stream) == 0, rabit.last_error()
            torch.cuda.synchronize()
            assert stage_intact() and y_intact() and np.isfinite(y.numpy().astype(np.float64)).all()
        assert intact()
        assert lib.rabit_free(out) == 0
