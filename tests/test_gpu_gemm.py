"""GPU parity of the large-batch (tensor-core GEMM) form against the float64 CPU oracle, through
the C ABI, within  max_i |y_gpu - y_ref| <= 2e-3 * max_i sum_j sum_k |g_ki h_kj x_j| + 1e-5  per batch row."""
import numpy as np
import pytest

from synth import make_layer, make_x, make_planes_constant
from tests.gpu_util import run_layer, check_against_oracle

pytestmark = pytest.mark.gpu

GEMM = 3    # variant number of the tcgen05 GEMM


@pytest.mark.parametrize("K,M,N,batch", [
    (2, 128, 64, 17),        # one tile, one step
    (2, 256, 256, 40),
    (1, 200, 96, 64),        # ragged M, a last step with a single column tile
    (2, 1000, 1184, 300),    # several row tiles, four chunks of batch columns with a ragged tail, N % 64 == 32
    (2, 384, 2048, 512),
    (2, 2500, 512, 257),
    (3, 300, 352, 130),      # three paths: three chunks of batch columns, the last with a ragged tail
    (3, 128, 64, 17),
])
@pytest.mark.parametrize("variant", [0, GEMM])
def test_gemm_shapes(K, M, N, batch, variant):
    L = make_layer(M, N, K, key=(60, K, M, N))
    x = make_x(batch, N, key=(60, M, N, batch))
    y = run_layer(L, x, variant)
    check_against_oracle(L, x, y)


def test_gemm_matches_plain_kernel_closely():
    """Both device kernels see the same packed image; the GEMM keeps products exact and accumulates in fp32."""
    L = make_layer(512, 1024, 2, key=(61,))
    x = make_x(96, 1024, key=(61,))
    a = run_layer(L, x, GEMM).astype(np.float64)
    b = run_layer(L, x, 1).astype(np.float64)
    assert np.abs(a - b).max() <= 4e-3


def test_gemm_structured_inputs():
    K, M, N, batch = 2, 256, 320, 33
    L = make_layer(M, N, K, key=(62,))
    x = np.zeros((batch, N), dtype=np.float16)
    for b in range(batch):
        x[b, (b * 37) % N] = 1.0          # unit vectors: every output reads one column
    check_against_oracle(L, x, run_layer(L, x, GEMM))
    for bit in (0, 1):
        L.planes = make_planes_constant(K, M, N, bit)
        x = make_x(batch, N, key=(62, bit))
        check_against_oracle(L, x, run_layer(L, x, GEMM))
    y = run_layer(make_layer(M, N, K, key=(62, 9)), np.zeros((batch, N), dtype=np.float16), GEMM)
    assert not y.any()


def test_three_paths_large_batch():
    """K = 3 runs with three accumulators; automatic dispatch and the explicit variant agree with the oracle."""
    L = make_layer(160, 256, 3, key=(63,))
    x = make_x(48, 256, key=(63,))
    check_against_oracle(L, x, run_layer(L, x, 0))
    check_against_oracle(L, x, run_layer(L, x, GEMM))


@pytest.mark.parametrize("K,M,N,batch", [
    (2, 300, 640, 1),
    (2, 300, 640, 5),
    (3, 200, 352, 9),
    (2, 1000, 1184, 16),
])
def test_gemm_runs_small_batches_too(K, M, N, batch):
    """The tensor-core GEMM forced onto decode-sized batches (a pass of 16 columns, most of them zero fill)."""
    L = make_layer(M, N, K, key=(62, K, M, N))
    x = make_x(batch, N, key=(62, M, N, batch))
    y = run_layer(L, x, GEMM)
    check_against_oracle(L, x, y)


@pytest.mark.parametrize("batch", [2, 3, 4, 8, 9, 12, 16, 17, 32, 33])
def test_dispatch_by_batch(batch):
    """One or two rows take the table-driven GEMV, 3 to 8 the f16 tensor-core GEMV, more the GEMM.  Whichever kernel runs, the
    result is within tolerance and is exactly what that kernel gives when forced."""
    L = make_layer(14336, 512, 2, key=(63,))
    x = make_x(batch, 512, key=(63, batch))
    y_auto = run_layer(L, x, 0)
    check_against_oracle(L, x, y_auto)
    expect = 5 if batch <= 2 else 6 if batch <= 8 else GEMM
    y_forced = run_layer(L, x, expect)
    assert np.array_equal(y_auto.view(np.uint16), y_forced.view(np.uint16))


DEQ = 4     # variant number of the GEMM on dequantised fp16 weight tiles


@pytest.mark.parametrize("K,M,N,batch", [
    (2, 128, 64, 17),
    (1, 200, 96, 64),
    (2, 1000, 1184, 300),
    (2, 384, 2048, 512),
    (3, 300, 352, 130),
    (3, 1000, 1184, 300),
    (2, 300, 640, 5),
])
def test_dequantised_tile_gemm(K, M, N, batch):
    """Variant 4 forms sum_k +-g_k h_k per weight in fp16 and runs one contraction: every weight carries a relative
    rounding of about 2^-11 per partial product, so the result stays inside the tolerance (worst case half of it) but is
    not as close to the oracle as the exact-expansion GEMM."""
    L = make_layer(M, N, K, key=(64, K, M, N))
    x = make_x(batch, N, key=(64, M, N, batch))
    y = run_layer(L, x, DEQ)
    err, tol = check_against_oracle(L, x, y, tight=False)          # fp16-rounded weights: the mandated bound only
    y_exact = run_layer(L, x, GEMM)
    err_exact, _ = check_against_oracle(L, x, y_exact)
    assert err_exact.max() <= err.max() + 1e-3 * tol.max()        # the exact expansion is never noticeably worse


@pytest.mark.parametrize("K,M,N,batch,variant", [
    (2, 256, 4096, 64, GEMM),      # 2 row tiles, 64 steps: eight CTAs share each
    (2, 256, 4096, 300, GEMM),     # five chunks of batch columns, ragged
    (2, 200, 4160, 40, DEQ),       # ragged rows, 65 steps split unevenly
    (3, 256, 2048, 100, GEMM),     # three paths, two chunks, eight CTAs each
    (1, 384, 1024, 17, GEMM),      # 16 steps: one CTA per row tile
    (2, 1024, 8192, 512, GEMM),    # the 70B k/v projection at batch 512: 32 tasks of four CTAs
    (2, 19200, 1024, 20, GEMM),    # 150 row tiles on 148 SMs: contiguous ranges of 16-column groups
    (2, 19100, 1024, 20, DEQ),
    (2, 11008, 1024, 40, GEMM),    # 86 row tiles: more than half the SMs, one CTA each
])
def test_gemm_split_contraction_across_a_cluster(K, M, N, batch, variant):
    """Layers with few output tiles: the CTAs of a cluster split the contraction of a tile and add their partial
    results through distributed shared memory (fixed order, so the result is deterministic)."""
    L = make_layer(M, N, K, key=(65, K, M, N))
    x = make_x(batch, N, key=(65, M, N, batch))
    y = run_layer(L, x, variant)
    if M * N * batch <= 2 ** 31:
        check_against_oracle(L, x, y, tight=variant != DEQ)
    else:                                           # large case: sampled rows, at least one in every 128-row tile
        rng = np.random.default_rng(0)
        rows = np.unique(np.concatenate([np.arange(0, 4), np.arange(126, 131), np.arange(M - 3, M), rng.integers(0, M, 24),
                                         np.arange(0, M, 128) + rng.integers(0, 128, (M + 127) // 128)]))
        rows = rows[rows < M]
        check_against_oracle(L, x, y, tight=variant != DEQ, rows=rows)
    y2 = run_layer(L, x, variant)
    assert np.array_equal(y.view(np.uint16), y2.view(np.uint16))


@pytest.mark.parametrize("K,M,N,batch", [
    (1, 77000, 64, 9),       # four or five row tiles in every CTA's range, one step each
    (2, 38000, 544, 13),     # six (row tile, slice) pairs a CTA: parts of row tiles at both ends, a whole one between, last step half
    (3, 25700, 288, 16),     # one or two passes (more of them: test_short_passes_are_published_complete)
])
def test_several_row_tiles_in_a_range(K, M, N, batch):
    """Up to 16 rows: passes alternate between two sets of accumulators, and all but a CTA's last are published beside the next."""
    L = make_layer(M, N, K, key=(65, K, M, N))
    x = make_x(batch, N, key=(65, M, N, batch))
    check_against_oracle(L, x, run_layer(L, x, GEMM))


@pytest.mark.parametrize("batch", [16, 40, 64, 65])
@pytest.mark.parametrize("N", [64, 160, 320, 384, 448, 1024])
def test_one_path_accumulators(N, batch):
    """One operand per step: one, two or four accumulators up to 16 rows, by the steps of the shortest pass (a last slice of one to four steps, fewer
    steps than accumulators); one or two beyond (four: test_four_accumulators)."""
    L = make_layer(700, N, 1, key=(66, N))
    x = make_x(batch, N, key=(66, N, batch))
    check_against_oracle(L, x, run_layer(L, x, GEMM))


@pytest.mark.parametrize("K,M,N,batch,variant,split", [
    (1, 14336, 1536, 33, GEMM, 1), (1, 14336, 1536, 64, GEMM, 1),    # 24 steps, the fewest
    (1, 9000, 1600, 48, GEMM, 1),                                    # 25 steps: a unit more in the first accumulator
    (1, 300, 16384, 33, GEMM, 8), (1, 600, 15488, 20, GEMM, 8),      # over clusters: 32 steps a CTA, 30 or 31
    (1, 14336, 1536, 48, DEQ, 1), (1, 600, 16384, 20, DEQ, 8),
])
def test_four_accumulators(K, M, N, batch, variant, split):
    """One path, more than 16 rows, a long contraction: a fourth issuing warp, the sums of four accumulators added."""
    import torch
    from tests.test_gemm_plan import plan
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        p = plan([(M, N)], K, batch, deq=int(variant == DEQ))
        assert (p.n_acc, p.split, p.stream) == (4, split, 0)
    L = make_layer(M, N, K, key=(70, K, M, N))
    x = make_x(batch, N, key=(70, N, batch))
    check_against_oracle(L, x, run_layer(L, x, variant), tight=variant != DEQ)


@pytest.mark.parametrize("K,shapes,variant,passes", [
    (1, [(56832, 64)], 0, 3),           # three passes of one unit in every CTA: of the four expanding groups one has no unit at all
    (1, [(128256, 64)], 0, 7),
    (2, [(128256, 64)], 0, 7),
    (2, [(128256, 128)], GEMM, 7),
    (2, [(128256, 64)], 4, 7),          # (dequantised: one unit a step)
    (3, [(57000, 64)], 0, 4),           # three paths: a fourth group that never has a unit
    (3, [(77000, 64)], 0, 5),
    (3, [(40000, 288)], GEMM, 3),
    (1, [(14336, 64)] * 4, 0, 4),
    (2, [(11008, 64)] * 4, 0, 3),
    (3, [(14336, 512)] * 3, 0, 3),
])
def test_short_passes_are_published_complete(K, shapes, variant, passes):
    """Ranges of several short passes, whose expanding warps are far ahead of the MMAs when they come to publish the last one: it must not be read
    before its MMAs are done.  Other activations in every call, and another layer in between, so that what an earlier launch left in
    tensor memory is never the right answer."""
    import torch
    import paper_2602_05367_b200 as rabit
    from tests.test_gemm_plan import plan
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 148:
        listed = plan(shapes, K, 16, deq=int(variant == 4)).passes[:, 0].tolist()
        assert max(listed.count(t) for t in set(listed)) == passes
    Ls = [make_layer(M, N, K, key=(67, i, K, M, N)) for i, (M, N) in enumerate(shapes)]
    between = make_layer(2560, 8192, K, key=(68, K))
    layers = [rabit.rabit_pack(L.planes, L.g, L.h) for L in Ls]
    other = rabit.rabit_pack(between.planes, between.g, between.h)
    xo = torch.from_numpy(make_x(16, 8192, key=(68,))).cuda()
    for layer in layers:
        layer.set_variant(variant)
    N = shapes[0][1]
    xs = [make_x(16, N, key=(67, N, i)) for i in range(4)]
    xd = [torch.from_numpy(x).cuda() for x in xs]
    ys = [[torch.zeros((16, M), dtype=torch.float16, device="cuda") for M, _ in shapes] for _ in xs]
    for i, x in enumerate(xd):
        if i & 1:
            rabit.rabit_linear(other, xo)
        if len(layers) == 1:
            rabit.rabit_linear(layers[0], x, ys[i][0])
        else:
            rabit.rabit_linear_group(layers, [x] * len(layers), ys[i])
    torch.cuda.synchronize()
    for x, y in zip(xs, ys):
        for L, layer, yl in zip(Ls, layers, y):
            assert layer.status() == 0, rabit.last_error()
            check_against_oracle(L, x, yl.cpu().numpy(), tight=variant != 4)
    for layer in layers + [other]:
        layer.free()


@pytest.mark.parametrize("K,batch,variant", [(1, 1, 0), (2, 2, 0), (3, 5, 0), (1, 9, 0), (2, 16, 0), (3, 16, 0), (1, 17, 0), (2, 40, 0), (3, 200, 0), (2, 16, DEQ), (2, 40, DEQ)])
def test_infinite_input_scale(K, batch, variant):
    """One infinite input scale: every output that it takes part in (all of them) is infinite or NaN, in every kernel."""
    M, N = 400, 1088
    L = make_layer(M, N, K, key=(69, K))
    L.h[K - 1, 77] = np.float16(np.inf)
    assert not np.isfinite(run_layer(L, make_x(batch, N, key=(69, batch)), variant)).any()
