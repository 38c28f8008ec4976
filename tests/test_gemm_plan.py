"""Host logic of the tcgen05 GEMM's work split, through the host-only view of it (no GPU): the passes that the kernel's own walk
yields must cover the layer exactly once, and the number of contributions at which an accumulate word counts as complete must
be the number that arrive.  The view and the kernel share the walk and the count."""
import collections
import ctypes
import random

import numpy as np
import pytest

import paper_2602_05367_b200 as rabit
from paper_2602_05367_b200 import binding

MAX_PASSES = 40000
Plan = collections.namedtuple("Plan", "tasks split stream seq max16 chunks stages n_acc passes")


def plan(shapes, K, batch, sms=148, deq=0, candidate=-1):
    lib = binding.raw_lib()
    M = np.array([s[0] for s in shapes], dtype=np.int32)
    N = np.array([s[1] for s in shapes], dtype=np.int32)
    head = np.zeros(8, dtype=np.int32)
    out = np.zeros((MAX_PASSES, 10), dtype=np.int32)
    n = lib.rabit_selftest_gemm_plan(len(shapes), M.ctypes.data, N.ctypes.data, K, deq, batch, sms, candidate, head.ctypes.data, out.ctypes.data, MAX_PASSES)
    return None if n < 0 else Plan(*(int(v) for v in head), out[:n])


def check_ranges(p, shapes, sms):
    """Contiguous ranges of (row tile, slice) pairs over all layers."""
    pairs = sum(-(-m // 128) * -(-n // 256) for m, n in shapes)
    assert 1 <= p.tasks <= min(sms, pairs) and p.split == 1
    assert len(set(p.passes[:, 0].tolist())) == p.tasks                               # no empty task
    assert sorted(p.passes[:, 0].tolist()) == p.passes[:, 0].tolist()
    at = 0
    for l, (m, n) in enumerate(shapes):
        steps = -(-n // 64)
        for rt in range(-(-m // 128)):
            lo, count, arrivals = 0, 0, set()
            while lo < steps:
                task, rank, pl, prt, c16, groups, s_lo, s_hi, path, arr = p.passes[at].tolist()
                assert (rank, pl, prt, c16, groups, path) == (0, l, rt, 0, 1, 0)
                assert s_lo == lo and s_lo % 4 == 0 and s_lo < s_hi <= steps and (s_hi % 4 == 0 or s_hi == steps)
                lo, count, at = s_hi, count + 1, at + 1
                arrivals.add(arr)
            assert arrivals == {count} and count <= 255
    assert at == len(p.passes)


def check_tiles(p, shape, K, batch):
    """Passes over 16-column groups, the steps of a pass shared by the CTAs of a cluster."""
    (m, n), n16 = shape, -(-batch // 16)
    steps, rts = -(-n // 64), -(-m // 128)
    cover = collections.defaultdict(list)
    for task, rank, l, rt, c16, groups, s_lo, s_hi, path, _ in p.passes.tolist():
        assert l == 0 and 0 <= rt < rts and 1 <= groups <= p.max16 and c16 + groups <= n16 and 0 <= rank < p.split
        for c in range(c16, c16 + groups):
            cover[rt, c, path].append((s_lo, s_hi, task, rank))
    assert set(cover) == {(rt, c, k) for rt in range(rts) for c in range(n16) for k in range(K if p.seq else 1)}
    for parts in cover.values():
        parts.sort()
        assert len(parts) == p.split and len({t for _, _, t, _ in parts}) == 1
        assert [r for _, _, _, r in parts] == list(range(p.split))
        assert parts[0][0] == 0 and parts[-1][1] == steps and all(a[1] == b[0] and a[0] < a[1] for a, b in zip(parts, parts[1:]))
    if p.split > 1:                                                                   # the exchange takes one pass (per path) of a task
        assert len(p.passes) == p.tasks * p.split * (K if p.seq else 1)
    assert 16 * p.max16 * (p.n_acc + p.seq) <= 512


def check(shapes, K, batch, sms=148, deq=0):
    p = plan(shapes, K, batch, sms, deq)
    assert p is not None
    if p.stream:
        check_ranges(p, shapes, sms)
    else:
        check_tiles(p, shapes[0], K, batch)
    return p


@pytest.mark.parametrize("K,M,N,batch,form", [
    (2, 28672, 8192, 16, "pairs"), (2, 4096, 4096, 9, "pairs"), (1, 1000, 8256, 16, "pairs"), (3, 33, 96, 9, "pairs"), (2, 129, 32, 16, "pairs"),
    (2, 200, 65280, 12, "pairs"),                                                     # 255 slices: the widest
    (2, 200, 65312, 12, "cluster"),                                                   # one more does not fit the arrival count
    (2, 14336, 4096, 48, "tiles"), (2, 128, 64, 17, "tiles"), (2, 28672, 8192, 512, "tiles"), (3, 13000, 2080, 209, "tiles"),
    (2, 20153, 2976, 46, "groups"), (2, 14336, 4096, 2048, "groups"), (3, 19544, 1440, 84, "groups"),
    (2, 300, 4096, 65, "cluster"), (3, 5000, 832, 24, "cluster"), (3, 5000, 13824, 200, "path after path"), (3, 2500, 8192, 200, "path after path"),
])
def test_the_split_covers_a_layer_once(K, M, N, batch, form):
    p = check([(M, N)], K, batch)
    assert form == ("pairs" if p.stream else "path after path" if p.seq else "cluster" if p.split > 1 else "tiles" if p.chunks else "groups")


def test_random_layers():
    rng = random.Random(7)
    for _ in range(400):
        K, sms, deq = rng.randint(1, 3), rng.choice((148, 148, 132, 7, 1)), rng.randint(0, 1)
        M, N = int(2 ** rng.uniform(0, 14)), 32 * max(1, int(2 ** rng.uniform(0, 9)))
        check([(M, N)], K, max(1, int(2 ** rng.uniform(0, 10))), sms, deq)


def test_random_groups_and_every_split_that_is_weighed():
    """Whatever the estimates prefer: a split that is weighed at all must be right.  (Layers of unlike widths, where equal parts
    for the widest one would be more tasks than there are pairs, among them.)"""
    rng = random.Random(8)
    groups = [[(128, 65280), (12800, 32)], [(128, 8192), (2560, 256), (2560, 256)]]
    for _ in range(250):
        groups.append([(int(2 ** rng.uniform(0, 13)), 32 * max(1, int(2 ** rng.uniform(0, 9)))) for _ in range(rng.randint(1, 4))])
    for shapes in groups:
        K, sms, batch = rng.randint(1, 3), rng.choice((148, 148, 132, 160, 5)), rng.randint(1, 16)
        check(shapes, K, batch, sms)
        for candidate in range(256):
            p = plan(shapes, K, batch, sms, candidate=candidate)
            if p is None:
                assert candidate >= 1
                break
            check_ranges(p, shapes, sms)


@pytest.mark.parametrize("K,M,N,tasks", [
    (2, 256, 512, 2), (2, 1024, 512, 8), (2, 2048, 512, 16), (3, 4096, 512, 32), (1, 3000, 1024, 24),    # publishing parts costs more than the slice it saves
    (2, 4096, 4096, 128), (3, 1024, 2048, 64), (1, 2048, 4096, 128),
    (2, 13824, 4096, 148), (3, 14336, 4096, 148),                                                        # a last pass in a range costs less than idle SMs
])
def test_what_the_estimates_choose_up_to_16_rows(K, M, N, tasks):
    """Splits that measure best on 148 SMs, most of them by 4 to 17 % over the one that a cheaper publishing or a dearer pass would choose."""
    assert plan([(M, N)], K, 16).tasks == tasks


@pytest.mark.parametrize("K,M,N,tasks", [(2, 700, 1024, 24), (2, 3000, 1024, 96)])
def test_what_they_choose_for_the_dequantised_form(K, M, N, tasks):
    """Its units take longer with every path: with those of one path such layers were not split, 700 x 1024 4.6 -> 5.7 us and 3000 x 1024 5.0 -> 5.75."""
    assert plan([(M, N)], K, 16, deq=1).tasks == tasks


@pytest.mark.parametrize("stream", [0, 1])
def test_nobody_waits_for_a_phase_further_off_than_the_next(stream):
    """A wait by parity cannot tell a phase from the one two before it, so a warp that waits for a barrier must wait for every phase
    of it in turn.  One phase completes per pass that the barrier belongs to; with ranges of pairs one group of warps publishes all passes but
    the last, another (which may come to it passes ahead of the MMAs) the last."""
    lib = binding.raw_lib()
    parity = ctypes.c_int()
    for passes in range(1, 12):
        ready = []
        for i in range(passes):
            ready.append((lib.rabit_selftest_gemm_ready(stream, i, passes, ctypes.byref(parity)), parity.value))
            assert ready[i][0] >= 0
        phase, of_bar = [], collections.Counter()
        for bar, _ in ready:
            phase.append(of_bar[bar])
            of_bar[bar] += 1
        for role in ([range(passes - 1), range(passes - 1, passes)] if stream else [range(passes)]):
            waited = collections.Counter()
            for i in role:
                bar, par = ready[i]
                assert phase[i] == waited[bar], f"pass {i} of {passes}: the wait is {phase[i] - waited[bar]} phases on from the last"
                assert par == phase[i] & 1
                waited[bar] += 1
    assert lib.rabit_selftest_gemm_ready(stream, 3, 3, ctypes.byref(parity)) == -1 and lib.rabit_selftest_gemm_ready(stream, 0, 1, None) == -1


def test_what_the_view_refuses():
    assert plan([(128, 64)], 4, 16) is None and plan([(128, 48)], 2, 16) is None and plan([(0, 64)], 2, 16) is None
    assert plan([(128, 64)] * 5, 2, 16) is None and plan([(128, 64)] * 2, 2, 17) is None and plan([(128, 64)], 2, 0) is None
    assert plan([(128, 64)], 2, 16, sms=513) is None and plan([(128, 64)], 2, 48, candidate=0) is None
    assert "rabit_selftest_gemm_plan" in rabit.last_error()
