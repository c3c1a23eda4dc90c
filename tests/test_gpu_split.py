"""How a launch's work is cut up: the segment search and the tile sizes at the
sizes where they can go wrong, element by element against the oracle."""
import numpy as np
import pytest
import torch

from parity import noise_abs_tol
from test_gpu_step import build_plan, compare, host_values, indices, make_params

pytestmark = pytest.mark.gpu


# The warp searches 32 table entries at a time: one step, the edges of one and two
# steps, and three steps, with tiles of one segment, of many and of the last one.
@pytest.mark.parametrize("nseg", [1, 2, 32, 33, 34, 65, 1023, 1026, 2500])
def test_segment_search(es, oracle, nseg):
    rng = np.random.default_rng(nseg)
    numels = [int(n) for n in rng.integers(1, 70, size=nseg)]
    numels[nseg // 2] = 3 * 8192 + 5
    numels[-1] = 8193
    tensors = make_params("bf16", numels, seed=nseg)
    plan, segs = build_plan(es, tensors)
    before = np.concatenate([host_values(t) for t in tensors])
    g = np.concatenate(indices(segs))
    es.es_perturb(plan, 21, 1e-3)
    torch.cuda.synchronize()
    got = np.concatenate([host_values(t) for t in tensors])
    compare("bf16", got, oracle.perturb(before, g, 21, 1e-3, "bf16"), f"{nseg} segments",
            noise_abs_tol([oracle.noise_at(21, g)], [1e-3]))
    plan.close()


# Passes whose CTAs have one row each, against the same tensors in a plan that a
# further, larger one takes out of that range, bit for bit: tables of one to three
# search steps, units at a segment's last elements, the high counter word changing
# inside the set, the largest set of one segment and the next one.
@pytest.mark.parametrize("dtype", ["bf16", "f32", "fp8"])
@pytest.mark.parametrize("nseg,total", [(1, 1), (1, 131_072), (1, 131_073), (2, 40), (3, 7_000),
                                        (31, 5_000), (32, 90_000), (33, 300),
                                        (40, 1_200_000), (1025, 40_000), (1100, 1_100_000)])
def test_one_row_passes(es, dtype, nseg, total):
    rng = np.random.default_rng(nseg + total)
    numels = [int(n) for n in rng.integers(1, max(2, 2 * total // nseg), size=nseg)]
    if nseg == 1:
        numels = [total]
    bases = [2**34 - 8 * (sum(numels) // 16)]
    for n in numels[:-1]:
        bases.append((bases[-1] + n + 7) // 8 * 8 + 8 * int(rng.integers(0, 3)))
    if dtype == "fp8":
        tensors = [torch.from_numpy(rng.integers(0, 120, size=n).astype(np.uint8)).cuda()
                   for n in numels]
        scales = [2.0**-9 * (1 + k % 5) for k in range(nseg)]
    else:
        tensors, scales = make_params(dtype, numels, seed=7), None
    more = torch.zeros(1 << 22, dtype=tensors[0].dtype, device="cuda")
    twins = [t.clone() for t in tensors]
    small = es.plan_from_tensors(tensors, bases, scales)
    large = es.plan_from_tensors(twins + [more], bases + [2**40], scales and scales + [1.0])
    for what in ("es_perturb", "es_restore_perturb", "flip"):
        for p in (small, large):
            if what == "es_perturb":
                es.es_perturb(p, 2**40 + 3, 1e-3)
            else:
                es.es_restore_perturb(p, 9, 1e-3, 9 if what == "flip" else 2**63, -1e-3)
        torch.cuda.synchronize()
        for x, y in zip(tensors, twins):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), what
    small.close()
    large.close()


# One segment long enough for runs of whole tiles and rows in every CTA, the
# high counter word changing inside it, against the same memory as many short
# segments (units found one by one): bit-identical everywhere, and equal to the
# oracle around the change, at both ends and on a sample.
@pytest.mark.parametrize("dtype", ["bf16", "f32", "fp8"])
@pytest.mark.parametrize("numel", [152 * 1024 * 64, 152 * 1024 * 64 + 4 * 1024 * 8 + 3])
def test_long_runs_equal_short_segments(es, oracle, dtype, numel):
    base = 2**34 - 8 * (numel // 17)
    scale = 2.0**-9
    if dtype == "fp8":
        rng = np.random.default_rng(3)
        codes = rng.integers(0, 120, size=numel).astype(np.uint8)
        a = torch.from_numpy(codes).cuda()
    else:
        (a,) = make_params(dtype, [numel], seed=3)
    b = a.clone()
    step = 8 * 1111 if dtype != "fp8" else 16 * 555
    pieces = [b[o:o + step] for o in range(0, numel, step)]
    scales = [scale] if dtype == "fp8" else None
    long_plan = es.plan_from_tensors([a], [base], scales)
    short_plan = es.plan_from_tensors(pieces, [base + o for o in range(0, numel, step)],
                                      scales and scales * len(pieces))
    edge = 2**34 - base
    at = np.unique(np.concatenate([
        np.arange(64), np.arange(edge - 9000, edge + 9000), np.arange(numel - 9000, numel),
        np.random.default_rng(4).integers(0, numel, size=20000)]))
    g = np.uint64(base) + at.astype(np.uint64)
    seeds = np.array([9, 2**40 + 1, 77, 4, 2**63, 5, 6, 8, 2**64 - 1], dtype=np.uint64)
    coeffs = np.array([2, -1, 0.5, 1, -0.5, 1.5, -2, 1, 0.25], dtype=np.float32) * np.float32(1e-3)

    def sample():
        return a.cpu().numpy()[at] if dtype == "fp8" else host_values(a)[at]

    def check(what, want, noise):
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), what
        if dtype == "fp8":
            from test_gpu_fp8 import assert_e4m3_close
            assert_e4m3_close(sample(), want, what, noise / scale)
        else:
            compare(dtype, sample(), want, what, noise)

    def both(call):
        before = sample()
        call(long_plan)
        call(short_plan)
        return before

    name, extra = ("e4m3", (scale,)) if dtype == "fp8" else (dtype, ())
    tol = noise_abs_tol([oracle.noise_at(9, g)], [1e-3])
    before = both(lambda p: es.es_perturb(p, 9, 1e-3))
    check("perturb", oracle.perturb(before, g, 9, 1e-3, name, *extra), tol)
    for second in (77, 9):
        both(lambda p: es.es_restore_perturb(p, 9, 1e-3, second, -1e-3))
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), "restore_perturb"
    # populations of 1 to 8 have passes of their own, 9 takes the seed loop
    for n in range(1, 10):
        before = both(lambda p: es.es_update(p, seeds[:n], coeffs[:n]))
        noise = noise_abs_tol([oracle.noise_at(int(s), g) for s in seeds[:n]], coeffs[:n])
        check(f"update {n}", oracle.update(before, g, seeds[:n], coeffs[:n], name, *extra), noise)
        # the fused call: one plan by it, the other by the two calls
        es.es_update_perturb(long_plan, seeds[:n], coeffs[:n], 5, 1e-3)
        es.es_update(short_plan, seeds[:n], coeffs[:n])
        es.es_perturb(short_plan, 5, 1e-3)
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), ("update_perturb", n)
    seeds, coeffs = seeds[:5], coeffs[:5]
    both(lambda p: es.es_update_perturb(p, seeds, coeffs, 5, 1e-3))
    both(lambda p: es.es_replay(p, np.tile(seeds, 30), np.tile(coeffs, 30), [1, 2, 3] * 25))
    torch.cuda.synchronize()
    assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), "update_perturb, replay"
    long_plan.close()
    short_plan.close()


# es_noise_fill for every way that index_base and out's 16-byte alignment can
# meet: the smallest counts, the edges of a row of 31 or 32 groups and of a pair of
# rows, and counts that fill every warp once and more often, across the change of the high counter
# word; bit-identical to one aligned fill, which the oracle checks.
@pytest.mark.parametrize("lead", [0, 1, 2, 3])
def test_noise_fill_alignments(es, oracle, lead):
    start = 2**34 - 4_000
    whole = torch.empty(3_000_016, device="cuda")
    es.es_noise_fill(31, start, whole.numel(), whole)
    at = np.unique(np.concatenate([np.arange(8_000), np.arange(0, whole.numel(), 97)]))
    want = oracle.noise_at(31, np.uint64(start) + at.astype(np.uint64))
    got = whole.cpu().numpy()[at].astype(np.float64)
    assert np.all(np.abs(got - want) <= 1e-5 * np.maximum(1.0, np.abs(want)))
    out = torch.empty(3_000_032, device="cuda")
    for skip in (0, 1, 2, 3, 3_998):
        for n in (1, 2, 3, 4, 5, 123, 124, 125, 127, 128, 129, 255, 256, 257, 4_001, 300_001,
                  452_353, 622_593, 904_703, 904_704, 904_705, 933_889, 3_000_001):
            if skip + n > whole.numel():
                continue
            out.fill_(7.0)
            es.es_noise_fill(31, start + skip, n, out[4 + lead:])
            torch.cuda.synchronize()
            assert torch.equal(out[4 + lead:4 + lead + n], whole[skip:skip + n]), (skip, n)
            assert torch.all(out[:4 + lead] == 7.0) and torch.all(out[4 + lead + n:] == 7.0)


# On both sides of the size from which a replayed generation gets a pass of its
# own: bit-identical to one es_update per generation.
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("numel", [2**25 - 8, 2**25])
def test_replay_passes(es, dtype, numel):
    a = torch.empty(numel, device="cuda").normal_(0.0, 0.02)
    a = a.to(torch.bfloat16) if dtype == "bf16" else a
    b = a.clone()
    counts = [1, 1, 2, 6, 1, 3, 140, 1, 2]
    seeds = np.arange(1, sum(counts) + 1, dtype=np.uint64)
    coeffs = np.linspace(-1e-3, 1e-3, seeds.size).astype(np.float32)
    coeffs[2:4] = [0.0, 1e-3]  # generation 2 has one non-zero seed
    plan_a, plan_b = es.plan_from_tensors([a]), es.plan_from_tensors([b])
    es.es_replay(plan_a, seeds, coeffs, counts)
    at = 0
    for n in counts:
        es.es_update(plan_b, seeds[at:at + n], coeffs[at:at + n])
        at += n
    torch.cuda.synchronize()
    assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    plan_a.close()
    plan_b.close()


# A launch may start before the kernel before it has ended. Behind every kind of
# work that a stream can hold (kernels of its own kind, other kernels, copies,
# fills, a join of two streams), eager and captured into a graph, the result is that
# of the same calls with the device synchronised in between.
@pytest.mark.parametrize("numel", [1000, 1 << 16, 3_000_001])
def test_launches_behind_other_work(es, numel):
    a = torch.empty(numel, device="cuda").normal_(0.0, 0.02)
    source, host = torch.randn(numel, device="cuda"), torch.randn(numel).pin_memory()
    start = a.clone()
    plan = es.plan_from_tensors([a])
    other = torch.empty(numel, device="cuda")
    seeds, coeffs = np.arange(6, dtype=np.uint64), np.full(6, 1e-3, dtype=np.float32)
    side = torch.cuda.Stream()

    def calls(wait):
        out = []
        for before in (lambda: a.copy_(start), lambda: a.copy_(host, non_blocking=True),
                       lambda: a.zero_(), lambda: a.add_(source),
                       lambda: es.es_noise_fill(5, 0, numel, a), lambda: fork()):
            before()
            wait()
            es.es_perturb(plan, 3, 1e-3)
            wait()
            es.es_restore_perturb(plan, 3, 1e-3, 4, 1e-3)
            wait()
            es.es_update(plan, seeds, coeffs)
            wait()
            es.es_update(plan, seeds[:2], coeffs[:2])
            wait()
            out.append(a.clone())
            wait()
        return out

    def fork():
        here = torch.cuda.current_stream()
        side.wait_stream(here)
        with torch.cuda.stream(side):
            es.es_noise_fill(6, 0, numel, other)
        a.mul_(0.5)
        here.wait_stream(side)

    want = calls(torch.cuda.synchronize)
    for got in (calls(lambda: None), calls(lambda: None)):
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(want, got))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = calls(lambda: None)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(want, got))
    plan.close()


# The same for every kernel that waits, in every storage type: the passes of one row,
# of runs and of several segments, sums alone and with a perturb, the seed loop in one
# generation, with a perturb and in several, the small sets' update, the fills and
# (eager only: a capture refuses them) es_perturb_noalloc's short and long tables.
@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("numel", [1000, 1 << 16, 3_000_001])
def test_every_kernel_behind_other_work(es, dtype, numel):
    torch.manual_seed(numel)
    values = torch.empty(3, numel, device="cuda").normal_(0.0, 0.02)
    scales = None
    if dtype == "bf16":
        values = values.to(torch.bfloat16)
    elif dtype == "fp8":
        values = (values * 2.0**9).to(torch.float8_e4m3fn).view(torch.uint8)
        scales = [2.0**-9]
    start, source, host = values[0].clone(), values[1].clone(), values[2].cpu().pin_memory()
    a = start.clone()
    # the same parameters as pieces of at least 16 elements
    step = max(16, numel // 70 // 16 * 16)
    bases = list(range(0, numel, step))
    pieces = [a[o:o + step] for o in bases]
    plan = es.plan_from_tensors([a], [0], scales)
    cut = es.plan_from_tensors(pieces, bases, scales and scales * len(pieces))
    segs = es.segments_from_tensors(pieces, bases)
    raw = {"f32": es.ES_FP32, "bf16": es.ES_BF16}.get(dtype)
    noise = torch.empty(numel, device="cuda")
    other = torch.empty(numel, device="cuda")
    seeds = np.arange(140, dtype=np.uint64) + 2**33
    coeffs = np.linspace(1e-3, 2e-3, 140).astype(np.float32)
    side = torch.cuda.Stream()

    def add(x):
        # another kernel that reads and writes the parameters
        if dtype == "fp8":
            a.bitwise_xor_(x & 1)
        else:
            a.add_(x)

    def fork():
        here = torch.cuda.current_stream()
        side.wait_stream(here)
        with torch.cuda.stream(side):
            es.es_noise_fill(6, 0, numel, other)
        add(source)
        here.wait_stream(side)

    def fill():
        es.es_noise_fill(5, 3, numel, a if dtype == "f32" else noise)
        if dtype != "f32":
            a.copy_(noise if dtype == "bf16" else source)

    calls_ = [
        lambda p: es.es_perturb(p, 3, 1e-3),
        lambda p: es.es_restore_perturb(p, 3, 1e-3, 4, 1e-3),
        lambda p: es.es_restore_perturb(p, 4, 1e-3, 4, -1e-3),
        lambda p: es.es_update(p, seeds[:6], coeffs[:6]),
        lambda p: es.es_update(p, seeds[:2], coeffs[:2]),
        lambda p: es.es_update_perturb(p, seeds[:2], coeffs[:2], 9, 1e-3),
        lambda p: es.es_update(p, seeds[:9], coeffs[:9]),
        lambda p: es.es_update(p, seeds[:129], coeffs[:129]),
        lambda p: es.es_update_perturb(p, seeds[:12], coeffs[:12], 9, 1e-3),
        lambda p: es.es_replay(p, seeds[:17], coeffs[:17], [2, 9, 1, 5]),
        lambda p: es.es_replay(p, seeds, coeffs, [70, 1, 69]),
    ]
    unplanned = [lambda: es.es_perturb_noalloc(segs[:40], raw, 8, 1e-3),
                 lambda: es.es_perturb_noalloc(segs, raw, 8, 1e-3)]

    def calls(wait, eager):
        out = []
        for before in (lambda: a.copy_(start), lambda: a.copy_(host, non_blocking=True),
                       lambda: a.zero_(), lambda: add(source), fill, fork):
            before()
            wait()
            for p in (plan, cut):
                for call in calls_:
                    call(p)
                    wait()
            for call in unplanned if eager and raw is not None else ():
                call()
                wait()
            out.append(a.clone())
            wait()
        return out

    def same(want, got):
        torch.cuda.synchronize()
        for x, y in zip(want, got):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))

    want = calls(torch.cuda.synchronize, True)
    for _ in range(2):
        a.copy_(start)
        same(want, calls(lambda: None, True))
    a.copy_(start)
    want = calls(torch.cuda.synchronize, False)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = calls(lambda: None, False)
    for _ in range(2):
        graph.replay()
        same(want, got)
    plan.close()
    cut.close()


# A kernel of another library behind a launch does not start early: it reads what the
# launch has written (es_noise_fill's buffer and an updated set, summed).
@pytest.mark.parametrize("numel", [1000, 1 << 16, 3_000_001])
def test_other_work_behind_launches(es, numel):
    a = torch.zeros(numel, device="cuda")
    plan = es.plan_from_tensors([a])
    out = torch.zeros(numel, device="cuda")
    seeds, coeffs = np.arange(9, dtype=np.uint64), np.full(9, 1e-3, dtype=np.float32)

    def calls(wait):
        got = []
        for call in (lambda: es.es_perturb(plan, 3, 1.0), lambda: es.es_update(plan, seeds, coeffs),
                     lambda: es.es_update(plan, seeds[:2], coeffs[:2]),
                     lambda: es.es_noise_fill(7, 1, numel, out)):
            a.zero_()
            out.zero_()
            wait()
            call()
            wait()
            got.append(a + out)
            wait()
        return got

    want = calls(torch.cuda.synchronize)
    for _ in range(3):
        got = calls(lambda: None)
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(want, got))
    plan.close()


# es_perturb_noalloc calls of up to 64 segments share nothing: on two streams at once,
# with different tables, each gives what its plan gives.
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_short_tables_on_two_streams(es, dtype):
    kind = es.ES_BF16 if dtype == "bf16" else es.ES_FP32
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    sets, twins, tables, plans = [], [], [], []
    for k, nseg in enumerate((64, 37)):
        tensors = make_params(dtype, [3_000 + 977 * i for i in range(nseg)], seed=k)
        twin = [t.clone() for t in tensors]
        plan, segs = build_plan(es, twin)
        sets.append(tensors)
        twins.append(twin)
        tables.append(es.segments_from_tensors(tensors, [s.index_base for s in segs]))
        plans.append(plan)
    torch.cuda.synchronize()
    for i in range(25):
        for k in (0, 1):
            es.es_perturb_noalloc(tables[k], kind, 100 * k + i, 1e-3, stream=streams[k])
    torch.cuda.synchronize()
    for i in range(25):
        for k in (0, 1):
            es.es_perturb(plans[k], 100 * k + i, 1e-3)
    torch.cuda.synchronize()
    for tensors, twin, plan in zip(sets, twins, plans):
        for x, y in zip(tensors, twin):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))
        plan.close()


# A plan is ready on every stream when it is handed out: used at once on a stream
# that does not synchronise with the default one and is still busy, its table (and
# FP8's scales) are those of the same call on a plan made long before.
@pytest.mark.parametrize("dtype", ["bf16", "fp8"])
def test_new_plan_on_a_busy_stream(es, dtype):
    n, pieces = 1 << 20, 900
    if dtype == "fp8":
        codes = np.random.default_rng(8).integers(0, 120, size=n).astype(np.uint8)
        a = torch.from_numpy(codes).cuda()
    else:
        (a,) = make_params("bf16", [n], seed=8)
    b, busy = a.clone(), torch.randn(1 << 24, device="cuda")
    step = n // pieces // 16 * 16
    bases = list(range(0, step * pieces, step))
    scales = [2.0**-9 * (1 + k % 7) for k in range(pieces)] if dtype == "fp8" else None
    old = es.plan_from_tensors([b[o:o + step] for o in bases], bases, scales)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for k in range(8):
        with torch.cuda.stream(side):
            busy.mul_(1.0)
            new = es.plan_from_tensors([a[o:o + step] for o in bases], bases, scales)
            es.es_perturb(new, k, 1e-3)
            es.es_perturb(old, k, 1e-3)
        torch.cuda.synchronize()
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), k
        new.close()
    old.close()


# The update of a small set, whose seeds are spread over warps: the same bits as
# in a plan that a further, larger tensor takes out of that range, and equal to the
# oracle; counts at the edges of a round of 8 and of 32 seeds, sets on both sides of
# the change between them and at the largest, ragged segments and a segment
# across the change of the high counter word.
@pytest.mark.parametrize("dtype", ["bf16", "f32", "fp8"])
@pytest.mark.parametrize("numels", [[1], [7, 1, 130, 16], [19_456], [19_457, 3], [5_000, 64_000]])
def test_small_set_update(es, oracle, dtype, numels):
    rng = np.random.default_rng(sum(numels))
    if dtype == "fp8":
        tensors = [torch.from_numpy(rng.integers(0, 120, size=n).astype(np.uint8)).cuda()
                   for n in numels]
        scales = [2.0**-9 * (k + 1) for k in range(len(numels))]
        more = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")
    else:
        tensors, scales = make_params(dtype, numels, seed=5), None
        more = torch.zeros(1 << 20, dtype=tensors[0].dtype, device="cuda")
    twins = [t.clone() for t in tensors]
    bases = [2**34 - 8 * (numels[0] // 16)]
    for n in numels[:-1]:
        bases.append((bases[-1] + n + 7) // 8 * 8 + 16)
    small = es.plan_from_tensors(tensors, bases, scales)
    large = es.plan_from_tensors(twins + [more], bases + [2**40], scales and scales + [1.0])

    def same(what):
        torch.cuda.synchronize()
        for x, y in zip(tensors, twins):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), what

    for n in (1, 4, 5, 7, 8, 9, 16, 31, 32, 33, 127, 128, 129):
        seeds = rng.integers(0, 2**63, size=n).astype(np.uint64)
        coeffs = (1e-3 * rng.standard_normal(n)).astype(np.float32)
        before = [t.cpu().numpy() if dtype == "fp8" else host_values(t) for t in tensors]
        for p in (small, large):
            es.es_update(p, seeds, coeffs)
        same(n)
        for k, t in enumerate(tensors if n in (5, 33) else []):
            g = np.arange(bases[k], bases[k] + numels[k], dtype=np.uint64)
            tol = noise_abs_tol([oracle.noise_at(int(s), g) for s in seeds], coeffs)
            if dtype == "fp8":
                from test_gpu_fp8 import assert_e4m3_close
                assert_e4m3_close(t.cpu().numpy(), oracle.update(before[k], g, seeds, coeffs, "e4m3",
                                                                 scales[k]), n, tol / scales[k])
            else:
                compare(dtype, host_values(t), oracle.update(before[k], g, seeds, coeffs, dtype),
                        f"{n} seeds", tol)
        for p in (small, large):
            es.es_update_perturb(p, seeds, coeffs, 77, 1e-3)
        same((n, "perturb"))
        counts = [n - n // 3, n // 3] if n >= 3 else [n]
        for p in (small, large):
            es.es_replay(p, seeds, coeffs, counts)
            es.es_replay(p, seeds, coeffs, [1] * n)
        same((n, "replay"))
    small.close()
    large.close()


# es_perturb_noalloc with its table in the launch's parameters (up to 64 segments) and
# in the static array (65), on a set of one SM's size and on one with long runs.
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("nseg,largest", [(1, 9_000_000), (64, 400), (64, 200_000), (65, 400)])
def test_noalloc_tables(es, dtype, nseg, largest):
    rng = np.random.default_rng(nseg)
    tensors = make_params(dtype, [int(n) for n in rng.integers(largest // 2, largest, size=nseg)])
    twins = [t.clone() for t in tensors]
    plan, segs = build_plan(es, tensors)
    segs_b = es.segments_from_tensors(twins, [s.index_base for s in segs])
    for sigma in (1e-3, -1e-3, 0.05):
        es.es_perturb(plan, 2**50 + 1, sigma)
        es.es_perturb_noalloc(segs_b, es.ES_BF16 if dtype == "bf16" else es.ES_FP32, 2**50 + 1,
                              sigma)
    torch.cuda.synchronize()
    for x, y in zip(tensors, twins):
        assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))
    plan.close()
