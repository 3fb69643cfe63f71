"""Edges of the size rules by which the library picks a kernel variant or the shape of a launch, against the oracle."""
import numpy as np
import pytest
import torch

from paper_2605_11354_b200 import binding as lt
from paper_2605_11354_b200 import workloads as wk

from oracle import sla_oracle as orc

import parity_util as pu
from test_gpu_parity import full_parity, oracle_subset, small_workload

pytestmark = pytest.mark.gpu


def launches(call):
    """Name, grid, block and shared memory of the kernels that call() launches, from a captured graph of it."""
    from cuda.bindings import driver

    def ok(result):
        assert result[0] == driver.CUresult.CUDA_SUCCESS, result[0]
        return result[1] if len(result) == 2 else result[1:]

    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = driver.CUgraph(graph.raw_cuda_graph())
    count = ok(driver.cuGraphGetNodes(raw))[1]
    found = []
    for node in ok(driver.cuGraphGetNodes(raw, count))[0]:
        if ok(driver.cuGraphNodeGetType(node)) == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            p = ok(driver.cuGraphKernelNodeGetParams(node))
            name = ok(driver.cuFuncGetName(p.func) if int(p.func) else driver.cuKernelGetName(p.kern)).decode()
            found.append((name, (p.gridDimX, p.gridDimY, p.gridDimZ), p.blockDimX, p.sharedMemBytes))
    return sorted(found)


@pytest.mark.parametrize("block,batch,heads,tokens", [(64, 37, 12, 128), (64, 89, 5, 65), (64, 23, 29, 200), (128, 89, 5, 100)])
def test_attention_grids_around_the_number_of_resident_ctas(block, batch, heads, tokens):
    """444, 445, 1334 and 445 attention tiles: three per SM are resident, from one more on CTAs take over tiles."""
    wl = small_workload(f"steal{batch}", batch=batch, heads=heads, tokens=tokens, block=block, crit=0.5, neg=0.3)
    inputs = wk.make_inputs(wl)
    eng, out = pu.run_gpu(inputs, wl)
    ref = oracle_subset(inputs, wl, list(range(heads)), cls=eng.plan.cls.cpu().numpy())
    rel, mx = pu.output_errors(out.cpu().numpy(), ref["out"])
    assert rel <= pu.REL_L2_TOL and mx <= pu.MAX_ABS_TOL
    again = torch.empty_like(out)
    eng.forward(torch.from_numpy(inputs["proj"]).cuda(), out=again)
    assert torch.equal(again, out)  # whichever CTA computes a tile


@pytest.mark.parametrize("crit,neg", [(0.0, 1.0), (1.0, 0.0), (0.4, 0.6)])
@pytest.mark.parametrize("block,batch,heads,tokens", [(64, 37, 12, 128), (64, 89, 5, 65), (128, 89, 5, 100), (64, 8, 16, 6397)])
def test_attention_without_products_on_grids_of_any_size(block, batch, heads, tokens, crit, neg):
    """444, 445, 445 and 6400 attention tiles that have nothing to multiply, in the forward (no critical and no marginal
    block) and in the linear branch alone (no marginal block, a dense plan among them): zeros in every row."""
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn((batch, heads, tokens, 64), device="cuda", generator=g).to(torch.bfloat16) for _ in range(3))
    proj = torch.randn((heads, 64, 64), device="cuda", generator=g)
    eng = lt.SlaForward(batch, heads, tokens, block, crit, neg, out_dtype=torch.bfloat16)
    assert eng.plan.k_marg == 0
    eng.run(q, k, v, proj)
    out = torch.full((batch, heads, tokens, 64), float("nan"), device="cuda")
    if crit == 0.0:
        eng.run(q, k, v, proj, out=out)
        torch.cuda.synchronize()
        assert eng.status.item() == 0 and torch.count_nonzero(out).item() == 0  # (NaN counts as non-zero)
        out.fill_(float("nan"))
    nbytes = lt.lite3r_train_workspace(eng.shape, crit, neg)
    raw = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    lt.lite3r_sla_linear_branch(eng.q8, eng.k8, eng.v8, eng.shape, eng.phi, eng.plan, out, raw[(-raw.data_ptr()) % 256:][:nbytes],
                                eng.status)
    torch.cuda.synchronize()
    assert eng.status.item() == 0 and torch.count_nonzero(out).item() == 0


@pytest.mark.parametrize("block", [64, 128])
def test_many_buffer_sets_in_turn(block):
    """Encoded tensor maps are kept for a few hundred buffers: more sets than that, at addresses that come and go, give the
    same bytes."""
    wl = small_workload(f"maps{block}", heads=2, tokens=300, block=block)
    inputs = wk.make_inputs(wl)
    first, hold = None, []
    for i in range(400):
        eng, out = pu.run_gpu(inputs, wl)
        first = out.clone() if first is None else first
        assert torch.equal(out, first)
        if i % 3:
            hold.append(eng)  # some buffers stay, the others' addresses are taken over


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("crit,neg", [(0.1, 0.6), (0.25, 0.75), (0.0, 0.5), (0.0, 1.0)])
@pytest.mark.parametrize("heads,tokens", [(16, 1374), (1, 30000)])
def test_calls_behind_event_waits(heads, tokens, crit, neg, captured):
    """Every kernel is a programmatic dependent, also where its stream has just waited for an event and, captured, where a
    graph's branches fork and join: two streams share one step (K and V quantised and the first half of the forward on a
    side stream, the plan on the main one), with summaries longer than the plan and the other way round, and with a copy
    in front.  What a kernel reads too early holds wrong values here, but no wrong index."""
    g = torch.Generator(device="cuda").manual_seed(2)
    sets = [[torch.randn((1, heads, tokens, 64), device="cuda", generator=g).to(torch.bfloat16) for _ in range(3)] for _ in range(2)]
    proj = torch.randn((heads, 64, 64), device="cuda", generator=g) / 8
    eng = lt.SlaForward(1, heads, tokens, 64, crit, neg)
    want = [eng.run(*x, proj).clone() for x in sets]
    q, k, v = (torch.empty_like(x) for x in sets[0])
    host = torch.empty_like(q, device="cpu").pin_memory()
    side = torch.cuda.Stream()

    def step():
        main = torch.cuda.current_stream()
        q.copy_(host, non_blocking=True)
        side.wait_stream(main)
        lt.lite3r_quantize_fp8(q, eng.shape, eng.q8, main)
        lt.lite3r_quantize_fp8(k, eng.shape, eng.k8, side)
        lt.lite3r_quantize_fp8(v, eng.shape, eng.v8, side)
        main.wait_stream(side)
        side.wait_stream(main)
        lt.lite3r_sla_forward_begin(eng.k8, eng.v8, proj, eng.shape, eng.phi, eng.plan, eng.workspace, eng.status, side)
        eng.make_plan(main)
        main.wait_stream(side)
        lt.lite3r_sla_forward_finish(eng.q8, eng.k8, eng.v8, eng.shape, eng.phi, eng.plan, eng.out, eng.workspace, eng.status, main)

    run = step
    if captured:
        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            step()
        run = graph.replay
    for i in range(12):
        for dst, src in zip((host, k, v), sets[i % 2]):
            dst.copy_(src)
        for t in (eng.workspace, eng.out.view(torch.uint8), eng.q8.codes, eng.k8.codes, eng.v8.codes):
            t.fill_(0xEE)
        eng.plan.cls.zero_()
        eng.plan.crit_idx.zero_()
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        assert eng.status.item() == 0 and torch.equal(eng.out, want[i % 2]), i


@pytest.mark.parametrize("call", ["run", "run_graph"])
def test_an_engine_changed_between_two_calls(call):
    """A step works on the buffers, strides, shape and settings of its call, not on those of the call before."""
    g = torch.Generator(device="cuda").manual_seed(3)
    B, H, N = 2, 4, 256
    args = [torch.randn((B, N, H, 64), device="cuda", generator=g) for _ in range(3)]
    proj = torch.randn((H, 64, 64), device="cuda", generator=g) / 8
    heads_first = [t.view(B, H, N, 64) for t in args]

    def fresh(x, phi="softmax", batch=B):
        return lt.SlaForward(batch, H, N, 64, 0.25, 0.25, phi=phi).run(*x, proj)

    eng = lt.SlaForward(B, H, N, 64, 0.25, 0.25)
    step = lambda x: getattr(eng, call)(*x, proj)  # noqa: E731
    assert torch.equal(step(heads_first), fresh(heads_first))
    mixed = [args[0].permute(0, 2, 1, 3), *heads_first[1:]]  # the same address with other strides
    assert torch.equal(step(mixed), fresh(mixed))
    held = []
    for obj, name in ((eng.q8, "codes"), (eng.k8, "scales"), (eng.k8, "colsum"), (eng.v8, "codes"), (eng.plan, "cls"),
                      (eng.plan, "crit_idx"), (eng, "workspace"), (eng, "out")):
        t = getattr(obj, name)
        old, new = t.view(t.shape), torch.zeros_like(t)
        held.append(old)
        t.set_(new)
        assert torch.equal(step(heads_first), fresh(heads_first)), name
        assert torch.count_nonzero(new) > 0, name  # the step wrote to the new storage
    eng.phi = lt.PHI_ELU1
    assert torch.equal(step(heads_first), fresh(heads_first, phi="elu1"))
    eng.phi = lt.PHI_SOFTMAX
    eng.shape.batch = 1
    eng.out.fill_(float("nan"))
    out = step(heads_first)
    assert torch.equal(out[:1], fresh([t[:1] for t in heads_first], batch=1)) and torch.isnan(out[1:]).all()


@pytest.mark.parametrize("blocks", [3, 32, 33, 64, 65])
def test_plan_rows_around_the_rank_limit(blocks):
    """Rows of up to 64 blocks are ranked by comparing all pairs (one or two entries per lane), longer ones selected
    through histograms."""
    wl = small_workload(f"rank{blocks}", heads=2, tokens=blocks * 64 - 3, crit=0.2, neg=0.3)
    full_parity(wl, wk.make_inputs(wl), query_blocks=pu.sample_blocks(wl, [0, 1], 4))


@pytest.mark.parametrize("spread", [1e-4, 3e-2])
@pytest.mark.parametrize("block,blocks", [(64, 150), (128, 131)])
def test_plan_scores_closer_than_their_approximation(spread, block, blocks):
    """Sixteen rows per CTA work on approximate scores: key blocks whose exact scores differ by less than the
    approximation's error have to come out in the exact order all the same."""
    g = np.random.default_rng(17)
    wl = small_workload(f"close{blocks}", heads=1, tokens=blocks * block - 5, block=block, crit=0.2, neg=0.5, src_dtype="f32")
    inputs = wk.make_inputs(wl)
    for name in ("q", "k"):
        inputs[name] = (1.0 + spread * g.standard_normal(inputs[name].shape)).astype(np.float32)
    plans = []
    try:
        for variant in (1, 3):
            lt.lite3r_plan_variant(variant)
            eng, _ = pu.run_gpu(inputs, wl)
            plans.append([t.cpu().numpy() for t in (eng.plan.cls, eng.plan.crit_idx, eng.plan.marg_idx)])
    finally:
        lt.lite3r_plan_variant(0)
    assert all(np.array_equal(a, b) for a, b in zip(*plans))


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("blocks", [81, 96, 97, 255, 256, 257, 513])
def test_plan_from_places_equals_plan_from_exact_keys(blocks, block):
    """Rows from the shortest that the approximate scores serve, around whole and ragged groups of 8 and 256 entries, a
    last block of one token, rows without a single place (queries of zero), lists that are empty, full, or share their
    threshold: the same plan bit for bit as from 64-bit keys of every entry."""
    g = np.random.default_rng(blocks)
    wl = small_workload(f"places{blocks}", heads=3, tokens=(blocks - 1) * block + 1, block=block, src_dtype="f32")
    inputs = wk.make_inputs(wl)
    inputs["q"][:, 0, 2 * block:3 * block] = 0.0
    inputs["k"][:, 1] *= np.exp(2.0 * g.standard_normal((1, wl.tokens, 1))).astype(np.float32)  # key blocks of very different scale
    inputs["k"][:, 2, block:2 * block] = inputs["k"][:, 2, :block]
    try:
        for crit, neg in ((0.1, 0.6), (0.0, 0.4), (0.3, 0.7), (0.05, 0.0), (1.0, 0.0), (0.0, 1.0)):
            plans = []
            for variant in (1, 0, 2):
                lt.lite3r_plan_variant(variant)
                eng, _ = pu.run_gpu(inputs, wl, crit=crit, neg=neg)
                plans.append([t.cpu().numpy() for t in (eng.plan.cls, eng.plan.crit_idx, eng.plan.marg_idx)])
            for other in plans[1:]:
                assert all(np.array_equal(a, b) for a, b in zip(plans[0], other)), (crit, neg)
    finally:
        lt.lite3r_plan_variant(0)


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("blocks", [200, 257, 520])
def test_plan_ranges_too_full_for_a_list(blocks, block):
    """Many key blocks of a scale far above the others' and scores that differ by little leave most of a row in a few of the 16-bit
    places (up to 32 such key blocks are placed by themselves): more undecided entries at a threshold than a list holds, both thresholds among the same ones, ties that the exact
    keys leave, for critical and marginal blocks at once or one after the other.  The same plan bit for bit as from 64-bit
    keys of every entry."""
    g = np.random.default_rng(blocks)
    wl = small_workload(f"full{blocks}", heads=8, tokens=(blocks - 1) * block + 3, block=block, src_dtype="f32")
    inputs = wk.make_inputs(wl)
    q, k = inputs["q"], inputs["k"]
    k[:, 0, 3 * block + 1] *= 30.0
    k[:, 1, 3 * block + 1] *= 1000.0
    q[:, 2], k[:, 2] = (1.0 + 0.01 * g.standard_normal((2, 1) + q[:, 2].shape[1:])).astype(np.float32)
    period = 5 * block
    k[:, 3] = k[:, 3, np.arange(wl.tokens) % period]  # every block again and again
    k[:, 3, 3 * block + 1] *= 300.0
    for head, large, times in ((4, 32, 50.0), (5, 33, 50.0), (6, 40, 2000.0)):  # as many as have their places made exactly, and more
        k[:, head, 5 * block:(5 + large) * block:block] *= times
    k[:, 7, -1] *= 100.0  # the last block, of three tokens
    try:
        for crit, neg in ((0.1, 0.6), (0.0, 0.4), (0.3, 0.7), (0.05, 0.0), (0.3, 0.69), (0.01, 0.98)):
            plans = []
            for variant in (1, 3, 2):
                lt.lite3r_plan_variant(variant)
                eng, _ = pu.run_gpu(inputs, wl, crit=crit, neg=neg)
                plans.append([t.cpu().numpy() for t in (eng.plan.cls, eng.plan.crit_idx, eng.plan.marg_idx)])
            for other in plans[1:]:
                assert all(np.array_equal(a, b) for a, b in zip(plans[0], other)), (crit, neg)
    finally:
        lt.lite3r_plan_variant(0)


@pytest.mark.parametrize("scale", [float("inf"), float("nan"), 3e38, 0.0])
def test_plan_with_extreme_scales(scale):
    """A key block whose scale is not finite, next to overflow or zero, for ordinary queries and a block of zeros (zero times
    infinity among its scores): the same plan bit for bit as from 64-bit keys of every entry."""
    wl = small_workload("extreme", heads=2, tokens=140 * 64 - 7, crit=0.1, neg=0.6)
    inputs = wk.make_inputs(wl)
    inputs["q"][:, 0, 3 * 64:4 * 64] = 0.0
    eng, _ = pu.run_gpu(inputs, wl)
    eng.k8.scales[0, 0, 9] = scale
    plans = []
    try:
        for variant in (1, 3, 2):
            lt.lite3r_plan_variant(variant)
            eng.plan.cls.fill_(-1)
            eng.make_plan()
            plans.append([t.cpu().numpy().copy() for t in (eng.plan.cls, eng.plan.crit_idx, eng.plan.marg_idx)])
    finally:
        lt.lite3r_plan_variant(0)
    for other in plans[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(plans[0], other))


@pytest.mark.parametrize("times", [10.0, 30.0])
def test_plan_time_with_one_large_key(times):
    """One key token that much larger than the others (an attention sink) leaves fewer places to all other blocks.  687 blocks
    took 4.4 and 15 times as long with it; placed by itself it leaves the others theirs, and the time is 1.25 times."""
    shape = lt.Shape(1, 16, 687 * 64, 64, 64)
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k = (torch.randn((1, 16, shape.tokens, 64), device="cuda", generator=g) for _ in range(2))
    q8, k8, plan = lt.alloc_fp8(shape, "cuda"), lt.alloc_fp8(shape, "cuda"), lt.alloc_plan(shape, 0.05, 0.75, "cuda")
    lt.lite3r_quantize_fp8(q, shape, q8)

    def shortest():
        lt.lite3r_quantize_fp8(k, shape, k8)
        best = float("inf")
        for _ in range(6):
            start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            start.record()
            for _ in range(10):
                lt.lite3r_sla_plan(q8, k8, shape, 0.05, 0.75, plan)
            end.record()
            end.synchronize()
            best = min(best, start.elapsed_time(end))
        return best

    plain = shortest()
    k[:, :, 7 * 64 + 3] *= times
    assert shortest() < 2.0 * plain


def test_plan_rows_per_cta_around_one_cta_per_sm():
    """Eight rows per CTA as long as that is one CTA per SM, sixteen from one row more on: the same plan as from 64-bit keys."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for blocks in (8 * sms, 8 * sms + 1):
        wl = small_workload(f"rows{blocks}", heads=1, tokens=blocks * 64 - 9, crit=0.05, neg=0.6)
        inputs = wk.make_inputs(wl)
        eng, _ = pu.run_gpu(inputs, wl)
        (_, grid, threads, _), = launches(eng.make_plan)
        assert (threads, grid[0]) == ((256, sms) if blocks == 8 * sms else (512, -(-blocks // 16)))
        got = [t.clone() for t in (eng.plan.cls, eng.plan.crit_idx, eng.plan.marg_idx)]
        try:
            lt.lite3r_plan_variant(1)
            eng.make_plan()
        finally:
            lt.lite3r_plan_variant(0)
        assert all(torch.equal(x, y) for x, y in zip(got, (eng.plan.cls, eng.plan.crit_idx, eng.plan.marg_idx)))


@pytest.mark.parametrize("blocks", [13592, 13593])
def test_plan_of_the_longest_rows(blocks):
    """The longest row that fits as 16-bit places and the first that gets one row per CTA (from there on the kernel that the
    hook forces as variant 4): classes and lists of sampled rows from exact scores."""
    tokens, kc = blocks * 64 - 5, round(0.002 * blocks)
    shape = lt.Shape(1, 1, tokens, 64, 64)
    g = torch.Generator(device="cuda").manual_seed(blocks)
    q8, k8 = lt.alloc_fp8(shape, "cuda"), lt.alloc_fp8(shape, "cuda")
    for out in (q8, k8):
        lt.lite3r_quantize_fp8(torch.randn((1, 1, tokens, 64), device="cuda", generator=g, dtype=torch.bfloat16), shape, out)
    k8.colsum[0, 0, 7] = k8.colsum[0, 0, 3]  # a tie
    k8.scales[0, 0, 7] = k8.scales[0, 0, 3]
    plan = lt.alloc_plan(shape, 0.002, 0.99, "cuda")
    calls = []
    try:
        for variant in (0, 4):
            lt.lite3r_plan_variant(variant)
            plan.cls.fill_(-1)
            lt.lite3r_sla_plan(q8, k8, shape, 0.002, 0.99, plan)
            calls.append(launches(lambda: lt.lite3r_sla_plan(q8, k8, shape, 0.002, 0.99, plan)))
            rows = torch.tensor([0, 1, blocks // 2, blocks - 2, blocks - 1], device="cuda")
            valid = torch.full((blocks,), 64.0, device="cuda", dtype=torch.float64)
            valid[-1] = 59.0
            scores = q8.colsum[0, 0, rows].double() @ k8.colsum[0, 0].double().T * (k8.scales[0, 0].double() / valid)
            rank = torch.argsort(torch.argsort(-scores, dim=1, stable=True), dim=1)
            want = torch.where(rank < plan.k_crit, 2, torch.where(rank < blocks - plan.k_neg, 1, 0)).to(torch.int8)
            assert plan.k_crit == kc and torch.equal(plan.cls[0, 0, rows], want)
            assert torch.equal(plan.crit_idx[0, 0, rows].long(), (want == 2).nonzero()[:, 1].view(len(rows), -1))
            assert torch.equal(plan.marg_idx[0, 0, rows].long(), (want == 1).nonzero()[:, 1].view(len(rows), -1))
    finally:
        lt.lite3r_plan_variant(0)
    assert (calls[0] == calls[1]) == (blocks > 13592)


@pytest.mark.parametrize("blocks", [64, 65, 128, 129, 193])
def test_aggregation_inside_one_sequence(blocks):
    """Key chunks of 64 that end with, before and after the row, row tiles of 128 full and ragged."""
    wl = small_workload(f"agg{blocks}", heads=3, tokens=blocks * 64, crit=0.05, neg=0.2)
    full_parity(wl, wk.make_inputs(wl), query_blocks=pu.sample_blocks(wl, [0, 2], 6))


@pytest.mark.parametrize("batch,heads,blocks", [(40, 5, 1), (67, 3, 2), (50, 4, 3), (31, 7, 5), (40, 11, 21), (3, 2, 260)])
def test_aggregation_tiles_of_persistent_ctas(batch, heads, blocks):
    """Row tiles that run through many sequences of one to five key blocks (also fewer than four, where a step of four rows
    skips whole sequences), and several tiles per CTA, inside a sequence and through the boundaries: ring and accumulators
    go round."""
    wl = small_workload(f"aggp{blocks}", batch=batch, heads=heads, tokens=blocks * 64 - 7, crit=0.0 if blocks == 1 else 0.2,
                        neg=0.0 if blocks < 3 else 0.3)
    full_parity(wl, wk.make_inputs(wl), query_blocks=pu.sample_blocks(wl, [0, heads - 1], min(150, batch * blocks)))


@pytest.mark.parametrize("batch,heads,blocks", [(3, 43, 1), (32, 32, 1), (23, 3, 5), (16, 4, 15), (28, 1, 36), (9, 3, 37), (6, 19, 9),
                                                 (32, 64, 1), (31, 7, 5), (16, 4, 22), (41, 7, 7), (64, 4, 8), (3, 683, 1)])
def test_aggregation_tiles_whose_masks_are_made_at_once(batch, heads, blocks):
    """Tiles through the (b, h) boundaries, one or two to a CTA: 129 rows, 1024 rows (the most that are one tile per SM), rows that
    start at every byte of a word, tiles that begin and end inside a sequence, 1026 rows, where there are more tiles than SMs,
    up to 2048 rows, where there are twice as many, tiles of one to four chunks (two tiles then go once or twice around the ring), and
    2049 rows, where the general form follows.  The same output from class bytes at odd addresses."""
    wl = small_workload(f"once{blocks}", batch=batch, heads=heads, tokens=blocks * 64 - 7, crit=0.0 if blocks == 1 else 0.2,
                        neg=0.0 if blocks < 3 else 0.3)
    inputs = wk.make_inputs(wl)
    eng, out = full_parity(wl, inputs, query_blocks=pu.sample_blocks(wl, [0, heads - 1], min(60, batch * blocks)))
    proj, want, cls = torch.from_numpy(inputs["proj"]).cuda(), out.clone(), eng.plan.cls
    for shift in (1, 2, 3):
        raw = torch.ones(cls.numel() + 8, dtype=torch.int8, device="cuda")  # marginal all round
        eng.plan.cls = raw[shift:shift + cls.numel()].view(cls.shape)
        eng.plan.cls.copy_(cls)
        assert torch.equal(eng.forward(proj, out=torch.empty_like(out)), want), shift
    assert int(eng.status.item()) == 0


@pytest.mark.parametrize("batch,heads,tokens,block,crit", [(1, 16, 1374, 64, 0.25), (3, 5, 3001, 128, 0.15), (1, 16, 832, 64, 0.1),
                                                           (1, 12, 1374, 128, 0.25), (2, 16, 1374, 64, 0.25), (1, 4, 12016, 64, 0.15),
                                                           (1, 8, 629, 64, 0.15), (1, 8, 3000, 64, 0.05), (1, 8, 4122, 64, 0.1)])
def test_aggregation_beside_the_attention_kernel(batch, heads, tokens, block, crit):
    """Attention grids that fit on the SMs a narrower aggregation leaves free, and grids that do not: the same output every
    time, and the same sums over the marginal blocks as from a plan without critical blocks, whose aggregation gets all SMs."""
    wl = small_workload("beside", batch=batch, heads=heads, tokens=tokens, block=block, crit=crit, neg=0.5)
    inputs = wk.make_inputs(wl)
    eng, out = pu.run_gpu(inputs, wl)
    want = out.clone()
    offsets = lt.lite3r_workspace_layout(eng.shape, wl.crit, wl.neg)
    sums = eng.workspace[offsets[1]:offsets[3]]
    proj = torch.from_numpy(inputs["proj"]).cuda()
    for _ in range(3):
        sums.fill_(0xEE)
        eng.forward(proj, out=out)
        assert torch.equal(out, want)
    beside = sums.clone()
    plan = eng.plan
    plan.k_crit, plan.k_neg = 0, plan.k_crit + plan.k_neg
    sums.fill_(0xEE)
    lt.lite3r_sla_forward(eng.q8, eng.k8, eng.v8, proj, eng.shape, eng.phi, plan, out, eng.workspace, eng.status)
    assert int(eng.status.item()) == 0
    assert torch.equal(sums, beside)


@pytest.mark.parametrize("batch,heads,tokens,block,crit", [(1, 16, 1374, 64, 0.25), (3, 5, 3001, 128, 0.15), (1, 2, 512, 64, 0.25)])
def test_stage_times_are_those_of_the_launches_of_any_call(batch, heads, tokens, block, crit):
    """Grid, block and shared memory of every kernel of a forward, without and with stage times."""
    eng = lt.SlaForward(batch, heads, tokens, block, crit, 0.5)
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k, v = (torch.randn((batch, heads, tokens, 64), device="cuda", generator=g) for _ in range(3))
    proj = torch.randn((heads, 64, 64), device="cuda", generator=g)
    eng.run(q, k, v, proj)
    torch.cuda.synchronize()

    plain = launches(lambda: eng.forward(proj))
    lt.profile_enable(True)
    try:
        timed = launches(lambda: eng.forward(proj))
    finally:
        lt.profile_enable(False)
    assert len(plain) == 3 and timed == plain


@pytest.mark.parametrize("heads,tokens,crit", [(8, 629, 0.15), (8, 1374, 0.25), (16, 832, 0.1), (8, 3000, 0.05)])
def test_aggregation_leaves_room_for_the_attention_grid(heads, tokens, crit):
    """Where one round of tiles through the (b, h) boundaries leaves SMs on which the whole attention grid fits, three CTAs to
    an SM, the aggregation takes no more than that, although tiles inside the (b, h) are shorter for themselves."""
    eng = lt.SlaForward(1, heads, tokens, 64, crit, 0.6)
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k, v = (torch.randn((1, heads, tokens, 64), device="cuda", generator=g) for _ in range(3))
    proj = torch.randn((heads, 64, 64), device="cuda", generator=g)
    eng.run(q, k, v, proj)
    grids = {name: grid[0] for name, grid, *_ in launches(lambda: eng.forward(proj))}
    aggregation, = (n for name, n in grids.items() if "aggregate" in name)
    attention, = (n for name, n in grids.items() if "attention" in name)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert attention <= 3 * (sms - aggregation)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("rows,d_in,d_out", [(18944, 256, 256), (18945, 256, 256), (9473, 1024, 512), (2500, 1152, 1984)])
def test_linear_tiles_around_one_per_sm(rows, d_in, d_out, dtype):
    """148 tiles of 128 x 256 are one per SM; from one more on, pairs of CTAs take tiles of 256 x 256: an odd number of row
    tiles, last tiles of one row, last column tiles of less than half a tile."""
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((rows, d_in), device="cuda", generator=g)
    w = torch.randn((d_out, d_in), device="cuda", generator=g) / d_in ** 0.5
    (xc, xs), (wc, ws) = lt.lite3r_quantize_rows_fp8(x), lt.lite3r_quantize_rows_fp8(w)
    y, status = torch.empty((rows, d_out), device="cuda", dtype=dtype), torch.zeros(1, dtype=torch.int32, device="cuda")
    lt.lite3r_linear_fp8(xc, xs, wc, ws, None, y, status)
    pick = sorted({0, 1, rows - 1, *range(127, rows, 64)})
    ref = orc.linear_fp8(*(t.cpu().numpy() for t in (xc[pick], xs.reshape(-1)[pick], wc, ws)))
    assert status.item() == 0
    tol = 1e-5 if dtype == torch.float32 else 5e-3
    np.testing.assert_allclose(y[pick].float().cpu().numpy(), ref, rtol=tol, atol=1e-5 * np.abs(ref).max())


@pytest.mark.parametrize("low", [1, 3, -2])
def test_codes_next_to_rounding_boundaries_at_scales_that_take_a_second_correction(low):
    """Scales whose last 20 bits are nearly zero: fp32 values whose quotient lies within 2^-46 of the middle of two fp32
    values next to an e4m3 rounding boundary, in a block tile and in rows."""
    block = 64
    tiles = []
    for t in range(8, 16):
        scale = np.float32((t << 20) + low) * np.float32(2.0 ** -20)
        amax = scale * np.float32(448.0)
        while (amax + np.float32(1e-8)) / np.float32(448.0) > scale:
            amax = np.nextafter(amax, np.float32(0.0))
        while (amax + np.float32(1e-8)) / np.float32(448.0) < scale:
            amax = np.nextafter(amax, np.float32(np.inf))
        if (amax + np.float32(1e-8)) / np.float32(448.0) != scale:
            continue  # no largest magnitude gives this scale
        values = [amax]
        for m in range(16, 32):
            for side in (-1, 1):
                exact = ((m << 20) + side) * ((t << 20) + low)  # the quotient's middle times the scale
                k = exact.bit_length() - 24
                for x in (exact >> k, (exact >> k) + 1):
                    values += [np.float32(np.ldexp(float(x), k - 40 - e)) for e in (-3, 0, 5)]
        values = [v for v in values if v <= amax]
        tile = np.resize(np.array(values, dtype=np.float32), block * 64)
        tile[1::2] *= np.float32(-1.0)
        tile[0] = amax
        tiles.append(tile.reshape(block, 64))
    assert len(tiles) >= 3
    x = np.stack(tiles).reshape(1, 1, -1, 64)
    shape = lt.Shape(1, 1, x.shape[2], 64, block)
    got = lt.alloc_fp8(shape, "cuda")
    lt.lite3r_quantize_fp8(torch.from_numpy(x).cuda(), shape, got)
    codes, scales = orc.quantize_fp8_blocks(x, block)
    assert np.array_equal(got.scales.cpu().numpy().view(np.uint32), scales.view(np.uint32))
    assert np.array_equal(got.codes.cpu().numpy(), codes)
    rows = x.reshape(len(tiles), -1)[:, :1024]
    got_codes, got_scales = lt.lite3r_quantize_rows_fp8(torch.from_numpy(np.ascontiguousarray(rows)).cuda())
    assert np.array_equal(got_codes.cpu().numpy(), codes.reshape(len(tiles), -1)[:, :1024])
    assert np.array_equal(got_scales.cpu().numpy().view(np.uint32).ravel(), scales.view(np.uint32).ravel())


@pytest.mark.parametrize("block,crit,read", [(64, 0.1, False), (64, 0.2, True), (128, 0.1, True), (64, 0.0, False)])
def test_key_norms_are_made_for_more_than_one_step(block, crit, read):
    """The largest norms of the key blocks spare the maxima of a tile's steps after the first: they are written where there is
    one (one critical block of 128 tokens is two steps)."""
    wl = small_workload("norms", heads=2, tokens=10 * block, block=block, crit=crit, neg=0.3)
    inputs = wk.make_inputs(wl)
    eng, out = pu.run_gpu(inputs, wl)
    start = lt.lite3r_workspace_layout(eng.shape, wl.crit, wl.neg)[3] + 2 * 10 * block * 64 * 2  # behind the fp16 values
    norms = eng.workspace[start:start + 2 * 10 * 4].view(torch.float32)
    norms.fill_(float("nan"))
    again = eng.forward(torch.from_numpy(inputs["proj"]).cuda(), out=torch.empty_like(out))
    assert torch.equal(again, out)
    assert torch.isnan(norms).all() if not read else (norms > 0).all()


@pytest.mark.parametrize("block,blocks", [(64, 65), (128, 129)])
def test_key_norms_are_the_largest_of_each_block(block, blocks):
    """One large key in every block, in every row of it in turn (the last block has five), so that each warp, lane and row that
    takes part in the maximum decides it once; queries of very different length inside a warp.  The norms against those of
    the codes, the output against the oracle."""
    g = np.random.default_rng(block)
    wl = small_workload(f"norm{block}", heads=2, tokens=(blocks - 1) * block + 5, block=block, crit=0.1, neg=0.3, src_dtype="f32")
    inputs = wk.make_inputs(wl)
    for head in range(2):
        row = np.arange(blocks) * block + (np.arange(blocks) if head == 0 else block - 1 - np.arange(blocks)) % block
        row[-1] = (blocks - 1) * block + (4 if head == 0 else 0)
        inputs["k"][:, head, row] *= 12.0
    inputs["q"] *= np.exp(1.5 * g.standard_normal((1, 2, wl.tokens, 1)) - 1.5).astype(np.float32)
    eng, out = full_parity(wl, inputs, query_blocks=pu.sample_blocks(wl, [0, 1], 24))
    start = lt.lite3r_workspace_layout(eng.shape, wl.crit, wl.neg)[3] + 2 * blocks * block * 64 * 2  # behind the fp16 values
    norms = eng.workspace[start:start + 2 * blocks * 4].view(torch.float32).view(2, blocks)
    codes = eng.k8.codes.view(torch.float8_e4m3fn).double().view(2, blocks, block, 64)
    want = codes.pow(2).sum(-1).amax(-1).sqrt()
    # 64 squares and their sums in single precision, halved by the root, and the root's own rounding
    torch.testing.assert_close(norms.double(), want, rtol=34 * 2.0 ** -24, atol=0.0)


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("climb", [7.9, 8.1, 14.8, 15.2, 15.95, 16.1, 40.0])
def test_attention_with_and_without_a_row_maximum(climb, block):
    """A step whose scores cannot beat the row's reference by more than 2^15 (norm of the query times largest norm of the key
    block) goes without a maximum.  Query and key rows share a direction, so that the bound is nearly reached: a second
    critical block 2^climb above the first, on both sides of the rescale threshold (8), of the bound (15) and of the
    largest fp16 number (16); a ragged last block."""
    g = np.random.default_rng(block)
    wl = small_workload(f"climb{climb}", heads=2, tokens=8 * block - 9, block=block, crit=0.5, neg=0.25, src_dtype="f32")
    inputs = wk.make_inputs(wl)
    top = 1.0 + climb / np.log2(np.e)
    level = np.repeat(np.array([1.0, top, top - 0.5, 0.9, 0.2, 0.1, -0.1, -0.2]), block)[:wl.tokens]
    for name, along in (("q", 8.0), ("k", level[None, None, :, None])):
        inputs[name] = (along / 8.0 + 0.02 * g.standard_normal(inputs[name].shape)).astype(np.float32)
    eng, _ = full_parity(wl, inputs)
    assert (eng.plan.crit_idx.cpu().numpy() == np.arange(4)).all()


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("ones,first,last", [(42, 0x41F0F633, 0x41F0F63C), (23, 0x42DC3CE9, 0x42DC3CEE), (39, 0x4317517A, 0x4317517C)])
def test_attention_bound_is_not_rounded_below_the_scores(ones, first, last, block):
    """Scores of 3e7 to 2e8 (base 2), where neighbouring fp32 numbers are 2 to 16 apart.  The last block's single key lies 2^16
    or more above the reference, past the largest fp16 number, but with these scales the norms' product, rounded to nearest,
    is not above the reference plus 15: taken for the bound, the probability is infinite.  All values are one, so every
    softmax gives one."""
    eng = lt.SlaForward(1, 1, 2 * block + 1, block, 2 / 3, 0.0)
    assert (eng.plan.k_crit, eng.plan.k_marg) == (2, 1)
    row = torch.zeros(64, dtype=torch.uint8, device="cuda")
    row[:ones] = 0x7E  # 448
    for t in (eng.q8, eng.k8, eng.v8):
        t.codes.zero_()
        t.scales.fill_(1.0)
    eng.q8.codes[0, 0, :2 * block + 1] = row
    eng.q8.scales.fill_(0.75)
    eng.k8.codes[0, 0, :block] = row
    eng.k8.codes[0, 0, 2 * block] = row
    bits = torch.tensor([first, 0x3F800000, last], dtype=torch.int32, device="cuda")
    eng.k8.scales[0, 0] = bits.view(torch.float32)
    eng.v8.codes[0, 0, :2 * block + 1] = 0x38  # 1
    eng.plan.cls[0, 0] = torch.tensor([2, 1, 2], dtype=torch.int8)
    eng.plan.crit_idx[0, 0] = torch.tensor([0, 2], dtype=torch.int32)
    eng.plan.marg_idx[0, 0] = 1
    out = eng.forward(torch.zeros((1, 64, 64), device="cuda"))
    assert int(eng.status.item()) == 0
    # probabilities are rounded to fp16 in the product and not in the sum: 2^-11
    torch.testing.assert_close(out, torch.ones_like(out), rtol=2.0 ** -10, atol=0.0)
