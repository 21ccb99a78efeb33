"""GPU parity of a plan's layers that are launched together (one preparation, one GEMM kernel over all their tiles) against
the oracle: shapes at the edges of tiles, of the row forms of the quantization and of a unit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_11446_b200 import binding as B, synth
from gpu_util import DevLayer, to_dev_bf16, bf16_to_np

pytestmark = pytest.mark.gpu
SEED = synth.BASE_SEED + 77

# (M, K, N, bits) a layer. Rows around the 128 of a CTA and the 256 of a pair; K of one k-block, of the last row length that
# one (1280), two (2560) and four warps hold, and of the longest; widths that 128, 192 and 256 divide, alone and together.
EDGES = [(33, 128, 128, 4), (127, 1280, 192, 3), (128, 1408, 256, 8), (129, 2560, 384, 4), (255, 2688, 128, 3),
         (256, 4608, 576, 8), (257, 256, 1152, 16), (40, 4608, 768, 16), (513, 384, 320 + 64, 4)]
STACKS = {
    "edges": EDGES,
    "three": [(300, 384, 384, 4), (300, 384, 1152, 3), (300, 384, 128, 8)],
    # more layers than a unit takes, one without a tile width (N = 320: layer by layer) and one small-M layer among them
    "many": [(100 + 7 * i, 256, 384, (3, 4, 8, 16)[i % 4]) for i in range(18)] + [(64, 256, 320, 4), (8, 256, 384, 4)]
            + [(70, 256, 256, (8, 3, 4)[i]) for i in range(3)],
    "tiles": [(4100, 128, 2304, 3), (4100, 128, 2304, 8), (1, 256, 128, 16), (2050, 1152, 384, 4)],
}


def _reference(x, K, w, s_w, bias, bits, clip, act_bits):
    if clip == 100000 and act_bits == 8:
        q, s_a = oracle.daq(x)[:2]
    else:
        q, s_a = oracle.daq_robust(x, oracle.clip_rank(clip / 1000, K), act_bits)[:2]
    return oracle.epilogue(oracle.gemm_i32(q, w), s_a, s_w, bias)


@pytest.mark.parametrize("clip,act_bits", [(100000, 8), (99900, 8), (99900, 5)])
@pytest.mark.parametrize("name", list(STACKS))
def test_layers_launched_together_match_the_oracle(name, clip, act_bits):
    if name != "edges" and act_bits != 8:
        pytest.skip("one stack is enough for the reduced activation bits")
    stack = STACKS[name]
    ws_, keep, host = [], [], []
    for l, (M, K, N, bits) in enumerate(stack):
        bias = synth.bias(SEED, l, N) if l % 3 else None
        if bits == 16:
            w = (np.random.default_rng(l).standard_normal((N, K)) * 0.05).astype(np.float32)
            w = (w.view(np.uint32) >> 16).astype(np.uint16)
            wd, bd = to_dev_bf16(w), None if bias is None else to_dev_bf16(bias)
            keep += [wd, bd]
            ws_.append(B.dp_weight(N, K, 16, 0, wd.data_ptr(), None, None if bd is None else bd.data_ptr()))
            host.append((w, None, bias))
        else:
            w, s_w = synth.weights(SEED, l, N, K, bits)
            keep.append(DevLayer(w, s_w, bias, bits))
            ws_.append(keep[-1].w)
            host.append((w, s_w, bias))
    plan = B.dp_plan_create(ws_, [s[0] for s in stack], B.DP_FLAG_GROUP_SMALL_M)
    try:
        B.dp_plan_set_daq(plan, clip, 9 if act_bits < 8 else 0, [act_bits] * 3 if act_bits < 8 else None)
        xs = [synth.activations(SEED, l, 0, M, K, 1.0, n_out=max(1, K // 100)) for l, (M, K, _, _) in enumerate(stack)]
        xd = [to_dev_bf16(x) for x in xs]
        # three steps in one call (each unit runs ahead of the one before it, over both parts of the workspace)
        ys = [[torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda") for M, _, N, _ in stack] for _ in range(3)]
        ws = torch.full((B.dp_plan_workspace(plan),), 0x5A, dtype=torch.uint8, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        B.dp_plan_run(plan, [0, 1, 2], 0, B.ptr_array([t.data_ptr() for t in xd]),
                      B.ptr_array([t.data_ptr() for y in ys for t in y]), ws, status, flags=B.DP_PLAN_SAME_X)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        for l, (M, K, N, bits) in enumerate(stack):
            w, s_w, bias = host[l]
            got = bf16_to_np(ys[0][l])
            if bits == 16:
                # bf16 rounding plus an ulp of slack, and K fp32 additions each within 2^-24 of at most the absolute
                # sum, a factor 2 for truncating alignment inside the tensor core
                f = lambda b: (b.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
                exact = f(xs[l]) @ f(w).T + (0.0 if bias is None else f(bias))
                bound = 2.0 ** -8 * np.abs(exact) + K * 2.0 ** -23 * (np.abs(f(xs[l])) @ np.abs(f(w)).T)
                assert np.all(np.abs(f(got) - exact) <= bound), (l, stack[l])
            else:
                assert np.array_equal(got, _reference(xs[l], K, w, s_w, bias, bits, clip, act_bits)), (l, stack[l])
            for i in (1, 2):
                assert torch.equal(ys[i][l].view(torch.int16), ys[0][l].view(torch.int16)), (i, l, stack[l])
    finally:
        B.dp_plan_destroy(plan)


def _layer(l, K, N, bits, group=0):
    """(weight, what holds its memory) of a layer of 3, 4, 8 or 16 bits, group-wise with `group`."""
    bias = synth.bias(SEED, l, N)
    if bits == 16:
        wt = torch.from_numpy((np.random.default_rng(l).standard_normal((N, K)) * 0.05).astype(np.float32)).bfloat16().cuda()
        keep = (wt, to_dev_bf16(bias))
        return B.make_weight(wt, keep[1], keep[1], N, K, 16), keep  # (no scales: that pointer is not read)
    w, s_w = synth.weights(SEED, l, N, K, bits)
    keep = DevLayer(w, s_w, bias, bits)
    if not group:
        return keep.w, keep
    s = torch.from_numpy((np.random.default_rng(l).random((N, K // group)) * 4e-3 + 1e-4).astype(np.float32)).cuda()
    return B.make_weight(keep.qweight, s, keep.bias, N, K, bits, group), (keep, s)


# name: (M, K, N, bits, group) a layer, and which layer's output each one reads (None: an input of its own). What feeds a unit
# takes long, the layers that read it little.
def _fed(bits):
    b = lambda l: bits[l % len(bits)]
    behind = [(300, 1152, 384, b(l), 0) for l in range(3)]
    return {
        "behind_group_wise": ([(6000, 1152, 1152, 4, 32)] + behind, [None, 0, 0, 0]),
        "behind_one_by_one": ([(6000, 1152, 1152 + 64, 8, 0)] + behind, [None, 0, 0, 0]),
        "behind_small_m": ([(8, 1152, 6912, 8, 0)] * 4 + [(144, 384, 256, b(l), 0) for l in range(3)],
                           [None] * 4 + [3, 3, 3]),
        "unit_behind_unit": ([(2000, 384, 384, b(l), 0) for l in range(48)],
                             [None] * 16 + [15 - l for l in range(16)] + [15 + (5 * l) % 16 for l in range(16)]),
        # the first unit's outputs feed the third, beside which they could only run if the second did not wait
        "unit_two_back": ([(2000, 384, 384, b(l), 0) for l in range(48)], [None] * 32 + [l for l in range(16)]),
    }


@pytest.mark.parametrize("bits,clip", [((16,), 100000), ((8,), 100000), ((3, 4), 99900), ((16, 4, 8), 100000)],
                         ids=["sixteen", "eight", "packed_percentile", "mixed"])
@pytest.mark.parametrize("feed", list(_fed((8,))))
def test_units_wait_for_what_feeds_them(feed, bits, clip):
    """Layers launched together that read outputs of the launch before them, whatever that is, over two steps: the bits of
    a plan that runs one kernel at a time."""
    stack, src = _fed(bits)[feed]
    layers = [_layer(l, K, N, b, g) for l, (_, K, N, b, g) in enumerate(stack)]
    x0 = [to_dev_bf16(synth.activations(SEED, l, 0, M, K, 1.0, n_out=3)) for l, (M, K, *_) in enumerate(stack)]
    got = []
    for flags in (B.DP_FLAG_NO_PDL, 0):
        plan = B.dp_plan_create([w for w, _ in layers], [s[0] for s in stack], flags | B.DP_FLAG_GROUP_SMALL_M)
        try:
            B.dp_plan_set_daq(plan, clip, 0)
            ws = torch.full((B.dp_plan_workspace(plan),), 0x5A, dtype=torch.uint8, device="cuda")
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            ys = [torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for M, _, N, *_ in stack]
            # (the end of the output, whose tiles are the last to be written)
            xp = B.ptr_array([x0[l].data_ptr() if s is None else ys[s].view(-1)[-x0[l].numel():].data_ptr()
                              for l, s in enumerate(src)])
            for _ in range(3):
                for t in ys:
                    t.zero_()
                B.dp_plan_run(plan, [0, 1], 0, xp, B.ptr_array([t.data_ptr() for t in ys]), ws, status,
                              flags=B.DP_PLAN_SAME_X | B.DP_PLAN_SAME_Y)
                torch.cuda.synchronize()
                assert int(status.item()) == 0
                got.append([t.view(torch.int16).clone() for t in ys])
        finally:
            B.dp_plan_destroy(plan)
    for run in got[1:]:
        for l, (a, b) in enumerate(zip(got[0], run)):
            assert torch.equal(a, b), (l, stack[l])


@pytest.mark.parametrize("bits", [(16,), (8, 3)], ids=["sixteen", "quantized"])
@pytest.mark.parametrize("small", [True, False], ids=["small_m_between", "units_only"])
def test_steps_that_write_one_set_of_outputs(bits, small):
    """Three steps with inputs of their own and one set of outputs, with and without the grouped small-M launch in front of
    each step's unit: what stays is the last visited step's."""
    stack = [(2048, 768, 768, bits[l % len(bits)], 0) for l in range(4)] + ([(8, 768, 4608, 4, 0)] * 3 if small else [])
    layers = [_layer(l, K, N, b, g) for l, (_, K, N, b, g) in enumerate(stack)]
    xs = [[to_dev_bf16(synth.activations(SEED, l, t, M, K, 1.0, n_out=3)) for l, (M, K, *_) in enumerate(stack)] for t in range(3)]
    got = []
    for flags in (B.DP_FLAG_NO_PDL, 0):
        plan = B.dp_plan_create([w for w, _ in layers], [s[0] for s in stack], flags | B.DP_FLAG_GROUP_SMALL_M)
        try:
            ws = torch.full((B.dp_plan_workspace(plan),), 0x5A, dtype=torch.uint8, device="cuda")
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            for _ in range(3):
                ys = [torch.zeros((M, N), dtype=torch.bfloat16, device="cuda") for M, _, N, *_ in stack]
                torch.cuda.synchronize()
                B.dp_plan_run(plan, [0, 1, 2], 0, B.ptr_array([t.data_ptr() for x in xs for t in x]),
                              B.ptr_array([t.data_ptr() for t in ys]), ws, status, flags=B.DP_PLAN_SAME_Y)
                torch.cuda.synchronize()
                assert int(status.item()) == 0
                got.append([t.view(torch.int16) for t in ys])
        finally:
            B.dp_plan_destroy(plan)
    for run in got[1:]:
        for l, (a, b) in enumerate(zip(got[0], run)):
            assert torch.equal(a, b), (l, stack[l])


@pytest.mark.parametrize("flags", [B.DP_FLAG_GROUP_SMALL_M, 0, B.DP_FLAG_GROUP_SMALL_M | B.DP_FLAG_CTA_PAIR,
                                   B.DP_FLAG_GROUP_SMALL_M | B.DP_FLAG_FUSED_DAQ],
                         ids=["units", "small_m_between", "named_variant", "daq_in_gemm"])
@pytest.mark.parametrize("bit_choices", [(3, 4, 8), (4, 16), (16,)])
def test_launch_count_is_that_of_a_captured_step(bit_choices, flags):
    from cuda.bindings import runtime
    from paper_2511_11446_b200.workloads import DitStack
    stack = DitStack(seed=SEED, batch=2, tokens=128, blocks=5, T=2, keep=1, bit_choices=bit_choices, flags=flags)
    try:
        stack.run(1)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(graph):
            stack.run(1)
        err, _, n = runtime.cudaGraphGetNodes(runtime.cudaGraph_t(graph.raw_cuda_graph()))
        assert err == runtime.cudaError_t.cudaSuccess
        assert n == stack.launches_per_timestep()
        assert int(stack.status.item()) == 0
    finally:
        stack.close()


@pytest.mark.parametrize("sizes,units", [
    ("aaa", [0, 0, 0]), ("aaaa", [-1] * 4), ("aaaaa", [-1] * 5), ("aaaaaa", [0] * 3 + [1] * 3),
    ("aaaaaaa", [0] * 3 + [1] * 3 + [-1]), ("aaac", [-1] * 4), ("aaacaaa", [0] * 3 + [-1] + [1] * 3),
    ("aaacaaac", [-1] * 8), ("cccc" + "aaa" + "bb", [-1] * 9), ("c" + "s" * 17, [-1] + [0] * 16 + [-1]), ("sssgaaa", [0] * 3 + [-1] + [1] * 3)])
def test_which_layers_are_launched_together(sizes, units):
    """Three layers of size a fill a unit, two of size b, none of size c; g is a group-wise layer. Layers go together where at
    least four times as many are in units of three or more as there are pieces left between or behind them."""
    K, N = {"s": 128, "a": 128, "b": 256, "c": 640, "g": 128}, 128
    rows = {"s": 300, "a": 130048, "b": 100000, "c": 130048, "g": 300}
    layers = [_layer(l, K[s], N, 8, 64 if s == "g" else 0) for l, s in enumerate(sizes)]
    plan = B.dp_plan_create([w for w, _ in layers], [rows[s] for s in sizes])
    try:
        assert [B.dp_plan_layer_unit(plan, l) for l in range(len(sizes))] == units
    finally:
        B.dp_plan_destroy(plan)


@pytest.mark.parametrize("Ms,K,named,before,after", [
    ([130048] * 4, 128, [3], [-1] * 4, [0] * 3 + [-1]),             # the piece behind a unit is what kept it from being one
    ([300] * 6, 128, [2], [0] * 6, [-1] * 3 + [0] * 3),
    ([300] * 6, 128, [4, 1, 2], [0] * 6, [-1] * 6)])
def test_units_after_variants_have_been_named(Ms, K, named, before, after):
    """Layers whose variant is named leave their unit, whatever is asked of the plan first: its units, its workspace, a run."""
    layers = [_layer(l, K, 128, 8) for l in range(len(Ms))]
    x = torch.ones((max(Ms), K), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for ask in ("units", "workspace", "run"):
        plan = B.dp_plan_create([w for w, _ in layers], Ms)
        try:
            units = lambda: [B.dp_plan_layer_unit(plan, l) for l in range(len(Ms))]
            assert units() == before
            room = B.dp_plan_workspace(plan)
            for l in named:
                B.dp_plan_set_layer_flags(plan, l, B.DP_FLAG_TILE_N(128))
            if ask == "workspace":
                assert B.dp_plan_workspace(plan) >= room
            elif ask == "run":
                fresh = B.dp_plan_create([w for w, _ in layers], Ms, B.DP_FLAG_NO_PDL)
                ys = []
                for p in (fresh, plan):
                    ys.append([torch.zeros((M, 128), dtype=torch.bfloat16, device="cuda") for M in Ms])
                    ws = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
                    B.dp_plan_run(p, [0], 0, B.ptr_array([x.data_ptr()] * len(Ms)), B.ptr_array([t.data_ptr() for t in ys[-1]]),
                                  ws, status)
                torch.cuda.synchronize()
                B.dp_plan_destroy(fresh)
                assert int(status.item()) == 0 and all(torch.equal(a, b) for a, b in zip(*ys))
            assert units() == after
        finally:
            B.dp_plan_destroy(plan)


@pytest.mark.parametrize("blocks,bit_choices", [(2, (3, 4, 8)), (2, (4, 8, 16)), (1, (4,))])
def test_saved_variants_leave_the_units_as_they_are(blocks, bit_choices):
    from paper_2511_11446_b200.workloads import DitStack
    args = dict(seed=SEED, batch=2, tokens=128, blocks=blocks, T=2, keep=1, bit_choices=bit_choices)
    first = DitStack(flags=B.DP_FLAG_AUTOTUNE | B.DP_FLAG_GROUP_SMALL_M, **args)
    again = DitStack(variants=first.layer_variants(), **args)
    try:
        units = [[B.dp_plan_layer_unit(s.plan, l) for l in range(len(s.table))] for s in (first, again)]
        assert units[0] == units[1] and max(units[0]) >= 0
        assert again.launches_per_timestep() == first.launches_per_timestep()
    finally:
        first.close()
        again.close()
