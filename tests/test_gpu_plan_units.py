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
