"""The work that users of this library have it do, as timed cases: single quantized linears, one
transformer block's linears layer by layer, a block with its neighbouring operators fused, and whole
plans, from one conditioning vector to tens of thousands of tokens.

Kinds
  linear   dp_wq_linear on bf16 tokens (quantization, weight expansion, GEMM, dequantisation)
  shared   dp_daq_quantize once, then two linears of half the width on the codes (several consumers of
           one input quantize it once)
  block    the five linears of a block through dp_wq_linear, one call each
  fused    a block with its neighbours taken in: LayerNorm + modulation + quantization in front of qkv
           and fc1, gated residual adds behind proj and fc2
  plan     a whole stack through dp_plan_run, one retained timestep a pass

A case's "bits" are the widths its layers go through in turn (3, 4, 8, or 16 = kept in bf16).
"group" > 0: one weight scale per that many input channels, "zeros": with zero-points. "clip" < 100000:
the percentile clip of the activation quantization in 1/1000 %, with the activation bits "abits" of the
three time bins. Attention and GELU between the linears are other code's work, so their outputs are
inputs here.
"""
import torch

from paper_2511_11446_b200 import binding as B

STEPS = 50  # timesteps that a plan's schedule and its time bins refer to


# ---- the cases ------------------------------------------------------------------------------------

def listed():
    return [
        # the conditioning vector of one image through one adaLN modulation layer: a few megabytes of
        # weights, so launch latency and the rate of the weight stream
        _linear("adaln_m1_b4", 1, 1152, 6912, "4"),
        # attention projection of one 256-pixel image: the smallest token linear, all latency
        _linear("proj_m256_b8", 256, 1152, 1152, "8"),
        # a 4-bit MLP layer at the batch that samplers run (8 x 256 tokens)
        _linear("fc1_m2048_b4", 2048, 1152, 4608, "4"),
        # one input for several consumers (query and key-value of 3 bits), quantized once; a ragged token count
        dict(name="shared_m1333_b3", kind="shared", M=1333, K=1152, N=3456, bits="3"),
        # the MLP output layer at a ragged batch: the longest contraction
        _linear("fc2_m3001_b3", 3001, 4608, 1152, "3"),
        # all five linears of a block at batch 16, called layer by layer as a model's forward pass does
        _block("block_m4096_b48", 256, 16, 1152, "4,8,4,8,4"),
        # a block of 512-pixel images, batch 32: throughput
        _block("block_m32768_b348", 1024, 32, 1152, "3,8,4,8,3"),
        # group-wise scales with zero-points, the storage format that GPTQ-style quantizers write
        _block("block_m2048_g128z", 256, 8, 1152, "4", group=128, zeros=True),
        # a block with LayerNorm, modulation and residual adds taken into the linears, a ragged token count
        dict(name="fused_m2056_b48", kind="fused", tokens=257, batch=8, width=1152, bits="8,4"),
        # a sampler's whole step, mixed bit plan, batch 8
        _plan("plan_m2048_b348", 256, 8, 1152, 28, "4,8,3,4,8,3,3,8"),
        # the same stack for a single image: launches and host work count
        _plan("plan_m256_b348", 256, 1, 1152, 28, "4,8,3,4,8,3,3,8"),
        # a plan that keeps its most sensitive layers in 16 bits and clips activations at a percentile,
        # with fewer activation bits in the later time bins, batch 4
        _plan("plan_m1024_b48f_clip", 256, 4, 1152, 28, "4,4,16,4,8,4,4,16,4", clip=99900, abits="8,6,4"),
    ]


def draw(rng):
    width = rng.choice((384, 768, 1024, 1152))
    kind = rng.choice(("linear", "linear", "linear", "shared", "block", "block", "block", "fused", "plan", "plan"))
    if kind == "shared":
        return dict(kind="shared", M=_spread(rng, 64, 16384), K=width, N=width * rng.choice((3, 4, 6)),
                    bits=rng.choice(("3", "4", "8")))
    if kind == "linear":
        K, N = rng.choice(((width, 3 * width), (width, width), (width, 4 * width), (4 * width, width), (width, 6 * width)))
        group = rng.choice((0, 0, 0, 32, 64, 128))
        return _linear(None, _spread(rng, 1, 16384 if K > 1152 else 32768), K, N,
                       rng.choice(("3", "4", "8") if group else ("3", "4", "8", "4", "8", "16")),
                       group=group, zeros=group > 0 and rng.random() < 0.5)
    tokens = rng.choice((64, 100, 256, 257, 333, 576, 1024))
    if kind == "plan":
        batch = rng.randint(1, max(1, min(32, 4096 // tokens)))
        clip, abits = rng.choice(((100000, ""), (100000, ""), (99900, "8,6,4"), (100000, "8,8,6")))
        return _plan(None, tokens, batch, width, rng.randint(12, 28) if batch * tokens <= 2048 else 12,
                     _widths(rng, (3, 4, 8, 4, 8, 16), 7), clip=clip, abits=abits)
    batch = rng.randint(1, min(32, 16384 // tokens))
    if kind == "fused":
        return dict(kind="fused", tokens=tokens, batch=batch, width=width, bits=_widths(rng, (3, 4, 8), 4))
    group = rng.choice((0, 0, 64, 128))
    return _block(None, tokens, batch, width, _widths(rng, (3, 4, 8), 5), group=group, zeros=group > 0 and rng.random() < 0.5)


def _linear(name, M, K, N, bits, group=0, zeros=False):
    return _named(name, dict(kind="linear", M=M, K=K, N=N, bits=bits, group=group, zeros=zeros))


def _block(name, tokens, batch, width, bits, group=0, zeros=False):
    return _named(name, dict(kind="block", tokens=tokens, batch=batch, width=width, bits=bits, group=group, zeros=zeros))


def _plan(name, tokens, batch, width, blocks, bits, clip=100000, abits=""):
    return _named(name, dict(kind="plan", tokens=tokens, batch=batch, width=width, blocks=blocks, bits=bits, clip=clip,
                             abits=abits))


def _named(name, case):
    return dict(name=name, **case) if name else case


def _spread(rng, lo, hi):
    """A size spread over its logarithm, odd as often as not."""
    return max(lo, min(hi, round(lo * (hi / lo) ** rng.random())))


def _widths(rng, choices, n):
    return ",".join(str(rng.choice(choices)) for _ in range(n))


def _block_shapes(case):
    """(M, K, N) of a block's linears in call order: qkv, proj, fc1, fc2, adaLN modulation."""
    m, h = case["tokens"] * case["batch"], case["width"]
    return [(m, h, 3 * h), (m, h, h), (m, h, 4 * h), (m, 4 * h, h), (case["batch"], h, 6 * h)]


# ---- inputs -----------------------------------------------------------------------------------------

def _tokens(gen, M, K, sigma=1.0, gelu=False):
    """bf16 activations: normal with 1 % of the channels x 20, or (fc2's input) GELU of a normal."""
    x = torch.randn(M, K, generator=gen, device="cuda")
    if gelu:
        x = torch.nn.functional.gelu(x)
    else:
        x *= sigma
        x[:, torch.randint(K, (max(1, K // 100),), generator=gen, device="cuda")] *= 20.0
    return x.to(torch.bfloat16)


def _pack(codes, bits):
    """Offset-binary codes [N][K] (uint8) as a little-endian bit stream per row."""
    N, K = codes.shape
    if bits == 4:
        c = codes.view(N, K // 2, 2)
        return (c[..., 0] | (c[..., 1] << 4)).contiguous()
    c = codes.view(N, K // 8, 8).to(torch.int32)
    word = sum(c[..., j] << (3 * j) for j in range(8))
    return torch.stack([(word >> s) & 0xFF for s in (0, 8, 16)], -1).to(torch.uint8).view(N, K * 3 // 8)


class _Layer:
    """One layer's constants as a loaded checkpoint leaves them on the GPU."""

    def __init__(self, gen, K, N, bits, group=0, zeros=False):
        self.K, self.N, self.bits, self.group, self.z = K, N, bits, group, None
        self.bias = (torch.randn(N, generator=gen, device="cuda") * 0.01).to(torch.bfloat16)
        w = torch.randn(N, K, generator=gen, device="cuda") * 0.02
        if bits == 16:
            self.q, self.s = w.to(torch.bfloat16), torch.ones(N, device="cuda")
        else:
            half = 1 << (bits - 1)
            v = w.view(N, -1, group or K)
            if zeros:  # asymmetric: the range of a group onto the codes 0 .. 2^bits - 1
                lo, hi = v.amin(-1, keepdim=True), v.amax(-1, keepdim=True)
                s = (hi - lo) / (2 * half - 1)
                z = (-lo / s).round().clamp(0, 2 * half - 1)
                u = (v / s + z).round().clamp(0, 2 * half - 1)
                self.z = z.view(N, -1).to(torch.uint8)
            else:
                s = v.abs().amax(-1, keepdim=True) / (half - 1)
                u = (v / s).round() + half
            u = u.view(N, K).to(torch.int16)
            self.s = s.view(N, -1).contiguous() if group else s.view(N).contiguous()
            self.q = (u - 128).to(torch.int8) if bits == 8 else _pack(u.to(torch.uint8), bits)
        self.w = B.make_weight(self.q, self.s, self.bias, N, K, bits, group, self.z)

    def workspace(self, M, flags=0):
        n = B.dp_wq_linear_workspace_grouped(M, self.w) if self.group else B.dp_wq_linear_workspace(
            M, self.N, self.K, self.bits, flags)
        return torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")


class _Plan:
    def __init__(self, layers, Ms, case):
        self.layers = layers
        self.handle = B.dp_plan_create([l.w for l in layers], Ms, B.DP_FLAG_AUTOTUNE | B.DP_FLAG_GROUP_SMALL_M)
        if case["clip"] < 100000 or case["abits"]:
            bits = [int(b) for b in case["abits"].split(",")] if case["abits"] else None
            B.dp_plan_set_daq(self.handle, case["clip"], STEPS if bits else 0, bits)
        self.workspace = torch.empty(B.dp_plan_workspace(self.handle), dtype=torch.uint8, device="cuda")

    def __del__(self):
        B.dp_plan_destroy(self.handle)


def _out(M, N):
    return torch.empty(M, N, dtype=torch.bfloat16, device="cuda")


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    bits = [int(b) for b in case["bits"].split(",")]
    s = {"case": case, "status": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if case["kind"] == "linear":
        M, K, N = case["M"], case["K"], case["N"]
        layer = _Layer(gen, K, N, bits[0], case["group"], case["zeros"])
        s.update(layers=[layer], x=[_tokens(gen, M, K)], y=[_out(M, N)], ws=layer.workspace(M))
    elif case["kind"] == "shared":
        M, K, N = case["M"], case["K"], case["N"] // 2
        s.update(layers=[_Layer(gen, K, N, bits[0]) for _ in range(2)], x=_tokens(gen, M, K), y=[_out(M, N) for _ in range(2)],
                 q=torch.empty(M, K, dtype=torch.int8, device="cuda"), s_a=torch.empty(M, device="cuda"))
    elif case["kind"] == "block":
        shapes = _block_shapes(case)
        layers = [_Layer(gen, K, N, bits[i % len(bits)], case["group"], case["zeros"]) for i, (_, K, N) in enumerate(shapes)]
        ws = [l.workspace(M) for l, (M, _, _) in zip(layers, shapes)]
        s.update(layers=layers, x=[_tokens(gen, M, K, gelu=i == 3) for i, (M, K, _) in enumerate(shapes)],
                 y=[_out(M, N) for M, _, N in shapes], ws=max(ws, key=lambda t: t.numel()))
    elif case["kind"] == "fused":
        M, h = case["tokens"] * case["batch"], case["width"]
        layers = [_Layer(gen, K, N, bits[i % len(bits)]) for i, (_, K, N) in enumerate(_block_shapes(case)[:4])]
        ws = [l.workspace(M, B.DP_FLAG_FORCE_MMA | B.DP_FLAG_UNPACK_FIRST) for l in layers]
        mod = (torch.randn(6, case["batch"], h, generator=gen, device="cuda") * 0.5).to(torch.bfloat16)
        s.update(layers=layers, mod=mod, x=_tokens(gen, M, h), attn=_tokens(gen, M, h, 0.5),
                 act=_tokens(gen, M, 4 * h, gelu=True), y=[_out(M, l.N) for l in layers],
                 q=[torch.empty(M, h, dtype=torch.int8, device="cuda") for _ in range(2)],
                 s_a=[torch.empty(M, device="cuda") for _ in range(2)], ws=max(ws, key=lambda t: t.numel()))
    else:
        shapes, n = _block_shapes(case), case["blocks"]
        layers, Ms, xp, yp = [], [], [], []
        x = [torch.empty(n, M, K, dtype=torch.bfloat16, device="cuda") for M, K, _ in shapes]
        y = [torch.empty(n, M, N, dtype=torch.bfloat16, device="cuda") for M, _, N in shapes]
        t = seed % STEPS
        for b in range(n):
            for i, (M, K, N) in enumerate(shapes):
                layers.append(_Layer(gen, K, N, bits[len(layers) % len(bits)]))
                Ms.append(M)
                x[i][b] = _tokens(gen, M, K, 0.5 + 2.0 * t / STEPS, gelu=i == 3)
                xp.append(x[i][b].data_ptr())
                yp.append(y[i][b].data_ptr())
        s.update(plan=_Plan(layers, Ms, case), layers=layers, x=x, y=y, xp=B.ptr_array(xp), yp=B.ptr_array(yp), steps=[t])
    return s


# ---- one pass -----------------------------------------------------------------------------------------

def run(state):
    s, case = state, state["case"]
    kind, status = case["kind"], state["status"]
    if kind == "plan":
        B.dp_plan_run(s["plan"].handle, s["steps"], 0, s["xp"], s["yp"], s["plan"].workspace, status)
        return s["y"]
    if kind in ("linear", "block"):
        for layer, x, y in zip(s["layers"], s["x"], s["y"]):
            B.dp_wq_linear(layer.w, x, layer.K, None, x.shape[0], y, layer.N, s["ws"], device_status=status)
        return s["y"]
    if kind == "shared":
        M, K = case["M"], case["K"]
        B.dp_daq_quantize(s["x"], M, K, K, s["q"], K, s["s_a"])
        for layer, y in zip(s["layers"], s["y"]):
            B.dp_wq_linear(layer.w, s["q"], K, s["s_a"], M, y, layer.N, None, device_status=status)
        return s["y"] + [s["q"], s["s_a"]]
    tokens, h = case["tokens"], case["width"]
    M = tokens * case["batch"]
    qkv, proj, fc1, fc2 = s["layers"]
    (shift1, scale1, gate1, shift2, scale2, gate2), ws = s["mod"], s["ws"]
    B.dp_ln_modulate_daq(s["x"], M, h, h, shift1, scale1, tokens, 1e-6, s["q"][0], h, s["s_a"][0])
    B.dp_wq_linear(qkv.w, s["q"][0], h, s["s_a"][0], M, s["y"][0], 3 * h, None, device_status=status)
    B.dp_wq_linear_residual(proj.w, s["attn"], h, M, s["x"], h, gate1, tokens, s["y"][1], h, ws, ws.numel(), status)
    B.dp_ln_modulate_daq(s["y"][1], M, h, h, shift2, scale2, tokens, 1e-6, s["q"][1], h, s["s_a"][1])
    B.dp_wq_linear(fc1.w, s["q"][1], h, s["s_a"][1], M, s["y"][2], 4 * h, None, device_status=status)
    B.dp_wq_linear_residual(fc2.w, s["act"], 4 * h, M, s["y"][1], h, gate2, tokens, s["y"][3], h, ws, ws.numel(), status)
    return s["y"] + s["q"] + s["s_a"]


# ---- what a pass cannot do without ----------------------------------------------------------------------

def _linear_work(M, K, N, bits, group=0, zeros=False, x_bytes=2):
    scales = N * (K // group if group else 1)
    weights = N * K * bits // 8 + 2 * N + (0 if bits == 16 else 4 * scales) + (scales if zeros else 0)
    return x_bytes * M * K + weights + 2 * M * N, 2 * M * N * K


def work(case):
    bits = [int(b) for b in case["bits"].split(",")]
    if case["kind"] == "linear":
        parts = [_linear_work(case["M"], case["K"], case["N"], bits[0], case["group"], case["zeros"])]
    elif case["kind"] == "shared":
        M, K, N = case["M"], case["K"], case["N"] // 2
        parts = [_linear_work(M, K, N, bits[0], x_bytes=0)] * 2 + [(3 * M * K + 4 * M, 0)]
    elif case["kind"] == "fused":
        M, h = case["tokens"] * case["batch"], case["width"]
        parts = [_linear_work(m, K, N, bits[i % len(bits)], x_bytes=2 if i in (1, 3) else 0)
                 for i, (m, K, N) in enumerate(_block_shapes(case)[:4])]
        # the residual stream in once (its later readers find what this pass wrote), codes and scales
        # of the two normalizations out, modulation vectors in
        parts += [(2 * M * h + 2 * (M * h + 4 * M) + 12 * case["batch"] * h, 0)]
    else:
        group, zeros = case.get("group", 0), case.get("zeros", False)
        shapes = _block_shapes(case) * case.get("blocks", 1)
        parts = [_linear_work(M, K, N, bits[i % len(bits)], group, zeros) for i, (M, K, N) in enumerate(shapes)]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """Quantized layers: codes, scales and accumulators are integers or single roundings and the fp32
    sequence behind them is part of the interface, so outputs are the same bits whatever kernel ran.
    Layers kept in bf16: fp32 sums of up to 4608 products in another order, then one bf16 rounding;
    against sums in double 0.3 % of the outputs differ, by one bf16 ulp (2^-7): 1.7e-4 in the 2-norm."""
    if "16" in case["bits"].split(","):
        return {"rel": 7e-4, "max": 0.016}
    return "exact"
