"""The contractions that users of this library run, as measurable cases.

`listed()` are named representatives, `draw(rng)` gives further ones of the same ranges.  A case is a dict of plain
values: `op` names the entry point, the rest its sizes, accumulation order, quantiser formats and operand bytes.
Networks (`convnet`, `encoder`) are all LBA calls of one forward pass, in order; the glue between them (ReLU, pooling,
re-quantisation) is the user's own PyTorch code and not part of the case, so every call gets operands with the
distribution it sees there: half-normal activations, He-normal weights, Gaussian token features with outlier columns.
"""
import torch

from paper_2401_14110_b200 import (ORDER_CHUNKED, ORDER_SEQUENTIAL, PAPER_CHUNK, ROUND_FLOOR, ROUND_NEAREST_EVEN,
                                   code_domain_formats, m4e3_input_formats)
from paper_2401_14110_b200 import binding, synth, workloads

MAX_MACS = 1 << 36  # of a drawn case: below the largest listed one in time, whatever its formats


def _case(op, order="chunk", man=7, exp=4, rounding="floor", wa="e4m3", **sizes):
    return dict(op=op, order=order, man=man, exp=exp, rounding=rounding, wa=wa, **sizes)


def listed():
    return [
        # one small contraction, the size of a unit of work in a notebook or a test: latency and launches are all of it
        _case("gemm", order="seq", M=64, N=64, K=576, per_channel=False, bias=False, name="gemm_small_seq"),
        # classifier head of one batch: few rows, per-channel weight scales and a bias
        _case("gemm", M=32, N=1000, K=512, per_channel=True, bias=True, name="classifier_b32"),
        # forward pass of a small convolution network (stem on 3-channel images, 3x3 and strided 1x1 layers, classifier)
        _case("convnet", arch="resnet18", batch=32, hw=224, name="resnet18_b32"),
        # a deeper one, mostly 1x1 convolutions, fed the paper's own weight/activation bytes (Q_prod cuts mantissas)
        _case("convnet", arch="resnet50", batch=16, hw=224, wa="m4e3", name="resnet50_b16_m4e3"),
        # the six linear layers of a transformer encoder layer at a training batch
        _case("encoder", tokens=4096, name="bert_linears_4096"),
        # the two matrix products inside its attention: scores and context of every head
        _case("attention", heads=384, seq=128, dim=64, name="attention_384x128"),
        # the largest single contraction, 12-bit accumulator in the paper's order
        _case("gemm", M=8192, N=8192, K=8192, per_channel=False, bias=False, name="gemm_8192"),
        # points of an accumulator-format sweep: nearest-even rounding, and a mantissa that cuts the products
        _case("gemm", M=4096, N=4096, K=4096, rounding="rne", per_channel=False, bias=False, name="sweep_4096_rne"),
        _case("gemm", M=4096, N=4096, K=4096, man=5, exp=5, per_channel=False, bias=False, name="sweep_4096_m5e5"),
        # sizes that no tile divides, rows that are not 16-byte aligned
        _case("gemm", M=1111, N=777, K=1203, per_channel=True, bias=True, name="gemm_ragged"),
        # backward direction: the overflow masks and the difference masks that fine-tuning re-computes, on an
        # encoder's first feed-forward layer and on a projection
        _case("ste", ste="of", M=4096, N=3072, K=768, name="ste_of_ffn"),
        _case("ste", ste="diff", order="seq", M=4096, N=768, K=768, name="ste_diff_proj"),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    op = rng.choice(["gemm"] * 6 + ["convnet", "encoder", "attention", "ste", "ste"])
    order = rng.choice(["chunk", "chunk", "seq"])
    if op == "gemm":
        man, exp, rounding, wa = rng.choice([(7, 4, "floor", "e4m3")] * 4 + [
            (7, 4, "rne", "e4m3"), (10, 5, "rne", "e4m3"), (5, 5, "rne", "e4m3"), (4, 4, "floor", "e4m3"),
            (10, 6, "floor", "e4m3"), (5, 6, "floor", "e4m3"), (7, 4, "floor", "m4e3"), (10, 5, "floor", "m4e3")])
        while True:
            M, N, K = _log_int(rng, 16, 8192), _log_int(rng, 32, 8192), _log_int(rng, 64, 8192)
            if rng.random() < 0.6:  # most layers have multiples of 16; the rest are ragged
                M, N, K = M, -(-N // 16) * 16, -(-K // 16) * 16
            if M * N * K <= MAX_MACS:
                break
        return _case("gemm", order, man, exp, rounding, wa, M=M, N=N, K=K, per_channel=rng.random() < 0.5,
                     bias=rng.random() < 0.5)
    if op == "convnet":
        arch = rng.choice(["resnet18", "resnet50"])
        return _case("convnet", order, wa=rng.choice(["e4m3", "m4e3"]), arch=arch, hw=32 * rng.randint(4, 8),
                     batch=_log_int(rng, 1, 32 if arch == "resnet18" else 12))
    if op == "encoder":
        return _case("encoder", order, tokens=_log_int(rng, 128, 8192))
    if op == "attention":
        return _case("attention", order, heads=12 * _log_int(rng, 1, 40), seq=rng.choice([64, 100, 128, 197, 256, 384]), dim=64)
    ste = rng.choice(["of", "diff"])
    return _case("ste", order, ste=ste, M=_log_int(rng, 64, 4096), N=16 * _log_int(rng, 4, 192), K=16 * _log_int(rng, 4, 96))


# ------------------------------------------------------------------ inputs
def _formats(case):
    rounding = ROUND_NEAREST_EVEN if case["rounding"] == "rne" else ROUND_FLOOR
    make = m4e3_input_formats if case["wa"] == "m4e3" else code_domain_formats
    return make(case["man"], case["exp"], rounding)


def _order(case):
    return ORDER_CHUNKED if case["order"] == "chunk" else ORDER_SEQUENTIAL


class _Source:
    """Random tensors on the GPU from one seed, encoded as operand bytes with their scales."""

    def __init__(self, seed, wa):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)
        self.wa = wa

    def normal(self, *shape, std=1.0):
        return torch.randn(shape, generator=self.gen, device="cuda") * std

    def features(self, *shape, gain=20.0):
        """Gaussian token features with 1 % of outlier columns."""
        t = self.normal(*shape)
        cols = torch.randperm(shape[-1], generator=self.gen, device="cuda")[: max(1, shape[-1] // 100)]
        t[..., cols] *= gain
        return t

    def act(self, t):
        codes, scale = (synth.quantise_m4e3_per_tensor if self.wa == "m4e3" else synth.quantise_per_tensor)(t)
        return codes.contiguous(), scale

    def weight(self, w, per_channel=True):
        if self.wa == "m4e3" or not per_channel:
            return self.act(w)
        codes, scale = synth.quantise_per_channel(w)
        return codes.contiguous(), scale.contiguous()


def _gemm_state(src, M, N, K, per_channel=True, bias=False, outliers=False):
    a, sa = src.act(src.features(M, K) if outliers else src.normal(M, K))
    b, sb = src.weight(src.normal(N, K, std=0.02 if outliers else 1.0), per_channel)
    return a, b, sa, sb, src.normal(N, std=0.1) if bias else None


def _conv_out(size, spec):
    return (size + 2 * spec.pad - spec.k) // spec.stride + 1


def _convnet_state(src, arch, batch, hw):
    specs = {"resnet18": workloads.resnet18_convs, "resnet50": workloads.resnet50_convs}[arch]()
    calls = []
    for i, spec in enumerate(specs):
        h = hw * spec.h_in // 224
        t = src.normal(batch, h, h, spec.c_in)
        x, sx = src.act(t if i == 0 else t.relu_())
        fan_in = spec.k * spec.k * spec.c_in
        w, sw = src.weight(src.normal(spec.c_out, spec.k, spec.k, spec.c_in, std=(2.0 / fan_in) ** 0.5))
        calls.append((x, w, sx, sw, (spec.stride, spec.stride), (spec.pad, spec.pad)))
    c = specs[-1].c_out
    x, sx = src.act(src.normal(batch, c).abs_())
    w, sw = src.weight(src.normal(1000, c, std=(1.0 / c) ** 0.5))
    return calls, (x, w, sx, sw, src.normal(1000, std=0.1))


def prepare(case, seed):
    src = _Source(seed, case["wa"])
    prod, acc = _formats(case)
    state = {"case": case, "prod": prod, "acc": acc, "order": _order(case)}
    op = case["op"]
    if op in ("gemm", "ste"):
        state["gemm"] = _gemm_state(src, case["M"], case["N"], case["K"], case.get("per_channel", True), case.get("bias", False))
    elif op == "convnet":
        state["convs"], state["fc"] = _convnet_state(src, case["arch"], case["batch"], case["hw"])
    elif op == "encoder":
        state["linears"] = [_gemm_state(src, m, n, k, bias=True, outliers=True)
                            for _, m, n, k in workloads.bert_base_linears(case["tokens"])]
    else:
        z, s, d = case["heads"], case["seq"], case["dim"]
        q, sq = src.act(src.normal(z, s, d))
        k, sk = src.act(src.normal(z, s, d))
        p, sp = src.act(torch.softmax(src.normal(z, s, s), dim=-1))
        vt, sv = src.act(src.normal(z, d, s))
        state["attention"] = (q, k, sq, sk), (p, vt, sp, sv)
    return state


def run(state):
    prod, acc, order, case = state["prod"], state["acc"], state["order"], state["case"]
    op = case["op"]
    if op == "gemm":
        a, b, sa, sb, bias = state["gemm"]
        return binding.lba_gemm(a, b, sa, sb, bias, prod, acc, order, PAPER_CHUNK)
    if op == "ste":
        a, b = state["gemm"][:2]
        diff = case["ste"] == "diff"
        return binding.lba_gemm_ste_mask(a, b, prod, acc, order, PAPER_CHUNK, ste=binding.STE_DIFF if diff else binding.STE_OF,
                                         eps1=4.0 if diff else 0.0, eps2=2.0 ** -7 if diff else 0.0)
    if op == "convnet":
        outs = [binding.lba_conv2d(x, w, sx, sw, None, stride, pad, prod, acc, order, PAPER_CHUNK)
                for x, w, sx, sw, stride, pad in state["convs"]]
        x, w, sx, sw, bias = state["fc"]
        return outs + [binding.lba_gemm(x, w, sx, sw, bias, prod, acc, order, PAPER_CHUNK)]
    if op == "encoder":
        return [binding.lba_gemm(a, b, sa, sb, bias, prod, acc, order, PAPER_CHUNK) for a, b, sa, sb, bias in state["linears"]]
    return [binding.lba_gemm_batched(a, b, sa, sb, None, prod, acc, order, PAPER_CHUNK) for a, b, sa, sb in state["attention"]]


# ------------------------------------------------------------------ what a pass cannot do without
def _gemm_work(M, N, K, Z=1, out_bytes=None):
    return Z * (M * K + N * K) + (4 * Z * M * N if out_bytes is None else out_bytes), 2 * Z * M * N * K


def work(case):
    op = case["op"]
    if op == "gemm":
        parts = [_gemm_work(case["M"], case["N"], case["K"])]
    elif op == "ste":
        M, N, K = case["M"], case["N"], case["K"]
        words = -(-K // 32) + (-(-(-(-K // PAPER_CHUNK)) // 32) if case["order"] == "chunk" else 0)
        parts = [_gemm_work(M, N, K, out_bytes=4 * M * N * words)]
    elif op == "convnet":
        specs = {"resnet18": workloads.resnet18_convs, "resnet50": workloads.resnet50_convs}[case["arch"]]()
        B, parts = case["batch"], [_gemm_work(case["batch"], 1000, 512 if case["arch"] == "resnet18" else 2048)]
        for s in specs:
            h = case["hw"] * s.h_in // 224
            ho, k = _conv_out(h, s), s.k * s.k * s.c_in
            parts.append((B * h * h * s.c_in + s.c_out * k + 4 * B * ho * ho * s.c_out, 2 * B * ho * ho * s.c_out * k))
    elif op == "encoder":
        parts = [_gemm_work(m, n, k) for _, m, n, k in workloads.bert_base_linears(case["tokens"])]
    else:
        z, s, d = case["heads"], case["seq"], case["dim"]
        parts = [_gemm_work(s, s, d, z), _gemm_work(s, d, s, z)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


def tolerance(case):
    # every addition is rounded once, in a fixed order, to a stated format: one bit pattern is correct
    return "exact"
