"""The work that users of libmqgrad have it do, as cases that can be timed.

A case names a path through the public calls (`path`), sizes, the bit width and the options of that path:

  worker      one worker encodes its gradient for the wire: mqg_quantize
  server      the server applies W received buffers: mqg_server_step, or unfused mqg_dequant_accumulate + mqg_apply
  loop        one iteration with simulated workers: a quantize call per worker (or one batched call), then the server step
  layers      the same for a gradient of many tensors with one scale per tensor
  paper_cnn   two large matrices quantized as a whole, the other tensors applied uncompressed, worker by worker
  downlink    the server's re-quantization of the mean and the worker's update from it
  minmax, l2, onebit     an iteration with one of the codec variants

Every result is fixed bit for bit by the codec's definition (reproducible draws, fixed order of every sum), so all
outputs are compared exactly.
"""
import itertools
import math

import torch

import paper_1804_08066_b200 as mqg
from paper_1804_08066_b200 import workloads as wl

PHILOX_SEED = 2


def listed():
    return [
        # A worker process that sends one small gradient: latency of a single call.
        {"name": "worker_small", "path": "worker", "n": 100_013, "W": 1, "bits": 4, "bucket": 512, "dtype": "f32"},
        # The training loop of this package: its CNN (620,362 parameters), four workers, a call per worker.
        {"name": "loop_cnn_620k", "path": "loop", "n": 620_362, "W": 4, "bits": 3, "bucket": 2048, "dtype": "f32",
         "batched": False},
        # The small benchmark configuration, all workers in one call, then the server.
        {"name": "loop_1M_batched", "path": "loop", "n": 1 << 20, "W": 4, "bits": 2, "bucket": 512, "dtype": "f32",
         "batched": True},
        # A worker in earnest: one bf16 gradient of an odd size that no tile divides.
        {"name": "worker_bf16_ragged", "path": "worker", "n": 6_543_217, "W": 1, "bits": 6, "bucket": 1024, "dtype": "bf16"},
        # The headline configuration, each side on its own: encode of eight gradients, and the server's pass over them.
        {"name": "encode_25M_w8", "path": "encode", "n": 25_000_000, "W": 8, "bits": 4, "bucket": 2048, "dtype": "f32",
         "batched": True},
        {"name": "server_25M_w8", "path": "server", "n": 25_000_000, "W": 8, "bits": 2, "bucket": 2048, "dtype": "f32",
         "form": "step"},
        # The layered configuration: AlexNet-shaped tensors, one scale per tensor, eight workers.
        {"name": "layers_alexnet_w8", "path": "layers", "tensors": "alexnet", "W": 8, "bits": 4, "dtype": "f32",
         "batched": True},
        # The model of the paper's evaluation: two large matrices quantized, everything else uncompressed.
        {"name": "paper_cnn_w3", "path": "paper_cnn", "W": 3, "bits": 5, "dtype": "f32"},
        # The stress configuration (bf16, sixteen workers, bucket 4096) at a quarter of its 10^9 elements, every worker with
        # a gradient of its own.
        {"name": "loop_bf16_250M_w16", "path": "loop", "n": 250_000_000, "W": 16, "bits": 4, "bucket": 4096,
         "dtype": "bf16", "batched": True},
        # The downlink half of an iteration at the headline size.
        {"name": "downlink_25M_w8", "path": "downlink", "n": 25_000_000, "W": 8, "bits": 4, "bucket": 2048, "dtype": "f32"},
        # The (min, max) codec, unfused on the server (a sum that is inspected before it is applied).
        {"name": "minmax_9M_w8", "path": "minmax", "n": 9_000_001, "W": 8, "bits": 8, "bucket": 4096, "dtype": "f32",
         "batched": True, "form": "unfused"},
        # One bit with error feedback: each of four workers keeps its residual.
        {"name": "onebit_9M_w4", "path": "onebit", "n": 9_000_001, "W": 4, "bits": 1, "bucket": 2048, "dtype": "f32"},
    ]


BUCKETS = (256, 512, 768, 1024, 2048, 3072, 4096, 8192)
MOST_VALUES = 400_000_000          # W * n of a drawn case
MOST_ELEMENTS = 60_000_000         # n of a drawn case


def draw(rng):
    path = rng.choice(("worker", "worker", "server", "encode", "loop", "loop", "layers", "downlink", "minmax", "l2", "onebit"))
    W = 1 if path == "worker" else rng.choice((2, 3, 4, 8, 8, 16)) if path == "encode" else rng.choice((1, 2, 3, 4, 8, 8, 16))
    n = int(round(math.exp(rng.uniform(math.log(3_000), math.log(min(MOST_ELEMENTS, MOST_VALUES // W))))))
    if rng.random() < 0.4:
        n = max(2048, n // 2048 * 2048)
    case = {"path": path, "n": n, "W": W, "bits": 1 if path == "onebit" else rng.randint(1, 8), "bucket": rng.choice(BUCKETS),
            "dtype": rng.choice(("f32", "f32", "bf16"))}
    if path in ("worker", "encode", "loop", "server", "minmax") and rng.random() < 0.1:
        case["bucket"] = 16384     # longer than one tile of any kernel: two passes over the gradient
    if path in ("encode", "loop", "layers", "minmax", "l2"):
        case["batched"] = rng.random() < 0.6
    if path in ("server", "minmax"):
        case["form"] = rng.choice(("step", "step", "unfused", "sum"))
    if path == "l2":
        case["layers"] = rng.random() < 0.4
    if path == "layers" or case.get("layers"):
        case["tensors"] = "split"
        case["parts"] = rng.choice((2, 5, 16, 40))
        del case["bucket"]
    return case


def _sizes(case):
    """Tensor sizes of a layered gradient, in order."""
    if case["tensors"] == "alexnet":
        return wl.alexnet_segments()[1]
    # `parts` tensors of very unlike sizes, every second one as short as a bias vector; sizes are multiples of eight
    # (channel counts) unless n is odd, in which case hardly any tensor starts on an aligned address
    n, parts = case["n"], case["parts"]
    weight = [((7 * i) % 13 + 1) ** 2 if i % 2 == 0 else 0.05 for i in range(parts)]
    sizes = [max(8, int(n * w / sum(weight))) for w in weight]
    sizes = [s | 1 for s in sizes] if n % 2 else [s // 8 * 8 for s in sizes]
    return sizes


def _offsets(sizes, bits):
    """Element offsets of the tensors and word offsets of their bit streams."""
    seg = [0, *itertools.accumulate(sizes)]
    code = [0, *itertools.accumulate(mqg.mqg_code_words(s, bits) for s in sizes)]
    return seg, code


def _gradient(n, dtype, gen, sizes=None):
    """Laplace(0, 1e-4) in fp32; Student-t(3) * 1e-4 with 0.1 % zeros in bf16 (heavy tails, as accumulated bf16
    gradients have); with `sizes` every tensor N(0, sigma), sigma log-uniform in [1e-5, 1e-2]."""
    out = torch.empty(n, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    if sizes is not None:
        sigma = torch.rand(len(sizes), generator=gen, device="cuda").mul_(3).sub_(5).mul_(math.log(10)).exp_()
        lo = 0
        for j, s in enumerate(sizes):
            out[lo:lo + s] = torch.randn(s, generator=gen, device="cuda") * sigma[j]
            lo += s
        return out
    step = 1 << 26
    for lo in range(0, n, step):
        m = min(step, n - lo)
        if dtype == "f32":
            u = torch.rand(m, generator=gen, device="cuda").sub_(0.5)
            out[lo:lo + m] = torch.log1p(u.abs().mul_(-2).clamp_(min=-1 + 2.0 ** -24)).mul_(u.sign()).mul_(-1e-4)
        else:
            x = torch.randn(m, generator=gen, device="cuda")
            x.div_(torch.randn(3, m, generator=gen, device="cuda").square_().sum(0).div_(3.0).sqrt_()).mul_(1e-4)
            x[torch.rand(m, generator=gen, device="cuda") < 1e-3] = 0.0
            out[lo:lo + m] = x
    return out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.path, s.W, s.bits = case, case["path"], case["W"], case["bits"]
    s.step = itertools.count(1)                    # the iteration number keys the draws
    s.lr = 0.1 / s.W
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if s.path == "paper_cnn":
        seg, s.n = wl.paper_cnn_layout()
        sizes = [int(seg[1] - seg[0]), int(seg[2] - seg[1])]
        s.seg, s.code = _offsets(sizes, s.bits)
        s.nq = s.seg[-1]
        grad_sizes = [*sizes, *(math.prod(shape) for shape in wl.PAPER_CNN_UNCOMPRESSED)]
    elif "tensors" in case:
        grad_sizes = _sizes(case)
        s.seg, s.code = _offsets(grad_sizes, s.bits)
        s.n = s.seg[-1]
    else:
        grad_sizes, s.seg, s.n, s.bucket = None, None, case["n"], case["bucket"]
    s.grads = [_gradient(s.n, case["dtype"], gen, grad_sizes) for _ in range(s.W)]
    if s.seg is not None:
        words, nscales = s.code[-1], len(s.seg) - 1
    else:
        words, nscales = mqg.mqg_code_words(s.n, s.bits), mqg.mqg_num_buckets(s.n, s.bucket)
    if s.path in ("minmax", "onebit"):
        nscales *= 2
    s.codes = [torch.zeros(words, dtype=torch.int32, device="cuda") for _ in range(s.W)]
    s.scales = [torch.zeros(nscales, dtype=torch.float32, device="cuda") for _ in range(s.W)]
    if s.path not in ("worker", "encode"):
        s.params = torch.randn(s.n, generator=gen, device="cuda").mul_(0.05)
    if case.get("form") in ("unfused", "sum"):
        s.acc = torch.zeros(s.n, dtype=torch.float32, device="cuda")
    if s.path == "onebit":
        s.residuals = [torch.zeros(s.n, dtype=torch.float32, device="cuda") for _ in range(s.W)]
    if s.path == "l2" and s.seg is not None:
        s.workspace = torch.zeros(max(1, mqg.mqg_l2_workspace_floats(s.seg)), dtype=torch.float32, device="cuda")
    if s.path in ("server", "downlink"):           # what has arrived from the workers
        for w in range(s.W):
            mqg.mqg_quantize(s.grads[w], s.n, s.bits, s.bucket, PHILOX_SEED, s.codes[w], s.scales[w], worker=w)
        s.grads = None
    if s.path == "downlink":
        s.down_codes, s.down_scales = torch.zeros_like(s.codes[0]), torch.zeros_like(s.scales[0])
    return s


def _server(s):
    form = s.case.get("form", "step")
    if s.path in ("minmax", "onebit"):
        step, total = mqg.mqg_server_step_minmax, mqg.mqg_dequant_accumulate_minmax
    else:
        step, total = mqg.mqg_server_step, mqg.mqg_dequant_accumulate
    if form == "step":
        step(s.codes, s.scales, s.W, s.bits, s.n, s.bucket, s.params, s.lr)
        return [s.params]
    if form == "sum":
        step(s.codes, s.scales, s.W, s.bits, s.n, s.bucket, s.params, s.lr, acc_out=s.acc)
    else:
        total(s.codes, s.scales, s.W, s.bits, s.n, s.acc, s.bucket)
        mqg.mqg_apply(s.params, s.acc, s.lr, s.n)
    return [s.params, s.acc]


def _encode(s, m):
    """Every worker's gradient of iteration m, in one call or a call per worker."""
    batched = s.case.get("batched", False)
    if s.path == "minmax":
        if batched:
            mqg.mqg_quantize_workers_minmax(s.grads, s.W, s.n, s.bits, s.bucket, s.codes, s.scales)
        else:
            for w in range(s.W):
                mqg.mqg_quantize_minmax(s.grads[w], s.n, s.bits, s.bucket, s.codes[w], s.scales[w])
    elif s.path == "onebit":
        for w in range(s.W):
            mqg.mqg_quantize_1bit_ef(s.grads[w], s.residuals[w], s.n, s.bucket, s.codes[w], s.scales[w])
    elif s.path == "l2" and s.seg is not None:
        for w in range(s.W):
            mqg.mqg_quantize_segments_l2(s.grads[w], s.seg, s.code, s.bits, PHILOX_SEED, s.codes[w], s.scales[w],
                                         s.workspace, worker=w, step=m)
    elif s.seg is not None:
        if batched:
            mqg.mqg_quantize_segments_workers(s.grads, s.W, s.seg, s.code, s.bits, PHILOX_SEED, s.codes, s.scales, step=m)
        else:
            for w in range(s.W):
                mqg.mqg_quantize_segments(s.grads[w], s.seg, s.code, s.bits, PHILOX_SEED, s.codes[w], s.scales[w],
                                          worker=w, step=m)
    elif batched:
        all_workers = mqg.mqg_quantize_workers_l2 if s.path == "l2" else mqg.mqg_quantize_workers
        all_workers(s.grads, s.W, s.n, s.bits, s.bucket, PHILOX_SEED, s.codes, s.scales, step=m)
    else:
        one = mqg.mqg_quantize_l2 if s.path == "l2" else mqg.mqg_quantize
        for w in range(s.W):
            one(s.grads[w], s.n, s.bits, s.bucket, PHILOX_SEED, s.codes[w], s.scales[w], worker=w, step=m)


def run(s):
    m = next(s.step)
    if s.path == "server":
        return _server(s)
    if s.path == "downlink":
        mqg.mqg_server_requantize(s.codes, s.scales, s.W, s.bits, s.n, s.bucket, 1.0 / s.W, PHILOX_SEED,
                                  s.down_codes, s.down_scales, worker=s.W, step=m)
        mqg.mqg_server_step([s.down_codes], [s.down_scales], 1, s.bits, s.n, s.bucket, s.params, 0.1)
        return [s.down_codes, s.down_scales, s.params]
    _encode(s, m)
    if s.path in ("worker", "encode"):
        return [s.codes, s.scales]
    if s.seg is None:
        updated = _server(s)
    else:
        mqg.mqg_server_step_segments(s.codes, s.scales, s.W, s.bits, s.seg, s.code, s.params, s.lr)
        updated = [s.params]
        if s.path == "paper_cnn":
            for w in range(s.W):
                mqg.mqg_apply(s.params[s.nq:], s.grads[w][s.nq:], s.lr, s.n - s.nq)
    return [s.codes, s.scales, s.residuals if s.path == "onebit" else None, *updated]


def work(case):
    path, W, bits = case["path"], case["W"], case["bits"]
    size = 4 if case["dtype"] == "f32" else 2
    if path == "paper_cnn":
        seg, n = wl.paper_cnn_layout()
        n, coded, nscales = int(n), int(seg[-1]), 2
    elif "tensors" in case:
        sizes = _sizes(case)
        n = coded = sum(sizes)
        nscales = len(sizes)
    else:
        n = coded = case["n"]
        nscales = mqg.mqg_num_buckets(n, case["bucket"])
    wire = coded * bits / 8 + 4 * nscales * (2 if path in ("minmax", "onebit") else 1)   # of one worker
    encode = {"bytes": W * (size * n + wire), "flops": 4 * W * coded}
    decode = {"bytes": W * wire + 8 * n, "flops": (3 * W + 2) * n}
    if path in ("worker", "encode"):
        parts = [encode]
    elif path == "server":
        parts = [decode]
    elif path == "downlink":
        parts = [{"bytes": W * wire + 2 * wire + 8 * n, "flops": (3 * W + 10) * n}]
    else:
        parts = [encode, decode]
        if path == "onebit":
            parts.append({"bytes": 8 * W * n, "flops": 4 * W * n})       # the residuals, in and out
    if case.get("form") in ("unfused", "sum"):
        parts.append({"bytes": 4 * n, "flops": 0})                       # the sum, written
    return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}


def tolerance(case):
    return "exact"
