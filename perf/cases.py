"""The workloads this framework's speed is judged on.

Every case is work a user of the library has it do through ``pipeline.Round`` (or through the two
calls of ``dq`` that a worker and a server on different GPUs use), over layouts of the networks in
``workloads.py`` and over flat gradients from a few thousand elements to gigabytes.

A case names
    call     what one pass is:
             "round"    Round.step_fused: Algorithm 1's order, the next b chosen on the device
             "update"   the same round with the parameter update of Eq. 2 in it
             "fourcall" Round.step: norms, bit rule on this step's norms, quantize, average
             "encode"   norms and codes only: the worker's side, one gradient on its own GPU
             "decode"   the average only: the server's side, from packed words
             "host"     Round.step_host: pinned host gradients in, pinned host average out
    layout   "flat" (one tensor of ``d`` elements), "resnet18", "vgg16" or "text" (the tensor lists
             of ``workloads.py``, every size divided by ``shrink``)
    M        workers, ``bucket`` elements per norm (0: one norm per tensor), ``norm`` "l2" or "linf"
    b        bits per code; where a round chooses b itself, the rule is calibrated so that it lands there
"""
import numpy as np
import torch

from paper_2107_14575_b200 import dq, workloads
from paper_2107_14575_b200.pipeline import Round

SEED = 2107          # seed of the rounding draws; the inputs have their own
T = 100              # length of the schedule the rule is asked for

NETWORKS = {
    "resnet18": workloads.resnet18_cifar_segments,
    "vgg16": workloads.vgg16_cifar_segments,
    "text": workloads.text_classifier_segments,
}


def _case(name, call, layout, M, bucket, b, d=0, shrink=1, norm="l2"):
    return {"name": name, "call": call, "layout": layout, "d": d, "shrink": shrink, "M": M, "bucket": bucket,
            "norm": norm, "b": b}


def listed():
    return [
        # a single small layer's gradient, ragged: launches and host work decide
        _case("round_layer_70k", "round", "flat", 4, 512, 8, d=70001),
        # a small network with many tensors, most of them far shorter than a bucket
        _case("round_resnet18_small", "round", "resnet18", 4, 512, 4, shrink=32),
        # CIFAR ResNet-18, eight workers, at the bit width its schedule starts with
        _case("round_resnet18", "round", "resnet18", 8, 512, 4),
        # VGG-16, sixteen workers, long buckets, heavy-tailed gradients, parameters updated by the server step
        _case("update_vgg16", "update", "vgg16", 16, 2048, 5),
        # text classifier: 97 % of the embedding rows have no gradient
        _case("round_text", "round", "text", 16, 1024, 4),
        # the bench's workload: 8 GiB of gradients per round
        _case("round_flat_8gib", "round", "flat", 32, 512, 4, d=1 << 26),
        # largest magnitude instead of the l2 norm, short buckets, the high end of the schedule's b
        _case("round_linf_4m", "round", "flat", 4, 128, 8, d=4194307, norm="linf"),
        # the normalisation Eq. 5 writes: one norm per tensor, which takes a second pass over the gradients
        _case("round_whole_tensor", "round", "resnet18", 8, 0, 8),
        # b from this step's own norms; a bucket length that is not a power of two
        _case("fourcall_vgg16_odd_bucket", "fourcall", "vgg16", 8, 480, 6, shrink=2),
        # one worker per GPU: its own gradient to codes, before the words leave for the server
        _case("encode_worker_16m", "encode", "flat", 1, 512, 6, d=16777259),
        # one server shard: the words of sixteen workers to the averaged gradient
        _case("decode_server_8m", "decode", "flat", 16, 512, 4, d=8388617),
        # gradients that live in pinned host memory
        _case("host_resnet18", "host", "resnet18", 4, 512, 4),
    ]


def draw(rng):
    call = rng.choice(["round", "round", "round", "update", "fourcall", "encode", "encode", "decode", "decode"])
    layout = rng.choice(["flat", "flat", "flat", "resnet18", "vgg16", "text"])
    M = 1 if call == "encode" and rng.random() < 0.5 else rng.choice([1, 2, 3, 4, 6, 8, 12, 16, 24, 32])
    bucket = rng.choice([0, 32, 96, 128, 256, 480, 512, 512, 512, 1024, 1024, 2048, 2048, 4096])
    if call == "encode" and bucket == 0:
        bucket = 512
    norm = "linf" if rng.random() < 0.2 else "l2"
    b = rng.choice([2, 3, 4, 4, 4, 5, 5, 6, 7, 8, 8, 10, 12, 16])
    c = _case("", call, layout, M, bucket, b, norm=norm)
    del c["name"]
    if layout == "flat":
        # over the logarithm of the size, mostly odd; at most 2^30 elements over all workers
        top = min(1 << 27, (1 << 30) // M)
        d = int(3000 * (top / 3000) ** rng.random())
        c["d"] = d | 1 if rng.random() < 0.7 else max(32, d // 1024 * 1024)
    else:
        c["shrink"] = int(64 ** rng.random())
    return c


# --------------------------------------------------------------------------------------------------
def _segments(case):
    if case["layout"] == "flat":
        return [case["d"]]
    return [max(1, n // case["shrink"]) for n in NETWORKS[case["layout"]]()]


def _gradients(case, L, segments, gen):
    """[M, D32] fp32 on the GPU: the distributions of ``workloads.py``, zero between the tensors."""
    dev = "cuda"
    shape = (case["M"], L.D32)
    if case["layout"] == "flat":
        g = torch.randn(shape, generator=gen, device=dev)
        g[:, case["d"]:] = 0.0
        return g
    # one number per element: the tensor's scale, 0 on the padding
    scale = torch.zeros(L.D32, device=dev)
    last = max(len(segments) - 1, 1)
    for i, (o, n) in enumerate(zip(L.offsets, segments)):
        scale[o: o + n] = 1e-2 * (10.0 ** (-i / last) if case["layout"] == "resnet18" else 1.0)
    if case["layout"] == "resnet18":                         # Laplace
        u = torch.rand(shape, generator=gen, device=dev).sub_(0.5)
        g = u.sign().mul_(-1).mul_(torch.log1p(u.abs().clamp_(max=0.4999999).mul_(-2.0)))
    else:
        g = torch.randn(shape, generator=gen, device=dev)
    if case["layout"] == "vgg16":                            # one entry in a hundred is 100 times larger
        big = torch.rand(shape, generator=gen, device=dev) < 0.01
        g = torch.where(big, g * 100.0, g)
    g.mul_(scale)
    if case["layout"] == "text":                             # 3 % of the embedding rows have a gradient
        rows = segments[0] // 300
        if rows:
            keep = torch.rand((case["M"], rows, 1), generator=gen, device=dev) < 0.03
            g[:, : rows * 300].view(case["M"], rows, 300).mul_(keep)
    return g


class _State:
    """What a user's training loop keeps: the round with its buffers, the rule's constants, the step counter."""


def prepare(case, seed):
    segments = _segments(case)
    norm = dq.NORM_LINF if case["norm"] == "linf" else dq.NORM_L2
    s = _State()
    s.call, s.step = case["call"], 0
    s.rnd = rnd = Round(segments, case["bucket"], case["M"], norm=norm)
    L = rnd.layout
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    s.grads = _gradients(case, L, segments, gen)
    # eps_hat such that x of Eq. 17 lies half a level below s(b) (alpha = 1: constant norms keep b)
    rnd.norms_(s.grads)
    g2 = float((rnd.norms.double() ** 2).sum().item()) / case["M"]
    s.eps_hat = T * g2 / ((1 << (case["b"] - 1)) - 1.5) ** 2
    rnd.bits_(dq.Rule.dynamic(T, 0, s.eps_hat, 1.0))
    assert rnd.bits() == case["b"], (rnd.bits(), case["b"])
    s.words = rnd.packed[:, : L.packed_words(case["b"])]     # the part of the stream b bits use
    if case["call"] == "update":
        s.params = torch.randn(L.D32, generator=gen, device="cuda").mul_(0.05)
    if case["call"] == "decode":
        rnd.norms_quantize_(s.grads, SEED, 0)
        s.grads = None
    if case["call"] == "host":
        s.grads = s.grads.cpu().pin_memory()
    return s


def run(s):
    rnd, step = s.rnd, s.step
    s.step = step + 1
    if s.call == "decode":
        rnd.average_()
        return rnd.out
    if s.call == "encode":
        rnd.norms_quantize_(s.grads, SEED, step)
        return rnd.norms, s.words
    rule = dq.Rule.dynamic(T, step % T, s.eps_hat, 1.0)
    if s.call == "round":
        out = rnd.step_fused(s.grads, rule, SEED, step)
    elif s.call == "update":
        out = rnd.step_fused(s.grads, rule, SEED, step, params=s.params, lr=1e-2)
    elif s.call == "fourcall":
        out = rnd.step(s.grads, rule, SEED, step)
    else:
        return rnd.step_host(s.grads, rule, SEED, step)
    return out, rnd.norms, s.words, rnd.dev_b


def _sizes(case):
    """(elements of all tensors, buckets) of one worker."""
    segments = _segments(case)
    per = case["bucket"]
    return sum(segments), sum(-(-n // per) if per else 1 for n in segments)


def work(case):
    d, nb = _sizes(case)
    M, b, call = case["M"], case["b"], case["call"]
    grads, norms, words, out = 4 * M * d, 4 * M * nb, M * d * b // 8, 4 * d
    # per element: 2 operations for its norm, 4 for its code (scale, draw, add, floor), and on the
    # server's side 2 for its share of the average
    if call == "decode":
        return {"bytes": words + norms + out, "flops": 2 * M * d}
    if call == "encode":
        return {"bytes": grads + norms + words, "flops": 6 * M * d}
    if call == "host":
        return {"bytes": grads + out, "flops": 8 * M * d}
    if call == "update":
        return {"bytes": grads + norms + words + 2 * out, "flops": 8 * M * d + 2 * d}
    return {"bytes": grads + norms + words + out, "flops": 8 * M * d}


def tolerance(case):
    # Against norms formed from 64-bit sums, norms and averages move by 2-norms of 2e-9 to 8e-8 and single
    # values by at most 1.6e-6 of their size or of the rms.  A code changes where its draw lies that close
    # to its position on the grid: up to 1.3e-5 of the words (16 bits), none at all with exact norms.
    # (One such change moves its average by a whole level, which the limits below do not allow for: the
    # sums of a bucket are taken in the library's own order.)
    words = 0.0 if case["norm"] == "linf" or case["call"] in ("decode", "host") else 5e-5
    return {"rel": 4e-7, "max": 8e-6, "differ": words}
