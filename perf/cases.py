"""The timed cases of this library: one compress + average step of every compressor family.

One pass is what a data-parallel training step does with the library: `mlmc_compress_*` turns the M workers' gradients
into their messages, `mlmc_aggregate*` averages the messages into the dense gradient.  The step number advances from
pass to pass, so every pass draws its own levels.  `prepare` makes the gradients (seeded, synthetic: per-layer scales,
Gaussian or heavy-tailed entries) and what a training program keeps between steps: the context, the message buffers and
the dense output.
"""
import torch

from paper_2507_05508_b200 import binding as B
from paper_2507_05508_b200 import workloads as wl

MAX_LEVELS = 32
FIXED_POINT = "1,2,4,8,16,23"      # bits kept by the fixed-point levels
RTN_WIDTHS = "2,4,8,16"            # grid widths of the round-to-nearest levels
MANTISSA = {"f32": "1,2,4,8,16,23", "bf16": "1,2,4,7"}
MOST_ENTRIES = 8 * 124_439_808     # entries (M * d) of the largest listed cases
MOST_SORTED = 16 * 11_689_512      # entries of the largest listed s-Top-k case with adaptive probabilities


def _case(kind, d, M, dtype="f32", adaptive=False, dist="normal", scale="segments", segments=0, lo=1e-4, hi=1e-1,
          outliers=False, k_den=0, seg_len=0, bits=""):
    return {"kind": kind, "d": d, "M": M, "dtype": dtype, "adaptive": adaptive, "dist": dist, "scale": scale,
            "segments": segments, "lo": lo, "hi": hi, "outliers": outliers, "k_den": k_den, "seg_len": seg_len,
            "bits": bits}


def listed():
    transformer = dict(segments=148, lo=1e-5, hi=1e-1, outliers=True)  # 124M parameters, fp32, rare large coordinates
    resnet18 = dict(segments=62)
    cases = {
        # the smallest step: one small tensor (an embedding, a classifier head) compressed by itself; latency counts
        "topk_fixed_65k": _case("topk", 65_536, 4, scale="coord_loguniform", lo=1e-3, hi=1.0, k_den=1024),
        # a single layer of odd length, adaptive probabilities
        "topk_adaptive_700k": _case("topk", 700_001, 3, adaptive=True, k_den=10_000, **transformer),
        # a mixed-precision layer: bf16 gradients, odd length
        "bitwise_adaptive_bf16_400k": _case("bitwise", 400_003, 6, "bf16", True, "student_t3", segments=161,
                                            bits=FIXED_POINT),
        # a small model with the bit-wise compressor at its optimal fixed probabilities
        "bitwise_fixed_1m": _case("bitwise", 1_048_576, 8, dist="student_t3", scale="const", lo=1e-2, hi=1e-2,
                                  bits=FIXED_POINT),
        # ResNet-18-sized gradients, levels drawn from fixed probabilities
        "topk_fixed_12m": _case("topk", 11_689_512, 16, k_den=1000, **resnet18),
        # the same gradients in segments of 0.1 % of the sorted vector, fixed probabilities over 1000 levels
        "stopk_fixed_12m": _case("stopk", 11_689_512, 16, seg_len=11_690, **resnet18),
        # segments of 1 %, adaptive probabilities: the paper's Adaptive MLMC-Top-k runs
        "stopk_adaptive_12m": _case("stopk", 11_689_512, 16, adaptive=True, seg_len=116_896, **resnet18),
        # ResNet-50-sized bf16 gradients of 32 workers, adaptive probabilities
        "topk_adaptive_bf16_26m": _case("topk", 25_557_032, 32, "bf16", True, "student_t3", segments=161, k_den=2000),
        # GPT-2-small-sized gradients through each family: the largest steps
        "topk_adaptive_124m": _case("topk", 124_439_808, 8, adaptive=True, k_den=10_000, **transformer),
        "bitwise_adaptive_124m": _case("bitwise", 124_439_808, 8, adaptive=True, bits=FIXED_POINT, **transformer),
        "floatbits_124m": _case("floatbits", 124_439_808, 8, bits=MANTISSA["f32"], **transformer),
        "rtn_adaptive_124m": _case("rtn", 124_439_808, 8, adaptive=True, bits=RTN_WIDTHS, **transformer),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def draw(rng):
    """A layer, a bucket or a whole model: 8 thousand to 125 million parameters, 2 to 32 workers."""
    kind = rng.choice(["topk", "topk", "stopk", "bitwise", "floatbits", "rtn"])
    dtype = rng.choice(["f32", "f32", "bf16"])
    adaptive = kind != "floatbits" and rng.random() < 0.6
    M = rng.choice([2, 3, 4, 5, 8, 16, 32])
    most = MOST_SORTED if kind == "stopk" and adaptive else MOST_ENTRIES * (3 if kind == "rtn" else 4) // 4
    d = int(round(8192 * (125e6 / 8192) ** rng.random()))
    d = min(d, most // M)
    if rng.random() < 0.5:
        d |= 1
    k_den = rng.choice([20, 100, 1000, 2000, 10_000]) if kind == "topk" else 0
    seg_len = max(1, int(d * rng.choice([0.001, 0.005, 0.01, 0.05, 0.1]))) if kind == "stopk" else 0
    bits = {"bitwise": rng.choice([FIXED_POINT, "1,2,3,4,5,6,7,8"]), "floatbits": MANTISSA[dtype],
            "rtn": rng.choice([RTN_WIDTHS, "2,3,4,8"])}.get(kind, "")
    return _case(kind, d, M, dtype, adaptive, rng.choice(["normal", "student_t3"]), segments=rng.choice([62, 148, 161]),
                 lo=rng.choice([1e-5, 1e-4]), hi=1e-1, outliers=rng.random() < 0.3, k_den=k_den, seg_len=seg_len, bits=bits)


def _bits(case):
    return [int(x) for x in case["bits"].split(",")]


def _widths(bits):
    return [b - a for a, b in zip([0] + bits[:-1], bits)]


def _workload(case, seed):
    return wl.Workload(case["kind"], case["kind"], case["d"], case["M"], case["dtype"], case["adaptive"], seed, 0,
                       case["dist"], case["scale"], case["lo"], case["hi"],
                       segments=min(case["segments"], max(1, case["d"] // 8)),
                       outlier_frac=1e-3 if case["outliers"] else 0.0, outlier_mult=100.0, k_den=case["k_den"],
                       seg_len=case["seg_len"])


def _levels(case):
    if case["kind"] == "stopk":
        return -(-case["d"] // case["seg_len"])
    if case["kind"] == "topk":
        return len(wl.topk_schedule(_workload(case, 0)))
    return len(_bits(case)) + (case["kind"] == "rtn")


class State:
    """Gradients, and what a training program keeps from step to step."""

    def __init__(self, case, seed):
        w = _workload(case, seed)
        d, M = case["d"], case["M"]
        self.kind, self.d, self.M, self.seed, self.step, self.ctx = case["kind"], d, M, seed, 0, None
        g = wl.gradients(w, 0, "cuda")
        per16 = 16 // g.element_size()
        if d % per16:  # rows start on 16-byte boundaries
            rows = torch.zeros((M, -(-d // per16) * per16), dtype=g.dtype, device="cuda")
            rows[:, :d] = g
            g = rows[:, :d]
        self.g = g
        L = _levels(case)
        self.p = None if case["adaptive"] or self.kind == "floatbits" else list(wl.geometric_probs(L))
        if self.kind == "topk":
            self.sched = wl.topk_schedule(w)
            self.out = B.TopkBuffers(M, wl.max_band(self.sched))
        elif self.kind == "stopk":
            self.sched = case["seg_len"]
            self.out = B.TopkBuffers(M, min(self.sched, d))
        else:
            self.sched = _bits(case)
            if self.kind == "rtn":
                self.out = B.RtnBuffers(M, d)
            else:
                buffers = B.BitBuffers if self.kind == "bitwise" else B.FloatBuffers
                self.out = buffers(M, d, max(_widths(self.sched)))
        if self.kind in ("topk", "stopk"):  # a message shorter than its buffer leaves the rest as it was
            self.out.idx.zero_()
            self.out.val.zero_()
        self.dense = torch.zeros(d, dtype=torch.float32, device="cuda")
        self.ctx = B.mlmc_create(torch.cuda.current_device(), d, M, MAX_LEVELS)

    def __del__(self):
        if self.ctx is not None:
            B.mlmc_destroy(self.ctx)


def prepare(case, seed):
    return State(case, seed)


def run(s):
    step, s.step = s.step, s.step + 1
    out = s.out
    if s.kind == "topk":
        B.mlmc_compress_topk(s.ctx, s.g, s.sched, s.p, s.seed, step, out)
        B.mlmc_aggregate(s.ctx, B.MLMC_TOPK, out, None, s.M, s.d, s.dense)
    elif s.kind == "stopk":
        B.mlmc_compress_stopk(s.ctx, s.g, s.sched, s.p, s.seed, step, out)
        B.mlmc_aggregate(s.ctx, B.MLMC_TOPK, out, None, s.M, s.d, s.dense)
    elif s.kind == "bitwise":
        B.mlmc_compress_bitwise(s.ctx, s.g, s.sched, s.p, s.seed, step, out)
        B.mlmc_aggregate(s.ctx, B.MLMC_BITWISE, out, s.sched, s.M, s.d, s.dense)
    elif s.kind == "floatbits":
        B.mlmc_compress_floatbits(s.ctx, s.g, s.sched, s.p, s.seed, step, out)
        B.mlmc_aggregate_floatbits(s.ctx, out, s.sched, s.M, s.d, s.dense)
    else:
        B.mlmc_compress_rtn(s.ctx, s.g, s.sched, s.p, s.seed, step, out)
        B.mlmc_aggregate_rtn(s.ctx, out, s.M, s.d, s.dense)
    head = {"level": out.level, "p_sel": out.p_sel, "dense": s.dense}
    if s.kind in ("topk", "stopk"):
        return dict(head, idx=out.idx, val=out.val, count=out.count)
    if s.kind == "bitwise":
        return dict(head, planes=out.planes, gmax=out.gmax)
    if s.kind == "floatbits":
        return dict(head, planes=out.planes, expo=out.expo)
    return dict(head, val=out.val, c=out.c)


def _message_bytes(case):
    """Bytes of one worker's message: its mean over the fixed probabilities, or its smallest size where the probabilities
    follow from the data."""
    d, kind, L = case["d"], case["kind"], _levels(case)
    if kind == "rtn":
        return 4.0 * d
    if kind == "stopk":
        return 8.0 * min(case["seg_len"], d)
    if kind == "topk":
        ks = wl.topk_schedule(_workload(case, 0))
        sizes = [8.0 * (b - a) for a, b in zip([0] + ks[:-1], ks)]
    else:
        sizes = [(1 + w) * 4.0 * -(-d // 32) + (d if kind == "floatbits" else 0) for w in _widths(_bits(case))]
    if case["adaptive"]:
        return min(sizes)
    if kind == "floatbits":
        bits = _bits(case)
        weights = [2.0 ** -a - 2.0 ** -b for a, b in zip([0] + bits[:-1], bits)]
    else:
        weights = list(wl.geometric_probs(L))
    return sum(s * w for s, w in zip(sizes, weights)) / sum(weights)


def work(case):
    """The gradients read once, the messages and the dense mean written once; one operation per entry, and for adaptive
    probabilities a square and a sum more."""
    entries = case["M"] * case["d"]
    return {"bytes": float(entries * (2 if case["dtype"] == "bf16" else 4) + case["M"] * _message_bytes(case) + 4 * case["d"]),
            "flops": float(entries * (3 if case["adaptive"] else 1))}


def tolerance(case):
    """Levels, indices, counts, planes and exponent bytes are exact; message values and means are fp32 (one or two
    roundings per value, M additions per mean), probabilities fp64."""
    return {"rel": 1e-6, "max": 1e-5}
