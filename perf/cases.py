"""Performance cases of the library: what its users run, through the Python binding's public calls.

Three kinds of use are covered, each over its real range of sizes:
  - whole networks (`binding.Network.run`): the layer tables of the benchmark workloads, from one image per request to
    the throughput batch, with every table option (8 bit, mixed 4/8 bit, INT32 residual stream, Inception modules);
  - one convolution layer (`Handle.conv2d`): the layers a caller with its own graph runner issues one by one;
  - one memory-bound layer (`Handle.residual_add`, `Handle.concat_requant`).
All results are integers and are compared exactly.
"""
from __future__ import annotations

import math

import torch

from paper_2011_10680_b200 import binding, inputs


# --------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------
def _network(name, table, batch, image_hw):
    return {"name": name, "kind": "network", "table": table, "batch": batch, "image_hw": image_hw}


def _conv(name, n, hw, cin, cout, k, stride, bits, out_bits, residual):
    return {"name": name, "kind": "conv", "n": n, "hw": hw, "cin": cin, "cout": cout, "k": k, "stride": stride,
            "bits": bits, "out_bits": out_bits, "residual": residual}


def listed():
    return [
        # throughput serving / offline scoring: the headline workload
        _network("resnet50_int8_b256", "resnet50", 256, 224),
        # the same with the last two stages at 4 bit (the paper's mixed-precision deployment)
        _network("resnet50_mixed_b256", "resnet50_mixed", 256, 224),
        # the dataflow of Fig. 2 as drawn, residual stream kept in INT32 between blocks; a medium batch
        _network("resnet50_int32stream_b64", "resnet50_int32", 64, 224),
        # concatenating networks: Inception modules with 4-bit convolutions and INT32 pooling branches
        _network("inception_int4_b256", "inception", 256, 71),
        # a small batch of a small network: online serving with light batching
        _network("resnet18_int8_b8", "resnet18", 8, 224),
        # one request, one image: latency
        _network("resnet50_int8_b1", "resnet50", 1, 224),
        # what a dynamic batcher hands over: an odd batch of a smaller image size, mixed precision
        _network("resnet50_mixed_b13_192", "resnet50_mixed", 13, 192),
        # the smallest call: one layer of one image (the single-layer benchmark configuration)
        _conv("conv3x3_64_56_b1", 1, 56, 64, 64, 3, 1, 8, 8, False),
        # the longest reduction of the layer sweep at a large batch: bound by the tensor cores
        _conv("conv3x3_512_7_b256", 256, 7, 512, 512, 3, 1, 8, 8, False),
        # a packed 4-bit layer with the fused residual add at an odd batch
        _conv("conv1x1_256_1024_14_b37_int4_res", 37, 14, 256, 1024, 1, 1, 4, 8, True),
        # the stored-tensor residual add of a caller that does not fuse it
        {"name": "add_u8_56_256_b64", "kind": "add", "n": 64, "hw": 56, "ch": 256, "main_bits": 8, "res_bits": 8, "out_bits": 8},
        # one concatenation of an Inception 35x35 module, a dyadic pair per channel
        {"name": "concat_35_b256", "kind": "concat", "n": 256, "hw": 35, "ch": 64, "ch2": 96, "pool_ch": 64, "per_channel": True},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    named = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        c = _draw_one(rng)
        if c not in named:
            return c


def _draw_one(rng):
    u = rng.random()
    if u < 0.5:
        table = rng.choice(["resnet50", "resnet50", "resnet50_mixed", "resnet18", "resnet50_int32", "inception"])
        if table == "inception":
            hw = rng.choice([55, 63, 71, 79, 87])
            top = min(256, int(256 * 71 * 71 / (hw * hw)))
        else:
            hw = 224 if rng.random() < 0.3 else rng.randrange(96, 257, 8)
            top = min(256, int((64 if table == "resnet50_int32" else 256) * 224 * 224 / (hw * hw)))
        return {"kind": "network", "table": table, "batch": _log_uniform(rng, 1, top), "image_hw": hw}
    if u < 0.75:
        while True:
            c = {"kind": "conv", "n": _log_uniform(rng, 1, 256), "hw": _log_uniform(rng, 7, 112),
                 "cin": _log_uniform(rng, 16, 1024), "cout": _log_uniform(rng, 16, 2048), "k": rng.choice([1, 1, 3]),
                 "stride": rng.choice([1, 1, 1, 2]), "bits": rng.choice([8, 8, 4]), "out_bits": rng.choice([8, 8, 4, 32]),
                 "residual": rng.random() < 0.3}
            for key in ("cin", "cout"):            # channel counts of real layers: multiples of 16, of 32 from 256 up
                step = 16 if c[key] < 256 else 32
                c[key] = max(step, c[key] // step * step)
            c["residual"] = c["residual"] and c["out_bits"] == 8
            ho = _out(c["hw"], c["k"], c["stride"])
            pixels = c["n"] * ho * ho
            if (pixels * c["cout"] * c["k"] * c["k"] * c["cin"] <= 2.5e11 and pixels * c["cout"] <= 1.5e8
                    and c["n"] * c["hw"] ** 2 * c["cin"] <= 3e8):
                return c
    if u < 0.875:
        while True:
            c = {"kind": "add", "n": _log_uniform(rng, 1, 256), "hw": _log_uniform(rng, 7, 112),
                 "ch": max(16, _log_uniform(rng, 16, 2048) // 16 * 16), "main_bits": rng.choice([8, 8, 32]),
                 "res_bits": rng.choice([0, 8, 8, 32]), "out_bits": rng.choice([8, 8, 4, 32])}
            if c["n"] * c["hw"] ** 2 * c["ch"] <= 2.1e8:
                return c
    hw = rng.choice([17, 35, 35, _log_uniform(rng, 8, 40)])
    ch = rng.choice([64, 192]) if hw <= 17 else 64
    return {"kind": "concat", "n": _log_uniform(rng, 1, 256), "hw": hw, "ch": ch, "ch2": ch * 3 // 2 if hw > 17 else ch,
            "pool_ch": rng.choice([32, 64, 192]), "per_channel": rng.random() < 0.5}


# --------------------------------------------------------------------------------------------
# State
# --------------------------------------------------------------------------------------------
def _out(hw, k, stride):
    return (hw + 2 * (k // 2) - k) // stride + 1


def _table(case, seed):
    if case["table"] == "inception":
        return inputs.inception_table(seed, conv_bits=4, image_hw=case["image_hw"])
    return inputs.resnet_table(18 if case["table"] == "resnet18" else 50, seed, mixed=case["table"] == "resnet50_mixed",
                               image_hw=case["image_hw"], int32_stream=case["table"] == "resnet50_int32")


class _Draw:
    """Seeded device tensors with the value ranges of the quantizers."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def ints(self, lo, hi, shape, dtype):
        return torch.randint(lo, hi, shape, generator=self.g, device="cuda", dtype=torch.int32).to(dtype)

    def acts(self, shape, ch, bits):
        """Activations: uniform unsigned 8-bit, packed unsigned 4-bit (two per byte), or signed INT32 accumulators."""
        if bits == 32:
            return self.ints(-(1 << 20), 1 << 20, (*shape, ch), torch.int32)
        return self.ints(0, 256, (*shape, ch * bits // 8), torch.uint8)

    def pairs(self, ch, lo, hi, uniform=False):
        """Dyadic pairs (b, c) of `ch` channels, c in [lo, hi]; uniform: one pair for all of them."""
        b, c = self.ints(1 << 30, (1 << 31) - 1, (1 if uniform else ch,), torch.int32), self.ints(lo, hi + 1, (1 if uniform else ch,), torch.int32)
        return (b.expand(ch).contiguous(), c.expand(ch).contiguous()) if uniform else (b, c)


def _empty(n, hw, ch, bits):
    dtype = torch.int32 if bits == 32 else torch.uint8
    return torch.empty((n, hw, hw, ch if bits != 4 else ch // 2), dtype=dtype, device="cuda")


def prepare(case, seed):
    d = _Draw(seed)
    s = dict(case=case, hq=binding.Handle(0))
    if case["kind"] == "network":
        s["net"] = binding.Network(s["hq"], _table(case, seed), case["batch"])
        s["images"] = d.ints(0, 256, (case["batch"], case["image_hw"], case["image_hw"], 3), torch.uint8)
        s["logits"] = torch.empty(s["net"].logits_shape, dtype=torch.int32, device="cuda")
    elif case["kind"] == "conv":
        n, hw, cin, cout, k, bits = (case[f] for f in ("n", "hw", "cin", "cout", "k", "bits"))
        ho = _out(hw, k, case["stride"])
        s["x"] = d.acts((n, hw, hw), cin, bits)
        if bits == 8:
            s["wgt"] = d.ints(-127, 128, (cout, k, k, cin), torch.int8)
        else:
            lo, hi = (d.ints(-7, 8, (cout, k, k, cin // 2), torch.int32) & 15 for _ in range(2))
            s["wgt"] = (lo | (hi << 4)).to(torch.uint8)
        s["bias"] = d.ints(-(1 << 15), (1 << 15) + 1, (cout,), torch.int32)
        # shifts that spread the accumulators over the output range: their typical size is sqrt(K) * input * weight
        spread = math.log2(math.sqrt(k * k * cin) * (128 * 73 if bits == 8 else 7.5 * 4.3))
        c = int(round(spread)) + 30 - {8: 7, 4: 3, 32: 7}[case["out_bits"]]
        s["b"], s["c"] = d.pairs(cout, c - 1, c + 2)
        s["res"] = s["rb"] = s["rc"] = None
        if case["residual"]:
            s["res"] = d.acts((n, ho, ho), cout, 8)
            s["rb"], s["rc"] = d.pairs(cout, 30, 33)
        s["out"] = _empty(n, ho, cout, case["out_bits"])
    elif case["kind"] == "add":
        shape, ch = (case["n"], case["hw"], case["hw"]), case["ch"]
        down = 4 if case["out_bits"] == 4 else 0
        for key, pair, bits in (("main", ("mb", "mc"), case["main_bits"]), ("res", ("rb", "rc"), case["res_bits"])):
            s[key] = s[pair[0]] = s[pair[1]] = None
            if bits:
                s[key] = d.acts(shape, ch, bits)
                lo = 30 if bits == 8 or case["out_bits"] == 32 else 42
                s[pair[0]], s[pair[1]] = d.pairs(ch, lo + down, lo + down + 3)
        s["out"] = _empty(case["n"], case["hw"], ch, case["out_bits"])
    else:
        s["branches"] = []
        for ch, bits in ((case["ch"], 8), (case["ch"], 8), (case["ch2"], 8), (case["pool_ch"], 32)):
            b, c = d.pairs(ch, *((44, 48) if bits == 32 else (30, 33)), uniform=not case["per_channel"])
            s["branches"].append({"x": d.acts((case["n"], case["hw"], case["hw"]), ch, bits), "bits": bits,
                                  "signed": int(bits == 32), "ch": ch, "b": b, "c": c})
        s["out"] = _empty(case["n"], case["hw"], 2 * case["ch"] + case["ch2"] + case["pool_ch"], 8)
    return s


_STREAM = []


def _inference_stream():
    """The program's one inference stream: networks are replayed as graphs on a stream of their own, in order."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _range(bits):
    return (-(1 << 31), (1 << 31) - 1) if bits == 32 else (0, (1 << bits) - 1)


def run(s):
    case, hq = s["case"], s["hq"]
    if case["kind"] == "network":
        with torch.cuda.stream(_inference_stream()):
            st, out = s["net"].run(s["images"], s["logits"]), s["logits"]
    elif case["kind"] == "conv":
        qmin, qmax = _range(case["out_bits"])
        k, out = case["k"], s["out"]
        st = hq.conv2d(s["x"], case["bits"], 0, case["cin"], s["wgt"], case["cout"], k, k, case["stride"], k // 2, s["bias"],
                       s["b"], s["c"], out, case["out_bits"], int(case["out_bits"] == 32), s["res"], 8, 0, s["rb"], s["rc"],
                       1, qmin, qmax)
    elif case["kind"] == "add":
        qmin, qmax = _range(case["out_bits"])
        out = s["out"]
        st = hq.residual_add(s["main"], case["main_bits"], int(case["main_bits"] == 32), s["mb"], s["mc"],
                             s["res"], case["res_bits"], int(case["res_bits"] == 32), s["rb"], s["rc"], case["ch"],
                             1, qmin, qmax, out, case["out_bits"], int(case["out_bits"] == 32))
    else:
        out = s["out"]
        st = hq.concat_requant(s["branches"], 1, 0, 255, out, 8, 0)
    if st != binding.HQ_OK:
        raise RuntimeError(binding.status_string(st))
    return out


# --------------------------------------------------------------------------------------------
# Least work and tolerance
# --------------------------------------------------------------------------------------------
_COST = {}


def _network_cost(case):
    """Multiply-accumulates of one image, parameter bytes (weights, bias, dyadic pairs): a function of the table's shapes."""
    key = (case["table"], case["image_hw"])
    if key not in _COST:
        layers = _table(case, 0)["layers"]
        macs = sum(l["macs"] for l in layers)
        params = sum(l["params"] * l["bits"] // 8 + 12 * l["cout"] for l in layers if l["op"] in ("conv", "linear"))
        _COST[key] = (macs, params, layers[-1]["cout"])
    return _COST[key]


def work(case):
    if case["kind"] == "network":
        macs, params, classes = _network_cost(case)
        b = case["batch"]
        return {"bytes": b * case["image_hw"] ** 2 * 3 + params + b * classes * 4, "flops": 2 * macs * b}
    if case["kind"] == "conv":
        ho = _out(case["hw"], case["k"], case["stride"])
        pixels, kk = case["n"] * ho * ho, case["k"] ** 2 * case["cin"]
        # a 1x1 / stride 2 layer reads the sampled pixels only
        in_pixels = pixels if case["k"] == 1 else case["n"] * case["hw"] ** 2
        return {"bytes": (in_pixels * case["cin"] + case["cout"] * kk) * case["bits"] // 8 + 12 * case["cout"]
                + pixels * case["cout"] * (case["out_bits"] / 8 + (1 if case["residual"] else 0)),
                "flops": 2 * pixels * case["cout"] * kk}
    if case["kind"] == "add":
        values = case["n"] * case["hw"] ** 2 * case["ch"]
        return {"bytes": values * (case["main_bits"] + case["res_bits"] + case["out_bits"]) // 8, "flops": 2 * values}
    pixels = case["n"] * case["hw"] ** 2
    stored = 2 * case["ch"] + case["ch2"]
    return {"bytes": pixels * (2 * stored + 5 * case["pool_ch"]), "flops": 2 * pixels * (stored + case["pool_ch"])}


def tolerance(case):
    return "exact"
