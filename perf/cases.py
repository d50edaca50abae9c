"""Performance cases of the DHQ forward path: what a program that uses this library has it do.

Three kinds of pass:
  forward  `dhq_forward` on coordinates and results in device memory, with a handle that the program
           prepared (and, for per-tensor activation scales, calibrated) once: rendering an image, a
           preview or a set of query points, over and over.
  host     `dhq_forward_host` on pinned host buffers: the same for a program whose data live on the host.
  open     from fp32 weights to the image: `dhq_prepare`, `dhq_calibrate`, `dhq_forward`,
           `dhq_destroy` - quantizing a newly arrived network and decoding it once.

Coordinates are pixel grids on [-1, 1]^2 or scattered points; networks are SIREN-initialised from the
seed, in the repository's own shapes (2 inputs, hidden width 64 to 512, 1 to 4 outputs).
"""
from __future__ import annotations

import math
import weakref

import torch

import paper_2508_13478_b200 as dhq
from dhq_inputs import siren_init

OMEGA0 = 30.0
GABOR_S0 = 10.0
FLOAT = dhq.DHQ_BITS_FLOAT
ROTATIONS = {"input": dhq.DHQ_ROT_INPUT, "both": dhq.DHQ_ROT_BOTH, "none": dhq.DHQ_ROT_NONE}


def _case(kind, rows, cols, width, hidden, d_out, w_bits=8, a_bits=8, per_channel=False, per_token=False,
          rotation="input", gabor=False, scatter=False):
    return {"kind": kind, "rows": rows, "cols": cols, "width": width, "hidden": hidden, "d_out": d_out,
            "w_bits": w_bits, "a_bits": a_bits, "per_channel": per_channel, "per_token": per_token,
            "rotation": rotation, "gabor": gabor, "scatter": scatter}


def listed():
    fine = {"per_channel": True, "per_token": True}
    cases = [
        # a thumbnail or a tile of a small grey-level network: launch latency counts
        ("thumb-w64", _case("forward", 64, 64, 64, 3, 1)),
        # a handful of scattered samples of an RGB network (picking, a line profile): one partial wave
        ("query-w256", _case("forward", 1, 1000, 256, 3, 3, scatter=True)),
        # an ordinary small RGB picture, scales per tensor
        ("image-w256", _case("forward", 256, 256, 256, 3, 3)),
        # deeper network, the finer scales (per output channel, per token)
        ("image-w256-fine", _case("forward", 512, 512, 256, 5, 3, **fine)),
        # the same network shape in 4-bit codes on a larger picture
        ("image-w256-4bit", _case("forward", 1024, 1024, 256, 5, 3, 4, 4, **fine)),
        # the largest: a wide network over a whole 2048 x 2048 picture
        ("large-w512", _case("forward", 2048, 2048, 512, 4, 3)),
        # wavelet network of intermediate width, without the rotation (the uniform quantizer that is
        # compared against), picture of odd size, grey level
        ("wavelet-w128-odd", _case("forward", 611, 437, 128, 4, 1, rotation="none", gabor=True)),
        # the two-sided transform with the finer scales
        ("two-sided-w256-fine", _case("forward", 512, 512, 256, 5, 3, rotation="both", **fine)),
        # the fp32 network, for the quality of the quantized one to be judged against
        ("fp32-w256", _case("forward", 256, 256, 256, 3, 3, FLOAT, FLOAT)),
        # weight-only quantization of the wide network
        ("w8a32-w512", _case("forward", 512, 512, 512, 4, 3, 8, FLOAT)),
        # pinned host buffers in and out, picture of odd size
        ("host-w256-odd", _case("host", 511, 767, 256, 3, 3)),
        # a network arrives, is quantized, calibrated on its picture and decoded once
        ("open-w256", _case("open", 256, 256, 256, 3, 3)),
    ]
    return [dict(c, name=name) for name, c in cases]


def draw(rng):
    kind = rng.choices(["forward", "float", "host", "open"], [6, 2, 1.5, 1.5])[0]
    width = rng.choice([64, 128, 256, 256, 512])
    hidden = rng.randint(2, 6)
    c = _case("forward" if kind == "float" else kind, 1, 1, width, hidden, rng.choice([1, 1, 2, 3, 3, 3, 4]))
    if kind == "float":
        c["w_bits"], c["a_bits"] = rng.choice([FLOAT, 8, 4]), FLOAT
        c["rotation"] = rng.choice(["input", "input", "none"])
    else:
        c["w_bits"], c["a_bits"] = rng.choice([(8, 8), (8, 8), (8, 8), (6, 6), (4, 4)])
        c["per_channel"], c["per_token"] = rng.choice([(False, False), (False, False), (True, True), (True, True), (True, False), (False, True)])
        c["rotation"] = rng.choices(["input", "none", "both"], [5, 1, 1])[0]
        c["gabor"] = rng.random() < 0.15
    # whole pictures up to 2048 x 2048 on the fused path; the others up to the work of their listed case
    macs = hidden * width * width
    if kind == "float":
        most = 512 * 512 * 4 * 512 * 512 / macs
    elif c["rotation"] == "both" and c["per_channel"]:
        most = 512 * 512 * 5 * 256 * 256 / macs
    elif kind == "open":
        most = 1024 * 1024
    else:
        most = 2048 * 2048 * 4 * 512 * 512 / macs
    most = min(most, 2048 * 2048)
    n = math.exp(rng.uniform(math.log(64), math.log(most)))
    if kind in ("forward", "float") and n <= 4096 and rng.random() < 0.5:
        c["scatter"], c["cols"] = True, int(n)
    else:
        c["rows"] = max(1, int(math.sqrt(n * math.exp(rng.uniform(-0.7, 0.7)))))
        c["cols"] = max(1, int(n / c["rows"]))
    return c


def _dims(case):
    return tuple([2] + [case["width"]] * case["hidden"] + [case["d_out"]])


def _grid(rows, cols):
    def axis(n):
        if n == 1:
            return torch.zeros(1, dtype=torch.float32, device="cuda")
        return (-1.0 + 2.0 * torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1)).float()
    gy, gx = torch.meshgrid(axis(rows), axis(cols), indexing="ij")
    return torch.stack((gy, gx), dim=-1).reshape(-1, 2).contiguous()


def _granularity(fine):
    return dhq.DHQ_GRAN_CHANNEL_OR_TOKEN if fine else dhq.DHQ_GRAN_TENSOR


class State:
    def __init__(self, case, seed):
        self.kind = case["kind"]
        self.handle = None
        self.dims = _dims(case)
        weights, biases = siren_init(self.dims, OMEGA0, seed)
        self.weights = [torch.from_numpy(w).cuda() for w in weights]
        self.biases = [torch.from_numpy(b).cuda() for b in biases]
        self.options = {
            "omega0": OMEGA0, "w_bits": case["w_bits"], "a_bits": case["a_bits"],
            "w_gran": _granularity(case["per_channel"]), "a_gran": _granularity(case["per_token"]),
            "rotation": ROTATIONS[case["rotation"]],
            "activation": dhq.DHQ_ACT_GABOR if case["gabor"] else dhq.DHQ_ACT_SINE,
            "act_s0": GABOR_S0 if case["gabor"] else 0.0,
        }
        n = case["rows"] * case["cols"]
        if case["scatter"]:
            gen = torch.Generator(device="cuda").manual_seed(seed)
            self.coords = torch.rand((n, 2), generator=gen, device="cuda") * 2.0 - 1.0
        else:
            self.coords = _grid(case["rows"], case["cols"])
        if self.kind != "open":
            self.handle = dhq.dhq_prepare(self.dims, self.weights, self.biases, **self.options)
            weakref.finalize(self, dhq.dhq_destroy, self.handle)
            # per-tensor activation scales are frozen on the picture (a no-op for the other handles)
            dhq.dhq_calibrate(self.handle, _grid(256, 256) if case["scatter"] else self.coords)
        self.out = torch.empty((n, case["d_out"]), device="cuda")
        if self.kind == "host":
            self.coords = self.coords.cpu().pin_memory()
            self.out = torch.empty((n, case["d_out"])).pin_memory()
        torch.cuda.synchronize()


def prepare(case, seed):
    return State(case, seed)


def run(state):
    if state.kind == "forward":
        dhq.dhq_forward(state.handle, state.coords, state.out)
    elif state.kind == "host":
        dhq.dhq_forward_host(state.handle, state.coords, state.out)
    else:
        handle = dhq.dhq_prepare(state.dims, state.weights, state.biases, **state.options)
        dhq.dhq_calibrate(handle, state.coords)
        dhq.dhq_forward(handle, state.coords, state.out)
        dhq.dhq_destroy(handle)
    return state.out


def work(case):
    dims, n = _dims(case), case["rows"] * case["cols"]
    macs = sum(a * b for a, b in zip(dims, dims[1:]))
    flops = 2.0 * macs
    if case["w_bits"] != FLOAT and case["rotation"] != "none":
        flops += case["hidden"] * case["width"] * math.log2(case["width"])
    if case["rotation"] == "both":
        flops += case["hidden"] * case["width"] * math.log2(case["width"])
    # weights as the pass finds them: fp32 before quantization, else one byte a code and the scales
    fp32 = case["kind"] == "open" or case["w_bits"] == FLOAT
    weights = 4 * (macs + sum(dims[1:])) if fp32 else macs + 8 * sum(dims[1:])
    return {"bytes": 8.0 * n + 4.0 * case["d_out"] * n + weights, "flops": flops * n}


def tolerance(case):
    if case["a_bits"] == FLOAT:
        # sums of up to 512 fp32 products in another order, through a chain of sines
        return {"rel": 2e-5}
    # A phase that differs in its last bit moves a value across a rounding boundary of the activation
    # quantizer now and then: one code step there, a wider step with fewer bits, which spreads over
    # the outputs of that coordinate.  The limits are 1.5 to 2 times what two implementations within
    # 1e-5 per layer were seen to differ by on 65,536 coordinates of 5-layer networks (the two-sided
    # transform with an fp32 and with an fp64 epilogue, width 512: 1.3e-3, 2.2e-3, 8.1e-3 at 8, 6, 4
    # bits, largest single differences 0.05, 0.12, 0.42 of the result's root mean square).
    return {8: {"rel": 2e-3, "max": 0.1}, 6: {"rel": 4e-3, "max": 0.25}, 4: {"rel": 1.5e-2, "max": 0.8}}[case["a_bits"]]
