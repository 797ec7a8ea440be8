"""What this framework is used for, as measurable cases: networks handed over as graphs, compiled once and run many times.

A case is one network at one batch size, input resolution and storage type:

  net       "v1" | "v2"  MobileNetV1 / MobileNetV2 classification (1001 classes)
            "seg"        the MobileNetV2 backbone at output stride 16 with the segmentation head and its bilinear up-sampling
            "fire"       the fire-module network (2x2, 3x3 and stride-3 convolutions, concatenation)
            "block"      one depthwise-separable block, the smallest graph anybody hands over
  batch     images per call
  size      height and width of the input image
  storage   "f16" (fp16 storage, fp32 accumulation) | "f32" (fp32 throughout: the validation mode)
  source    "device": NHWC images resident on the GPU, results left there, through Executable.run
            "host":   images and results in pinned host memory, through HostPipeline.submit

Weights are the networks' own seeded ones (random: there are no trained models here); images are uniform in [-1, 1] and
representable in fp16, as in the repository's tests and benchmark.
"""
import math

import torch

from paper_1907_01989_b200 import api
from paper_1907_01989_b200 import workloads as wl
from paper_1907_01989_b200.pipeline import HostPipeline

_MAKE = {"v1": wl.mobilenet_v1, "v2": wl.mobilenet_v2, "seg": wl.mobilenet_v2_segmentation, "fire": wl.fire_network,
         "block": lambda batch, size: wl.separable_block(batch, size, size)}
_STORAGE = {"f16": (api.GI_F16, torch.float16), "f32": (api.GI_F32, torch.float32)}


def listed():
    def case(name, net, batch, size, storage="f16", source="device"):
        return {"name": name, "net": net, "batch": batch, "size": size, "storage": storage, "source": source}

    return [
        # one separable block on one small feature map: what a call costs when there is next to nothing to compute
        case("block_b1", "block", 1, 32),
        # one camera frame through the classifier: the latency case the paper's engine was built for
        case("v2_b1", "v2", 1, 224),
        # one frame through the segmentation network: odd planes (257, 129, 65, 33) and dilated layers
        case("seg_b1", "seg", 1, 513),
        # a handful of requests served together, at a reduced resolution
        case("v2_b8_192", "v2", 8, 192),
        # the same for the older network, at a batch that a server collects under load
        case("v1_b32_160", "v1", 32, 160),
        # images as they come: an odd resolution (every plane is odd) and a batch that fills nothing evenly
        case("v2_b21_205", "v2", 21, 205),
        # throughput: the repository's headline benchmark
        case("v2_b256", "v2", 256, 224),
        # throughput of the older network, whose last layers are bound by arithmetic
        case("v1_b256", "v1", 256, 224),
        # throughput of segmentation: large planes, and an output far larger than its input
        case("seg_b16", "seg", 16, 513),
        # full 2x2 / 3x3 convolutions and concatenations in many small launches
        case("fire_b64", "fire", 64, 96),
        # fp32 storage: a few images checked against the fp16 path
        case("v2_f32_b2", "v2", 2, 224, storage="f32"),
        # images decoded on the host, answers read back: the end-to-end path
        case("v2_host_b64", "v2", 64, 224, source="host"),
    ]


def draw(rng):
    """A case of the same ranges: any network, resolutions from the usual ones or any whole number in the range, batch
    sizes spread over their logarithm up to the work of the largest listed case of that network."""
    net = rng.choices(["v2", "v1", "seg", "fire", "block"], weights=[6, 4, 2, 2, 1])[0]
    usual, lo, hi, most, pixels = {
        "v2": ([96, 128, 160, 192, 224], 65, 288, 256, 256 * 224 * 224),
        "v1": ([96, 128, 160, 192, 224], 65, 288, 256, 256 * 224 * 224),
        "seg": ([129, 257, 321, 385, 513], 97, 513, 16, 16 * 513 * 513),
        "fire": ([64, 96, 128], 33, 160, 256, 256 * 96 * 96),
        "block": ([16, 32, 64], 7, 112, 64, 64 * 112 * 112),
    }[net]
    size = rng.choice(usual) if rng.random() < 0.4 else rng.randint(lo, hi)
    storage = "f32" if rng.random() < 0.1 else "f16"
    source = "host" if storage == "f16" and net in ("v1", "v2") and rng.random() < 0.1 else "device"
    if storage == "f32":
        pixels //= 128
    most = max(1, min(most, pixels // (size * size)))
    batch = min(most, int(math.exp(rng.uniform(0.0, math.log(most + 1)))))
    return {"net": net, "batch": batch, "size": size, "storage": storage, "source": source}


def prepare(case, seed):
    spec = _MAKE[case["net"]](case["batch"], size=case["size"])
    storage, dtype = _STORAGE[case["storage"]]
    graph, _ = api.graph_from_spec(spec, storage)
    ex = graph.compile()
    ex.bind("cuda:0")
    gen = torch.Generator(device="cuda:0").manual_seed(seed)
    shape_in = (spec.batch,) + tuple(spec.shapes[spec.inputs[0]])
    shape_out = (spec.batch,) + tuple(spec.shapes[spec.outputs[0]])
    x = torch.rand(shape_in, generator=gen, device="cuda:0").mul_(2).sub_(1).half().to(dtype)
    if case["source"] == "host":
        pipe = HostPipeline(ex, [shape_in], [shape_out], dtype, "cuda:0")
        return {"pipe": pipe, "x": x.cpu().pin_memory(), "y": torch.empty(shape_out, dtype=dtype).pin_memory()}
    return {"ex": ex, "x": x, "y": torch.empty(shape_out, dtype=dtype, device="cuda:0")}


def run(state):
    if "pipe" in state:
        state["pipe"].submit([state["x"]], [state["y"]])
    else:
        state["ex"].run([state["x"]], [state["y"]])
    return state["y"]


def work(case):
    """Images in, results out and the weights once; two operations per multiply-add of every convolution."""
    spec = _MAKE[case["net"]](case["batch"], size=case["size"])
    elem = 2 if case["storage"] == "f16" else 4
    values, flops = 0, 0
    for t in spec.inputs + spec.outputs:
        values += spec.batch * math.prod(spec.shapes[t])
    for op in spec.ops:
        if op.weights is not None:
            values += op.weights.size
            per_output = op.weights.size // op.cout
            flops += 2 * spec.batch * math.prod(spec.shapes[op.output]) * per_output
    return {"bytes": values * elem, "flops": flops}


# Four times what the same path shows when its sums are taken in another order (every 1x1 kernel against every other, and the
# CPU oracle, which accumulates in double): (relative error, largest difference).  In fp16 storage the differences are single
# roundings of stored values that fall the other way and are carried on; "max" is a few units in the last place.
_F16 = {"block": (1e-4, 4e-3), "fire": (6e-4, 4e-3), "v1": (1.1e-3, 4e-3), "v2": (1.4e-3, 5e-3), "seg": (2.4e-3, 1.3e-2)}
_F32 = (2e-6, 1e-5)


def tolerance(case):
    rel, largest = _F32 if case["storage"] == "f32" else _F16[case["net"]]
    return {"rel": rel, "max": largest}
