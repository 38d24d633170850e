"""What the library's speed is measured on: whole inference passes of the workload graphs through xenos_graph_run.

A program that serves one of these models builds the graph once, links it, compiles it for its largest batch, binds a
workspace and then calls ``Graph.run`` for every batch of images; that call, with its images and results in device
memory, is one pass.  The graphs are the five workload graphs and one operator benchmark of ``xenos_workloads`` at the
sizes the benchmark names, and the same graphs at other image sizes, widths, batches and image types.
"""
import torch

from paper_2302_00282_b200 import binding as xb
from xenos_workloads import graphs
from xenos_workloads.feed import graph_from_spec


def listed():
    return [
        # The smallest call: one fp32 conv3x3 -> conv1x1 -> max-pool chain of one 32 x 32 feature map (the fp32
        # workload of the benchmark); launch latency decides.
        dict(name="chain_f32_b1", graph="chain", hw=32, cin=16, cmid=32, cout=32, batch=1),
        # The same chain as a batch job on larger maps: the fp32 arithmetic decides.
        dict(name="chain_f32_b32", graph="chain", hw=75, cin=32, cmid=64, cout=64, batch=32),
        # Single-image serving of the three classifiers (the latency setting of the paper), bf16 images.
        dict(name="mobilenet_b1", graph="mobilenet", hw=224, width=1.0, classes=1000, batch=1, image="bf16"),
        dict(name="resnet18_b1", graph="resnet18", hw=224, base=64, classes=1000, batch=1, image="bf16"),
        dict(name="squeezenet_b1", graph="squeezenet", hw=224, scale=1, classes=1000, batch=1, image="bf16"),
        # Batched serving of the three classifiers (the throughput setting).
        dict(name="mobilenet_b32", graph="mobilenet", hw=224, width=1.0, classes=1000, batch=32, image="bf16"),
        dict(name="resnet18_b32", graph="resnet18", hw=224, base=64, classes=1000, batch=32, image="bf16"),
        dict(name="squeezenet_b32", graph="squeezenet", hw=224, scale=1, classes=1000, batch=32, image="bf16"),
        # A slimmer model on smaller, odd-sized fp32 images and an odd batch: ragged tiles everywhere, an image pitch
        # that is no multiple of 16 bytes.
        dict(name="mobilenet_ragged", graph="mobilenet", hw=157, width=0.5, classes=101, batch=7, image="f32"),
        # A fine-tuned ResNet-18 with few classes on larger fp32 images.
        dict(name="resnet18_hw288_b9", graph="resnet18", hw=288, base=64, classes=37, batch=9, image="f32"),
        # One operator alone: the 1x1 convolution + global average of the operator benchmark, NHWC features in.
        dict(name="op_cbr_avgpool_b32", graph="op_avgpool", hw=7, cin=1024, cout=1024, batch=32),
        # The largest: the bottleneck graph on 512 x 512 images, batch 64.
        dict(name="resnet50_b64", graph="resnet50", hw=512, base=64, batch=64, image="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["chain", "mobilenet", "mobilenet", "resnet18", "resnet18", "squeezenet", "squeezenet", "resnet50", "op_avgpool"])
    if kind == "chain":
        return dict(graph="chain", hw=_log_int(rng, 16, 96), cin=8 * rng.randint(1, 6), cmid=8 * rng.randint(1, 8),
                    cout=8 * rng.randint(1, 8), batch=_log_int(rng, 1, 48))
    if kind == "op_avgpool":
        return dict(graph="op_avgpool", hw=rng.randint(4, 11), cin=64 * rng.randint(4, 24), cout=8 * rng.randint(16, 160),
                    batch=_log_int(rng, 1, 64))
    # image sizes: half of them multiples of 32, as models are mostly fed, the others any
    size = (lambda lo, hi: 32 * rng.randint(-(-lo // 32), hi // 32) if rng.random() < 0.5 else rng.randint(lo, hi))
    image = rng.choice(["bf16", "bf16", "f32"])
    if kind == "resnet50":
        return dict(graph="resnet50", hw=size(128, 512), base=rng.choice([32, 64, 64]), batch=_log_int(rng, 1, 32), image=image)
    hw, batch, classes = size(128, 320), _log_int(rng, 1, 64), rng.choice([10, 100, 365, 1000])
    if kind == "mobilenet":
        return dict(graph=kind, hw=hw, width=rng.choice([0.25, 0.5, 0.75, 1.0, 1.0]), classes=classes, batch=batch, image=image)
    if kind == "resnet18":
        return dict(graph=kind, hw=hw, base=rng.choice([32, 64, 64]), classes=classes, batch=batch, image=image)
    # (a convolution makes the class scores here, and its channels are a multiple of 8)
    return dict(graph="squeezenet", hw=hw, scale=rng.choice([1, 1, 2]), classes=8 * (-(-classes // 8)), batch=batch, image=image)


def _spec(c):
    kind = c["graph"]
    if kind == "chain":
        return graphs.single_chain(c["hw"], c["cin"], c["cmid"], c["cout"])
    if kind == "mobilenet":
        return graphs.mobilenet_v1(c["hw"], c["width"], c["classes"])
    if kind == "resnet18":
        return graphs.resnet18(c["hw"], c["base"], c["classes"])
    if kind == "squeezenet":
        return graphs.squeezenet11(c["hw"], c["classes"], c["scale"])
    if kind == "resnet50":
        return graphs.resnet50_stress(c["hw"], c["base"])
    spec = graphs.GraphSpec("op_cbr_avgpool", (c["cin"], c["hw"], c["hw"]))
    spec.gap("ap", spec.cbr("c", "input", c["cout"], 1, 1, 0))
    return spec


def _params(spec, rng):
    """Weights with the distributions of ``graphs.make_params`` (He-normal weights, BatchNorm statistics around one)."""
    def normal(shape, std):
        return (torch.randn(shape, generator=rng, device="cuda") * std).cpu().numpy()

    def uniform(shape, lo, hi):
        return (torch.rand(shape, generator=rng, device="cuda") * (hi - lo) + lo).cpu().numpy()

    out = {}
    for o in spec.ops:
        if o["kind"] in ("conv", "fc"):
            k, cg = (o["k"], o["cin"] // o["groups"]) if o["kind"] == "conv" else (1, o["cin"])
            shape = (o["cout"], cg, k, k) if o["kind"] == "conv" else (o["cout"], cg)
            out[o["name"]] = dict(w=normal(shape, (2.0 / (cg * k * k)) ** 0.5))
            if o["bias"]:
                out[o["name"]]["b"] = uniform((o["cout"],), -0.1, 0.1)
        elif o["kind"] == "bn":
            n = (o["c"],)
            out[o["name"]] = dict(gamma=uniform(n, 0.5, 1.5), beta=uniform(n, -0.1, 0.1), mean=normal(n, 0.1), var=uniform(n, 0.5, 1.5))
    return out


def prepare(case, seed):
    spec, batch = _spec(case), case["batch"]
    fp32 = spec.precision == "fp32"
    nhwc = not fp32 and spec.in_shape[0] >= 8
    rng = torch.Generator(device="cuda")
    rng.manual_seed(seed)
    # images ~ U[-1, 1]
    c, h, w = spec.in_shape
    x = torch.rand((batch, h, w, c) if nhwc else (batch, c, h, w), generator=rng, device="cuda") * 2 - 1
    if not fp32 and case.get("image") != "f32":
        x = x.to(torch.bfloat16)
    in_dtype = xb.DTYPE_F32 if x.dtype == torch.float32 else xb.DTYPE_BF16
    g, _ = graph_from_spec(spec, _params(spec, rng), in_dtype=in_dtype, in_layout=xb.LAYOUT_NHWC if nhwc else xb.LAYOUT_NCHW)
    g.link()
    nbytes = g.compile(batch, xb.PRECISION_FP32_CUDA_CORE if fp32 else xb.PRECISION_BF16_TENSOR)
    ws = torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    g.bind(ws.data_ptr(), ws.numel(), stream)
    shape = spec.shapes[spec.output]
    if len(shape) == 1:
        out = torch.empty((batch, shape[0]), dtype=torch.float32, device="cuda")
    elif fp32:
        out = torch.empty((batch,) + tuple(shape), dtype=torch.float32, device="cuda")
    else:
        out = torch.empty((batch, shape[1], shape[2], shape[0]), dtype=torch.bfloat16, device="cuda")
    return dict(graph=g, workspace=ws, images=x, out=out, batch=batch, stream=stream)


def run(state):
    state["graph"].run(state["batch"], [state["images"].data_ptr()], [state["out"].data_ptr()], state["stream"])
    return state["out"]


def work(case):
    """Images, parameters and results, each moved once; two operations per multiply-accumulate."""
    spec, batch = _spec(case), case["batch"]
    fp32 = spec.precision == "fp32"
    c, h, w = spec.in_shape
    es_in = 4 if fp32 or case.get("image") == "f32" else 2
    es_w = 4 if fp32 else 2
    shape = spec.shapes[spec.output]
    n_out = 1
    for d in shape:
        n_out *= d
    es_out = 4 if fp32 or len(shape) == 1 else 2
    params = 0
    for o in spec.ops:
        if o["kind"] == "conv":
            params += o["cout"] * (o["cin"] // o["groups"]) * o["k"] ** 2 * es_w + 4 * o["cout"]
        elif o["kind"] == "fc":
            params += o["cout"] * o["cin"] * es_w + 4 * o["cout"]
    return dict(bytes=batch * (c * h * w * es_in + n_out * es_out) + params, flops=2.0 * batch * spec.macs())


def tolerance(case):
    if case["graph"] == "chain":
        return dict(rel=1e-5, max=1e-4)      # fp32 sums of a few hundred products
    if case["graph"] == "op_avgpool":
        return dict(rel=1e-3, max=1e-2)      # one product of bf16 operands; the averaged map may be rounded to bf16 or not
    # every stored activation is rounded to bf16; sums formed in another order move some of them by one step
    # (the bottleneck graph passes through 53 such tensors)
    return dict(rel=2e-2 if case["graph"] == "resnet50" else 1e-2, max=0.25)
