"""Workloads of the library, each one pass through its public entry points.

Five kinds of work, as programs that use the library have them:

  step     merge a run of convolutions (dc_merge_chain) and run the merged layer on a batch (dc_conv_forward)
  conv     one dense layer on its own: a merged layer whose weights were packed once, a 1x1 layer, a wide 5x5 layer
  dw       one depthwise layer that the compression left alone
  block    one unmerged inverted-residual block (dc_block_forward)
  net      the depth-compressed MobileNetV2-1.0 as one captured CUDA graph: its forward, or its merges and its forward

Feature maps are NHWC.  bf16 is what the merged network is served in, fp32 is the library's accuracy path.  Shapes are
those of the four single-run workloads, of the VGG-style runs and of the network in paper_2301_12187_b200/inputs.py,
and of the same layers at other resolutions and batch sizes.
"""
import functools
import math

import torch

from paper_2301_12187_b200 import dc
from paper_2301_12187_b200 import inputs as I
from paper_2301_12187_b200.network import CompressedNetwork

BF16_BYTES_MAX, BF16_FLOPS_MAX = 2.5e8, 4e10     # bounds on one drawn layer
F32_BYTES_MAX, F32_FLOPS_MAX = 1.5e8, 4e9
PLAN_SEED = 0                                    # the seeded choice of removed activations


# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # The paper's unit of work: one block's three layers merged (skip folded), then the merged 3x3 on 64 images.
        dict(name="step_block56", kind="step", form="blocks", c_in=24, c_mid=144, c_out=24, blocks=1, stride=1, skip=True,
             n=64, h=56, w=56, dtype="bf16"),
        # A deep block merged for a small batch: 160 -> 960 -> 160 at 7x7, where the merge is most of the work.
        dict(name="step_deep7", kind="step", form="blocks", c_in=160, c_mid=960, c_out=160, blocks=1, stride=1, skip=True,
             n=8, h=7, w=7, dtype="bf16"),
        # Two dense 3x3 layers of a VGG-style network merged to one 5x5 when a model is loaded, and its first image.
        dict(name="step_vgg256", kind="step", form="dense", c_in=256, c_mid=256, c_out=256, blocks=1, stride=1, skip=False,
             n=1, h=56, w=56, dtype="bf16"),
        # A merged layer in service: a stride-2 block's 3x3 at 56x56, the paper's batch of 128.
        dict(name="conv_s2_56", kind="conv", c_in=24, c_out=32, k=3, stride=2, residual=False, act=1, n=128, h=56, w=56,
             dtype="bf16"),
        # A merged 3x3 with its skip input at a resolution that gives odd map sides (200 / 8 = 25) and an odd batch.
        dict(name="conv_odd25", kind="conv", c_in=32, c_out=32, k=3, stride=1, residual=True, act=0, n=51, h=25, w=25,
             dtype="bf16"),
        # The widest work of the path: a merged 5x5 of 128 channels at 112x112, tensor-bound.
        dict(name="conv_vgg128", kind="conv", c_in=128, c_out=128, k=5, stride=1, residual=False, act=1, n=32, h=112, w=112,
             dtype="bf16"),
        # The fp32 path: the merged 5x5 of two blocks (32 -> 32 at 28x28), as it is run to check a compression's accuracy.
        dict(name="conv_f32_28", kind="conv", c_in=32, c_out=32, k=5, stride=1, residual=False, act=0, n=32, h=28, w=28,
             dtype="f32"),
        # A depthwise layer between two merged ones.
        dict(name="dw_56", kind="dw", c=144, k=3, stride=1, act=1, n=64, h=56, w=56, dtype="bf16"),
        # A block that the selector left unmerged.
        dict(name="block_14", kind="block", c_in=64, c_mid=384, c_out=64, stride=1, skip=True, n=128, h=14, w=14, dtype="bf16"),
        # The compressed network on one image: latency and launches.
        dict(name="net_1", kind="net", mode="forward", n=1, res=224, n_remove=17),
        # The network's forward at the paper's batch size.
        dict(name="net_128", kind="net", mode="forward", n=128, res=224, n_remove=17),
        # Merges and forward in one piece (weights changed, network run again), at a resolution whose maps have odd sides.
        dict(name="net_step_20", kind="net", mode="step", n=20, res=200, n_remove=17),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _sides(rng, lo=7, hi=112):
    h = _log_int(rng, lo, hi)
    return h, max(lo, min(hi, h + (rng.randint(-5, 5) if rng.random() < 0.3 else 0)))      # mostly square images


def _shrink(case, key="n"):
    """Fewer images until the case is within the bounds (then smaller maps)."""
    b_max, f_max = (F32_BYTES_MAX, F32_FLOPS_MAX) if case["dtype"] == "f32" else (BF16_BYTES_MAX, BF16_FLOPS_MAX)
    while True:
        wk = work(case)
        over = max(wk["bytes"] / b_max, wk["flops"] / f_max)
        if over <= 1.0 or (case["n"] == 1 and case["h"] <= 14):
            return case
        if case["n"] > 1:
            case["n"] = max(1, int(case["n"] / max(over, 1.01)))
        else:
            case["h"], case["w"] = max(7, case["h"] // 2), max(7, case["w"] // 2)


def draw(rng):
    kind = rng.choice(["step", "step", "conv", "conv", "conv", "dw", "block", "net", "net"])
    n = _log_int(rng, 1, 128)
    h, w = _sides(rng)
    if kind == "net":
        res = rng.randint(96, 224)
        return dict(kind="net", mode=rng.choice(["forward", "forward", "step"]), n=n, res=res, n_remove=rng.randint(10, 24))
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    if kind == "step":
        if rng.random() < 0.3:
            c = [8 * _log_int(rng, 4, 32) for _ in range(3)]
            return _shrink(dict(kind="step", form="dense", c_in=c[0], c_mid=c[1], c_out=c[2], blocks=1, stride=1, skip=False,
                                n=n, h=h, w=w, dtype=dtype))
        c = 8 * _log_int(rng, 2, 20)
        stride = 2 if rng.random() < 0.3 else 1
        skip = stride == 1 and rng.random() < 0.6
        blocks = 2 if skip and c <= 64 and rng.random() < 0.5 else 1
        c_out = c if skip else 8 * _log_int(rng, 2, 20)
        return _shrink(dict(kind="step", form="blocks", c_in=c, c_mid=6 * c, c_out=c_out, blocks=blocks, stride=stride,
                            skip=skip, n=n, h=h, w=w, dtype=dtype))
    if kind == "conv":
        k = rng.choice([1, 1, 3, 3, 3, 5])
        hi = {1: 120, 3: 40, 5: 20}[k]
        c_in, c_out = 8 * _log_int(rng, 2, hi), 8 * _log_int(rng, 2, hi)
        stride = 2 if k > 1 and rng.random() < 0.25 else 1
        return _shrink(dict(kind="conv", c_in=c_in, c_out=c_out, k=k, stride=stride, residual=stride == 1 and rng.random() < 0.3,
                            act=rng.randint(0, 1), n=n, h=h, w=w, dtype=dtype))
    if kind == "dw":
        return _shrink(dict(kind="dw", c=8 * _log_int(rng, 2, 120), k=5 if rng.random() < 0.25 else 3,
                            stride=2 if rng.random() < 0.3 else 1, act=rng.randint(0, 1), n=n, h=h, w=w, dtype=dtype))
    c = 8 * _log_int(rng, 2, 20)
    stride = 2 if rng.random() < 0.3 else 1
    skip = stride == 1 and rng.random() < 0.6
    return _shrink(dict(kind="block", c_in=c, c_mid=6 * c, c_out=c if skip else 8 * _log_int(rng, 2, 40), stride=stride,
                        skip=skip, n=n, h=h, w=w, dtype=dtype))


# --------------------------------------------------------------------------- work and tolerance


def _ext(h, k, s, p):
    return (h + 2 * p - k) // s + 1


def _es(case):
    return 4 if case["dtype"] == "f32" else 2


def _conv_work(n, h, w, c_in, c_out, k, s, p, es, w_es, extra_y=0):
    """One dense convolution: x and the weights read once, y written once, extra_y further maps of y's size."""
    out = n * _ext(h, k, s, p) * _ext(w, k, s, p) * c_out
    return n * h * w * c_in * es + (1 + extra_y) * out * es + c_out * c_in * k * k * w_es, 2.0 * out * c_in * k * k


def _run_geometry(case):
    """(k, stride, pad) of the merged layer of a step case."""
    if case["form"] == "dense":
        return 5, 1, 2
    return (3, case["stride"], 1) if case["blocks"] == 1 else (5, 1, 2)


@functools.lru_cache(maxsize=None)
def _plan(res, n_remove):
    net = I.mobilenet_v2(seed=0, batch=1, res=res)
    acts, ops = I.plan_spans(net, seed=PLAN_SEED, n_remove=n_remove)
    shapes = [(s.c_in, s.c_out, s.groups, s.k, s.stride, s.pad) for s in net.layers]
    return shapes, [(tuple(o.layers), o.add_from) for o in ops]


def _net_work(case):
    """Sum over the launch groups of the plan, each reading its input (and skip input) and its weights once and writing
    its output once; three untouched layers of one block are still three groups here, their maps counted."""
    shapes, ops = _plan(case["res"], case["n_remove"])
    n, h = case["n"], case["res"]
    nbytes = flops = 0.0
    for layers, add_from in ops:
        k, s, p = 1, 1, 0
        for i in layers:
            _, _, _, k2, s2, p2 = shapes[i]
            k, p, s = k + (k2 - 1) * s, p + p2 * s, s * s2
        c_in, c_out = shapes[layers[0]][0], shapes[layers[-1]][1]
        depthwise = all(shapes[i][2] > 1 for i in layers)
        ho = _ext(h, k, s, p)
        taps = k * k * (1 if depthwise else c_in)
        nbytes += 2.0 * n * h * h * c_in + 2.0 * n * ho * ho * c_out * (2 if add_from > -2 else 1) + 2.0 * c_out * taps
        flops += 2.0 * n * ho * ho * c_out * taps
        if case["mode"] == "step" and len(layers) > 1:
            nbytes += sum(4.0 * shapes[i][1] * (shapes[i][0] // shapes[i][2]) * shapes[i][3] ** 2 for i in layers)
            nbytes += 6.0 * c_out * taps                       # the merged kernel in fp32 and its packed copy
            hid = max(max(shapes[i][:2]) for i in layers)
            flops += 2.0 * c_out * hid * c_in * k * k          # one contraction over the widest inner layer
        h = ho
    return {"bytes": nbytes, "flops": flops}


def work(case):
    kind = case["kind"]
    if kind == "net":
        return _net_work(case)
    n, h, w, es = case["n"], case["h"], case["w"], _es(case)
    if kind == "conv":
        k, s = case["k"], case["stride"]
        b, f = _conv_work(n, h, w, case["c_in"], case["c_out"], k, s, k // 2, es, es, extra_y=int(case["residual"]))
    elif kind == "dw":
        k, s, c = case["k"], case["stride"], case["c"]
        out = n * _ext(h, k, s, k // 2) * _ext(w, k, s, k // 2) * c
        b, f = (n * h * w * c + out) * es + 4.0 * k * k * c, 2.0 * out * k * k
    elif kind == "block":
        ci, cm, co, s = case["c_in"], case["c_mid"], case["c_out"], case["stride"]
        ho, wo = _ext(h, 3, s, 1), _ext(w, 3, s, 1)
        b = (n * h * w * ci + n * ho * wo * co + ci * cm + cm * co) * es + 36.0 * cm
        f = 2.0 * n * (h * w * ci * cm + ho * wo * (9 * cm + cm * co))
    else:
        ci, cm, co = case["c_in"], case["c_mid"], case["c_out"]
        k, s, p = _run_geometry(case)
        b, f = _conv_work(n, h, w, ci, co, k, s, p, es, es)    # the forward; its packed weights are written and read
        if case["form"] == "dense":
            b += 4.0 * 9 * cm * (ci + co)
            f += 2.0 * 81 * ci * cm * co                       # every product of two taps once
        else:
            b += case["blocks"] * 4.0 * cm * (ci + co + 9)
            f += case["blocks"] * 2.0 * 9 * ci * cm * co
            if case["blocks"] == 2:
                f += 2.0 * 81 * co * co * ci                   # the two merged 3x3 kernels composed
        b += (4 + es) * co * ci * k * k
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    """What another implementation at the same precision shows: about four times the measured distance of the path from
    itself in 64 bits.  fp32: at most 1.1e-6 (largest element 8.1e-6).  bf16, weights, inputs and outputs rounded to 8
    bits: 2.4e-3 (1.4e-2); a block, whose inner maps are rounded as well, 3.8e-3 (2.2e-2).  The network, some thirty
    layers of it, 1.8e-2: less than twice that is left to it."""
    if case["kind"] == "net":
        return {"rel": 3e-2, "max": 0.5}
    if case["dtype"] == "f32":
        return {"rel": 4e-6, "max": 4e-5}
    return {"rel": 1.5e-2, "max": 0.09} if case["kind"] == "block" else {"rel": 1e-2, "max": 0.06}


# --------------------------------------------------------------------------- preparing and running


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, shape, dtype=torch.float32, std=1.0):
    return (torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) * std).to(dtype)


def _torch_dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _packed(wf, g, code):
    out = torch.empty(dc.packed_bytes(g, code), dtype=torch.uint8, device="cuda")
    dc.pack_weights(wf, g, code, out)
    return out


def _layer(gen, c_in, c_out, k, s, groups, code):
    """Geometry, packed weights (variance 1 / fan-in) and bias of one layer."""
    g = dc.geom(c_in, c_out, groups, k, s, k // 2)
    fan_in = (c_in // groups) * k * k
    wf = _randn(gen, (c_out, c_in // groups, k, k), std=fan_in ** -0.5)
    return g, _packed(wf, g, code), _randn(gen, (c_out,), std=0.1)


def _specs(case, seed):
    ci, cm, co = case["c_in"], case["c_mid"], case["c_out"]
    mk = functools.partial(I.make_layer, seed)
    if case["form"] == "dense":
        return [mk(0, ci, cm, 3, 1, 1), mk(1, cm, co, 3, 1, 1)], []
    specs, residuals = [], []
    for _ in range(case["blocks"]):
        i = len(specs)
        specs += [mk(i, ci, cm, 1, 1, 0), mk(i + 1, cm, cm, 3, case["stride"], 1, depthwise=True), mk(i + 2, cm, co, 1, 1, 0)]
        if case["skip"]:
            residuals.append((i, i + 2))
    return specs, residuals


def prepare(case, seed):
    kind = case["kind"]
    gen = _generator(seed)
    st = dict(kind=kind)
    if kind == "net":
        net = I.mobilenet_v2(seed=seed, batch=case["n"], res=case["res"])
        acts, ops = I.plan_spans(net, seed=PLAN_SEED, n_remove=case["n_remove"])
        cn = CompressedNetwork(net, acts, ops)
        x = _randn(gen, cn.in_shape, torch.bfloat16)
        cn.merge()
        graph = cn.capture(x) if case["mode"] == "forward" else cn.capture_step(x)
        st.update(cn=cn, x=x, graph=graph, y=cn.ops[-1].y)
        return st
    dt = _torch_dtype(case)
    code = dc.dtype_code(dt)
    n, h, w = case["n"], case["h"], case["w"]
    if kind == "step":
        specs, residuals = _specs(case, seed)
        layers = [dc.DeviceLayer(s) for s in specs]
        g, ws_bytes = dc.merge_query(layers, residuals)
        st.update(layers=layers, residuals=residuals, g=g, code=code,
                  wm=torch.empty((g.c_out, g.c_in, g.k, g.k), device="cuda"), bias=torch.empty((g.c_out,), device="cuda"),
                  packed=torch.empty(dc.packed_bytes(g, code), dtype=torch.uint8, device="cuda"),
                  merge_ws=torch.empty(ws_bytes, dtype=torch.uint8, device="cuda"), act=dc.ACT_IDENTITY, residual=None)
    elif kind == "conv":
        g, packed, bias = _layer(gen, case["c_in"], case["c_out"], case["k"], case["stride"], 1, code)
        st.update(g=g, packed=packed, bias=bias, act=case["act"], residual=None)
    elif kind == "dw":
        g, packed, bias = _layer(gen, case["c"], case["c"], case["k"], case["stride"], case["c"], dc.F32)
        st.update(g=g, packed=packed, bias=bias, act=case["act"])
    else:
        ci, cm, co, s = case["c_in"], case["c_mid"], case["c_out"], case["stride"]
        parts = [_layer(gen, ci, cm, 1, 1, 1, code), _layer(gen, cm, cm, 3, s, cm, dc.F32), _layer(gen, cm, co, 1, 1, 1, code)]
        ptr = [t.data_ptr() for _, pk, b in parts for t in (pk, b)]
        blk = dc.Block(ci, cm, co, 1, 3, s, 1, int(case["skip"]), dc.ACT_RELU6, dc.ACT_RELU6, *ptr)
        st.update(parts=parts, blk=blk, y=torch.empty((n, _ext(h, 3, s, 1), _ext(w, 3, s, 1), co), dtype=dt, device="cuda"),
                  ws=torch.zeros(dc.block_workspace_bytes(n, h, w, blk, code), dtype=torch.uint8, device="cuda"),
                  x=_randn(gen, (n, h, w, ci), dt))
        return st
    g = st["g"]
    st["x"] = _randn(gen, (n, h, w, g.c_in), dt)
    shape = (n, _ext(h, g.k, g.stride, g.pad), _ext(w, g.k, g.stride, g.pad), g.c_out)
    st["y"] = torch.empty(shape, dtype=dt, device="cuda")
    st["ws"] = torch.zeros(dc.conv_workspace_bytes(), dtype=torch.uint8, device="cuda")
    if case.get("residual"):
        st["residual"] = _randn(gen, shape, dt)
    return st


def run(st):
    kind = st["kind"]
    if kind == "net":
        st["graph"].replay()
        return st["y"]
    if kind == "block":
        dc.block_forward(st["x"], st["blk"], st["y"], st["ws"])
        return st["y"]
    g = st["g"]
    if kind == "dw":
        dc.dwconv_forward(st["x"], g.k, g.stride, g.pad, st["packed"], st["bias"], st["act"], st["y"])
        return st["y"]
    if kind == "step":
        dc.merge_chain(st["layers"], st["residuals"], st["wm"], st["bias"], st["packed"], st["code"], st["merge_ws"])
    dc.conv_forward(st["x"], g, st["packed"], st["bias"], st["act"], st["residual"], st["y"], st["ws"])
    return (st["wm"], st["bias"], st["y"]) if kind == "step" else st["y"]
