"""What the speed of this package is measured on: the work its users have it do, through its public entry points.

Five kinds of work:
  step      one training iteration of all simulated nodes (TrainStep): forward, backward, SGD half-step and gossip mix,
            then the mixed model becomes the next iteration's parameters, as a training loop does it
  product   the 8-bit contraction of one conv / linear layer: forward, backward-data and backward-weight
  gossip    the decentralized update of a parameter vector that some other program computed the gradient of
  quantize  a tensor to 8-bit codes and back
  norm      one normalization layer, forward and backward
Sizes come from the package's workloads, sweeps and tests, or are generic.
"""
import math

import torch

from paper_2111_09389_b200 import api, workloads
from paper_2111_09389_b200.step import TrainStep


def listed():
    return [
        # ---- training iterations
        # one conv layer on 4 nodes, launched call by call: nothing but latency (a first experiment, a unit of a larger loop)
        dict(name="step_conv_4x8", kind="step", net="conv", nodes=4, batch=8, graph=False),
        # the usual experiment: 16 nodes, uncompressed gossip, batches arriving from pinned host memory one ahead
        dict(name="step_resnet20_16x32_host", kind="step", net="resnet20", nodes=16, batch=32, host=True),
        # the largest experiment: 40 nodes, top 1 % of the flattened update
        dict(name="step_resnet20_40x32_top1", kind="step", net="resnet20", nodes=40, batch=32, keep=0.01, groups=2),
        # odd sizes, launched call by call: layer-wise top-k with 8-bit messages
        dict(name="step_resnet20_7x19_layers_q8", kind="step", net="resnet20", nodes=7, batch=19, keep=0.01,
             layerwise=True, bits=8, graph=False),
        # the wide network: 9.2 M parameters per node
        dict(name="step_vgg11_8x32", kind="step", net="vgg11", nodes=8, batch=32),
        # ---- contractions
        # the largest matrix product of the sweep
        dict(name="linear_8192", kind="product", nodes=1, B=8192, H=1, cin=8192, cout=8192, R=1, stride=1, affine=False),
        # a linear layer with class-count-like widths (1000 is no multiple of 16)
        dict(name="linear_4x1500_1000x1000", kind="product", nodes=4, B=1500, H=1, cin=1000, cout=1000, R=1, stride=1,
             affine=False),
        # a convolution at the sweep's batch
        dict(name="conv_256x56x56_c256", kind="product", nodes=1, B=256, H=56, cin=256, cout=256, R=3, stride=1,
             affine=False),
        # zero-point operands, the other quantization scheme, on a layer of the wide network
        dict(name="conv_affine_8x32x16x16_c128", kind="product", nodes=8, B=32, H=16, cin=128, cout=128, R=3, stride=1,
             affine=True),
        # ---- the update, the quantizer and a comparison layer alone
        dict(name="gossip_16x8652k_top1", kind="gossip", algo="choco", nodes=16, d=32 * 270410, segs=1, keep=0.01, bits=32),
        dict(name="quantize_8x4m_stochastic", kind="quantize", nodes=8, n=1 << 22, affine=False, stochastic=True),
        dict(name="norm_evonorm_8x64x32x32_c64", kind="norm", layer="evonorm_s0", nodes=8, B=64, H=32, C=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 5 + ["product"] * 4 + ["gossip", "quantize", "norm"])
    if kind == "step":
        net = rng.choice(["conv", "resnet20", "resnet20", "resnet20", "vgg11"])
        nodes = _log(rng, 2, 8 if net == "vgg11" else 40)
        c = dict(kind="step", net=net, nodes=nodes, batch=_log(rng, 4, 32), graph=rng.random() < 0.6)
        if nodes >= 32:
            c["groups"] = 2
        if net != "conv" and rng.random() < 0.5:
            c.update(keep=rng.choice([0.01, 0.1]), layerwise=rng.random() < 0.5)
        if rng.random() < 0.25:
            c["bits"] = 8
        if rng.random() < 0.2:
            c["stochastic"] = True                       # layer gradients rounded stochastically
        elif net != "conv" and rng.random() < 0.2:
            c["recompute"] = True                        # only 8-bit tensors kept between the passes
        if net != "conv" and rng.random() < 0.25:
            c["host"] = True
        return c
    if kind == "product":
        affine = rng.random() < 0.25
        ragged = rng.random() < 0.4
        # ragged: any channel count, at sizes a classifier or a first layer has; else multiples of 16
        most = 6e9 if ragged else 8192.0 ** 3 / (4 if affine else 1)
        wide = (lambda lo, hi: _log(rng, lo, hi)) if ragged else (lambda lo, hi: max(16, _log(rng, lo, hi) // 16 * 16))
        while True:
            nodes = _log(rng, 1, 16)
            if rng.random() < 0.5:
                c = dict(kind="product", nodes=nodes, B=_log(rng, 16, 8192), H=1, cin=wide(64, 8192), cout=wide(10, 8192),
                         R=1, stride=1, affine=affine)
            else:
                c = dict(kind="product", nodes=nodes, B=_log(rng, 8, 256), H=_log(rng, 4, 56), cin=wide(3, 512),
                         cout=wide(16, 512), R=rng.choice([3, 3, 3, 1]), stride=rng.choice([1, 1, 1, 2]), affine=affine)
            ho = _out(c)
            macs = _macs(c)
            if 1e6 <= macs <= most and nodes * c["B"] * (c["H"] ** 2 * c["cin"] + ho ** 2 * c["cout"]) <= 4.2e8:
                return c
    if kind == "gossip":
        nodes = _log(rng, 2, 40)
        d = min(_log(rng, 1000, 32 * 270410), 16 * 32 * 270410 // nodes)
        return dict(kind="gossip", algo=rng.choice(["choco", "choco", "deepsqueeze", "dense"]), nodes=nodes, d=d,
                    segs=rng.choice([1, 1, 20]), keep=rng.choice([0.01, 0.1]), bits=rng.choice([32, 8]))
    if kind == "quantize":
        nodes = _log(rng, 1, 40)
        return dict(kind="quantize", nodes=nodes, n=min(_log(rng, 1000, 1 << 24), (1 << 25) // nodes),
                    affine=rng.random() < 0.3, stochastic=rng.random() < 0.5)
    while True:
        c = dict(kind="norm", layer=rng.choice(["range_evonorm", "range_evonorm", "evonorm_s0", "range_bn"]),
                 nodes=_log(rng, 1, 40), B=_log(rng, 2, 128), H=_log(rng, 4, 56), C=8 * _log(rng, 2, 64))
        if c["layer"] == "range_evonorm":                 # that layer takes widths with few odd factors only
            c["C"] = rng.choice([16, 32, 48, 64, 96, 128, 160, 192, 256, 320, 384, 512])
        if c["nodes"] * c["B"] * c["H"] ** 2 * c["C"] <= 8 * 64 * 32 * 32 * 64:
            return c


# ---------------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return globals()["_prepare_" + case["kind"]](case, g)


def run(state):
    return state["run"](state)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


# ---- training iterations
def _network(net):
    return {"conv": workloads.single_conv_ops, "resnet20": workloads.resnet20_ops, "vgg11": workloads.vgg11_ops}[net]()


def _parameters(ops, d, nodes, g):
    """Kaiming-uniform weights, norm scales 1, offsets 0; every node 1 % off a common draw."""
    base = torch.zeros(d, device="cuda")
    for op in ops:
        if op["op"] in ("conv", "linear"):
            fan = op["cin"] * (op["R"] * op["S"] if op["op"] == "conv" else 1)
            w = base[op["w_off"]:op["w_off"] + fan * op["cout"]]
            w.copy_((torch.rand(w.shape, generator=g, device="cuda") * 2 - 1) * math.sqrt(6.0 / fan))
    params = base * (1 + 0.01 * _randn(g, nodes, d))
    for op in ops:
        if op["op"] == "ren":
            params[:, op["p_off"]:op["p_off"] + 2 * op["C"]] = 1.0
    return params


def _prepare_step(c, g):
    ops, d = _network(c["net"])
    nodes, batch, conv = c["nodes"], c["batch"], c["net"] == "conv"
    in_shape = (16, 16, 16) if conv else (32, 32, 3)
    seg = workloads.layer_segments(ops, d).tolist() if c.get("layerwise") else [0, d]
    keep = c.get("keep")
    seg_k = [hi - lo if keep is None else max(1, int((hi - lo) * keep)) for lo, hi in zip(seg[:-1], seg[1:])]
    st = TrainStep(ops, d, nodes, batch, in_shape, lr=0.1, gamma=1.0 if keep is None else 0.1, seg_offsets=seg, seg_k=seg_k,
                   has_labels=not conv, input_grad=conv, message_bits=c.get("bits", 32),
                   grad_rounding=int(c.get("stochastic", False)), seed=7, recompute_norm_input=c.get("recompute", False),
                   node_groups=c.get("groups", 1))
    st.params.copy_(_parameters(ops, d, nodes, g))
    lag = _randn(g, nodes, d) * torch.where(torch.rand(nodes, d, generator=g, device="cuda") < 0.05, 1e-2, 1e-4)
    st.x_hat.copy_(st.params - lag)                       # public copies lag the models by a heavy-tailed residual
    st.Wmix.copy_(torch.from_numpy(workloads.ring_matrix(nodes)))
    x = _randn(g, nodes, batch, *in_shape)
    st.x.copy_(x)
    if conv:
        st.dy.copy_(_randn(g, nodes, batch, 16, 16, 16))
    else:
        labels = torch.randint(0, 10, (nodes, batch), generator=g, device="cuda", dtype=torch.int32)
        st.labels.copy_(labels)
    state = dict(run=_run_step, st=st, step=st.run)
    x_hat = st.x_hat.clone()
    if c.get("graph", True):
        st.capture()                                      # runs one step: the public copies are put back
        st.x_hat.copy_(x_hat)
        state["step"] = st.replay
    if c.get("host"):
        state["host"] = [x.cpu().pin_memory(), labels.cpu().pin_memory()]
        state["loss_host"] = torch.empty(nodes).pin_memory()
        st.upload(*state["host"])
    return state


def _run_step(s):
    st = s["st"]
    if "host" in s:
        st.step_from_upload(s["step"])
        st.upload(*s["host"])                             # the next batch, while this step computes
        s["loss_host"].copy_(st.loss, non_blocking=True)
    else:
        s["step"]()
    st.params.copy_(st.x_out)
    return dict(logits=st.out, loss=None if st.labels is None else st.loss, grads=st.grads, x_half=st.x_half, x_hat=st.x_hat, x=st.x_out,
                input_grad=st.input_grad_out if st.input_grad else None)


# ---- contractions
def _out(c):
    return (c["H"] + 2 * (c["R"] // 2) - c["R"]) // c["stride"] + 1


def _macs(c):
    return c["nodes"] * c["B"] * _out(c) ** 2 * c["cin"] * c["cout"] * c["R"] ** 2


def _prepare_product(c, g):
    n, B, H, Ho, cin, cout, R = c["nodes"], c["B"], c["H"], _out(c), c["cin"], c["cout"], c["R"]
    desc = api.conv_desc(n, B, H, H, cin, cout, R, R, c["stride"], R // 2)
    lo, hi, dt = (0, 256, torch.uint8) if c["affine"] else (-127, 128, torch.int8)

    def codes(*shape):
        return torch.randint(lo, hi, shape, generator=g, device="cuda", dtype=dt)

    def scale():
        return torch.rand(n, generator=g, device="cuda") * 0.01 + 0.001
    s = dict(run=_run_product, desc=desc, affine=c["affine"], A=codes(n, B, H, H, cin), W=codes(n, cout, R, R, cin),
             E=codes(n, B, Ho, Ho, cout), sA=scale(), sW=scale(), sE=scale(), Y=torch.empty(n, B, Ho, Ho, cout, device="cuda"),
             dA=torch.empty(n, B, H, H, cin, device="cuda"), dW=torch.empty(n, cout * R * R * cin, device="cuda"),
             status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if c["affine"]:
        need = (api.lpdt_qconv_fwd_affine_workspace_size, api.lpdt_qconv_bwd_data_affine_workspace_size,
                api.lpdt_qconv_bwd_weight_affine_workspace_size)
        size = max(f(desc) for f in need)
        s.update({z: torch.randint(100, 156, (n,), generator=g, device="cuda", dtype=torch.int32) for z in ("zA", "zW", "zE")})
    else:
        size = max(api.lpdt_qconv_workspace_size(desc, which) for which in (0, 1, 2))
    s["ws"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    return s


def _run_product(s):
    d, kw, stride = s["desc"], dict(ws=s["ws"], dev_status=s["status"]), s["dW"].shape[1]
    if s["affine"]:
        api.lpdt_qconv_fwd_affine(d, s["A"], s["sA"], s["zA"], s["W"], s["sW"], s["zW"], Y=s["Y"], **kw)
        api.lpdt_qconv_bwd_data_affine(d, s["E"], s["sE"], s["zE"], s["W"], s["sW"], s["zW"], dA=s["dA"], **kw)
        api.lpdt_qconv_bwd_weight_affine(d, s["E"], s["sE"], s["zE"], s["A"], s["sA"], s["zA"], dW=s["dW"],
                                         dw_node_stride=stride, **kw)
    else:
        api.lpdt_qconv_fwd(d, s["A"], s["sA"], s["W"], s["sW"], Y=s["Y"], **kw)
        api.lpdt_qconv_bwd_data(d, s["E"], s["sE"], s["W"], s["sW"], dA=s["dA"], **kw)
        api.lpdt_qconv_bwd_weight(d, s["E"], s["sE"], s["A"], s["sA"], dW=s["dW"], dw_node_stride=stride, **kw)
    return s["Y"], s["dA"], s["dW"]


# ---- the decentralized update alone
def _prepare_gossip(c, g):
    n, d = c["nodes"], c["d"]
    seg = [d * i // c["segs"] for i in range(c["segs"] + 1)]
    x = _randn(g, 1, d) * 0.1 + _randn(g, n, d) * 0.01
    s = dict(run=_run_gossip, algo=c["algo"], n=n, d=d, seg=seg, k=[max(1, int((hi - lo) * c["keep"])) for lo, hi in zip(seg, seg[1:])],
             bits=c["bits"], x=x, grad=_randn(g, n, d) * 1e-2, x_half=torch.empty_like(x), x_out=torch.empty_like(x),
             W=torch.from_numpy(workloads.ring_matrix(n)).cuda(), msg=torch.empty(n, len(seg) - 1, device="cuda"),
             status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    lag = _randn(g, n, d) * 1e-2
    s["public"] = lag if c["algo"] == "deepsqueeze" else x - lag        # error buffer, or public copies
    s["ws"] = torch.empty(api.lpdt_gossip_mix_workspace_size(n, d, len(seg) - 1), dtype=torch.uint8, device="cuda")
    return s


def _run_gossip(s):
    n, d, x, half, out, pub = s["n"], s["d"], s["x"], s["x_half"], s["x_out"], s["public"]
    if s["algo"] == "dense":
        api.lpdt_sgd_gossip_mix(n, d, x, s["grad"], 0.1, half, pub, out, s["W"], 1.0)
    else:
        api.lpdt_sgd_update(n * d, x, s["grad"], 0.1, half)
        if s["algo"] == "deepsqueeze":
            api.lpdt_deepsqueeze_mix(n, d, half, pub, out, s["W"], 0.1, s["seg"], s["k"], s["ws"], s["bits"], s["msg"],
                                     s["status"])
        elif s["bits"] == 8:
            api.lpdt_gossip_mix_q8(n, d, half, pub, out, s["W"], 0.1, s["seg"], s["k"], s["msg"], s["ws"], s["status"])
        else:
            api.lpdt_gossip_mix(n, d, half, pub, out, s["W"], 0.1, s["seg"], s["k"], s["ws"], s["status"])
    s["x"], s["x_out"] = out, x                           # the mixed model is the next iteration's
    return half, pub, out


# ---- quantizer
def _prepare_quantize(c, g):
    n, m = c["nodes"], c["n"]
    code = torch.uint8 if c["affine"] else torch.int8
    return dict(run=_run_quantize, case=c, x=_randn(g, n, m), q=torch.empty(n, m, dtype=code, device="cuda"),
                scale=torch.empty(n, device="cuda"), zero=torch.zeros(n, dtype=torch.int32, device="cuda") if c["affine"] else None,
                y=torch.empty(n, m, device="cuda"),
                ws=torch.empty(api.lpdt_quantize_workspace_size(n), dtype=torch.uint8, device="cuda"))


def _run_quantize(s):
    n, m = s["x"].shape
    api.lpdt_quantize(s["x"], n, m, m, s["q"], s["scale"], s["ws"], mode=int(s["case"]["affine"]),
                      rounding=int(s["case"]["stochastic"]), seed=11, zero_point=s["zero"])
    api.lpdt_dequantize(s["q"], n, m, s["scale"], s["y"], zero_point=s["zero"])
    return s["q"], s["scale"], s["zero"], s["y"]


# ---- normalization layers
def _prepare_norm(c, g):
    n, B, H, C = c["nodes"], c["B"], c["H"], c["C"]
    f = dict(device="cuda")
    shape = (n, B, H, H, C)
    stat = (n, C) if c["layer"] == "range_bn" else (n, B, C // 8)
    s = dict(run=_run_norm, case=c, x=_randn(g, *shape), dy=_randn(g, *shape), y=torch.empty(shape, **f), dx=torch.empty(shape, **f),
             v=1 + 0.1 * _randn(g, n, C), gamma=1 + 0.1 * _randn(g, n, C), beta=0.1 * _randn(g, n, C), a=torch.empty(stat, **f),
             b=torch.empty(stat, **f), mean=torch.empty(stat, **f), ia=torch.empty(stat, dtype=torch.int32, **f),
             ib=torch.empty(stat, dtype=torch.int32, **f), dv=torch.zeros(n, C, **f), dgamma=torch.empty(n, C, **f),
             dbeta=torch.empty(n, C, **f), amax=torch.zeros(2, n, **f))
    size = {"range_evonorm": lambda: api.lpdt_range_evonorm_bwd_workspace_size(n, B, C),
            "evonorm_s0": lambda: api.lpdt_evonorm_s0_bwd_workspace_size(n, B, C),
            "range_bn": lambda: api.lpdt_range_bn_workspace_size(n, C)}[c["layer"]]()
    s["ws"] = torch.empty(max(size, 256), dtype=torch.uint8, **f)
    return s


def _run_norm(s):
    c, ws = s["case"], s["ws"]
    n, B, H, C = c["nodes"], c["B"], c["H"], c["C"]
    x, dy, y, dx, a, b, mean = s["x"], s["dy"], s["y"], s["dx"], s["a"], s["b"], s["mean"]
    v, gamma, beta, dv, dg, db = s["v"], s["gamma"], s["beta"], s["dv"], s["dgamma"], s["dbeta"]
    if c["layer"] == "range_evonorm":
        api.lpdt_fill_zero(s["amax"])                     # per-node ranges for the quantizers behind the layer
        api.lpdt_range_evonorm_fwd(n, B, H, H, C, C // 8, 1e-5, x, v, gamma, beta, C, y, a, b, s["ia"], s["ib"],
                                   amax_out=s["amax"][0])
        api.lpdt_range_evonorm_bwd(n, B, H, H, C, C // 8, 1e-5, dy, x, v, gamma, C, a, b, s["ia"], s["ib"], dx, dv, dg, db, C,
                                   ws, amax_out=s["amax"][1])
        return y, dx, dv, dg, db, a, b, s["amax"]
    if c["layer"] == "evonorm_s0":
        api.lpdt_evonorm_s0_fwd(n, B, H, H, C, C // 8, 1e-5, x, v, gamma, beta, C, y, a, b)
        api.lpdt_evonorm_s0_bwd(n, B, H, H, C, C // 8, 1e-5, dy, x, v, gamma, C, a, b, dx, dv, dg, db, C, ws)
        return y, dx, dv, dg, db, a, b
    api.lpdt_range_bn_fwd(n, B, H, H, C, 1e-5, x, gamma, beta, C, y, mean, a, b, s["ia"], s["ib"], ws)
    api.lpdt_range_bn_bwd(n, B, H, H, C, 1e-5, dy, x, gamma, C, mean, a, b, s["ia"], s["ib"], dx, dg, db, C, ws)
    return y, dx, dg, db, mean, a, b


# ---------------------------------------------------------------------------------------------------------------------
def work(case):
    """Inputs read once, results written once; multiply and add counted apart."""
    c, kind = case, case["kind"]
    if kind == "step":
        ops, d = _network(c["net"])
        images, conv = c["nodes"] * c["batch"], c["net"] == "conv"
        first = [op for op in ops if op["op"] == "conv"][:1]
        macs = 3 * workloads.conv_macs(ops, images) - (0 if conv else workloads.conv_macs(first, images))
        # images, dy / labels and input gradient; parameters, public copies in; gradients, half-step, public copies, model out
        io = images * (3 * 4 * 16 ** 3 if conv else 4 * (3 * 32 * 32 + 1)) + 24 * c["nodes"] * d
        return dict(bytes=io, flops=2 * macs)
    if kind == "product":
        n_in, n_out = c["nodes"] * c["B"] * c["H"] ** 2 * c["cin"], c["nodes"] * c["B"] * _out(c) ** 2 * c["cout"]
        n_w = c["nodes"] * c["cout"] * c["cin"] * c["R"] ** 2
        return dict(bytes=5 * (n_in + n_out + n_w), flops=6 * _macs(c))
    if kind == "gossip":
        return dict(bytes=24 * c["nodes"] * c["d"], flops=10 * c["nodes"] * c["d"])
    if kind == "quantize":
        return dict(bytes=9 * c["nodes"] * c["n"], flops=4 * c["nodes"] * c["n"])
    n = c["nodes"] * c["B"] * c["H"] ** 2 * c["C"]
    return dict(bytes=16 * n, flops=40 * n)


def tolerance(case):
    """The integer codes are exact by contract: every value that decides one is a fixed sequence of rounded fp32
    operations, so two correct implementations differ only by the last bit of the sums (measured against the fp64
    oracle and between summation orders: below 2e-7 for the products, the mix and the steps, 2e-6 for the sums of the
    comparison layers).  A step is not judged more loosely than that: a parameter moved by one ulp changes codes, and
    through twenty layers the gradients by 10 %."""
    return {"step": {"rel": 1e-5}, "product": {"rel": 5e-7}, "gossip": {"rel": 1e-6}, "quantize": "exact",
            "norm": {"rel": 1e-5}}[case["kind"]]


# ---------------------------------------------------------------------------------------------------------------------
def exact(case, seed):
    """What run() returns for these inputs, in 64 bits.  None for a training iteration: its result follows from integer
    codes that are decided in 32 bits (see tolerance), and so do stochastic codes and 8-bit messages."""
    make = {"product": _exact_product, "gossip": _exact_gossip, "quantize": _exact_quantize, "norm": _exact_norm}
    if case["kind"] not in make or (case["kind"] == "gossip" and case["bits"] == 8 and case["algo"] != "dense"):
        return None
    return make[case["kind"]](case, prepare(case, seed))


def _exact_product(c, s):
    n, H, Ho, R, st = c["nodes"], c["H"], _out(c), c["R"], c["stride"]
    pad = R // 2
    # output rows whose tap at offset t lies inside the image, and the input rows that they read
    taps = []
    for t in range(R):
        o = [i for i in range(Ho) if 0 <= i * st + t - pad < H]
        taps.append((slice(o[0], o[-1] + 1), slice(o[0] * st + t - pad, o[-1] * st + t - pad + 1, st)) if o else None)
    Y, dA, dW = (torch.zeros(s[k].shape, dtype=torch.float64, device="cuda") for k in ("Y", "dA", "dW"))
    dW = dW.view(n, c["cout"], R, R, c["cin"])
    for i in range(n):
        A, W, E = (s[k][i].double() - (float(s["z" + k][i]) if c["affine"] else 0.0) for k in "AWE")
        for r in range(R):
            for q in range(R):
                if taps[r] is None or taps[q] is None:
                    continue
                (oh, ih), (ow, iw) = taps[r], taps[q]
                a, e, w = A[:, ih, iw], E[:, oh, ow], W[:, r, q]
                Y[i][:, oh, ow] += a @ w.t()
                dA[i][:, ih, iw] += e @ w
                dW[i][:, r, q] += e.reshape(-1, c["cout"]).t() @ a.reshape(-1, c["cin"])
        sA, sW, sE = (float(s[k][i]) for k in ("sA", "sW", "sE"))
        Y[i] *= sA * sW
        dA[i] *= sE * sW
        dW[i] *= sE * sA
    return Y, dA, dW.reshape(n, -1)


def _exact_gossip(c, s):
    lr, gamma = (0.1, 1.0) if c["algo"] == "dense" else (0.1, 0.1)
    half, pub, W = s["x"].double() - lr * s["grad"].double(), s["public"].double(), s["W"].double()
    v = half + pub if c["algo"] == "deepsqueeze" else half - pub
    if c["algo"] != "dense":
        sent = torch.zeros_like(v)
        for lo, hi, k in zip(s["seg"], s["seg"][1:], s["k"]):
            for row, out in zip(v[:, lo:hi], sent[:, lo:hi]):
                at = row.abs().topk(k).indices
                out[at] = row[at]
        if c["algo"] == "deepsqueeze":
            return half, v - sent, half + gamma * (W @ sent - sent)
        v = sent
    pub = pub + v
    return half, pub, half + gamma * (W @ pub - W.sum(1, keepdim=True) * pub)


def _exact_quantize(c, s):
    x = s["x"].double()
    if c["affine"]:
        lo, hi = x.amin(1, True).clamp(max=0), x.amax(1, True).clamp(min=0)
        scale = (hi - lo) / 255
        zero = (-lo / scale).round().clamp(0, 255)
        q = ((x / scale).round() + zero).clamp(0, 255)
    else:
        scale = x.abs().amax(1, True) / 127
        zero, q = torch.zeros_like(scale), (x / scale).round().clamp(-127, 127)
    y = (q - zero) * scale
    drawn = c["stochastic"]
    return None if drawn else q, scale.flatten(), zero.flatten() if c["affine"] else None, None if drawn else y


def _exact_norm(c, s):
    n, B, H, C, eps = c["nodes"], c["B"], c["H"], c["C"], 1e-5
    out = []
    for i in range(n):                                    # node by node: a fraction of the memory
        x = s["x"][i].double().requires_grad_()
        v, g, b = (s[k][i].double().requires_grad_() for k in ("v", "gamma", "beta"))
        if c["layer"] == "range_bn":
            f = x.view(-1, C)
            hi, lo = (f.gather(0, (f * k).detach().argmax(0, keepdim=True))[0] for k in (1, -1))
            mu = f.mean(0)
            y = g * (x - mu) / ((hi - lo) / math.sqrt(2 * math.log(B)) + eps) + b
            stats = (mu, lo, hi)
        else:
            f = x.view(B, H * H, C // 8, 8).transpose(1, 2).reshape(B, C // 8, -1)
            if c["layer"] == "evonorm_s0":
                stats = (f.mean(-1), f.var(-1, unbiased=False))
                D, h = (stats[1] + eps).sqrt(), torch.sigmoid(v * x)
            else:
                hi, lo = (f.gather(-1, (f * k).detach().argmax(-1, keepdim=True))[..., 0] for k in (1, -1))
                stats = (lo, hi)
                D, h = (hi - lo) / math.sqrt(2 * math.log(8)) + eps, ((v * x + 3) / 6).clamp(0, 1)
            y = g * x * h / D.repeat_interleave(8, 1)[:, None, None] + b
        wrt = (x, g, b) if c["layer"] == "range_bn" else (x, v, g, b)
        grads = torch.autograd.grad(y, wrt, s["dy"][i].double())
        extra = (y.detach().abs().max(), grads[0].abs().max()) if c["layer"] == "range_evonorm" else ()
        out.append([t.detach() for t in (y, *grads, *stats)] + ([torch.stack(extra)] if extra else []))
    r = [torch.stack(t) for t in zip(*out)]
    if c["layer"] == "range_evonorm":
        r[-1] = r[-1].t().contiguous()
    return tuple(r)
