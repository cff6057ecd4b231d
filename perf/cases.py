"""The timed work of this framework: PalQuant layers, the quantisers of a training step
and whole networks, each through the entry points that a program calls.

Activations entering a layer are half-normal (a ReLU's output), weights are
He-initialised, images are N(0, 1), steps are the LSQ initialisation 2 mean / sqrt(Qp);
everything is drawn on the GPU from the seed.  A case is a dict of plain values:

kind "layer"    one PalQuant layer (group convolution, rescale, optional shortcut, ReLU,
                output permutation, requantisation).  entry: "codes" takes codes in,
                "on_load" takes fp32 activations through the fused call, "two_calls"
                quantises in a call of its own first, "bounds" does so with learned
                bounds l < u.  fmt: the code format ("nhwc", "c16", "f4").  out: "codes"
                or "both" (fp32 and codes).
kind "front"    the first block of a stage: conv1 3x3 stride 2 (codes out) and the 1x1
                stride-2 downsample of the same codes (fp32 out).
kind "qat"      the quantisers' part of one layer's training step: fake quantisation of
                its activations and weights, forward and backward, learned bounds.
kind "network"  the ResNet-18-shaped network, images to logits, as one eager forward or
                as the replay of its CUDA graph.
"""
import math

import numpy as np
import torch

from paper_2208_01944_gb300 import binding as B
from paper_2208_01944_gb300.resnet18 import PalQuantResNet18

FORMATS = {"nhwc": B.PQ_CODES_INT8, "c16": B.PQ_CODES_C16, "f4": B.PQ_CODES_C32F4}
WIDTHS = (64, 128, 256, 512)  # per-group widths of the ResNet-18-shaped network
CLASSES = 1000


def listed():
    layer = dict(kind="layer", k=3, stride=1, pad=1, bits=2, shuffle="cyclic", shortcut=False)
    return [
        # One image through a small layer in the plain layout, every output taken: the
        # latency of a call, as in interactive use or while bringing a model up.
        dict(layer, name="layer 1x28 nhwc", N=1, H=28, W=28, G=2, cin=32, cout=32, entry="two_calls", fmt="nhwc",
             out="both"),
        # ResNet-18 stage 1 with G = 4: the benchmarked step, fp32 in and the next layer's codes out.
        dict(layer, name="step 64x56 c16", N=64, H=56, W=56, G=4, cin=64, cout=64, entry="on_load", fmt="c16",
             out="codes"),
        # Many narrow groups on packed 2-bit codes, inside a network (codes in, codes out).
        dict(layer, name="layer 128x28 g8 f4", N=128, H=28, W=28, G=8, cin=64, cout=64, entry="codes", fmt="f4",
             out="codes"),
        # Two wide groups of 4-bit codes: the most arithmetic per byte.
        dict(layer, name="layer 128x28 b4 c16", N=128, H=28, W=28, G=2, cin=256, cout=256, bits=4, entry="codes",
             fmt="c16", out="codes"),
        # A block's second convolution at the largest image: fp32 shortcut in, fp32 and codes out.
        dict(layer, name="conv2 128x56 f4", N=128, H=56, W=56, G=2, cin=64, cout=64, entry="codes", fmt="f4",
             shortcut=True, out="both"),
        # The stride-2 entry of stage 3.
        dict(kind="front", name="front 128x28 f4", N=128, H=28, W=28, G=2, cin=128, cout=256, bits=2, fmt="f4"),
        # The last stage: small images, wide groups, the largest weights.
        dict(layer, name="layer 128x7 f4", N=128, H=7, W=7, G=2, cin=512, cout=512, entry="codes", fmt="f4",
             out="codes"),
        # A MobileNetV2-shaped pointwise layer.
        dict(layer, name="pointwise 256x14 c16", N=256, H=14, W=14, G=4, cin=96, cout=96, k=1, pad=0, entry="codes",
             fmt="c16", out="codes"),
        # A user's own layer: image and channel sizes that no tile divides, an odd number of
        # groups in an order of its own, 3-bit codes, bounds learned in training.
        dict(layer, name="ragged 20x37x45 nhwc", N=20, H=37, W=45, G=3, cin=96, cout=80, bits=3, shuffle="explicit",
             entry="bounds", fmt="nhwc", out="both"),
        # Training: the quantisers of the benchmarked layer, both directions.
        dict(kind="qat", name="qat 64x56", N=64, H=56, W=56, G=4, cin=64, cout=64, k=3, bits=2),
        # One image through the network as it is served: the replay of its graph.
        dict(kind="network", name="network 1", N=1, size=224, G=2, placement="block", graph=True),
        # A full batch through the network, launched as it is written.
        dict(kind="network", name="network 128", N=128, size=224, G=2, placement="block", graph=False),
    ]


def _log_int(rng, lo, hi):
    """A whole number in [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["layer"] * 6 + ["pointwise"] * 2 + ["front", "qat", "network"])
    if kind == "network":
        return dict(kind="network", N=_log_int(rng, 1, 96), size=rng.choice([160, 192, 224]), G=2,
                    placement=rng.choice(["block", "block", "paper"]), graph=rng.random() < 0.5)
    size = _log_int(rng, 7, 56)
    other = max(7, min(60, size + rng.randint(-3, 3)))
    if kind == "qat":
        G = rng.choice([1, 2, 3, 4, 8])
        cin = 16 * _log_int(rng, 1, 32 // G)
        n = _log_int(rng, 1, max(1, min(64, 51_000_000 // (size * other * G * cin))))
        return dict(kind="qat", N=n, H=size, W=other, G=G, cin=cin, cout=16 * _log_int(rng, 1, 16),
                    k=rng.choice([1, 3]), bits=rng.choice([2, 3, 4]))
    fmt = rng.choice(["f4", "f4", "c16", "c16", "nhwc"])
    G = rng.choice([1, 2, 3, 4, 8])
    step = 64 if fmt == "f4" else 32
    cin = step * _log_int(rng, 1, max(1, 512 // (step * max(1, G // 2))))
    cout = cin if rng.random() < 0.5 else step * _log_int(rng, 1, max(1, 512 // (step * max(1, G // 2))))
    bits = 2 if fmt == "f4" else rng.choice([2, 2, 3, 4])
    # at most 51 M activations on either side and 240 G operations
    most = min(128, 51_000_000 // (size * other * G * max(cin, cout)),
               120_000_000_000 // (size * other * G * cin * cout * 9))
    n = _log_int(rng, 1, max(1, most))
    if kind == "front":  # a stage's entry doubles the width
        cin = max(64, min(cin, 256))
        n = max(1, min(n, 25_000_000 // (size * other * G * cin)))
        return dict(kind="front", N=n, H=size, W=other, G=G, cin=cin, cout=2 * cin, bits=bits,
                    fmt="c16" if fmt == "nhwc" else fmt)
    k = 1 if kind == "pointwise" else 3
    shortcut = rng.random() < 0.3
    entry = rng.choice(["codes", "codes", "two_calls", "bounds"])
    if k == 3 and fmt != "nhwc" and max(cin, cout) <= 128 and not shortcut and rng.random() < 0.3:
        entry = "on_load"
    return dict(kind="layer", N=n, H=size, W=other, G=G, cin=cin, cout=cout, k=k, stride=1, pad=k // 2, bits=bits,
                shuffle=rng.choice(["none", "cyclic", "cyclic", "explicit"]), shortcut=shortcut, entry=entry, fmt=fmt,
                out="both" if shortcut else rng.choice(["codes", "codes", "both"]))


# ---------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _half_normal(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda").abs_()


def _he(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda").mul_(math.sqrt(2.0 / math.prod(shape[2:])))


def _steps(t, bits, signed=False):
    """Per-group LSQ steps 2 mean / sqrt(Qp) of t [G, ...] or of activations [..., G, C]."""
    mean = t.double().abs().flatten(1).mean(1) if signed else t.double().flatten(0, -3).mean((0, 2))
    qp = (1 << (bits - 1)) - 1 if signed else (1 << bits) - 1
    return (2.0 * mean / math.sqrt(qp)).float().cpu().numpy()


def _inverse(s):
    return (1.0 / s.astype(np.float64)).astype(np.float32)


def _on_gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _per_channel(v, C):
    """A value per group as a row of one per channel (fp32)."""
    return _on_gpu(np.repeat(np.asarray(v, dtype=np.float32), C))


def _quantise(x, inv, G, bits):
    """Codes clamp(rint(x inv), 0, Qp) of fp32 activations [..., G C], one fp32 product."""
    return torch.round(x * _per_channel(inv, x.shape[-1] // G)).clamp_(0, (1 << bits) - 1).to(torch.uint8)


def _quantise_bounds(x, lo, up, G, bits, dtype=torch.float32):
    """Codes rint(clip((x - l) / (u - l), 0, 1) Qp) with learned bounds."""
    C = x.shape[-1] // G
    l, u = _per_channel(lo, C).to(dtype), _per_channel(up, C).to(dtype)
    t = ((x.to(dtype) - l) * (1.0 / (u - l))).clamp_(0, 1)
    return torch.round(t * ((1 << bits) - 1)).to(torch.uint8)


def _to_format(q, fmt):
    """NHWC codes in a code format's bytes."""
    N, H, W, C = q.shape
    if fmt == "nhwc":
        return q.contiguous()
    if fmt == "c16":
        return q.view(N, H, W, C // 16, 16).permute(0, 3, 1, 2, 4).contiguous()
    b = q.view(N, H, W, C // 32, 16, 2).permute(0, 3, 1, 2, 4, 5)
    return (b[..., 0] | (b[..., 1] << 4)).contiguous()


def _empty_codes(N, H, W, C, fmt):
    shape = {"nhwc": (N, H, W, C), "c16": (N, C // 16, H, W, 16), "f4": (N, C // 32, H, W, 16)}[fmt]
    return torch.empty(shape, dtype=torch.uint8, device="cuda")


def _out(n, k, s, p):
    return (n + 2 * p - k) // s + 1


def _destination(case):
    """Destination group of each group."""
    G = case["G"]
    if case["shuffle"] == "cyclic":
        return [(g + 1) % G for g in range(G)]
    if case["shuffle"] == "explicit":
        return [G - 1 - g for g in range(G)]
    return list(range(G))


def _shuffle(case):
    if case["shuffle"] == "explicit":
        return B.shuffle(3, 0, _destination(case))
    return B.shuffle(1, 1) if case["shuffle"] == "cyclic" else B.shuffle(0, 0)


def _next_steps(case):
    """The next layer's input steps: the mean of ReLU(N(0, 2)) (with a shortcut about twice
    that), a little different in each group."""
    mean = 1.2 if case.get("shortcut") else 0.56
    qp = (1 << case["bits"]) - 1
    return np.array([2.0 * mean / math.sqrt(qp) * (1.0 + 0.05 * g) for g in range(case["G"])], dtype=np.float32)


def _bounds(case):
    G = case["G"]
    lo = np.array([0.02 + 0.01 * g for g in range(G)], dtype=np.float32)
    return lo, np.array([2.0 + 0.1 * g for g in range(G)], dtype=np.float32)


def _layer_inputs(case, seed):
    """What a layer gets, and the plain quantities behind it."""
    gen = _generator(seed)
    N, H, W, G, cin, cout, k, bits = (case[n] for n in ("N", "H", "W", "G", "cin", "cout", "k", "bits"))
    Ho, Wo = _out(H, k, case["stride"], case["pad"]), _out(W, k, case["stride"], case["pad"])
    x = _half_normal((N, H, W, G * cin), gen)
    w = _he((G, cout, k, k, cin), gen)
    r = dict(x=x, w=w, s_w=_steps(w, bits, signed=True), Ho=Ho, Wo=Wo, shape=(N, Ho, Wo, G * cout))
    if case["entry"] == "bounds":
        lo, up = _bounds(case)
        r.update(lo=lo, up=up, s_a=((up - lo) / ((1 << bits) - 1)).astype(np.float32))
    else:
        r["s_a"] = _steps(x.view(N, H, W, G, cin), bits)
        r["inv_a"] = _inverse(r["s_a"])
    r["shortcut"] = _half_normal(r["shape"], gen) if case["shortcut"] else None
    return r


def _pack(w, d, s_w):
    n = B.palquant_packed_weight_bytes(d)
    wp = torch.empty(n, dtype=torch.uint8, device="cuda")
    B.palquant_pack_weights(w.cpu().numpy(), d, _inverse(s_w), wp, n)
    return wp


# --------------------------------------------------------------------- prepare
def prepare(case, seed):
    state = {"layer": _prepare_layer, "front": _prepare_front, "qat": _prepare_qat,
             "network": _prepare_network}[case["kind"]](case, seed)
    state["run"] = {"layer": _run_layer, "front": _run_front, "qat": _run_qat,
                    "network": _run_network}[case["kind"]]
    return state


def _prepare_layer(case, seed):
    r = _layer_inputs(case, seed)
    N, H, W, G, cin, cout, bits, fmt = (case[n] for n in ("N", "H", "W", "G", "cin", "cout", "bits", "fmt"))
    d = B.layer_desc(N, H, W, G, cin, cout, case["k"], case["stride"], case["pad"], bits, bits, bits, 1,
                     code_format=FORMATS[fmt])
    shuf = _shuffle(case)
    s_next = _next_steps(case)
    m_out, m_req = B.palquant_epilogue_scales(G, r["s_w"], r["s_a"], 1.0, s_next, shuf)
    if case["shortcut"]:  # the codes come from the fp32 sum: fl(1/s) of the destination group
        m_req = _inverse(s_next)[_destination(case)]
    st = dict(case=case, d=d, shuf=shuf, m_out=m_out, m_req=m_req, wp=_pack(r["w"], d, r["s_w"]),
              shortcut=r["shortcut"], y=None, q_out=_empty_codes(N, r["Ho"], r["Wo"], G * cout, fmt))
    if case["out"] == "both":
        st["y"] = torch.empty(r["shape"], device="cuda")
    if case["entry"] == "codes":
        st["q"] = _to_format(_quantise(r["x"], r["inv_a"], G, bits), fmt)
    else:
        st["x"] = r["x"]
        st["q"] = None if case["entry"] == "on_load" else _empty_codes(N, H, W, G * cin, fmt)
        st.update({n: r[n] for n in ("inv_a", "lo", "up") if n in r})
    return st


def _run_layer(st):
    c = st["case"]
    if c["entry"] == "on_load":
        B.palquant_quantize_layer_fused(st["x"], st["inv_a"], st["wp"], st["d"], st["m_out"], st["m_req"], st["shuf"],
                                        st["shortcut"], None, st["y"], st["q_out"])
    else:
        if c["entry"] == "two_calls":
            B.palquant_quantize_act(st["x"], st["q"], c["N"], c["H"], c["W"], c["G"], c["cin"], c["bits"],
                                    st["inv_a"], code_format=FORMATS[c["fmt"]])
        elif c["entry"] == "bounds":
            B.palquant_quantize_act_lu(st["x"], st["q"], c["N"], c["H"], c["W"], c["G"], c["cin"], c["bits"],
                                       st["lo"], st["up"], code_format=FORMATS[c["fmt"]])
        B.palquant_layer_fused(st["q"], st["wp"], st["d"], st["m_out"], st["m_req"], st["shuf"], st["shortcut"], None,
                               st["y"], st["q_out"])
    out = {"codes": st["q_out"]}
    if st["y"] is not None:
        out["y"] = st["y"]
    return out


def _front_inputs(case, seed):
    gen = _generator(seed)
    N, H, W, G, cin, cout, bits = (case[n] for n in ("N", "H", "W", "G", "cin", "cout", "bits"))
    x = _half_normal((N, H, W, G * cin), gen)
    s_a = _steps(x.view(N, H, W, G, cin), bits)
    w1, wd = _he((G, cout, 3, 3, cin), gen), _he((G, cout, 1, 1, cin), gen)
    return dict(q=_quantise(x, _inverse(s_a), G, bits), s_a=s_a, w1=w1, wd=wd, s1=_steps(w1, bits, signed=True),
                sd=_steps(wd, bits, signed=True), shape=(N, _out(H, 3, 2, 1), _out(W, 3, 2, 1), G * cout))


def _prepare_front(case, seed):
    r = _front_inputs(case, seed)
    N, H, W, G, cin, cout, bits, fmt = (case[n] for n in ("N", "H", "W", "G", "cin", "cout", "bits", "fmt"))
    d1 = B.layer_desc(N, H, W, G, cin, cout, 3, 2, 1, bits, bits, bits, 1, code_format=FORMATS[fmt])
    dd = B.layer_desc(N, H, W, G, cin, cout, 1, 2, 0, bits, bits, bits, 0, code_format=FORMATS[fmt])
    none = B.shuffle(0, 0)
    m1, m_req1 = B.palquant_epilogue_scales(G, r["s1"], r["s_a"], 1.0, _next_steps(case), none)
    md, _ = B.palquant_epilogue_scales(G, r["sd"], r["s_a"], 1.0, None, none)
    return dict(d1=d1, dd=dd, none=none, m1=m1, m_req1=m_req1, md=md, wp1=_pack(r["w1"], d1, r["s1"]),
                wpd=_pack(r["wd"], dd, r["sd"]), q=_to_format(r["q"], fmt), q_out=_empty_codes(*r["shape"], fmt),
                down=torch.empty(r["shape"], device="cuda"))


def _run_front(st):
    B.palquant_layer_fused(st["q"], st["wp1"], st["d1"], st["m1"], st["m_req1"], st["none"], None, None, None,
                           st["q_out"])
    B.palquant_layer_fused(st["q"], st["wpd"], st["dd"], st["md"], None, st["none"], None, None, st["down"], None)
    return {"codes": st["q_out"], "down": st["down"]}


def _qat_inputs(case, seed):
    gen = _generator(seed)
    N, H, W, G, cin, cout, k = (case[n] for n in ("N", "H", "W", "G", "cin", "cout", "k"))
    lo, up = _bounds(case)
    wide = np.array([0.9 * math.sqrt(2.0 / (k * k * cin)) * (1.0 + 0.1 * g) for g in range(G)], dtype=np.float32)
    # activations [N H W, G cin] within [l, u], weights one row of G blocks within [-u, u]
    a = dict(P=N * H * W, Cg=cin, kind=0, l=lo, u=up, x=_half_normal((N * H * W, G * cin), gen))
    w = dict(P=1, Cg=cout * k * k * cin, kind=1, l=-wide, u=wide, x=_he((G, cout, k, k, cin), gen).view(1, -1))
    for t in (a, w):
        t["dy"] = torch.randn(t["x"].shape, generator=gen, device="cuda").mul_(1e-2)
    return a, w


def _prepare_qat(case, seed):
    parts = _qat_inputs(case, seed)
    G = case["G"]
    for t in parts:
        n = B.palquant_fake_quant_scratch_bytes(t["P"], G, t["Cg"])
        t.update(scratch=torch.empty(n, dtype=torch.uint8, device="cuda"), bytes=n, y=torch.empty_like(t["x"]),
                 dx=torch.empty_like(t["x"]), dl=torch.empty(G, dtype=torch.float64, device="cuda"),
                 du=torch.empty(G, dtype=torch.float64, device="cuda"))
    return dict(case=case, parts=parts)


def _run_qat(st):
    G, bits = st["case"]["G"], st["case"]["bits"]
    for t in st["parts"]:
        B.palquant_fake_quant_forward(t["x"], t["y"], t["P"], G, t["Cg"], bits, t["kind"], t["l"], t["u"])
    for t in reversed(st["parts"]):
        B.palquant_fake_quant_backward(t["x"], t["dy"], t["dx"], t["dl"], t["du"], t["P"], G, t["Cg"], bits,
                                       t["kind"], t["l"], t["u"], t["scratch"], t["bytes"])
    return [{n: t[n] for n in ("y", "dx", "dl", "du")} for t in st["parts"]]


def _network_inputs(case, seed):
    gen = _generator(seed)
    N, size, G = case["N"], case["size"], case["G"]
    x = torch.randn((N, size, size, 3), generator=gen, device="cuda")
    params = {"stem": _he((1, G * WIDTHS[0], 7, 7, 3), gen)[0]}
    cin = WIDTHS[0]
    for s, w in enumerate(WIDTHS):
        if case["placement"] == "paper":
            params[f"s{s + 1}.csm"] = _he((G, cin, 1, 1, cin), gen)
        for b in range(2):
            name = f"s{s + 1}b{b + 1}"
            params[name + ".conv1"] = _he((G, w, 3, 3, cin), gen)
            params[name + ".conv2"] = _he((G, w, 3, 3, w), gen)
            if s > 0 and b == 0:
                params[name + ".down"] = _he((G, w, 1, 1, cin), gen)
            cin = w
    params["fc"] = torch.randn((CLASSES, G * WIDTHS[-1]), generator=gen, device="cuda").mul_(
        math.sqrt(1.0 / (G * WIDTHS[-1])))
    return x, params


_SERVING = []


def _serving_stream():
    if not _SERVING:
        _SERVING.append(torch.cuda.Stream())
    return _SERVING[0]


def _prepare_network(case, seed):
    x, params = _network_inputs(case, seed)
    stream = torch.cuda.current_stream()
    if case["graph"]:  # graphs are captured and replayed on the one stream that serves them
        stream = _serving_stream()
        stream.wait_stream(torch.cuda.current_stream())
    net = PalQuantResNet18({n: w.cpu().numpy() for n, w in params.items()}, case["N"], case["size"], case["size"],
                           G=case["G"], widths=WIDTHS, classes=CLASSES, bits=2, stream=stream,
                           placement=case["placement"])
    net.calibrate(x)
    if case["graph"]:
        net.capture(x)
    return dict(net=net, x=x, graph=case["graph"])


def _run_network(st):
    return {"logits": st["net"].replay() if st["graph"] else st["net"].forward(st["x"])}


def run(state):
    return state["run"](state)


# ------------------------------------------------------------------------ work
def _conv_ops(n, h, w, G, cout, k, cin):
    return 2.0 * n * h * w * G * cout * k * k * cin


def work(case):
    kind = case["kind"]
    if kind == "network":
        return _network_work(case)
    N, H, W, G, cin, cout, bits = (case[n] for n in ("N", "H", "W", "G", "cin", "cout", "bits"))
    if kind == "qat":
        elems = N * H * W * G * cin + G * cout * case["k"] ** 2 * cin
        # forward: x in, the value out; backward: x and its gradient in, the gradient out
        return {"bytes": 20.0 * elems, "flops": 14.0 * elems}
    per = 0.5 if case["fmt"] == "f4" else 1.0  # bytes of a code
    if kind == "front":
        pix = _out(H, 3, 2, 1) * _out(W, 3, 2, 1) * N
        return {"bytes": per * (N * H * W * G * cin + pix * G * cout + 10 * G * cout * cin) + 4.0 * pix * G * cout,
                "flops": _conv_ops(pix, 1, 1, G, cout, 3, cin) + _conv_ops(pix, 1, 1, G, cout, 1, cin)}
    k = case["k"]
    pix = N * _out(H, k, case["stride"], case["pad"]) * _out(W, k, case["stride"], case["pad"])
    outs = pix * G * cout
    return {"bytes": (per if case["entry"] == "codes" else 4.0) * N * H * W * G * cin + per * G * cout * k * k * cin
            + per * outs + (4.0 * outs if case["out"] == "both" else 0.0) + (4.0 * outs if case["shortcut"] else 0.0),
            "flops": _conv_ops(pix, 1, 1, G, cout, k, cin)}


def _network_work(case):
    """Images and weights in, logits out; every convolution's and the head's operations."""
    N, G, size = case["N"], case["G"], case["size"]
    h = _out(size, 7, 2, 3)
    ops = _conv_ops(N, h, h, 1, G * WIDTHS[0], 7, 3)
    weights = 4.0 * G * WIDTHS[0] * 147
    h = _out(h, 3, 2, 1)
    cin = WIDTHS[0]
    for s, w in enumerate(WIDTHS):
        if case["placement"] == "paper":
            ops += _conv_ops(N, h, h, G, cin, 1, cin)
            weights += 0.5 * G * cin * cin
        for b in range(2):
            h = _out(h, 3, 2, 1) if s > 0 and b == 0 else h
            ops += _conv_ops(N, h, h, G, w, 3, cin) + _conv_ops(N, h, h, G, w, 3, w)
            weights += 0.5 * G * 9 * w * (cin + w)
            if s > 0 and b == 0:
                ops += _conv_ops(N, h, h, G, w, 1, cin)
                weights += 0.5 * G * w * cin
            cin = w
    ops += 2.0 * N * CLASSES * G * cin
    return {"bytes": 4.0 * N * size * size * 3 + weights + 4.0 * CLASSES * G * cin + 4.0 * N * CLASSES, "flops": ops}


# ------------------------------------------------------------------- tolerance
def tolerance(case):
    if case["kind"] == "network":
        # The fp32 sums of the stem and the shortcuts decide codes; another order of them
        # moves a few codes across a rounding boundary, and those travel to the logits
        # (against 64 bits: up to 0.019, and 0.1 of the root mean square at most).
        return {"rel": 0.03, "max": 0.4}
    if case["kind"] == "qat":
        # Every rounding of the values and input gradients is defined; the bounds' gradients
        # are long sums that partly cancel (against 64 bits: 4e-7).
        return {"rel": 2e-6, "max": 1e-5}
    if case["kind"] == "front" or case["out"] == "both":
        # One or two fp32 roundings of an exact integer sum (against 64 bits: 3e-8, at most
        # 5e-7 of the root mean square); a code of such a sum may sit on a tie.
        return {"rel": 2e-7, "max": 2e-6, "differ": 2e-6}
    return "exact"  # codes: whole numbers


# ----------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if kind == "network":
        return {"logits": _exact_network(case, seed)}
    if kind == "qat":
        return _exact_qat(case, seed)
    G, bits = case["G"], case["bits"]
    if kind == "front":
        r = _front_inputs(case, seed)
        s_next = _next_steps(case)
        q = r["q"].double()
        m1, m_req1 = _scales64(r["s1"], r["s_a"], s_next)
        md, _ = _scales64(r["sd"], r["s_a"], s_next)
        acc = _conv64(q, _weights64(r["w1"], r["s1"], bits), 2, 1)
        codes = _requantise64(acc, m_req1, G, bits)
        down = _scale64(_conv64(q, _weights64(r["wd"], r["sd"], bits), 2, 0), md, G)
        return {"codes": _to_format(codes, case["fmt"]), "down": down}
    r = _layer_inputs(case, seed)
    if case["entry"] == "bounds":
        q = _quantise_bounds(r["x"], r["lo"], r["up"], G, bits).double()
    else:
        q = _quantise(r["x"], r["inv_a"], G, bits).double()
    dst = _destination(case)
    s_next = _next_steps(case)[dst]
    m_out, m_req = _scales64(r["s_w"], r["s_a"], s_next)
    acc = _conv64(q, _weights64(r["w"], r["s_w"], bits), case["stride"], case["pad"])
    y = _scale64(acc, m_out, G)
    if case["shortcut"]:
        y = torch.relu(y + r["shortcut"])
        codes = _requantise64(y, _inverse(s_next), G, bits)
    else:
        y = torch.relu(y)
        codes = _requantise64(acc, m_req, G, bits)
    out = {"codes": _to_format(_permute(codes, dst), case["fmt"])}
    if case["out"] == "both":
        out["y"] = _permute(y, dst)
    return out


def _scales64(s_w, s_a, s_next):
    """The multipliers that a layer is given: fp32 values of the 64-bit products."""
    m = s_w.astype(np.float64) * s_a.astype(np.float64)
    return m.astype(np.float32), (m / s_next.astype(np.float64)).astype(np.float32)


def _weights64(w, s_w, bits):
    """Signed weight codes of w [G, Cout, k, k, Cin]."""
    t = torch.round(w * _on_gpu(_inverse(s_w)).view(-1, 1, 1, 1, 1))
    return t.clamp_(-(1 << (bits - 1)), (1 << (bits - 1)) - 1).double()


def _conv64(q, w, stride, pad):
    """Group convolution of q [N, H, W, G Cin] (64-bit) with w [G, Cout, k, k, Cin]."""
    N, H, W, C = q.shape
    G, cout, k, _, cin = w.shape
    Ho, Wo = _out(H, k, stride, pad), _out(W, k, stride, pad)
    p = torch.nn.functional.pad(q, (0, 0, pad, pad, pad, pad))
    out = torch.zeros((N, Ho, Wo, G * cout), dtype=torch.float64, device=q.device)
    for i in range(k):
        for j in range(k):
            v = p[:, i:i + stride * (Ho - 1) + 1:stride, j:j + stride * (Wo - 1) + 1:stride]
            for g in range(G):
                out[..., g * cout:(g + 1) * cout] += v[..., g * cin:(g + 1) * cin] @ w[g, :, i, j].T
    return out


def _scale64(acc, m, G):
    return acc * _per_channel(m, acc.shape[-1] // G).double()


def _requantise64(t, m, G, bits):
    return torch.round(_scale64(t, m, G)).clamp_(0, (1 << bits) - 1).to(torch.uint8)


def _permute(t, dst):
    """Group g's channels to group dst[g]."""
    v = t.view(*t.shape[:-1], len(dst), -1)
    out = torch.empty_like(v)
    out[..., dst, :] = v
    return out.view(t.shape)


def _exact_qat(case, seed):
    G, qp = case["G"], (1 << case["bits"]) - 1
    got = []
    for t in _qat_inputs(case, seed):
        x, dy = (t[n].double().view(t["P"], G, t["Cg"]) for n in ("x", "dy"))
        l, u = (_on_gpu(t[n]).double().view(1, G, 1) for n in ("l", "u"))
        c = 2.0 if t["kind"] else 1.0
        s = (x - l) / (u - l)
        v = torch.round(s.clamp(0, 1) * qp) / qp
        inside = dy * ((s > 0) & (s < 1))
        k = c / (u - l)
        got.append({"y": (c * v - t["kind"]).view(t["x"].shape), "dx": (inside * k).view(t["x"].shape),
                    "dl": (inside * (x - u) * k / (u - l)).sum((0, 2)),
                    "du": -(inside * (x - l) * k / (u - l)).sum((0, 2))})
    return got


def _exact_network(case, seed):
    x, params = _network_inputs(case, seed)
    N, G, bits, paper = case["N"], case["G"], 2, case["placement"] == "paper"
    X = torch.relu(_conv64(x.double(), params["stem"].double()[None], 2, 3))
    X = torch.nn.functional.max_pool2d(X.permute(0, 3, 1, 2), 3, 2, 1).permute(0, 2, 3, 1).contiguous()
    cyclic, keep = [(g + 1) % G for g in range(G)], list(range(G))

    def steps(t):
        return _steps(t.view(*t.shape[:-1], G, -1), bits)

    def conv(q, name, s_in, stride, pad):
        w = params[name]
        s_w = _steps(w, bits, signed=True)
        acc = _conv64(q.double(), _weights64(w, s_w, bits), stride, pad)
        return acc, s_w.astype(np.float64) * s_in.astype(np.float64)

    s_in = steps(X)
    q = _requantise64(X, _inverse(s_in), G, bits)
    for s in range(len(WIDTHS)):
        if paper:  # the cyclic shuffle module: X + Conv1x1 of the permuted codes
            acc, m = conv(_permute(q, cyclic), f"s{s + 1}.csm", s_in[[(g - 1) % G for g in range(G)]], 1, 0)
            X = _scale64(acc, m.astype(np.float32), G) + X
            s_in = steps(X)
            q = _requantise64(X, _inverse(s_in), G, bits)
        for b in range(2):
            name, stride = f"s{s + 1}b{b + 1}", 2 if s > 0 and b == 0 else 1
            acc, m = conv(q, name + ".conv1", s_in, stride, 1)
            s_mid = steps(torch.relu(_scale64(acc, m.astype(np.float32), G)))
            mid = _requantise64(acc, (m / s_mid.astype(np.float64)).astype(np.float32), G, bits)
            if name + ".down" in params:
                acc, m = conv(q, name + ".down", s_in, stride, 0)
                X = _scale64(acc, m.astype(np.float32), G)
            acc, m = conv(mid, name + ".conv2", s_mid, 1, 1)
            X = torch.relu(_scale64(acc, m.astype(np.float32), G) + X)
            if not paper:
                X = _permute(X, cyclic)
            elif b == 1:  # the stage's channel shuffle
                X = X.view(*X.shape[:-1], G, -1).transpose(-1, -2).reshape(X.shape)
            s_in = steps(X)
            q = _requantise64(X, _inverse(s_in), G, bits)
    return X.mean((1, 2)) @ params["fc"].double().T
