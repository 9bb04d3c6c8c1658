"""Performance cases of the library: what a program that uses it has it do.

Every case goes through the public entry points (the C ABI's binding `ifq` and `DeviceStack`): single
quantized substructures (ifq_conv2bit), whole networks (ifq_forward, or a captured graph's replay),
the code pool (ifq_maxpool2bit) and the packing helpers at the boundary of a network.  Results are
integers (packed codes, int32 accumulators, fixed-point values), so the tolerance is "exact" and
exact() restates them in float64 / int64 torch.

Inputs are synthetic and seeded: uniform k-bit codes (uniform 8-bit pixels with a zero fourth channel
for an image), +-1 filters, and float parameters in the ranges of a trained layer (small filter
scales, batch-norm statistics matched to the layer's own spread, one channel in ten with a negative
batch-norm scale), so that the codes spread over every level.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1911_08076_gb300 import ifq, synth
from paper_1911_08076_gb300.stack import DeviceStack

DEV = "cuda"
OUT = {"codes": ifq.IFQ_OUT_CODES, "acc": ifq.IFQ_OUT_ACC, "both": ifq.IFQ_OUT_BOTH}
EPS = float(np.float32(1e-5))


def _conv(name, n, h, w, cin, cout, k, stride=1, pad=None, pool=0, kbits=2, in_bits=0, out="codes"):
    return {"name": name, "do": "conv", "n": n, "h": h, "w": w, "cin": cin, "cout": cout, "k": k, "stride": stride,
            "pad": k // 2 if pad is None else pad, "pool": pool, "kbits": kbits, "in_bits": in_bits, "out": out}


def listed():
    return [
        # one small layer, one image, codes and accumulators: a latency-bound call
        _conv("conv3x3_64_16x16_b1", 1, 16, 16, 64, 64, 3, out="both"),
        # an embedded-vision request: one image through the classifier body, replayed as a graph
        {"name": "resnet18_b1_graph", "do": "stack", "net": "resnet18", "batch": 1, "graph": True},
        # the classifier body at its usual batch, replayed as a graph
        {"name": "resnet18_b32_graph", "do": "stack", "net": "resnet18", "batch": 32, "graph": True},
        # the paper's AlexNet substructures (5x5, 3x3, overlapping pools, fully connected), called eagerly
        {"name": "alexnet_b128", "do": "stack", "net": "alexnet", "batch": 128, "graph": False},
        # the same network with 4-bit codes (the accuracy option)
        {"name": "alexnet_k4_b128_graph", "do": "stack", "net": "alexnet_k4", "batch": 128, "graph": True},
        # the face detector's backbone with its pools fused
        {"name": "tinyyolo_fused_b64_graph", "do": "stack", "net": "tinyyolo_fused", "batch": 64, "graph": True},
        # the half-width detector from 8-bit pixels to fixed-point detections
        {"name": "tinieryolo_full_fused_b64_graph", "do": "stack", "net": "tinieryolo_full_fused", "batch": 64,
         "graph": True},
        # large single layers
        _conv("conv3x3_256_56x56_b256", 256, 56, 56, 256, 256, 3),
        _conv("conv1x1_512_28x28_b256", 256, 28, 28, 512, 512, 1),
        # an odd layer: ragged map, channel counts that fill no tile, accumulators beside the codes
        _conv("conv3x3_72_100_37x45_b9_both", 9, 37, 45, 72, 100, 3, out="both"),
        # pooling on codes as its own call, larger than the L2 cache
        {"name": "pool2x2_32_208x208_b512", "do": "pool", "n": 512, "h": 208, "w": 208, "c": 32, "k": 2, "stride": 2,
         "pad": 0, "kbits": 2, "signed": True},
        # the boundary of a network: one code a byte packed into the library's format, and back
        {"name": "pack_unpack_208x208x16_b64", "do": "pack", "codes": 64 * 208 * 208 * 16, "kbits": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


NETS = {"resnet18": 32, "alexnet": 128, "alexnet_k3": 128, "alexnet_k4": 128, "resnet18_k4": 32, "tinyyolo": 64,
        "tinyyolo_fused": 64, "tinieryolo_fused": 64, "tinieryolo_full_fused": 64}


def draw(rng):
    do = rng.choice(["conv", "conv", "conv", "stack", "stack", "pool", "pack"])
    if do == "stack":
        net = rng.choice(sorted(NETS))
        return {"do": "stack", "net": net, "batch": _log(rng, 1, NETS[net]), "graph": rng.random() < 0.6}
    if do == "pool":
        kbits = rng.choice([2, 2, 3, 4])
        k, stride, pad = rng.choice([(2, 2, 0), (2, 2, 0), (3, 2, 0), (2, 1, 1)])
        while True:
            c = {"do": "pool", "n": _log(rng, 1, 512), "h": _log(rng, 6, 208), "w": _log(rng, 6, 208),
                 "c": 4 * _log(rng, 2, 128), "k": k, "stride": stride, "pad": pad, "kbits": kbits,
                 "signed": rng.random() < 0.7}
            if c["n"] * c["h"] * c["w"] * c["c"] <= 512 * 208 * 208 * (32 if kbits == 2 else 16):
                return c
    if do == "pack":
        return {"do": "pack", "codes": 4 * _log(rng, 1 << 12, 1 << 25), "kbits": rng.choice([2, 2, 3, 4])}
    while True:
        kbits, in_bits = rng.choice([(2, 0), (2, 0), (2, 0), (3, 0), (4, 0), (2, 8)])
        k, stride = rng.choice([(3, 1), (3, 1), (3, 1), (1, 1), (5, 1), (3, 2), (1, 2)])
        if in_bits == 8:   # a first layer on pixels
            cin, cout, k = 4, rng.choice([8, 16, 32, 64]), 3
        elif rng.random() < 0.6:   # widths of the usual networks
            cin, cout = 2 ** rng.randint(3, 10), 2 ** rng.randint(3, 10)
        else:
            unit = 4 if kbits == 2 else 8
            cin, cout = unit * _log(rng, 2, 512 // unit), 4 * _log(rng, 2, 256)
        h = _log(rng, 5, 112)
        w = h if rng.random() < 0.5 else _log(rng, 5, 112)
        out = rng.choice(["codes", "codes", "codes", "both", "acc"])
        pool = 2 if rng.random() < 0.3 else 0
        c = _conv("", _log(rng, 1, 256), h, w, cin, cout, k, stride, k // 2, pool, kbits, in_bits, out)
        del c["name"]
        ho, wo = (h - 1) // stride + 1, (w - 1) // stride + 1
        if pool and (out != "codes" or ho % 2 or wo % 2):
            continue
        if (255 if in_bits == 8 else 2 ** kbits - 1) * k * k * cin > 196608:
            continue
        wk = work(c)
        # no dearer than the largest listed layer, narrow channel counts included
        if wk["flops"] <= 9e11 and wk["bytes"] <= 4e8 and c["n"] * ho * wo * max(64, k * k * cin) * max(64, cout) <= 4e11:
            return c


# ------------------------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1911 + seed)
    return g


def _codes(g, shape, kbits):
    return torch.randint(0, 1 << kbits, shape, dtype=torch.uint8, device=DEV, generator=g)


def _pixels(g, shape):
    x = torch.randint(0, 256, shape, dtype=torch.uint8, device=DEV, generator=g)
    x[..., 3:] = 0
    return x


def _filters(g, cout, k, cin):
    return torch.randint(0, 2, (cout, k, k, cin), dtype=torch.int8, device=DEV, generator=g) * 2 - 1


def _pack(codes, kbits):
    """uint8 codes [..., C] -> packed [..., C*f/8] (f = 2 for 2-bit codes, 4 for 3- and 4-bit ones)."""
    f = 2 if kbits == 2 else 4
    per = 8 // f
    q = codes.reshape(codes.shape[:-1] + (codes.shape[-1] // per, per))
    out = q[..., 0].clone()
    for i in range(1, per):
        out |= q[..., i] << (f * i)
    return out


def _params(rng, cout, K, kbits, in_bits):
    """Float parameters of a layer in a trained layer's ranges (see the module's docstring)."""
    L = (1 << kbits) - 1
    step = 1.5 / L                                     # quantizer step of the input and output codes
    delta = 1.0 / 255.0 if in_bits == 8 else step
    m2 = 0.75 * 255 * 511 / 6 if in_bits == 8 else L * (2 * L + 1) / 6   # mean square of an input value
    alpha = rng.uniform(0.005, 0.05, cout).astype(np.float32)
    sd = alpha.astype(np.float64) * delta * math.sqrt(m2 * K)
    gamma = np.abs(rng.normal(1.0, 0.3, cout)) * np.where(rng.random(cout) < 0.1, -1.0, 1.0)
    return {"alpha": alpha, "gamma": gamma.astype(np.float32),
            "beta": rng.normal(0.0, 0.5, cout).astype(np.float32),
            "mean": (rng.normal(0.0, 0.1, cout) * sd).astype(np.float32),
            "var": (sd * sd * rng.uniform(0.8, 1.25, cout)).astype(np.float32),
            "delta_in": float(np.float32(delta)), "q_base": float(np.float32(step)),
            "q_offset": float(np.float32(-step / 2))}


def _conv_inputs(c, seed):
    g, rng = _gen(seed), np.random.default_rng(seed)
    shape = (c["n"], c["h"], c["w"], c["cin"])
    x = _pixels(g, shape) if c["in_bits"] == 8 else _codes(g, shape, c["kbits"])
    w = _filters(g, c["cout"], c["k"], c["cin"])
    return x, w, _params(rng, c["cout"], c["k"] ** 2 * c["cin"], c["kbits"], c["in_bits"])


def _stack_inputs(c, seed):
    wl = synth.get(c["net"], c["batch"])
    g, rng = _gen(seed), np.random.default_rng(seed)
    shape = (wl.batch, wl.h, wl.w, wl.c)
    x = _pixels(g, shape) if wl.in_bits == 8 else _codes(g, shape, wl.kbits)
    ws, ps = [], []
    for l in wl.layers:
        conv = l.kind == "conv"
        ws.append(_filters(g, l.cout, l.k, l.cin) if conv else None)
        ps.append(_params(rng, l.cout, l.k * l.k * l.cin, wl.kbits, l.in_bits) if conv else None)
    return wl, x, ws, ps


def prepare(case, seed):
    do = case["do"]
    if do == "conv":
        x, w, p = _conv_inputs(case, seed)
        k, cin, cout, kbits = case["k"], case["cin"], case["cout"], case["kbits"]
        K, mode = k * k * cin, OUT[case["out"]]
        d = ifq.conv_desc(case["n"], case["h"], case["w"], cin, cout, k, case["stride"], case["pad"], mode,
                          pool=case["pool"], kbits=kbits, in_bits=case["in_bits"])
        K_fold = -(-255 * K // ((1 << kbits) - 1)) if case["in_bits"] == 8 else K
        T, s = ifq.ifq_fold_layer(K_fold, p["alpha"], p["gamma"], p["beta"], p["mean"], p["var"], p["delta_in"], None,
                                  EPS, p["q_base"], p["q_offset"], kbits)
        bits = torch.empty((cout, (K + 31) // 32), dtype=torch.int32, device=DEV)
        ifq.ifq_pack_signs(w.view(cout, K), bits, cout, K)
        prep = torch.empty(ifq.ifq_weights_prep_bytes(d), dtype=torch.uint8, device=DEV)
        ifq.ifq_pack_weights(d, bits, prep)
        ho, wo = ifq.ifq_conv_out_shape(d)
        f = 2 if kbits == 2 else 4
        yc = torch.empty((case["n"], ho, wo, cout * f // 8), dtype=torch.uint8, device=DEV) if mode & 1 else None
        ya = torch.empty((case["n"], ho, wo, cout), dtype=torch.int32, device=DEV) if mode & 2 else None
        return {"do": do, "d": d, "x": x if case["in_bits"] == 8 else _pack(x, kbits), "prep": prep,
                "thr": torch.from_numpy(T).to(DEV), "sign": torch.from_numpy(s).to(DEV), "yc": yc, "ya": ya}
    if do == "stack":
        wl, x, ws, ps = _stack_inputs(case, seed)
        params = [None if w is None else synth.ConvParams(w.cpu().numpy(), eps=EPS, **p) for w, p in zip(ws, ps)]
        st = DeviceStack(wl, params, device=DEV)
        xb = st.input_buffer()
        xb.copy_(x if wl.in_bits == 8 else _pack(x, wl.kbits))
        if case["graph"]:
            st.capture(xb)
        outs = [t for li in range(len(wl.layers)) for t in (st.y_codes.get(li), st.y_acc.get(li)) if t is not None]
        return {"do": do, "st": st, "x": xb, "graph": case["graph"], "outs": outs}
    if do == "pool":
        g, rng = _gen(seed), np.random.default_rng(seed)
        x = _codes(g, (case["n"], case["h"], case["w"], case["c"]), case["kbits"])
        sign = np.where(rng.random(case["c"]) < 0.1, -1, 1).astype(np.int8)
        d = ifq.pool_desc(case["n"], case["h"], case["w"], case["c"], case["k"], case["stride"], case["pad"],
                          case["kbits"])
        ho, wo = ifq.ifq_pool_out_shape(d)
        xp = _pack(x, case["kbits"])
        y = torch.empty((case["n"], ho, wo, xp.shape[-1]), dtype=torch.uint8, device=DEV)
        return {"do": do, "d": d, "x": xp, "sign": torch.from_numpy(sign).to(DEV) if case["signed"] else None, "y": y}
    codes = _codes(_gen(seed), (case["codes"],), case["kbits"])
    f = 2 if case["kbits"] == 2 else 4
    return {"do": do, "codes": codes, "kbits": case["kbits"], "n": case["codes"],
            "packed": torch.empty(case["codes"] * f // 8, dtype=torch.uint8, device=DEV),
            "back": torch.empty_like(codes)}


def run(state):
    do = state["do"]
    if do == "conv":
        ifq.ifq_conv2bit(state["d"], state["x"], state["prep"], state["thr"], state["sign"], state["yc"], state["ya"])
        return [t for t in (state["yc"], state["ya"]) if t is not None]
    if do == "stack":
        if state["graph"]:
            state["st"].replay()
        else:
            state["st"].forward(state["x"])
        return state["outs"]
    if do == "pool":
        ifq.ifq_maxpool2bit(state["d"], state["x"], state["sign"], state["y"])
        return [state["y"]]
    ifq.ifq_pack_codes_kbits(state["codes"], state["packed"], state["n"], state["kbits"])
    ifq.ifq_unpack_codes_kbits(state["packed"], state["back"], state["n"], state["kbits"])
    return [state["packed"], state["back"]]


# ------------------------------------------------------------------------------------ work


def _conv_work(n, h, w, cin, cout, k, stride, pad, pool, kbits, in_bits, out, read_x=True):
    f = 2 if kbits == 2 else 4
    ho, wo = (h + 2 * pad - k) // stride + 1, (w + 2 * pad - k) // stride + 1
    K, p = k * k * cin, max(1, pool)
    by = cout * K / 8 + cout * (4 * ((1 << kbits) - 1) + 1)   # one bit a weight, the thresholds and signs
    if read_x:
        by += n * h * w * cin * (1 if in_bits == 8 else f / 8)
    if out in ("codes", "both"):
        by += n * (ho // p) * (wo // p) * cout * f / 8
    if out in ("acc", "both"):
        by += n * ho * wo * cout * 4
    return by, 2.0 * n * ho * wo * cout * K


def work(case):
    do = case["do"]
    if do == "conv":
        by, fl = _conv_work(*[case[q] for q in ("n", "h", "w", "cin", "cout", "k", "stride", "pad", "pool", "kbits",
                                                "in_bits", "out")])
        return {"bytes": by, "flops": fl}
    if do == "stack":   # the input, every filter and every layer's output once
        wl = synth.get(case["net"], case["batch"])
        f = 2 if wl.kbits == 2 else 4
        by, fl = wl.batch * wl.h * wl.w * wl.c * (1 if wl.in_bits == 8 else f / 8), 0.0
        for l in wl.layers:
            if l.kind == "conv":
                b, o = _conv_work(wl.batch, l.h, l.w, l.cin, l.cout, l.k, l.stride, l.pad, l.pool, wl.kbits, l.in_bits,
                                  l.out, read_x=False)
                by, fl = by + b, fl + o
            elif l.kind == "pool":
                by += wl.batch * l.ho * l.wo * l.c * f / 8
            else:
                s = wl.layers[l.src]
                by += wl.batch * s.out_h * s.out_w * s.cout * 4
        return {"bytes": by, "flops": fl}
    if do == "pool":
        f = 2 if case["kbits"] == 2 else 4
        ho = (case["h"] + case["pad"] - case["k"]) // case["stride"] + 1
        wo = (case["w"] + case["pad"] - case["k"]) // case["stride"] + 1
        out = case["n"] * ho * wo * case["c"]
        return {"bytes": (case["n"] * case["h"] * case["w"] * case["c"] + out) * f / 8,
                "flops": float(out * case["k"] ** 2)}
    f = 2 if case["kbits"] == 2 else 4
    return {"bytes": 2.0 * (case["codes"] + case["codes"] * f / 8), "flops": float(2 * case["codes"])}


def tolerance(case):
    return "exact"   # every result is an integer (codes, accumulators, fixed-point values) with one right value


# ------------------------------------------------------------------------------------ exact values


def _thresholds(p, kbits):
    """Per-channel float64 bounds t and signs s: code = #{ i : s*A > t_i } (Eq. (7); the floor is left out,
    A being an integer)."""
    d = {q: np.asarray(p[q], np.float64) for q in ("alpha", "gamma", "beta", "mean", "var")}
    thr = p["q_base"] * np.arange(1, 1 << kbits, dtype=np.float64) + p["q_offset"]
    tau = ((thr[None, :] - d["beta"][:, None]) * np.sqrt(d["var"] + EPS)[:, None] / d["gamma"][:, None] +
           d["mean"][:, None]) / (d["alpha"] * p["delta_in"])[:, None]
    s = np.where(d["gamma"] < 0, -1.0, 1.0)
    return torch.from_numpy(tau * s[:, None]).to(DEV), torch.from_numpy(s).to(DEV)


def _quantize(a, p, kbits):
    t, s = _thresholds(p, kbits)
    sa = a * s
    out = torch.zeros(a.shape, dtype=torch.uint8, device=a.device)
    for i in range(t.shape[1]):
        out += sa > t[:, i]
    return out


def _exact_conv(x, w, p, stride, pad, pool, kbits, out):
    """(codes or None, accumulators or None) of one layer in float64, NHWC, a few images at a time."""
    n, h, wd, cin = x.shape
    cout, k = w.shape[0], w.shape[1]
    w2 = w.permute(0, 3, 1, 2).reshape(cout, -1).double()
    ho, wo = (h + 2 * pad - k) // stride + 1, (wd + 2 * pad - k) // stride + 1
    per = max(1, int(2e8 / (k * k * cin * ho * wo)))
    codes, accs = [], []
    for i in range(0, n, per):
        xi = x[i:i + per].permute(0, 3, 1, 2).double()
        a = torch.matmul(w2, F.unfold(xi, k, padding=pad, stride=stride)).view(-1, cout, ho, wo)
        if out in ("acc", "both"):
            accs.append(a.permute(0, 2, 3, 1).to(torch.int32))
        if out in ("codes", "both"):
            if pool > 1:
                a = F.max_pool2d(a, pool)
            codes.append(_quantize(a.permute(0, 2, 3, 1), p, kbits))
    return (torch.cat(codes) if codes else None), (torch.cat(accs) if accs else None)


def _exact_pool(x, sign, k, stride, pad):
    s = torch.ones(x.shape[-1], device=DEV) if sign is None else sign.to(DEV).float()
    v = (x.float() * s).permute(0, 3, 1, 2)
    v = F.pad(v, (0, pad, 0, pad), value=-1e9)
    return (F.max_pool2d(v, k, stride).permute(0, 2, 3, 1) * s).to(torch.uint8)


def _exact_fixed(acc, p, m):
    q = 1 << m
    mul = np.floor(p["alpha"].astype(np.float64) * q) * math.floor(p["delta_in"] * q)
    v = (torch.from_numpy(mul.astype(np.int64)).to(DEV) * acc.long()) >> m
    return v.clamp(-2 ** 31, 2 ** 31 - 1).to(torch.int32)


def exact(case, seed):
    do = case["do"]
    if do == "conv":
        x, w, p = _conv_inputs(case, seed)
        codes, acc = _exact_conv(x, w, p, case["stride"], case["pad"], case["pool"], case["kbits"], case["out"])
        return [t for t in (None if codes is None else _pack(codes, case["kbits"]), acc) if t is not None]
    if do == "stack":
        wl, x, ws, ps = _stack_inputs(case, seed)
        codes, accs, outs = {-1: x}, {}, []
        for li, l in enumerate(wl.layers):
            if l.kind == "conv":
                c, a = _exact_conv(codes[l.src], ws[li], ps[li], l.stride, l.pad, l.pool, wl.kbits, l.out)
                codes[li], accs[li] = c, a
            elif l.kind == "pool":
                s = np.where(ps[l.src]["gamma"] < 0, -1, 1).astype(np.int8)
                codes[li] = _exact_pool(codes[l.src], torch.from_numpy(s) if l.signed else None, l.k, l.stride, l.pad)
            else:
                accs[li] = _exact_fixed(accs[l.src], ps[l.src], l.m)
            outs += [t for t in (None if codes.get(li) is None else _pack(codes[li], wl.kbits), accs.get(li))
                     if t is not None]
        return outs
    if do == "pool":
        g, rng = _gen(seed), np.random.default_rng(seed)
        x = _codes(g, (case["n"], case["h"], case["w"], case["c"]), case["kbits"])
        sign = torch.from_numpy(np.where(rng.random(case["c"]) < 0.1, -1, 1).astype(np.int8))
        per = max(1, int(2e8 / (case["h"] * case["w"] * case["c"])))
        y = [_exact_pool(x[i:i + per], sign if case["signed"] else None, case["k"], case["stride"], case["pad"])
             for i in range(0, case["n"], per)]
        return [_pack(torch.cat(y), case["kbits"])]
    codes = _codes(_gen(seed), (case["codes"],), case["kbits"])
    return [_pack(codes, case["kbits"]), codes]
