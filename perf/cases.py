"""The calls a user of the library makes, as timed cases: 1-D signals from one packet to 2^24 codes, single convolution
layers of several widths and shapes, and the compact CNN at serving and at batch size.

All sums are integers and exact, so outputs are compared bit for bit.  Sizes are those of the repository's own workloads
(the 1-D sweep, the two benchmark layers, the compact CNN) or generic odd ones.  As in a C program on this interface,
buffers are the caller's: outputs and the layer workspace are allocated once and passed to every call.
"""
import torch

from paper_2208_00763_b200 import binding as hk
from paper_2208_00763_b200 import inputs
from paper_2208_00763_b200.network import CompactCnn


def _signal(name, n, K, p, q, fs, gs):
    return {"name": name, "kind": "conv1d", "n": n, "K": K, "p": p, "q": q, "fs": fs, "gs": gs}


def _layer(name, B, Ci, H, W, Co, K, pad, p, q, xs, ws, requant, zeros=0.0):
    return {"name": name, "kind": "conv2d", "B": B, "Ci": Ci, "H": H, "W": W, "Co": Co, "K": K, "pad": pad, "p": p, "q": q,
            "xs": xs, "ws": ws, "requant": requant, "zeros": zeros}


def listed():
    return [
        # one short packet through a three-tap filter: the smallest call, all latency
        _signal("signal_4k_u4_k3", 4096, 3, 4, 4, False, False),
        # the two ends of the bitwidth sweep on a long signal: 4-bit signed with three taps, 8-bit unsigned with seven
        _signal("signal_16m_s4_k3", 1 << 24, 3, 4, 4, True, True),
        _signal("signal_16m_u8_k7", 1 << 24, 7, 8, 8, False, False),
        # a long FIR filter on a signal of odd length, unsigned codes against signed taps
        _signal("signal_4m_u4s4_k31", 4194301, 31, 4, 4, False, True),
        # a signal that is kept compressed in memory (four 2-bit codes per byte)
        {"name": "dense_16m_u2_k5", "kind": "conv1d_dense", "n": 1 << 24, "K": 5, "p": 2, "q": 2, "fs": False, "gs": False},
        # packing alone: codes to words of the paper's 4-bit configuration (three codes per 32-bit word, ten bits apart)
        {"name": "pack_16m_u4", "kind": "pack", "n": 1 << 24, "bits": 4, "signed": False, "S": 10, "N": 3, "word": 32},
        # the two benchmark layers: a 56x56 layer with requantised output, a deep 14x14 layer after a ReLU with exact sums
        _layer("layer_56x56x64_s4", 32, 64, 56, 56, 64, 3, 1, 4, 4, True, True, True),
        _layer("layer_14x14x256_u4s4", 64, 256, 14, 14, 256, 3, 1, 4, 4, False, True, False, 0.3),
        # 8-bit codes on a map whose sizes divide nothing
        _layer("layer_37x53x48_s8", 8, 48, 37, 53, 40, 3, 1, 8, 8, True, True, False),
        # a 5x5 kernel on 2-bit codes, odd sizes again, requantised
        _layer("layer_45x61x24_u2s2_k5", 16, 24, 45, 61, 40, 5, 2, 2, 2, False, True, True),
        # the compact CNN: a batch for throughput (the largest case), and one image for latency
        {"name": "cnn_batch64", "kind": "cnn", "B": 64, "H": 160, "W": 320},
        {"name": "cnn_batch1", "kind": "cnn", "B": 1, "H": 160, "W": 320},
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], uniform over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["conv1d", "conv1d", "conv1d_dense", "pack", "conv2d", "conv2d", "conv2d", "conv2d", "cnn"])
    if kind == "conv1d":
        # the sweep's three kernel lengths as often as any other length up to 32 taps (accepted at every width)
        K = rng.choice([3, 5, 7]) if rng.random() < 0.5 else _log_int(rng, 1, 32)
        p = rng.randint(1, 8)
        q = p if rng.random() < 0.7 else rng.randint(1, 8)
        fs = rng.random() < 0.5
        gs = fs if rng.random() < 0.7 else not fs
        return {"kind": kind, "n": _log_int(rng, 2000, 1 << (24 if K <= 8 else 22)), "K": K, "p": p, "q": q, "fs": fs, "gs": gs}
    if kind == "conv1d_dense":
        p, signed = rng.choice([1, 2, 4]), rng.random() < 0.5
        return {"kind": kind, "n": _log_int(rng, 4000, 1 << 24), "K": rng.choice([3, 5, 7]), "p": p, "q": p, "fs": signed, "gs": signed}
    if kind == "pack":
        bits, word = rng.randint(1, 8), rng.choice([32, 64])
        S = rng.randint(bits, 2 * bits + 4)
        return {"kind": kind, "n": _log_int(rng, 4000, 1 << 24), "bits": bits, "signed": rng.random() < 0.5, "S": S,
                "N": min(12, (word - bits) // S + 1), "word": word}
    if kind == "conv2d":
        K = rng.choice([3, 3, 3, 3, 1, 5])
        p = rng.choice([4, 4, 4, 4, 1, 2, 3, 5, 6, 7, 8])
        xs = rng.random() < 0.5
        H, W = _log_int(rng, 7, 112), _log_int(rng, 7, 160)
        Ci, Co = _log_int(rng, 3, 256), _log_int(rng, 8, 256)
        B = _log_int(rng, 1, 64)
        # no more work than the batch of the CNN takes at the lowest rate of the width and kernel size
        most = (3e9 if p <= 4 else 1e9) if K == 3 else 6e8
        while B * Ci * Co * H * W * K * K > most:
            if B > 1:
                B = (B + 1) // 2
            elif Ci > 16:
                Ci = (Ci + 1) // 2
            else:
                H, W = (H + 1) // 2, (W + 1) // 2
        return {"kind": kind, "B": B, "Ci": Ci, "H": H, "W": W, "Co": Co, "K": K, "pad": K // 2, "p": p, "q": p, "xs": xs,
                "ws": xs or p > 1, "requant": p > 1 and rng.random() < 0.6, "zeros": 0.0 if xs else 0.3}
    return {"kind": "cnn", "B": _log_int(rng, 1, 48), "H": 16 * rng.randint(3, 10), "W": 16 * rng.randint(3, 20)}


def _codes(gen, shape, bits, signed, zeros=0.0, centred=False):
    """Uniform codes of this width, one per byte, on the GPU (optionally with a share of zeros, as after a ReLU, or with a
    mean of zero, as trained weights have: the lowest signed code is left out, or deep networks would end in zeros only)."""
    lo, hi = (-(1 << (bits - 1)), (1 << (bits - 1)) - 1) if signed else (0, (1 << bits) - 1)
    if centred and signed and bits > 1:
        lo += 1
    v = torch.randint(lo, hi + 1, shape, generator=gen, device="cuda", dtype=torch.int16)
    if zeros > 0.0:
        v = v * (torch.rand(shape, generator=gen, device="cuda") >= zeros)
    return v.to(torch.int8) if signed else v.to(torch.uint8).view(torch.int8)


def _dense(codes, bits):
    """Codes stored 8 / bits per byte, lowest bits first."""
    per = 8 // bits
    v = codes.view(torch.uint8) & ((1 << bits) - 1)
    v = torch.nn.functional.pad(v, (0, -v.numel() % per)).reshape(-1, per)
    out = torch.zeros(v.shape[0], dtype=torch.uint8, device="cuda")
    for i in range(per):
        out |= v[:, i] << (bits * i)
    return out


def _requant(c):
    """A shift that spreads the sums over the codes of the layer's width, and that width's range."""
    shift, spread = 0, 0.35 * 4 ** c["p"] * (c["Ci"] * c["K"] * c["K"]) ** 0.5
    while spread / (1 << shift) > (1 << c["p"]):
        shift += 1
    return (shift, -(1 << (c["p"] - 1)), (1 << (c["p"] - 1)) - 1) if c["xs"] else (shift, 0, (1 << c["p"]) - 1)


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": c}
    if c["kind"] in ("conv1d", "conv1d_dense"):
        f = _codes(gen, (c["n"],), c["p"], c["fs"])
        s["f"] = _dense(f, c["p"]) if c["kind"] == "conv1d_dense" else f
        s["g"] = _codes(gen, (c["K"],), c["q"], c["gs"])
        s["y"] = torch.empty(c["n"] + c["K"] - 1, dtype=torch.int32, device="cuda")
    elif c["kind"] == "pack":
        s["f"] = _codes(gen, (c["n"],), c["bits"], c["signed"])
    elif c["kind"] == "conv2d":
        s["x"] = _codes(gen, (c["B"], c["Ci"], c["H"], c["W"]), c["p"], c["xs"], c["zeros"])
        s["w"] = _codes(gen, (c["Co"], c["Ci"], c["K"], c["K"]), c["q"], c["ws"], centred=True)
        s["requant"] = _requant(c) if c["requant"] else None
        s["workspace"] = torch.empty(hk.conv2d_workspace_bytes(c["B"], c["Ci"], c["H"], c["W"], c["Co"], c["K"], c["pad"]),
                                     dtype=torch.uint8, device="cuda")
        Ho, Wo = c["H"] + 2 * c["pad"] - c["K"] + 1, c["W"] + 2 * c["pad"] - c["K"] + 1
        s["out"] = torch.empty((c["B"], c["Co"], Ho, Wo), dtype=torch.int8 if c["requant"] else torch.int32, device="cuda")
    else:
        ch = inputs.C5_CHANNELS
        weights = [_codes(gen, (ch[i + 1], ch[i], 3, 3), 4, True, centred=True).cpu().numpy() for i in range(8)]
        layers = [{"w": w, "pad": 1, "shift": inputs.C5_SHIFTS[i], "lo": 0, "hi": 15, "pool": inputs.C5_POOL[i], "p": 8 if i == 0 else 4,
                   "q": 4, "x_signed": False, "w_signed": True} for i, w in enumerate(weights)]
        s["net"] = CompactCnn(layers, _codes(gen, (inputs.C5_HEAD_CHANNELS, ch[8], 1, 1), 4, True, centred=True).cpu().numpy())
        s["x"] = _codes(gen, (c["B"], inputs.C5_CHANNELS[0], c["H"], c["W"]), 8, False)
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "conv1d":
        return hk.conv1d(s["f"], s["g"], c["p"], c["q"], c["fs"], c["gs"], out=s["y"])
    if c["kind"] == "conv1d_dense":
        return hk.conv1d_dense(s["f"], c["n"], s["g"], c["p"], c["q"], c["fs"], c["gs"], out=s["y"])
    if c["kind"] == "pack":
        return hk.pack(s["f"], c["bits"], c["signed"], c["S"], c["N"], c["word"])
    if c["kind"] == "conv2d":
        return hk.conv2d(s["x"], s["w"], c["pad"], c["p"], c["q"], c["xs"], c["ws"], requant=s["requant"], workspace=s["workspace"],
                         out=s["out"])
    head, _ = s["net"].forward(s["x"])
    return head


def _layer_work(B, Ci, H, W, Co, K, out_h, out_w):
    return 2.0 * B * Co * Ci * K * K * out_h * out_w


def work(case):
    """Inputs read once, outputs written once, one multiply and one add per product of the plain definition."""
    c = case
    if c["kind"] in ("conv1d", "conv1d_dense"):
        bits = 8 if c["kind"] == "conv1d" else c["p"]
        n_out = c["n"] + c["K"] - 1
        return {"bytes": c["n"] * bits / 8 + c["K"] + 4 * n_out, "flops": 2.0 * n_out * c["K"]}
    if c["kind"] == "pack":
        words = -(-c["n"] // c["N"])
        return {"bytes": c["n"] + words * c["word"] / 8, "flops": 2.0 * c["n"]}
    if c["kind"] == "conv2d":
        Ho, Wo = c["H"] + 2 * c["pad"] - c["K"] + 1, c["W"] + 2 * c["pad"] - c["K"] + 1
        return {"bytes": c["B"] * c["Ci"] * c["H"] * c["W"] + c["Co"] * c["Ci"] * c["K"] ** 2
                + c["B"] * c["Co"] * Ho * Wo * (1 if c["requant"] else 4),
                "flops": _layer_work(c["B"], c["Ci"], c["H"], c["W"], c["Co"], c["K"], Ho, Wo)}
    B, H, W, ch = c["B"], c["H"], c["W"], inputs.C5_CHANNELS
    flops, weights = 0.0, 0
    for i in range(8):
        flops += _layer_work(B, ch[i], H, W, ch[i + 1], 3, H, W)
        weights += 9 * ch[i] * ch[i + 1]
        if inputs.C5_POOL[i]:
            H, W = H // 2, W // 2
    flops += _layer_work(B, ch[8], H, W, inputs.C5_HEAD_CHANNELS, 1, H, W)
    weights += ch[8] * inputs.C5_HEAD_CHANNELS
    return {"bytes": B * ch[0] * c["H"] * c["W"] + weights + 4 * B * inputs.C5_HEAD_CHANNELS * H * W, "flops": flops}


def tolerance(case):
    return "exact"          # integer sums, packed words and requantised codes: one correct answer
