"""Performance cases of the decoder library: what a program that uses it has it do.

Each case is one call of a public entry point on inputs that are already on the
GPU: batches of noise realisations or syndromes of the toric code, packed
batches of mixed lattice sizes, rings of the repetition code, open-boundary
lattices, and the learned pre-decoder's inference (bf16 and FP8) and gradients.
Noise is drawn from torch's generator, so a case's inputs depend on its seed
alone.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2506_03266_gb300 as qca

# sizes and weights (per cent) of the mixed-size workload
MIX = "24:30,48:25,64:20,96:12,128:8,192:5"
# (c_out, c_in) of the pre-decoder's 3x3 circular convolutions
LAYERS = [(32, 2), (32, 32), (32, 32), (4, 32)]
SMOOTHING = 0.1  # label smoothing of the training loss


def listed():
    return [
        # a control loop's call: a few small codes, where launches and latency count
        {"name": "decode_L16_64", "kind": "decode", "L": 16, "shots": 64, "p": 0.05,
         "max_steps": 4096},
        # a threshold study's point on odd lattices
        {"name": "decode_L49_2000", "kind": "decode", "L": 49, "shots": 2000, "p": 0.06,
         "max_steps": 1000},
        # the plain decoder at the pre-decoder comparison's size
        {"name": "decode_L128_10000", "kind": "decode", "L": 128, "shots": 10000, "p": 0.04,
         "max_steps": 4096},
        # the headline workload, a fifth of its batch
        {"name": "decode_L256_20000", "kind": "decode", "L": 256, "shots": 20000, "p": 0.05,
         "max_steps": 4096},
        # the large-lattice stress
        {"name": "decode_L1024_512", "kind": "decode", "L": 1024, "shots": 512, "p": 0.05,
         "max_steps": 4096},
        # decoding measured syndromes, under the second reading of the tie and balance rules
        {"name": "syndrome_L64_5000", "kind": "syndrome", "L": 64, "shots": 5000, "p": 0.06,
         "max_steps": 1000, "tie_order": 1, "balance_rule": 1},
        # the packed batch of mixed sizes and noise rates
        {"name": "uneven_20000", "kind": "uneven", "mix": MIX, "shots": 20000, "p_lo": 0.01,
         "p_hi": 0.07, "max_steps": 4096},
        # the repetition code on rings, with its random moves
        {"name": "ring_L1024_20000", "kind": "ring", "L": 1024, "shots": 20000, "p": 0.3,
         "p_move": 0.1, "max_steps": 4096},
        # open (rough) boundaries
        {"name": "open_L64_5000", "kind": "open", "L": 64, "shots": 5000, "p": 0.05,
         "max_steps": 4096},
        # the pre-decoder's forward pass, bf16
        {"name": "logits_bf16_L128_1000", "kind": "logits", "L": 128, "shots": 1000, "p": 0.04,
         "precision": "bf16"},
        # the pre-decoder's forward pass, FP8
        {"name": "logits_fp8_L256_250", "kind": "logits", "L": 256, "shots": 250, "p": 0.05,
         "precision": "fp8"},
        # forward and backward of one training batch
        {"name": "gradients_L32_256", "kind": "gradients", "L": 32, "shots": 256, "p": 0.05},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shots(rng, L, lo, hi, most):
    """A batch of between lo and hi lattice sites, its logarithm uniform."""
    return max(1, min(most, _log_int(rng, lo, hi) // (L * L)))


def draw(rng):
    kind = rng.choice(["decode"] * 7 + ["syndrome"] * 2 + ["uneven"] * 3 +
                      ["ring", "open", "logits", "logits", "gradients"])
    if kind == "decode":
        part = rng.random()
        if part < 0.6:      # the usual sizes
            L = 4 * _log_int(rng, 2, 64)
        elif part < 0.8:    # any size, odd ones among them
            L = _log_int(rng, 5, 129)
        else:               # large lattices
            L = rng.choice([384, 512, 640, 768, 1024, _log_int(rng, 260, 700)])
        hi = 1 << (27 if L <= 256 and L % 4 == 0 else 24)
        return {"kind": kind, "L": L, "shots": _shots(rng, L, 1 << 14, hi, 20000),
                "p": round(rng.uniform(0.01, 0.055), 4), "max_steps": 1000}
    if kind == "syndrome":
        L = 4 * _log_int(rng, 3, 48)
        return {"kind": kind, "L": L, "shots": _shots(rng, L, 1 << 14, 1 << 24, 8000),
                "p": round(rng.uniform(0.01, 0.06), 4), "max_steps": 1000,
                "tie_order": rng.randrange(2), "balance_rule": rng.randrange(2)}
    if kind == "uneven":
        odd = rng.random() < 0.3
        sizes = set()
        while len(sizes) < 4:
            sizes.add(_log_int(rng, 9, 100) if odd else 4 * _log_int(rng, 3, 48))
        mix = ",".join("%d:%d" % (s, rng.randrange(10, 40)) for s in sorted(sizes))
        return {"kind": kind, "mix": mix, "shots": _log_int(rng, 100, 8000), "p_lo": 0.01,
                "p_hi": round(rng.uniform(0.03, 0.06), 4), "max_steps": 1000}
    if kind == "ring":
        L = _log_int(rng, 50, 4096)
        return {"kind": kind, "L": L, "shots": max(1, min(20000, _log_int(rng, 1 << 14, 1 << 24) // L)),
                "p": round(rng.uniform(0.1, 0.35), 3), "p_move": rng.choice([0.0, 0.1]),
                "max_steps": 4096}
    if kind == "open":
        L = _log_int(rng, 9, 100)
        return {"kind": kind, "L": L, "shots": _shots(rng, L, 1 << 14, 1 << 24, 8000),
                "p": round(rng.uniform(0.01, 0.05), 4), "max_steps": 1000}
    if kind == "logits":
        L = rng.choice([128, 256, _log_int(rng, 16, 300)])
        return {"kind": kind, "L": L, "shots": _shots(rng, L, 1 << 14, 1 << 24, 4000),
                "p": round(rng.uniform(0.02, 0.07), 4), "precision": rng.choice(["bf16", "fp8"])}
    L = rng.choice([24, 32, 48, 64])
    return {"kind": kind, "L": L, "shots": rng.randrange(16, 257),
            "p": round(rng.uniform(0.02, 0.07), 4)}


# ------------------------------------------------------------------ inputs

def _flips(shape, p, gen):
    """uint8 0 / 1 of the given shape, each 1 with probability p."""
    out = torch.empty(shape, dtype=torch.uint8, device="cuda")
    flat = out.view(-1)
    for a in range(0, flat.numel(), 1 << 26):
        part = flat[a:a + (1 << 26)]
        part.copy_(torch.rand(part.shape, generator=gen, device="cuda") < p)
    return out


def _noise(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return _flips((case["shots"], 2, case["L"], case["L"]), case["p"], gen)


def _anyons(N):
    """Parity of the four links incident to each site of the torus."""
    ex, ey = N[:, 0], N[:, 1]
    return ex ^ ex.roll(1, dims=2) ^ ey ^ ey.roll(1, dims=1)


def _sizes(case, seed):
    """Sizes of the batch's shots (the case's own) and their noise rates (the seed's)."""
    sizes, weights = zip(*(map(int, s.split(":")) for s in case["mix"].split(",")))
    w = np.array(weights, dtype=np.float64)
    L = np.random.default_rng(1000).choice(np.array(sizes, dtype=np.int32), size=case["shots"],
                                           p=w / w.sum())
    p = np.random.default_rng(seed).uniform(case["p_lo"], case["p_hi"], size=case["shots"]).astype(np.float32)
    return L.astype(np.int32), p


def _params(seed):
    """Flat weights and biases, uniform within 1 / sqrt(fan-in) times sqrt(3)."""
    rng = np.random.default_rng(seed)
    parts = []
    for co, ci in LAYERS:
        b = math.sqrt(3.0 / (9 * ci))
        parts += [rng.uniform(-b, b, co * ci * 9), rng.uniform(-0.1, 0.1, co)]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "ring":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s["errors"] = _flips((case["shots"], case["L"]), case["p"], gen)
    elif kind == "uneven":
        L, p = _sizes(case, seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        bits = torch.from_numpy(2 * L.astype(np.int64) ** 2).cuda()
        rate = torch.repeat_interleave(torch.from_numpy(p).cuda(), bits)
        s["errors"] = (torch.rand(rate.shape, generator=gen, device="cuda") < rate).to(torch.uint8)
        s["plan"] = qca.UnevenPlan(L)
    else:
        s["errors"] = _noise(case, seed)
    if kind == "syndrome":
        s["sigma"] = _anyons(s.pop("errors")).contiguous()
    if kind in ("logits", "gradients"):
        s["net"] = qca.Net(0)
        s["net"].set_params(_params(seed))
        if case.get("precision") == "fp8":
            s["net"].calibrate_fp8(s["errors"][:16].contiguous())
            s["net"].set_precision("fp8")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "decode":
        return qca.decode_batch(s["errors"], max_steps=case["max_steps"])
    if kind == "syndrome":
        return qca.decode_syndrome_batch(s["sigma"], max_steps=case["max_steps"], rng_seed=7,
                                         tie_order=case["tie_order"],
                                         balance_rule=case["balance_rule"])
    if kind == "uneven":
        return s["plan"].decode(s["errors"], max_steps=case["max_steps"])
    if kind == "ring":
        return qca.decode_1d_batch(s["errors"], max_steps=case["max_steps"], rng_seed=3,
                                   p_move=case["p_move"])
    if kind == "open":
        return qca.decode_open_batch(s["errors"], max_steps=case["max_steps"])
    if kind == "logits":
        return s["net"].logits(s["errors"])
    loss, grad = s["net"].gradients(s["errors"])
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------- work and exact values

def work(case):
    kind = case["kind"]
    n = case["shots"]
    if kind == "uneven":
        sites = float(np.sum(_sizes(case, 0)[0].astype(np.float64) ** 2))
    else:
        sites = n * case["L"] ** (1 if kind == "ring" else 2)
    forward = 2 * 9 * sum(co * ci for co, ci in LAYERS)  # per site
    if kind in ("decode", "open", "uneven"):   # links in, correction out, steps and flag
        return {"bytes": 4 * sites + 5 * n, "flops": 0}
    if kind == "syndrome":                     # anyons in, links out, steps, cuts, flag
        return {"bytes": 3 * sites + 7 * n, "flops": 0}
    if kind == "ring":
        return {"bytes": 2 * sites + 6 * n, "flops": 0}
    if kind == "logits":                       # links in, four fp32 logits out
        return {"bytes": 18 * sites, "flops": forward * sites}
    return {"bytes": 2 * sites + 4 * sum(9 * co * ci + co for co, ci in LAYERS),
            "flops": 3 * forward * sites}


def _weights64(seed):
    flat, out, o = torch.from_numpy(_params(seed)).double().cuda(), [], 0
    for co, ci in LAYERS:
        w = flat[o:o + 9 * co * ci].view(co, ci, 3, 3)
        o += 9 * co * ci
        out.append((w, flat[o:o + co]))
        o += co
    return flat, out


def _forward64(anyons, weights):
    x = torch.stack([anyons.double(), torch.ones_like(anyons, dtype=torch.float64)], dim=1)
    for i, (w, b) in enumerate(weights):
        x = F.conv2d(F.pad(x, (1, 1, 1, 1), mode="circular"), w, b)
        if i < len(weights) - 1:
            x = x.relu()
    return x


def _labels(a):
    """Class of each site: the direction (+x, -x, +y, -y) an anyon takes in the
    automaton's first step if its neighbour there moves back, else 4; 255
    where there is no anyon."""
    big = 9
    fields = []                                   # m^{+x}, m^{-x}, m^{+y}, m^{-y}
    for axis, sign in ((2, 1), (2, -1), (1, 1), (1, -1)):
        m = torch.full(a.shape, big, device=a.device)
        for d in (3, 2, 1):
            hit = torch.zeros_like(a)
            for j in range(-d, d + 1):
                hit |= a.roll((sign * d, j), dims=(axis, 3 - axis))
            m = torch.where(hit > 0, d, m)
        fields.append(m)
    px, mx, py, my = fields
    order = torch.stack([my, mx, px, py])         # ties go to the first
    first = order.argmin(dim=0)
    on_y = (first == 0) | (first == 3)
    up, um = torch.where(on_y, py, px), torch.where(on_y, my, mx)
    base = torch.where(on_y, 2, 0)
    # m^{+a} comes from the -a side: the anyon moves toward the smaller field
    move = torch.where(up < um, base + 1, torch.where(um < up, base, 4))
    move = torch.where((a > 0) & (order.amin(dim=0) < big), move, 4)
    label = torch.full(a.shape, 4, device=a.device)
    for k, (axis, step) in enumerate(((2, -1), (2, 1), (1, -1), (1, 1))):
        back = move.roll(step, dims=axis) == (k ^ 1)
        label = torch.where((move == k) & back, k, label)
    return torch.where(a > 0, label, 255)


def exact(case, seed):
    """Logits, loss and gradients in 64 bits; the decoders' outputs are whole numbers."""
    if case["kind"] == "logits":
        N = _noise(case, seed)
        _, weights = _weights64(seed)
        per = max(1, (1 << 20) // case["L"] ** 2)
        return torch.cat([_forward64(_anyons(part), weights) for part in N.split(per)])
    if case["kind"] == "gradients":
        a = _anyons(_noise(case, seed))
        flat, _ = _weights64(seed)
        flat.requires_grad_(True)
        weights, o = [], 0
        for co, ci in LAYERS:
            weights.append((flat[o:o + 9 * co * ci].view(co, ci, 3, 3),
                            flat[o + 9 * co * ci:o + 9 * co * ci + co]))
            o += 9 * co * ci + co
        z = _forward64(a, weights)
        z = torch.cat([z, torch.zeros_like(z[:, :1])], dim=1).permute(0, 2, 3, 1)
        label = _labels(a)
        on = label != 255
        loss = F.cross_entropy(z[on], label[on].long(), label_smoothing=SMOOTHING)
        loss.backward()
        return {"loss": float(loss.detach()), "grad": flat.grad}
    return None
