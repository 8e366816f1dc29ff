"""The work a user of the codec has it do, as measurable cases.

Every case goes through the public entry points of
``paper_1306_1373_gb300.dctgb`` (and ``rc`` for the seeded initial weights)
on seeded synthetic images: 1/f^beta noise with step edges, rounded to uint8.
A case is a dict of plain values; ``kind`` names the call:

  graph        one fused or two-pass batch graph over a grey plane and a
               4:2:0 frame, launch shape autotuned (the fast path of a
               program that codes the same buffers again and again)
  batch        one graph over many grey images of uneven sizes and qualities
  compress     direct dct_compress of one grey plane or 4:2:0 frame
  reconstruct  direct dct_reconstruct with the SSE against the original
  fused        direct dct_codec_fused (codes, reconstruction and SSE)
  rgb          dct_compress_rgb of an interleaved RGB frame
  exact        dct_exact_fused, the float32 exact-DCT pipeline
  entropy      dct_entropy_stats of a frame's codes (rate of the result)
  rate         dct_rate_control of a mixed 4:2:0 stream with a trained network
  train        one epoch of the rate controller's network
"""
import math

import numpy as np
import torch

from paper_1306_1373_gb300 import dctgb as D
from paper_1306_1373_gb300 import rc

DEV = "cuda"
STREAM_SIZES = ((1280, 720), (1920, 1080), (3840, 2160))


def listed():
    return [
        # The throughput case: one 8192 x 8192 grey scan and one 4K 4:2:0
        # frame at quality 75, codes + reconstruction + PSNR in one fused
        # graph replay (the repository's own benchmark workload).
        {"name": "graph_8k_4k420", "kind": "graph", "grey": 8192, "width": 3840, "height": 2160, "quality": 75,
         "two_pass": False},
        # A photo collection: 512 grey images, sides 64..2048 in multiples
        # of 8, quality 10..95, one graph launch.  The largest case.
        {"name": "batch_512_uneven", "kind": "batch", "n": 512, "lo": 64, "hi": 2048},
        # Separate forward and inverse kernels, as a program runs them that
        # keeps the paper's two-kernel structure: 4096 x 4096 + 4K 4:2:0.
        {"name": "twopass_4k_4k420", "kind": "graph", "grey": 4096, "width": 3840, "height": 2160, "quality": 75,
         "two_pass": True},
        # An encoder: one 4K 4:2:0 video frame to codes.
        {"name": "compress_4k420", "kind": "compress", "width": 3840, "height": 2160, "yuv": True, "quality": 75,
         "pad": 0, "stats": False},
        # A decoder with quality control: the same frame back, with its SSE,
        # at a high quality setting.
        {"name": "reconstruct_4k420", "kind": "reconstruct", "width": 3840, "height": 2160, "yuv": True,
         "quality": 90, "pad": 0},
        # The smallest everyday call: one 512 x 512 grey image at quality 50,
        # where launches and latency count.
        {"name": "fused_512", "kind": "fused", "width": 512, "height": 512, "yuv": False, "quality": 50, "pad": 0},
        # A photograph of arbitrary size as a file decoder hands it over:
        # tight rows of odd length, so no row but the first is aligned.
        {"name": "fused_ragged_2731x1823", "kind": "fused", "width": 2731, "height": 1823, "yuv": False,
         "quality": 85, "pad": 0},
        # A camera frame: 1080p interleaved RGB straight to 4:2:0 codes.
        {"name": "rgb_1080p", "kind": "rgb", "width": 1920, "height": 1080, "quality": 75, "pad": 0},
        # The exact-DCT pipeline beside the Cordic one (the paper's quality
        # comparison), on its largest image size.
        {"name": "exact_3072", "kind": "exact", "width": 3072, "height": 3072, "yuv": False, "quality": 75, "pad": 0},
        # Rate of a coded 4K frame: symbol statistics of its codes.
        {"name": "entropy_4k420", "kind": "entropy", "width": 3840, "height": 2160, "yuv": True, "quality": 75},
        # Rate control of a mixed 720p / 1080p / 2160p stream: learned
        # prediction, verification, bisection of the frames that miss.
        {"name": "rate_stream48", "kind": "rate", "frames": 48},
        # Training the controller: one epoch over 16,000 frames' features.
        {"name": "train_16000", "kind": "train", "n": 16000, "batch": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls, sizes spread over their logarithm, odd
    widths and padded pitches among them, qualities over the whole range."""
    kind = rng.choice(["graph", "graph", "batch", "batch", "compress", "compress", "reconstruct", "reconstruct",
                       "fused", "fused", "rgb", "exact", "entropy", "rate", "train"])
    quality = rng.randint(10, 98)
    if kind == "graph":
        w = _log_int(rng, 640, 3840)
        return {"kind": kind, "grey": _log_int(rng, 256, 8192), "width": w, "height": max(2, w * 9 // 16),
                "quality": quality, "two_pass": rng.random() < 0.4}
    if kind == "batch":
        return {"kind": kind, "n": _log_int(rng, 8, 384), "lo": 64, "hi": rng.choice([512, 1024, 2048])}
    if kind == "rate":
        return {"kind": kind, "frames": _log_int(rng, 6, 48)}
    if kind == "train":
        return {"kind": kind, "n": _log_int(rng, 600, 16000), "batch": rng.choice([64, 128, 256, 500])}
    w = _log_int(rng, 200, 4096)
    h = max(8, int(w * rng.uniform(0.5, 1.1)))
    if rng.random() < 0.5:      # sizes of screens and sensors; the others stay as drawn, odd ones among them
        w, h = (w + 7) // 8 * 8, (h + 7) // 8 * 8
    case = {"kind": kind, "width": w, "height": h, "quality": quality}
    if kind != "rgb":
        case["yuv"] = rng.random() < 0.5
    if kind != "entropy":
        case["pad"] = rng.choice([0, 0, 0, 5, 24])
    if kind == "compress":
        case["stats"] = rng.random() < 0.3
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + 12345) & ((1 << 62) - 1))
    return g


def _field(h, w, beta, g, std=40.0):
    """1/f^beta noise (power ~ f^-beta) of mean 128, float32."""
    spec = torch.fft.rfft2(torch.randn(h, w, generator=g, device=DEV))
    fy = torch.fft.fftfreq(h, device=DEV).view(-1, 1)
    fx = torch.fft.rfftfreq(w, device=DEV).view(1, -1)
    f = torch.sqrt(fx * fx + fy * fy)
    f[0, 0] = 1.0
    amp = f.pow(-beta / 2.0)
    amp[0, 0] = 0.0
    x = torch.fft.irfft2(spec * amp, s=(h, w))
    return 128.0 + std * (x / x.std().clamp_min(1e-12))


def _edges(img, rng, k):
    """Adds k half-plane steps of 20..80 levels."""
    h, w = img.shape
    yy = torch.arange(h, device=DEV, dtype=torch.float32).view(-1, 1)
    xx = torch.arange(w, device=DEV, dtype=torch.float32).view(1, -1)
    for _ in range(k):
        ang, x0, y0 = rng.uniform(0, 2 * math.pi), rng.uniform(0, w), rng.uniform(0, h)
        amp = rng.uniform(20.0, 80.0) * (1 if rng.random() < 0.5 else -1)
        img = img + amp * ((math.cos(ang) * (xx - x0) + math.sin(ang) * (yy - y0)) > 0)
    return img


def _u8(x, pad=0):
    """Rounded uint8 plane whose rows are `pad` bytes longer than its width."""
    h, w = x.shape
    out = torch.empty(h, w + pad, dtype=torch.uint8, device=DEV)[:, :w]
    out.copy_(x.round_().clamp_(0, 255))
    return out


def _rng(seed):
    return np.random.Generator(np.random.PCG64(int(seed) & 0xFFFFFFFF))


def _grey(h, w, seed, beta=2.0, pad=0):
    g, rng = _gen(seed), _rng(seed)
    return _u8(_edges(_field(h, w, beta, g), rng, int(rng.integers(2, 7))), pad)


def _frame(w, h, seed, beta=2.0, pad=0):
    """(Y, Cb, Cr) planes of a 4:2:0 frame; chroma is smoother."""
    g = _gen(3 * seed + 1)
    ch, cw = (h + 1) // 2, (w + 1) // 2
    return [_grey(h, w, 3 * seed, beta, pad)] + [_u8(_field(ch, cw, beta + 0.5, g, 16.0), pad) for _ in range(2)]


def _planes(case, seed):
    if case["yuv"]:
        return _frame(case["width"], case["height"], seed, pad=case.get("pad", 0))
    return [_grey(case["height"], case["width"], seed, pad=case.get("pad", 0))]


def _like(planes):
    out = []
    for p in planes:
        buf = torch.zeros(p.shape[0], p.stride(0), dtype=torch.uint8, device=DEV)
        out.append(buf[:, :p.shape[1]])
    return out


def _codes(planes):
    return torch.zeros(D.coeff_count([tuple(p.shape) for p in planes]), dtype=torch.int16, device=DEV)


def _plan(case, planes, max_batch=0):
    return D.Plan(max(p.shape[1] for p in planes), max(p.shape[0] for p in planes),
                  layout=D.DCT_LAYOUT_YUV420 if case.get("yuv") else D.DCT_LAYOUT_GRAY8, max_batch=max_batch)


def _batch_sizes(case, seed):
    """(width, height, quality, beta index) of every image of a batch: the
    sizes belong to the case, so that its work does not depend on the seed."""
    rng = np.random.Generator(np.random.PCG64(2 + case["n"] * 7919 + case["hi"]))
    ws = rng.integers(case["lo"] // 8, case["hi"] // 8 + 1, size=case["n"]) * 8
    hs = rng.integers(case["lo"] // 8, case["hi"] // 8 + 1, size=case["n"]) * 8
    qs = rng.integers(10, 96, size=case["n"])
    return [(int(w), int(h), int(q), int(i) % 8) for i, (w, h, q) in enumerate(zip(ws, hs, qs))]


def _stream_sizes(frames):
    rng = np.random.Generator(np.random.PCG64(4 + frames))
    return [STREAM_SIZES[int(k)] for k in rng.integers(0, 3, size=frames)]


def _rolled(field, h, w, rng):
    """A random window of a periodic field."""
    H, W = field.shape
    return torch.roll(field, (int(rng.integers(H)), int(rng.integers(W))), (0, 1))[:h, :w].contiguous()


def _stream(sizes, seed):
    """4:2:0 frames cut from periodic fields of beta 1..3, with edges."""
    g, rng = _gen(seed), _rng(seed + 77)
    fields = [_field(2160, 3840, b, g) for b in (1.0, 1.5, 2.0, 2.5, 3.0)]
    planes = []
    for w, h in sizes:
        k = int(rng.integers(len(fields)))
        planes.append(_u8(_edges(_rolled(fields[k], h, w, rng), rng, int(rng.integers(2, 7)))))
        for _ in range(2):
            planes.append(_u8((_rolled(fields[min(k + 1, 4)], h // 2, w // 2, rng) - 128.0) * 0.4 + 128.0))
    return planes


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _graph(planes, qualities, chroma, ops, autotune):
    n = len(planes)
    sizes = [D.coeff_count([tuple(p.shape)]) for p in planes]
    codes = torch.zeros(sum(sizes), dtype=torch.int16, device=DEV)
    recon = torch.zeros(sum(p.numel() for p in planes), dtype=torch.uint8, device=DEV)
    sse = torch.zeros(n, dtype=torch.int64, device=DEV)
    offs = np.cumsum([0] + [p.numel() for p in planes])
    recs = [recon[offs[i]:offs[i + 1]].view(p.shape) for i, p in enumerate(planes)]
    plan = D.Plan(max(p.shape[1] for p in planes), max(p.shape[0] for p in planes), max_batch=n)
    items = D.make_batch_items(planes, qualities, coeffs=list(codes.split(sizes)), recons=recs, chroma=chroma)
    D.dct_batch_prepare(plan, items, ops, sse=sse)
    if autotune:
        D.dct_autotune(plan)
    return {"plan": plan, "out": {"codes": codes, "recon": recon, "sse": sse}}


def prepare(case, seed):
    kind = case["kind"]
    all_ops = D.DCT_OP_COMPRESS | D.DCT_OP_RECONSTRUCT | D.DCT_OP_SSE
    if kind == "graph":
        planes = [_grey(case["grey"], case["grey"], seed)] + _frame(case["width"], case["height"], seed + 1)
        ops = all_ops | (D.DCT_OP_TWO_PASS if case["two_pass"] else 0)
        st = _graph(planes, [case["quality"]] * 4, [0, 0, 1, 1], ops, autotune=True)
    elif kind == "batch":
        g, rng = _gen(seed), _rng(seed + 5)
        fields = [_field(case["hi"], case["hi"], 1.0 + 2.0 * i / 7, g) for i in range(8)]
        sizes = _batch_sizes(case, seed)
        planes = [_u8(_edges(_rolled(fields[b], h, w, rng), rng, 2)) for w, h, _, b in sizes]
        st = _graph(planes, [q for _, _, q, _ in sizes], None, all_ops, autotune=False)
    elif kind in ("compress", "reconstruct", "fused", "exact"):
        planes = _planes(case, seed)
        plan = _plan(case, planes)
        st = {"plan": plan, "planes": D.PlaneArray(planes), "codes": _codes(planes),
              "sse": torch.zeros(len(planes), dtype=torch.int64, device=DEV)}
        if kind == "compress" and case["stats"]:
            st["stats"] = torch.zeros(len(planes), D.STATS_WORDS, dtype=torch.int64, device=DEV)
        if kind != "compress":
            recon = _like(planes)
            st["recon"] = D.PlaneArray(recon)
            st["recon_list"] = recon
        if kind == "reconstruct":
            D.dct_compress(plan, planes, case["quality"], coeffs=st["codes"])
    elif kind == "rgb":
        w, h = case["width"], case["height"]
        buf = torch.zeros(h, 3 * w + case["pad"], dtype=torch.uint8, device=DEV)
        rgb = torch.as_strided(buf, (h, w, 3), (3 * w + case["pad"], 3, 1))
        luma = _grey(h, w, seed).float()
        g = _gen(seed + 9)
        for c in range(3):
            rgb[:, :, c] = (luma + _field(h, w, 2.5, g, 24.0) - 128.0).round_().clamp_(0, 255).to(torch.uint8)
        st = {"plan": D.Plan(w, h, layout=D.DCT_LAYOUT_YUV420), "rgb": rgb,
              "codes": torch.zeros(D.rgb_coeff_count(h, w), dtype=torch.int16, device=DEV)}
    elif kind == "entropy":
        planes = _planes(case, seed)
        plan = _plan(case, planes)
        st = {"plan": plan, "codes": D.dct_compress(plan, planes, case["quality"]),
              "shapes": [tuple(p.shape) for p in planes]}
    elif kind == "rate":
        rng = _rng(seed + 31)
        sizes = _stream_sizes(case["frames"])
        planes = D.PlaneArray(_stream(sizes, seed))
        # the network: trained on other, 720p, frames with four targets each
        base = _stream([STREAM_SIZES[0]] * 48, 1000 + seed)
        train = [p for i in range(4) for p in base]
        plan = D.Plan(3840, 2160, layout=D.DCT_LAYOUT_YUV420, max_batch=max(len(planes), len(train)))
        targets = [float(t) for t in rng.uniform(30.0, 40.0, size=len(train) // 3)]
        train = D.PlaneArray(train)
        qual, _ = rc.label_by_bisection(plan, train, 3, targets)
        feats = D.dct_rate_features(plan, train, 3, targets)
        net, _ = rc.train_network(feats, qual, epochs=200, batch=64, seed=seed)
        st = {"plan": plan, "planes": planes, "net": net,
              "targets": [float(t) for t in rng.uniform(30.0, 40.0, size=case["frames"])]}
    elif kind == "train":
        feats, labels, order, params = _train_inputs(case, seed)
        net = D.Mlp(params, act_bf16=True, device=DEV)
        net.set_norm(feats)
        net.workspace(case["batch"])
        st = {"net": net, "feats": feats, "labels": labels, "order": order}
    else:
        raise ValueError(kind)
    st["case"] = case
    return st


def _train_inputs(case, seed):
    """Features, labels in 0..1, the epoch's order and initial weights."""
    n = case["n"]
    g, rng = _gen(seed), _rng(seed + 3)
    mix = torch.randn(12, D.DCT_MLP_INPUTS, generator=g, device=DEV)
    z = torch.randn(n, 12, generator=g, device=DEV)
    feats = 4.0 + z @ mix + 0.1 * torch.randn(n, D.DCT_MLP_INPUTS, generator=g, device=DEV)
    feats[:, -1] = 1.0
    labels = torch.sigmoid(z[:, 0] - 0.5 * z[:, 1] + 0.2 * z[:, 2] * z[:, 3])
    order = torch.as_tensor(rng.permutation(n).astype(np.int32)).to(DEV)
    return feats.contiguous(), labels.contiguous(), order, rc.init_params(seed & 0xFFFF)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("graph", "batch"):
        D.dct_batch_launch(state["plan"])
        return state["out"]
    if kind == "compress":
        D.dct_compress(state["plan"], state["planes"], case["quality"], coeffs=state["codes"], stats=state.get("stats"))
        return [state["codes"]] + ([state["stats"]] if "stats" in state else [])
    if kind == "reconstruct":
        D.dct_reconstruct(state["plan"], state["codes"], state["recon"], case["quality"], ref_planes=state["planes"],
                          sse=state["sse"])
        return state["recon_list"] + [state["sse"]]
    if kind in ("fused", "exact"):
        call = D.dct_codec_fused if kind == "fused" else D.dct_exact_fused
        call(state["plan"], state["planes"], case["quality"], coeffs=state["codes"], recon_planes=state["recon"],
             sse=state["sse"])
        return [state["codes"]] + state["recon_list"] + [state["sse"]]
    if kind == "rgb":
        return D.dct_compress_rgb(state["plan"], state["rgb"], case["quality"], coeffs=state["codes"])
    if kind == "entropy":
        return D.dct_entropy_stats(state["plan"], state["codes"], state["shapes"])
    if kind == "rate":
        r = D.dct_rate_control(state["plan"], state["planes"], 3, state["targets"], net=state["net"])
        return {"quality": r["quality"], "sse": r["sse"].astype(np.int64), "fell_back": r["fell_back"]}
    net = state["net"]
    losses = net.train_epoch(state["feats"], state["labels"], state["order"], batch=case["batch"], lr=2e-3)
    return {"losses": losses, "params": net.params, "m": net.m, "v": net.v}


# ---------------------------------------------------------------------------
# work and exact results
# ---------------------------------------------------------------------------

def _samples(case):
    """(samples, codes) of a case's planes."""
    kind = case["kind"]
    if kind == "batch":
        n = sum(w * h for w, h, _, _ in _batch_sizes(case, 0))
        return n, n
    shapes = []
    if kind == "graph":
        shapes.append((case["grey"], case["grey"]))
    if kind == "rate":
        for w, h in _stream_sizes(case["frames"]):
            shapes += [(h, w), (h // 2, w // 2), (h // 2, w // 2)]
    else:
        w, h = case["width"], case["height"]
        shapes.append((h, w))
        if kind in ("graph", "rgb") or case.get("yuv"):
            shapes += [((h + 1) // 2, (w + 1) // 2)] * 2
    return sum(h * w for h, w in shapes), D.coeff_count(shapes)


def work(case):
    """Bytes: each input read once and each output written once.  Operations
    per sample, of the arithmetic the definition asks for: 27 integer ones
    forward and 4 to quantise, 27 and 8 back, 2 for the SSE."""
    kind = case["kind"]
    if kind == "train":
        n, b = case["n"], case["batch"]
        steps = -(-n // b)
        params = D.DCT_MLP_PARAMS
        return {"bytes": n * (D.DCT_MLP_INPUTS + 2) * 4 + steps * 4 + 6 * params * 4, "flops": 6.0 * n * params}
    s, c = _samples(case)
    if kind in ("graph", "batch", "fused"):
        two = 2 * c if case.get("two_pass") else 0        # the inverse kernel of a two-pass graph reads the codes back
        return {"bytes": s * 2 + 2 * c + two, "flops": 61.0 * s}
    if kind == "exact":
        return {"bytes": s * 2 + 2 * c, "flops": 66.0 * s}
    if kind in ("compress", "rgb"):
        src = 3 * case["width"] * case["height"] if kind == "rgb" else s
        return {"bytes": src + 2 * c, "flops": 31.0 * s}
    if kind == "reconstruct":
        return {"bytes": 2 * s + 2 * c, "flops": 37.0 * s}
    if kind == "entropy":
        return {"bytes": 2 * c, "flops": 2.0 * c}
    # a frame's samples are read for its statistics and at least once more
    # to check the prediction
    return {"bytes": 2 * s, "flops": 61.0 * s}


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def exact(case, seed):
    """The training epoch in float64 (activations rounded to bfloat16, as the
    network is defined); the other cases return integers."""
    if case["kind"] != "train":
        return None
    feats, labels, order, params = _train_inputs(case, seed)
    x_all = feats.double()
    mean, std = x_all.mean(0), x_all.std(0, unbiased=False)
    std = torch.where(std < 1e-6, torch.ones_like(std), std)
    x_all, labels, order = (x_all - mean) / std, labels.double(), order.long()
    p = torch.as_tensor(params).to(DEV).double()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    n_in, hid = D.DCT_MLP_INPUTS, D.DCT_MLP_HIDDEN
    cuts = np.cumsum([hid * n_in, hid, hid * hid, hid, hid]).tolist()

    def gelu(a):
        return 0.5 * a * (1.0 + torch.erf(a / math.sqrt(2.0)))

    def gelu_grad(a):
        return 0.5 * (1.0 + torch.erf(a / math.sqrt(2.0))) + a * torch.exp(-0.5 * a * a) / math.sqrt(2.0 * math.pi)

    losses = []
    for t, b0 in enumerate(range(0, case["n"], case["batch"]), 1):
        idx = order[b0:b0 + case["batch"]]
        x, y_t = x_all[idx], labels[idx]
        w1, b1, w2, b2, w3 = (p[a:b] for a, b in zip([0] + cuts[:-1], cuts))
        w1, w2, b3 = w1.view(hid, n_in), w2.view(hid, hid), p[cuts[-1]:]
        a1 = x @ w1.t() + b1
        h1 = _bf16(gelu(a1))
        a2 = h1 @ w2.t() + b2
        h2 = _bf16(gelu(a2))
        y = torch.sigmoid(h2 @ w3 + b3)
        losses.append(((y - y_t) ** 2).mean())
        dz = 2.0 * (y - y_t) / len(idx) * y * (1.0 - y)
        d2 = dz[:, None] * w3 * gelu_grad(a2)
        d1 = (d2 @ w2) * gelu_grad(a1)
        g = torch.cat([(d1.t() @ x).reshape(-1), d1.sum(0), (d2.t() @ h1).reshape(-1), d2.sum(0), h2.t() @ dz,
                       dz.sum().reshape(1)])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - 2e-3 * (m / (1.0 - 0.9 ** t)) / ((v / (1.0 - 0.999 ** t)).sqrt() + 1e-8)
    return {"losses": torch.stack(losses), "params": p, "m": m, "v": v}
