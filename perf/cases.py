"""The work that users of this library have it do, as cases that can be timed and checked.

Each case is a call (or the few calls a program makes per pass) through the package's public entry
points: one pair for a preview, a recorded stream, a live camera loop, a batch of unrelated pairs, the
same from host memory, and the reverse mode of a training step.  Inputs are synthetic particle images of
the paper's kind (Gaussian particles of 2-3 px, 0.05-0.1 per pixel, a vortex plus a uniform shift),
rendered on the GPU from the seed alone; their integer accumulation makes them the same in every process.

`exact` restates the estimator in 64-bit torch without the package: the values the calls approximate.
"""
import math

import torch

import paper_2509_25924_gb300 as ofv
from paper_2509_25924_gb300.autograd import flow_fn

DEV = "cuda:0"

# Every case holds these; listed and drawn cases override some of them.
_BASE = dict(
    kind="pair",     # pair | stream | host | live | batch | grad
    H=1024, W=1024,
    n=2,             # frames of a stream, or pairs of a batch
    dtype="u16",     # u8 | u16 (12 bits) | f32
    store="f32",     # f32 | f16 | bf16: storage of the pyramid levels
    psl=2, kr=4, it=3, nr=0,
    ppp=0.08,        # particles per pixel
    peak=3.0,        # peak displacement of the vortex (px)
    warm=0,          # warm start of a stream from that many pairs back
    gauss=0.0,       # width of a Gaussian window (0: box)
    mask=False,      # a masked disk
    prefilter=False,
    derived=False,   # vorticity, recirculation area and probes of the fields too
    mix=0,           # batch: which sizes
)


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # Preview of a small pair, as a tool or a test harness computes it: launches and latency count.
        _case("pair_256_f32", H=256, W=256, dtype="f32", ppp=0.05),
        # One camera pair at the default parameters.
        _case("pair_1mp_u16"),
        # A cropped 8-bit pair at the paper's benchmark parameters (NR 2, KR 10); odd, ragged size.
        _case("pair_odd_u8_kr10", H=719, W=1283, dtype="u8", nr=2, kr=10, ppp=0.05),
        # The recorded 1 Mp time-resolved stream of the repository's benchmark, a part of it.
        _case("stream_1mp_u16", kind="stream", n=65),
        # The paper's own benchmark setting on a stream, with the quantities a monitoring display derives.
        _case("stream_1mp_u8_kr10", kind="stream", n=25, dtype="u8", nr=2, kr=10, ppp=0.05, derived=True),
        # A 4 Mp recording with 16-bit level storage.
        _case("stream_4mp_f16", kind="stream", H=2048, W=2048, n=9, store="f16", ppp=0.1),
        # Turbulence setting (small window, many iterations) on a warm-started time-resolved stream.
        _case("stream_1mp_kr2_warm", kind="stream", n=33, kr=2, nr=1, psl=1, it=4, warm=8, ppp=0.1, peak=2.0),
        # The live loop at the largest camera: one 21 Mp pair replayed as a CUDA graph.
        _case("live_21mp", kind="live", H=4096, W=5120, ppp=0.1, peak=4.0),
        # Unrelated pairs of unequal sizes in one persistent launch.
        _case("batch_32_uneven", kind="batch", n=32, mix=5, ppp=0.1, peak=2.0),
        # A recording in host memory, fields back to host memory (copies are part of the call).
        _case("host_1mp_u16", kind="host", n=25),
        # Reverse mode through autograd: a small training crop ...
        _case("grad_256_f32", kind="grad", H=256, W=256, dtype="f32", ppp=0.05),
        # ... and a full frame with the learnable 5x5 pre-filter and local normalization.
        _case("grad_1mp_prefilter", kind="grad", dtype="f32", nr=2, prefilter=True),
    ]


# Sizes of a batch's pairs: the benchmark's four classes, or odd crops.
_CLASSES = [(256, 256), (512, 512), (768, 1024), (1024, 1024)]


def _batch_sizes(c):
    g = torch.Generator().manual_seed(7919 + int(c["mix"]))
    out = []
    for _ in range(c["n"]):
        if c["mix"] % 2:
            out.append(_CLASSES[int(torch.randint(4, (1,), generator=g))])
        else:
            r = torch.rand(2, generator=g)
            out.append(tuple(int(math.exp(math.log(150) + float(x) * math.log(900 / 150))) for x in r))
    return out


def draw(rng):
    """One more case: kinds as listed, sizes over their logarithm, odd ones among them."""
    kind = rng.choice(["pair", "pair", "stream", "stream", "stream", "live", "batch", "host", "grad"])
    c = dict(_BASE, kind=kind)

    def size(lo, hi):
        s = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return s if rng.random() < 0.6 else (s + 15) // 16 * 16

    c["kr"] = rng.choice([2, 3, 4, 4, 5, 6, 8, 10])
    c["nr"] = rng.choice([0, 0, 1, 2, 3])
    c["psl"] = rng.choice([0, 1, 2, 2, 3])
    c["it"] = rng.choice([2, 3, 3, 4])
    c["dtype"] = rng.choice(["u8", "u16", "u16", "f32"])
    c["store"] = rng.choice(["f32", "f32", "f32", "f16", "bf16"])
    c["ppp"] = rng.choice([0.05, 0.08, 0.1])
    c["peak"] = round(rng.uniform(1.0, 2.0 if c["psl"] == 0 else 4.0), 2)
    if kind == "pair":
        c["H"], c["W"] = size(200, 3000), size(200, 3000)
        c["gauss"] = rng.choice([0.0, 0.0, 0.0, round(0.5 * c["kr"], 2)])
        c["mask"] = rng.random() < 0.15
    elif kind == "stream":
        c["H"], c["W"] = size(200, 1600), size(200, 1600)
        c["n"] = rng.randint(3, 26)
        c["warm"] = rng.choice([0, 0, 1, 4])
        c["derived"] = rng.random() < 0.3
    elif kind == "host":
        c["H"], c["W"] = size(200, 1100), size(200, 1100)
        c["n"] = rng.randint(3, 17)
    elif kind == "live":
        c["H"], c["W"] = size(400, 4000), size(400, 4000)
    elif kind == "batch":
        c["n"], c["mix"] = rng.randint(3, 24), rng.randint(0, 1000)
    else:
        c["H"], c["W"] = size(130, 900), size(130, 900)
        c["dtype"], c["store"] = "f32", "f32"
        c["prefilter"] = rng.random() < 0.5
        c["kr"] = max(3, c["kr"])  # a 5x5 window leaves gradients that 32-bit inputs do not determine
    if kind in ("batch",):
        c["psl"] = min(c["psl"], 2)
    return c


# --- inputs -------------------------------------------------------------------
def _field(c, H, W, x, y, g):
    """Displacement of a Rankine vortex at a seeded centre plus a seeded shift, at points (x, y)."""
    r = torch.rand(4, generator=g)
    cx, cy = W * (0.4 + 0.2 * float(r[0])), H * (0.4 + 0.2 * float(r[1]))
    R = max(16.0, 0.125 * min(H, W))
    sx, sy = 1.6 * float(r[2]) - 0.8, 1.6 * float(r[3]) - 0.8
    dx, dy = x - cx, y - cy
    rr = torch.sqrt(dx * dx + dy * dy).clamp_min(1e-6)
    ut = torch.where(rr < R, c["peak"] * rr / R, c["peak"] * R / rr)
    return -ut * dy / rr + sx, ut * dx / rr + sy


def _render(H, W, x, y, sig, amp, noise_gen, c):
    """Gaussian particles accumulated in integers (the order of the additions does not matter)."""
    acc = torch.zeros(H * W, dtype=torch.int32, device=x.device)
    xi, yi = torch.round(x), torch.round(y)
    inv = 0.5 / (sig * sig)
    for b in range(-3, 4):
        for a in range(-3, 4):
            px, py = xi + a, yi + b
            w = amp * torch.exp(-((px - x) ** 2 + (py - y) ** 2) * inv)
            ok = (px >= 0) & (px < W) & (py >= 0) & (py < H)
            idx = py.clamp(0, H - 1).long() * W + px.clamp(0, W - 1).long()
            acc.index_add_(0, idx, torch.where(ok, torch.round(w * (1 << 20)), torch.zeros_like(w)).int())
    img = (acc.float() * (1.0 / (1 << 20))).clamp_(0, 1)
    img = (img + 0.01 * torch.randn(H * W, generator=noise_gen, device=x.device)).clamp_(0, 1).view(H, W)
    if c["dtype"] == "u8":
        return torch.round(img * 255).to(torch.uint8)
    if c["dtype"] == "u16":
        return torch.round(img * 4095).to(torch.int16).view(torch.uint16)
    return img


def _frames(c, H, W, n, seed):
    """n consecutive frames: particles carried by the field, wrapped in a margin outside the view."""
    dev = DEV if torch.cuda.is_available() else "cpu"
    g = torch.Generator().manual_seed(seed)
    gd = torch.Generator(device=dev).manual_seed(seed + 1)
    m = 16.0
    np_ = int(c["ppp"] * (H + 2 * m) * (W + 2 * m))
    r = torch.rand(4, np_, generator=gd, device=dev, dtype=torch.float64)
    x, y = r[0] * (W + 2 * m) - m, r[1] * (H + 2 * m) - m
    sig = ((2.0 + r[2]) / 2.35482).float()
    amp = (0.5 + 0.5 * r[3]).float()
    out = []
    g0 = g.get_state()
    for f in range(n):
        out.append(_render(H, W, x.float(), y.float(), sig, amp, gd, c))
        g.set_state(g0)
        u, v = _field(c, H, W, x, y, g)
        x = torch.remainder(x + u + m, W + 2 * m) - m
        y = torch.remainder(y + v + m, H + 2 * m) - m
    return torch.stack(out)


def _params(c):
    return ofv.ofv_default_params(
        levels_psl=c["psl"], kernel_radius=c["kr"], iterations=c["it"], norm_radius=c["nr"],
        input={"u8": ofv.OFV_IN_U8, "u16": ofv.OFV_IN_U16, "f32": ofv.OFV_IN_F32}[c["dtype"]],
        bit_depth=8 if c["dtype"] == "u8" else 12,
        storage={"f32": ofv.OFV_STORE_F32, "f16": ofv.OFV_STORE_F16, "bf16": ofv.OFV_STORE_BF16}[c["store"]],
        prefilter=1 if c["prefilter"] else 0, warm_start=c["warm"],
        window=ofv.OFV_WINDOW_GAUSS if c["gauss"] else ofv.OFV_WINDOW_BOX, window_sigma=c["gauss"])


def _mask(c, H, W, dev):
    y = torch.arange(H, device=dev)[:, None] - 0.6 * H
    x = torch.arange(W, device=dev)[None, :] - 0.3 * W
    return (x * x + y * y >= (0.12 * min(H, W)) ** 2).to(torch.uint8)


def _weights(seed, dev):
    """A learnt 5x5 filter: near a small Gaussian blur."""
    k = torch.tensor([1.0, 4.0, 12.0, 4.0, 1.0], dtype=torch.float64)
    g = torch.Generator().manual_seed(seed + 3)
    w = torch.outer(k, k) / (k.sum() ** 2) + 0.004 * torch.randn(5, 5, generator=g, dtype=torch.float64)
    return w.float().to(dev)


def _loss_grads(seed, H, W, dev):
    g = torch.Generator(device=dev).manual_seed(seed + 4)
    return torch.randn(2, H, W, generator=g, device=dev)


def _probes(c, seed, dev):
    g = torch.Generator(device=dev).manual_seed(seed + 5)
    r = torch.rand(64, 2, generator=g, device=dev)
    return (r * torch.tensor([c["W"] - 1.0, c["H"] - 1.0], device=dev)).contiguous()


class _Graph:
    """A recorded graph and the handle it replays on, released together."""

    def __init__(self, flow, I1, I2, u, v):
        self.flow, self.keep = flow, (I1, I2, u, v)
        self.g = ofv.ofv_graph_create(flow.h, I1, I2, u, v)

    def __del__(self):
        try:
            ofv.ofv_graph_destroy(self.g)
        except Exception:
            pass


def prepare(case, seed):
    c, H, W = case, case["H"], case["W"]
    s = {"c": c}
    if c["kind"] == "batch":
        p = _params(c)
        s["pairs"] = []
        for k, (h, w) in enumerate(_batch_sizes(c)):
            f = _frames(c, h, w, 2, seed * 1000 + k)
            s["pairs"].append((f[0], f[1], torch.empty(h, w, device=DEV), torch.empty(h, w, device=DEV)))
        s["flow"] = ofv.Flow(256, 256, params=p)
        ofv.ofv_compute_batched(s["flow"].h, s["pairs"])  # a program tunes its layout once
        return s
    n = c["n"] if c["kind"] in ("stream", "host") else 2
    fr = _frames(c, H, W, n, seed)
    s["flow"] = ofv.Flow(H, W, params=_params(c))
    if c["mask"]:
        ofv.ofv_set_mask(s["flow"].h, _mask(c, H, W, DEV))
    if c["kind"] == "pair":
        s["I"] = (fr[0], fr[1])
    elif c["kind"] == "live":
        s["uv"] = torch.empty(2, H, W, device=DEV)
        s["I"] = (fr[0], fr[1])
        s["graph"] = _Graph(s["flow"], fr[0], fr[1], s["uv"][0], s["uv"][1])
    elif c["kind"] == "grad":
        s["I"] = (fr[0].clone().requires_grad_(True), fr[1].clone().requires_grad_(True))
        s["w"] = _weights(seed, DEV).requires_grad_(True) if c["prefilter"] else None
        s["g"] = _loss_grads(seed, H, W, DEV)
    elif c["kind"] == "host":
        s["frames"] = fr.cpu().pin_memory()
        s["uv"] = torch.empty(2, n - 1, H, W, pin_memory=True)
    else:
        s["frames"] = fr
        s["uv"] = torch.empty(2, n - 1, H, W, device=DEV)
        if c["derived"]:
            s["omega"] = torch.empty(n - 1, H, W, device=DEV)
            s["area"] = torch.empty(n - 1, dtype=torch.int64, device=DEV)
            s["xy"] = _probes(c, seed, DEV)
            s["ts"] = torch.empty(n - 1, 64, 2, device=DEV)
    return s


def run(state):
    s = state
    c = s["c"]
    H, W = c["H"], c["W"]
    if c["kind"] == "pair":
        return s["flow"](s["I"][0], s["I"][1])
    if c["kind"] == "live":
        ofv.ofv_graph_launch(s["graph"].g)
        return [s["uv"][0], s["uv"][1]]
    if c["kind"] == "batch":
        ofv.ofv_compute_batched(s["flow"].h, s["pairs"])
        # planar fields of all pairs, end to end (at most 64 outputs can be returned)
        return [torch.cat([p[k].view(-1) for p in s["pairs"]]) for k in (2, 3)]
    if c["kind"] == "grad":
        I1, I2 = s["I"]
        u, v = flow_fn(s["flow"], I1, I2, s["w"])
        wrt = [I1, I2] + ([s["w"]] if s["w"] is not None else [])
        return [u.detach(), v.detach(), *torch.autograd.grad([u, v], wrt, [s["g"][0], s["g"][1]])]
    fr, u, v = s["frames"], s["uv"][0], s["uv"][1]
    fn = ofv.ofv_compute_sequence_host if c["kind"] == "host" else ofv.ofv_compute_sequence
    fn(s["flow"].h, c["n"], fr, H * W * fr.element_size(), u, v, H * W)
    out = [u, v]
    if c["derived"]:
        m = c["n"] - 1
        ofv.ofv_vorticity(H, W, m, u, v, H * W, s["omega"])
        ofv.ofv_recirculation_area(H, W, m, u, H * W, None, s["area"])
        ofv.ofv_probe(H, W, m, u, v, H * W, 64, s["xy"], s["ts"])
        out += [s["omega"], s["area"].double(), s["ts"]]  # the area as a number: pixels at u = 0 may tie
    return out


def work(case):
    c = case
    ib = {"u8": 1, "u16": 2, "f32": 4}[c["dtype"]]
    sizes = _batch_sizes(c) if c["kind"] == "batch" else [(c["H"], c["W"])]
    seq = c["kind"] in ("stream", "host")
    frames, fields = (c["n"], c["n"] - 1) if seq else (2, 1)
    N = float(sum(h * w for h, w in sizes))
    levels = sum(0.25 ** l for l in range(c["psl"] + 1))
    # per pixel and iteration: two bilinear samples with gradients (48), their combination and the five
    # products (16), ten running window sums (20), the solve (16)
    flops = 100.0 * N * fields * levels * c["it"]
    nbytes = N * (frames * ib + fields * 8.0)
    if c["derived"]:
        nbytes += N * fields * 4.0
    if c["kind"] == "grad":
        flops *= 4.0  # forward, and its adjoint at about three times the operations
        nbytes += N * (8.0 + 8.0)  # dL/du, dL/dv in, dL/dI1, dL/dI2 out
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the difference seen between a pass and `exact` over the listed and drawn cases.

    32-bit storage: 1e-7 in the 2-norm at KR >= 3 and 9e-7 at KR 2, whose small windows leave single pixels
    nearly singular (3e-4 of the rms); vorticity subtracts neighbours (8e-6, 9e-4).  16-bit storage rounds
    the images themselves (f16 9e-5, bf16 4e-4).  Gradients: 2e-6 for the frames and 5e-5 for the pre-filter
    weights, sums of a million terms; a sample that lies on a cell boundary to the last bit may take the
    slope of either cell, which moves single pixels."""
    if case["kind"] == "grad":
        return {"rel": 2e-4, "max": 0.05}
    if case["store"] == "bf16":
        return {"rel": 2e-3, "max": 0.02}
    if case["store"] == "f16":
        return {"rel": 4e-4, "max": 4e-3}
    if case["derived"]:
        return {"rel": 4e-5, "max": 4e-3}
    return {"rel": 4e-6, "max": 2e-3}


# --- the same values in 64 bits, without the package ----------------------------
def _shift(P, a, b):
    """P(i+a, j+b), clamp-to-edge."""
    H, W = P.shape
    i = (torch.arange(H, device=P.device) + a).clamp(0, H - 1)
    j = (torch.arange(W, device=P.device) + b).clamp(0, W - 1)
    return P[i][:, j]


def _window(P, wts):
    """Truncated separable window sum, weights wts (2 r + 1 of them) along both axes."""
    r = (len(wts) - 1) // 2
    for dim in (0, 1):
        pad = torch.zeros_like(P.narrow(dim, 0, r)) if P.shape[dim] >= r else None
        Q = torch.cat([pad, P, pad], dim)
        P = sum(w * Q.narrow(dim, k, P.shape[dim]) for k, w in enumerate(wts))
    return P


def _sample(planes, px, py):
    """Bilinear samples of the planes at (px, py), clamp-to-edge taps."""
    H, W = planes[0].shape
    x0, y0 = torch.floor(px.detach()), torch.floor(py.detach())
    fx, fy = px - x0, py - y0
    x0, y0 = x0.clamp(-2, W + 1).long(), y0.clamp(-2, H + 1).long()
    xa, xb = x0.clamp(0, W - 1), (x0 + 1).clamp(0, W - 1)
    ya, yb = y0.clamp(0, H - 1) * W, (y0 + 1).clamp(0, H - 1) * W
    out = []
    for P in planes:
        f = P.reshape(-1)
        out.append((1 - fy) * ((1 - fx) * f[ya + xa] + fx * f[ya + xb]) + fy * ((1 - fx) * f[yb + xa] + fx * f[yb + xb]))
    return out


def _ingest(c, raw, w25):
    full = {"u8": 255.0, "u16": 4095.0, "f32": 1.0}[c["dtype"]]
    P = (raw.view(torch.int16) if raw.dtype == torch.uint16 else raw).double() / full
    if c["nr"]:
        one = [1.0] * (2 * c["nr"] + 1)
        n = _window(torch.ones_like(P), one)
        mu = _window(P, one) / n
        # centred at a constant first: the box variance then cancels nothing that matters in 64 bits
        Z = P - 0.25
        var = (_window(Z * Z, one) / n - (_window(Z, one) / n) ** 2).clamp_min(0)
        P = (P - mu) / torch.sqrt(var + float(torch.tensor(1e-2, dtype=torch.float32)) ** 2)
    if w25 is not None:
        P = sum(w25[a, b] * _shift(P, a - 2, b - 2) for a in range(5) for b in range(5))
    return P


def _pyramid(P, psl):
    k = [1 / 16, 4 / 16, 6 / 16, 4 / 16, 1 / 16]
    out = [P]
    for _ in range(psl):
        P = sum(w * _shift(P, a - 2, 0) for a, w in enumerate(k))[::2]
        P = sum(w * _shift(P, 0, b - 2) for b, w in enumerate(k))[:, ::2]
        out.append(P)
    return out


def _flow64(c, A, B, start=None, mask=None):
    """Gauss-Newton iterations of the symmetric SSD, coarse to fine, of two pyramids."""
    r = c["kr"]
    wts = [math.exp(-(d * d) / (2 * c["gauss"] ** 2)) if c["gauss"] else 1.0 for d in range(-r, r + 1)]
    u = v = None
    for l in range(c["psl"], -1, -1):
        P1, P2 = A[l], B[l]
        H, W = P1.shape
        y = torch.arange(H, device=P1.device, dtype=torch.float64)[:, None].expand(H, W)
        x = torch.arange(W, device=P1.device, dtype=torch.float64)[None, :].expand(H, W)
        f = 1 << l
        if u is not None:
            u, v = (2 * t for t in _sample([u, v], 0.5 * x, 0.5 * y))
        elif start is not None:
            u, v = start[0][::f, ::f] / f, start[1][::f, ::f] / f
        else:
            u = v = torch.zeros_like(P1)
        pl1, pl2 = ([P, 0.5 * (_shift(P, 0, 1) - _shift(P, 0, -1)), 0.5 * (_shift(P, 1, 0) - _shift(P, -1, 0))] for P in (P1, P2))
        keepers = None if mask is None else mask[::f, ::f].double()
        for _ in range(c["it"]):
            a, ax, ay = _sample(pl1, x - 0.5 * u, y - 0.5 * v)
            b, bx, by = _sample(pl2, x + 0.5 * u, y + 0.5 * v)
            gx, gy = 0.5 * (ax + bx), 0.5 * (ay + by)
            res = gx * u + gy * v - (b - a)
            q = [gx * gx, gx * gy, gy * gy, gx * res, gy * res]
            if keepers is not None:
                q = [keepers * t for t in q]
            sxx, sxy, syy, sxr, syr = (_window(t, wts) for t in q)
            tr, det = sxx + syy, sxx * syy - sxy * sxy
            keep = ~(tr > 1e-20) | (det <= 1e-6 * tr * tr)
            det = torch.where(keep, torch.ones_like(det), det)
            un, vn = (syy * sxr - sxy * syr) / det, (sxx * syr - sxy * sxr) / det
            u, v = torch.where(keep, u, un), torch.where(keep, v, vn)
    return u, v


def exact(case, seed):
    c, H, W = case, case["H"], case["W"]
    dev = DEV if torch.cuda.is_available() else "cpu"
    if c["kind"] == "batch":
        us, vs = [], []
        for k, (h, w) in enumerate(_batch_sizes(c)):
            f = _frames(c, h, w, 2, seed * 1000 + k)
            u, v = _flow64(c, *(_pyramid(_ingest(c, t, None), c["psl"]) for t in f))
            us.append(u.reshape(-1))
            vs.append(v.reshape(-1))
        return [torch.cat(us), torch.cat(vs)]
    n = c["n"] if c["kind"] in ("stream", "host") else 2
    fr = _frames(c, H, W, n, seed)
    if c["kind"] == "grad":
        w = _weights(seed, dev).double().requires_grad_(True) if c["prefilter"] else None
        I = [fr[k].double().requires_grad_(True) for k in (0, 1)]
        u, v = _flow64(c, *(_pyramid(_ingest(c, t, w), c["psl"]) for t in I))
        g = _loss_grads(seed, H, W, dev).double()
        return [u.detach(), v.detach(), *torch.autograd.grad([u, v], I + ([w] if w is not None else []), [g[0], g[1]])]
    mask = _mask(c, H, W, dev) if c["mask"] else None
    us, vs = [], []
    prev = _pyramid(_ingest(c, fr[0], None), c["psl"])
    for k in range(n - 1):
        cur = _pyramid(_ingest(c, fr[k + 1], None), c["psl"])
        start = (us[k - c["warm"]], vs[k - c["warm"]]) if c["warm"] and k >= c["warm"] else None
        u, v = _flow64(c, prev, cur, start, mask)
        if mask is not None:
            u, v = (torch.where(mask != 0, t, torch.full_like(t, math.nan)) for t in (u, v))
        us.append(u)
        vs.append(v)
        prev = cur
    if c["kind"] in ("pair", "live"):
        return [us[0], vs[0]]
    u, v = torch.stack(us), torch.stack(vs)
    out = [u.cpu(), v.cpu()] if c["kind"] == "host" else [u, v]
    if c["derived"]:
        dvdx, dudy = torch.gradient(v, dim=2)[0], torch.gradient(u, dim=1)[0]
        xy = _probes(c, seed, dev).double()
        ts = [torch.stack(_sample([u[k], v[k]], xy[:, 0], xy[:, 1]), 1) for k in range(n - 1)]
        out += [dvdx - dudy, (u < 0).sum((1, 2)).double(), torch.stack(ts)]
    return out
