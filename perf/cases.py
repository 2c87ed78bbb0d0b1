"""Workloads on which the speed of this library is measured.

A case is one call pattern of a program that uses the library: a frame (or a batch of frames) of a given size, scale
and dictionary, the coefficients a network has just produced, and one pass through the public entry points.  `path`
says which pattern:

    dense     every atom, sr_dict_regress_dense
    lists     the s strongest atoms of every pixel as index and value planes (kept by the program), then the
              regression from them: sr_dict_select followed by sr_dict_regress_selected
    fused     the same selection made inside the regression call, nothing stored
    subset    one atom subset with re-weights for every pixel: the inference rule of a compressed model; `planes` is
              "all" when the network still emits every plane and "kept" when it emits only the subset's
    producer  the regression fused with the network's last layer (features instead of coefficients)
    upsample  the up-sampled frame alone
    gram      the statistics of the atom search over sampled (or all) pixels
    search    the atom search itself on given statistics

Frames are fp32 in [0, 1], coefficients 1/D + N(0, 0.05) as binary16 or fp32, atoms Gaussians and differences of
Gaussians of unit sum.  Video and tiled programs have widths that are multiples of eight; photographs and test sets
have any width.
"""
import math

import torch
import torch.nn.functional as nnf

import paper_2303_08999_b200 as sr

CIN = 32                      # channels of the feature map in front of the network's last layer


def _frame(name, path, n, h, w, r, D=72, k=5, coef="f16", out="f32", c=3, **more):
    case = dict(path=path, n=n, c=c, h=h, w=w, r=r, D=D, k=k, coef=coef, out=out, **more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # a 64 x 64 training-size patch x2 with fp32 coefficients: the smallest call, where latency counts
        _frame("patch_dense_f32", "dense", 1, 64, 64, 2, coef="f32"),
        # a 180 x 320 frame x3 from a network that runs in fp32
        _frame("sd_dense_f32", "dense", 1, 180, 320, 3, coef="f32"),
        # one 1080p frame x4: every atom
        _frame("hd_dense", "dense", 1, 270, 480, 4),
        # the same frame with per-pixel lists of eight atoms that the program keeps
        _frame("hd_lists", "lists", 1, 270, 480, 4, s=8),
        # the same frame under the compressed model's rule, eight of 72 atoms
        _frame("hd_subset", "subset", 1, 270, 480, 4, s=8, planes="all"),
        # the same frame straight from the features of the network
        _frame("hd_producer", "producer", 1, 270, 480, 4, kc=3),
        # the up-sampled 1080p frame alone (what the network's residual is added to, and the preview)
        _frame("hd_upsample", "upsample", 1, 270, 480, 4),
        # a photograph of an odd size x3, written as an 8-bit image
        _frame("photo_dense", "dense", 1, 213, 321, 3, out="u8"),
        # four frames of 4K video x2 per call, every atom
        _frame("uhd_dense", "dense", 4, 1080, 1920, 2),
        # four frames of 4K video x2 per call, eight atoms per pixel chosen in the call, 8-bit output
        _frame("uhd_fused", "fused", 4, 1080, 1920, 2, s=8, out="u8"),
        # statistics for compressing a model: 100 000 pixels sampled from a 1080p frame
        _frame("compress_gram", "gram", 1, 270, 480, 4, samples=100000),
        # the search for the eight atoms to keep of 72
        dict(name="compress_search", path="search", D=72, s=8, step=16),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


MOST_COEF_BYTES = 4 * 72 * 2160 * 3840 * 2          # the largest listed coefficient tensor


def draw(rng):
    path = rng.choices(["dense", "lists", "fused", "subset", "producer", "upsample", "gram", "search"], [4, 2, 2, 2, 2, 1, 2, 1])[0]
    if path == "search":
        D = rng.randint(16, 64)
        return dict(path="search", D=D, s=rng.randint(4, max(4, D // 4)), step=rng.randint(12, 24))
    r, k = rng.choice([2, 3, 4]), rng.choice([3, 5, 5, 7])
    D, s = rng.choice([16, 32, 48, 64, 72, 72, 96, 128]), rng.choice([4, 8, 8, 16])
    coef = "f32" if rng.random() < 0.25 else "f16"
    out = rng.choice(["f32", "f32", "f16", "u8"])
    c = 1 if rng.random() < 0.2 else 3
    photo = rng.random() < 0.5                     # any width, one frame, up to 4K; else video: multiples of eight
    size = _log(rng, 16384, 8294400 if photo or coef == "f32" else 33177600)        # HR pixels in all
    if path == "gram":
        size = min(size, 2073600)
    n = 1 if photo else rng.choice([1, 1, 2, 4])
    size = max(size, 16384 * n)
    if path not in ("producer", "upsample"):
        size = min(size, MOST_COEF_BYTES / (D * (4 if coef == "f32" else 2)))
    aspect = rng.uniform(0.7, 2.0)
    h = max(8, int(math.sqrt(size / (n * r * r * aspect))))
    w = max(8, int(h * aspect))
    if not photo:
        h, w = max(8, h // 8 * 8), max(8, w // 8 * 8)
    case = _frame(None, path, n, h, w, r, D=D, k=k, coef=coef, out=out, c=c)
    if path in ("lists", "fused", "subset"):
        case["s"] = s
    if path == "subset":
        case["planes"] = rng.choice(["all", "kept"])
    if path == "producer":
        case.update(k=rng.choice([3, 5]) if r == 3 else k, coef="f16", kc=rng.choice([1, 3]))
    if path == "upsample":
        case.update(coef="f32", out="f32", D=1, k=1)
    if path == "gram":
        case.update(out="f32", samples=0 if size < 300000 and rng.random() < 0.3 else int(_log(rng, 2000, 100000)))
    return case


# ---- inputs ---------------------------------------------------------------------------------------------------------


def _dictionary(D, k, g):
    """D atoms of k x k: anisotropic rotated Gaussians, then differences of Gaussians, each of unit sum."""
    def u():
        return torch.rand(D, generator=g, device="cuda", dtype=torch.float64)

    s1, s2, th = 0.3 + 1.7 * u(), 0.3 + 1.7 * u(), math.pi * u()
    p = (k - 1) // 2
    y, x = torch.meshgrid(*[torch.arange(-p, p + 1, device="cuda", dtype=torch.float64)] * 2, indexing="ij")
    y, x = y.reshape(1, -1), x.reshape(1, -1)
    a = torch.cos(th)[:, None] * x + torch.sin(th)[:, None] * y
    b = torch.cos(th)[:, None] * y - torch.sin(th)[:, None] * x

    def gauss(m):
        e = torch.exp(-0.5 * ((a / (m * s1)[:, None]) ** 2 + (b / (m * s2)[:, None]) ** 2))
        return e / e.sum(1, keepdim=True)

    one = torch.ones_like(s1)
    atoms = gauss(one)
    wide = 2.0 * gauss(1.6 * one) - atoms           # of unit sum as well
    atoms[(D + 1) // 2:] = wide[(D + 1) // 2:]
    return atoms.float().contiguous()


def _importance(D, g):
    """How much each atom of a trained model matters: a few carry most of the energy."""
    order = torch.randperm(D, generator=g, device="cuda")
    return torch.exp(-4.0 * order.double() / D)


def _flags(case):
    return sr.SR_CLAMP01 | {"f32": 0, "f16": sr.SR_OUT_F16, "u8": sr.SR_OUT_U8}[case["out"]]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["path"] == "search":
        return _prepare_search(case, g)
    n, c, h, w, r, D, k = (case[x] for x in ("n", "c", "h", "w", "r", "D", "k"))
    H, W, path = h * r, w * r, case["path"]
    st = dict(case=case, lr=torch.rand(n, c, h, w, generator=g, device="cuda"))
    if path == "upsample":
        return st
    st["flags"] = _flags(case)
    st["dict"] = _dictionary(D, k, g)
    if path == "producer":
        kc = case["kc"]
        st["feat"] = torch.randn(n, h, w, CIN, generator=g, device="cuda").mul_(0.25).add_(0.5).half()
        wconv = torch.randn(D * r * r, CIN, kc, kc, generator=g, device="cuda") * (0.05 / math.sqrt(CIN * kc * kc * 0.3125))
        bias = torch.randn(D * r * r, generator=g, device="cuda") * 0.005 + 1.0 / D
        st["folded"] = sr.sr_producer_fold(wconv, bias, st["dict"], r, k)      # once per network, as a program does
        return st
    planes = case["s"] if case.get("planes") == "kept" else D
    dtype = torch.float32 if case["coef"] == "f32" else torch.float16
    st["coef"] = torch.randn(n, planes, H, W, generator=g, device="cuda", dtype=dtype).mul_(0.05).add_(1.0 / D)
    if path == "subset":
        s = case["s"]
        st["idx"] = torch.randperm(D, generator=g, device="cuda")[:s].sort().values.to(torch.uint8)
        st["gamma"] = (torch.rand(s, generator=g, device="cuda") + 0.5) * (D / s)
        st["flags"] |= sr.SR_IDX_GLOBAL | (sr.SR_COEF_COMPACT if case["planes"] == "kept" else 0)
    if path == "gram":
        st["coef"].mul_(_importance(D, g).to(dtype).view(1, D, 1, 1))
        up = nnf.interpolate(st["lr"], scale_factor=r, mode="bicubic", align_corners=False)
        st["target"] = (up + 0.01 * torch.randn(n, c, H, W, generator=g, device="cuda")).contiguous()
        m = min(case["samples"], n * H * W)
        st["samples"] = torch.randperm(n * H * W, generator=g, device="cuda")[:m].sort().values if m else None
    return st


def _prepare_search(case, g):
    """Statistics of D atoms' responses on 12 000 rows, in fp64: smooth 5 x 5 patches under the atoms, weighted by
    coefficients whose size differs from atom to atom."""
    D, m = case["D"], 12000
    atoms = _dictionary(D, 5, g).double()
    noise = torch.randn(m, 1, 9, 9, generator=g, device="cuda", dtype=torch.float64)
    patch = 0.5 + nnf.avg_pool2d(noise, 5, stride=1).reshape(m, 25)
    phi = 1.0 / D + 0.05 * torch.randn(m, D, generator=g, device="cuda", dtype=torch.float64)
    Z = phi * _importance(D, g) * (patch @ atoms.T)
    t = Z.sum(1) + 0.01 * torch.randn(m, generator=g, device="cuda", dtype=torch.float64)
    # kept to fp32 values, so that the inputs do not depend on the order of the sums that made them
    G, b, hh = ((Z.T @ Z).float().double(), (Z.T @ t).float().double(), (t @ t).reshape(1).float().double())
    return dict(case=case, G=((G + G.T) / 2).contiguous(), b=b, hh=hh, rows=float(m))


# ---- one pass -------------------------------------------------------------------------------------------------------


def run(st):
    case = st["case"]
    path = case["path"]
    if path == "search":
        return sr.sr_selection_search(st["G"], st["b"], st["hh"], st["rows"], case["s"] / case["D"], case["step"] / case["D"], 0.0, 1e-9)
    r, k = case["r"], case["k"]
    if path == "upsample":
        return sr.sr_bicubic_upsample(st["lr"], r)
    if path == "producer":
        return sr.sr_producer_regress(st["lr"], st["feat"], st["folded"], r, k, case["D"], case["kc"], st["flags"])
    if path == "dense":
        return sr.sr_dict_regress_dense(st["lr"], st["coef"], st["dict"], r, k, st["flags"])
    if path == "lists":
        idx, sel = sr.sr_dict_select(st["coef"], case["s"], want_sel=True)
        out = sr.sr_dict_regress_selected(st["lr"], sel, idx, None, st["dict"], r, k, case["s"], st["flags"] | sr.SR_COEF_COMPACT)
        return out, idx, sel
    if path == "fused":
        return sr.sr_dict_regress_selected(st["lr"], st["coef"], None, None, st["dict"], r, k, case["s"], st["flags"])
    if path == "subset":
        return sr.sr_dict_regress_selected(st["lr"], st["coef"], st["idx"], st["gamma"], st["dict"], r, k, case["s"], st["flags"])
    return sr.sr_selection_gram(st["lr"], st["coef"], st["dict"], st["target"], st["samples"], r, k)


def work(case):
    path = case["path"]
    if path == "search":
        D = case["D"]          # the statistics once; at least one sweep of coordinate descent and one re-fit per step
        steps = math.ceil((D - case["s"]) / case["step"])
        return {"bytes": 8 * (D * D + D + 1) + 5 * case["s"], "flops": steps * (2 * D * D + D * D * D / 3)}
    n, c, h, w, r, D, k = (case[x] for x in ("n", "c", "h", "w", "r", "D", "k"))
    px, kk = n * h * w * r * r, k * k
    cb, ob = (4 if case["coef"] == "f32" else 2), {"f32": 4, "f16": 2, "u8": 1}[case["out"]]
    io = 4 * n * c * h * w + ob * c * px
    if path == "upsample":     # separable: four taps per LR row of every HR column, then four per HR pixel
        return {"bytes": io, "flops": 2 * 4 * c * (px + px // r)}
    io += 4 * D * kk
    up = 8 * c * (px + px // r)
    if path == "dense":
        return {"bytes": io + px * D * cb, "flops": 2 * px * kk * (D + c) + up}
    if path == "lists":
        s = case["s"]
        return {"bytes": io + px * (D * cb + s * (1 + cb)), "flops": 2 * px * kk * (s + c) + up}
    if path == "fused":
        return {"bytes": io + px * D * cb, "flops": 2 * px * kk * (case["s"] + c) + up}
    if path == "subset":
        return {"bytes": io + px * case["s"] * cb, "flops": 2 * px * kk * (case["s"] + c) + up}
    if path == "producer":
        K = CIN * case["kc"] ** 2
        return {"bytes": io + 2 * n * h * w * CIN + 2 * K * r * r * kk, "flops": 2 * px * kk * (K + 1 + c) + up}
    m = min(case["samples"], px) or px
    rows = m * c
    return {"bytes": 4 * n * c * h * w + m * (D * cb + 4 * c) + (8 * m if case["samples"] else 0) + 8 * (D * D + D + 1),
            "flops": 2 * rows * (D * kk + D * (D + 1) / 2 + D)}


def tolerance(case):
    """About four times what the paths differ from the same arithmetic in fp64: 1.5e-7 with fp32 results, 2e-4 once
    they are rounded to binary16, 1.5e-5 of all 8-bit codes; with folded weights (rounded to binary16) 3e-5, 1.8e-4 and
    3e-3.  Indices, copied coefficients and the atom search have one right answer."""
    path, out = case["path"], case.get("out")
    if path == "search":
        return "exact"
    if path == "producer":
        return {"f32": {"rel": 1.5e-4}, "f16": {"rel": 8e-4}, "u8": {"differ": 0.01}}[out]
    return {"f32": {"rel": 1e-6, "differ": 0.0}, "f16": {"rel": 8e-4, "differ": 0.0}, "u8": {"rel": 1e-6, "differ": 1e-4}}[out]
