"""Representative workloads of the CMIF library: what its users run, with inputs, an FP64 reference and tolerances.

Every case goes through the Python entry points (``Plan``, ``VolumePlan``, ``Batch``).  A case is a dict:

kind        "map" (one pair, translation only), "rotation" (Alg. 1 over a set of angles), "batch" (uneven pairs, four
            angles each), "volume" (label volumes) or "weighted" (spatially weighted MI)
precision   "fp32", "split32", "fp64" or "auto" (the plan's transform arithmetic)
h, w, ...   sizes: h x w of A, hb x wb of B (equal unless given), d of volumes; ka, kb labels
mask        "ones" (none passed), "holes" (rectangular holes in both masks) or "disc" (a disc mask on B)
"""
import math

import numpy as np
import torch

import paper_2106_14699_gb300 as cm

PRECISIONS = {"fp32": cm.FP32, "split32": cm.SPLIT32, "fp64": cm.FP64, "auto": cm.AUTO}
DEVICE = "cuda"


def _map(name, h, w, ka, kb, precision="fp32", mask="ones", noise=0.1, **more):
    return dict(name=name, kind="map", h=h, w=w, hb=more.pop("hb", h), wb=more.pop("wb", w), ka=ka, kb=kb,
                precision=precision, mask=mask, noise=noise, nmi=more.pop("nmi", False),
                background=more.pop("background", 0.0), **more)


def listed():
    return [
        # the smallest call: a 64 x 64 patch, where launches and latency are all there is
        _map("map-64-k8", 64, 64, 8, 8, mask="disc", noise=0.05),
        # the same patch in FP64, the plan for guaranteed counts at any size
        _map("map-64-k8-fp64", 64, 64, 8, 8, "fp64", mask="disc", noise=0.05),
        # an ordinary registration of two 256 x 256 images with holes in their masks
        _map("map-256-k16-holes", 256, 256, 16, 16, mask="holes"),
        # the headline: one full map of two 1024 x 1024 images, 16 labels each
        _map("map-1024-k16", 1024, 1024, 16, 16),
        # unequal, odd sizes and label counts, normalised MI, a width beyond the 2048-point rows
        _map("map-331x1203-k5x24-nmi", 331, 1203, 5, 24, mask="holes", nmi=True),
        # slide-sized images with 32 labels, precision chosen per pair: the largest single map
        _map("map-834-k32-auto", 834, 834, 32, 32, "auto"),
        # a stained section: more than half of both images is one background label, so that pair needs the
        # second precision
        _map("map-900x1000-k8-background-auto", 900, 1000, 8, 8, "auto", background=0.6),
        # Alg. 1 as the paper runs it on 300 x 300 images: 50 angles, padded search window
        dict(name="rotation-300-k8-window", kind="rotation", h=300, w=300, ka=8, kb=8, precision="fp32", angles=50,
             window=True, mask="ones", noise=0.05),
        # a rotation search at 512 x 512 with 16 labels over the full shift range
        dict(name="rotation-512-k16", kind="rotation", h=512, w=512, ka=16, kb=16, precision="fp32", angles=12,
             window=False, mask="ones", noise=0.0),
        # many uneven pairs per request, each with its own angles and label counts
        dict(name="batch-8-uneven", kind="batch", pairs=8, side_lo=96, side_hi=768, angles=4, precision="fp32",
             layout=7),
        # two label volumes
        dict(name="volume-40x56x64-k8", kind="volume", d=40, h=56, w=64, ka=8, kb=8, precision="fp32", noise=0.1),
        # spatially weighted MI of two 256 x 256 images
        dict(name="weighted-200x256-k12", kind="weighted", h=200, w=256, ka=12, kb=12, precision="fp64", noise=0.1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "rotation", "rotation", "batch", "volume", "weighted"])
    if kind == "map":
        precision = rng.choice(["fp32", "fp32", "fp32", "auto", "split32", "fp64"])
        top = {"fp32": 1300, "auto": 1000, "split32": 300, "fp64": 256}[precision]
        h, w = _log_int(rng, 40, top), _log_int(rng, 40, top)
        # label counts: any up to 512 pixels wide; the customary multiples of 4 above
        ks = list(range(2, 17)) if w <= 512 else [4, 8, 12, 16, 24] + ([32] if precision == "auto" else [])
        case = _map(None, h, w, rng.choice(ks), rng.choice(ks), precision,
                    mask=rng.choice(["ones", "holes", "disc"]), nmi=rng.random() < 0.2)
        if rng.random() < 0.3:  # a template smaller than the image it is sought in
            case["hb"], case["wb"] = max(24, int(h * rng.uniform(0.3, 1.0))), max(24, int(w * rng.uniform(0.3, 1.0)))
        del case["name"]
        return case
    if kind == "rotation":
        k = rng.choice([4, 8, 11, 16])
        return dict(kind="rotation", h=_log_int(rng, 64, 512), w=_log_int(rng, 64, 512), ka=k, kb=k, precision="fp32",
                    angles=rng.randint(3, 12), window=rng.random() < 0.5, mask=rng.choice(["ones", "holes"]),
                    noise=0.05)
    if kind == "batch":
        return dict(kind="batch", pairs=rng.randint(2, 6), side_lo=96, side_hi=_log_int(rng, 200, 768), angles=4,
                    precision="fp32", layout=rng.randrange(1 << 20))
    if kind == "volume":
        return dict(kind="volume", d=rng.randint(3, 40), h=_log_int(rng, 16, 64), w=_log_int(rng, 16, 72),
                    ka=rng.randint(2, 8), kb=rng.randint(2, 8), precision="fp32", noise=0.1)
    return dict(kind="weighted", h=_log_int(rng, 40, 256), w=_log_int(rng, 40, 256), ka=rng.randint(2, 12),
                kb=rng.randint(2, 12), precision="fp64", noise=0.1)


# ---- inputs -------------------------------------------------------------------------------------------------------
# Quantised images are piecewise constant: Voronoi label fields, B the same scene relabelled, rotated, shifted and
# with label noise (the shapes and proportions of the library's own synthetic workloads).

def _field(rng, extent, n_cells):
    return np.stack([rng.uniform(0, e, n_cells) for e in extent], axis=1)


def _nearest(seeds, points):
    """Index of the nearest seed of every point (both float32 on the device), in pieces of at most 2^26 distances."""
    step = max(1, (1 << 26) // len(seeds))
    return torch.cat([torch.cdist(p, seeds, compute_mode="donot_use_mm_for_euclid_dist").argmin(1)
                      for p in points.split(step)])


def _grid(shape):
    axes = [torch.arange(n, device=DEVICE, dtype=torch.float32) for n in shape]
    return torch.stack(torch.meshgrid(*axes, indexing="ij"), dim=-1).reshape(-1, len(shape))


def _planted(rng, shape_a, shape_b, ka, kb, noise, angle=0.0, background=0.0):
    """Label images (or volumes) of one scene; rotating B by `angle` about its centre and shifting it lands it on A."""
    cells = max(20, int(np.prod(shape_a)) // 500)
    seeds = _field(rng, shape_a, cells)
    la = rng.integers(0, ka, cells)
    lb = rng.permutation(ka)[la] if ka == kb else rng.integers(0, kb, cells)
    if background:  # cells outside the tissue carry label 0 in both images
        bg = rng.random(cells) < background
        la, lb = np.where(bg, 0, la), np.where(bg, 0, lb)
    shift = np.array([rng.integers(-max(1, n // 8), max(1, n // 8) + 1) for n in shape_b], np.float64)
    sd = torch.tensor(seeds, dtype=torch.float32, device=DEVICE)
    la_d, lb_d = (torch.tensor(v, dtype=torch.int32, device=DEVICE) for v in (la, lb))
    a = la_d[_nearest(sd, _grid(shape_a))].reshape(shape_a).contiguous()
    pts = _grid(shape_b)
    if len(shape_b) == 2 and angle:
        cr, cc = (shape_b[0] - 1) / 2.0, (shape_b[1] - 1) / 2.0
        v, u = pts[:, 0] - cr, pts[:, 1] - cc
        pts = torch.stack([cr - u * math.sin(angle) + v * math.cos(angle),
                           cc + u * math.cos(angle) + v * math.sin(angle)], dim=-1)
    pts = pts - torch.tensor(shift, dtype=torch.float32, device=DEVICE)
    b = lb_d[_nearest(sd, pts)].reshape(shape_b).contiguous()
    if noise:
        hit = torch.tensor(rng.random(shape_b) < noise, device=DEVICE)
        b = torch.where(hit, torch.tensor(rng.integers(0, kb, shape_b), dtype=torch.int32, device=DEVICE), b)
    return a, b.contiguous()


def _holes(rng, h, w):
    m = np.ones((h, w), np.uint8)
    for _ in range(5):
        area, aspect = rng.uniform(0.02, 0.05) * h * w, rng.uniform(0.5, 2.0)
        hh = max(1, min(h, int(round(math.sqrt(area * aspect)))))
        ww = max(1, min(w, int(round(area / hh))))
        y, x = int(rng.integers(0, h - hh + 1)), int(rng.integers(0, w - ww + 1))
        m[y:y + hh, x:x + ww] = 0
    return torch.tensor(m, device=DEVICE)


def _disc(h, w):
    y, x = np.meshgrid(np.arange(h) - (h - 1) / 2.0, np.arange(w) - (w - 1) / 2.0, indexing="ij")
    return torch.tensor((y * y + x * x <= (0.44 * min(h, w)) ** 2).astype(np.uint8), device=DEVICE)


def _masks(rng, kind, ha, wa, hb, wb):
    if kind == "holes":
        return _holes(rng, ha, wa), _holes(rng, hb, wb)
    return None, _disc(hb, wb) if kind == "disc" else None


def _batch_layout(case):
    """Sizes and label counts of the pairs: part of the case, not of the seed."""
    rng = np.random.default_rng(case["layout"])
    lo, hi = math.log(case["side_lo"]), math.log(case["side_hi"])
    return [dict(h=int(round(math.exp(rng.uniform(lo, hi)))), w=int(round(math.exp(rng.uniform(lo, hi)))),
                 ka=int(rng.choice([8, 16, 24])), kb=int(rng.choice([8, 16, 24]))) for _ in range(case["pairs"])]


def _inputs(case, seed):
    """The tensors and host values of a case, by name (what both prepare and exact start from)."""
    rng = np.random.default_rng([seed, 2106])
    kind = case["kind"]
    if kind == "map":
        a, b = _planted(rng, (case["h"], case["w"]), (case["hb"], case["wb"]), case["ka"], case["kb"], case["noise"],
                        background=case["background"])
        ma, mb = _masks(rng, case["mask"], case["h"], case["w"], case["hb"], case["wb"])
        return dict(a=a, ma=ma, b=b, mb=mb)
    if kind == "rotation":
        shape = (case["h"], case["w"])
        step = 2 * math.pi / case["angles"]
        angles = step * np.arange(case["angles"]) + rng.uniform(0.1, 0.9) * step
        a, b = _planted(rng, shape, shape, case["ka"], case["kb"], case["noise"], angle=float(angles[1]))
        ma, mb = _masks(rng, case["mask"], *shape, *shape)
        return dict(a=a, ma=ma, b=b, mb=mb, angles=angles)
    if kind == "batch":
        pairs = []
        for p in _batch_layout(case):
            shape = (p["h"], p["w"])
            theta = rng.uniform(0.1, 6.1, case["angles"])
            a, b = _planted(rng, shape, shape, p["ka"], p["kb"], 0.1, angle=float(theta[0]))
            ma, mb = _masks(rng, "holes", *shape, *shape)
            pairs.append(dict(A=a, M_A=ma, B=b, M_B=mb, K_A=p["ka"], K_B=p["kb"], angles=theta, gamma=0.5))
        return dict(pairs=pairs)
    if kind == "volume":
        shape = (case["d"], case["h"], case["w"])
        a, b = _planted(rng, shape, shape, case["ka"], case["kb"], case["noise"])
        return dict(a=a, b=b)
    shape = (case["h"], case["w"])
    a, b = _planted(rng, shape, shape, case["ka"], case["kb"], case["noise"])
    # positive weights: where the weighted overlap is 0 the transforms' rounding errors would decide MI
    wa, wb = (torch.tensor(rng.uniform(0.05, 1.0, shape), device=DEVICE) for _ in range(2))
    return dict(a=a, wa=wa, b=b, wb=wb)


# ---- the library's side -------------------------------------------------------------------------------------------

def prepare(case, seed):
    s = _inputs(case, seed)
    s["kind"] = kind = case["kind"]
    f64 = dict(dtype=torch.float64, device=DEVICE)
    i32 = dict(dtype=torch.int32, device=DEVICE)
    prec = PRECISIONS[case["precision"]]
    if kind == "batch":
        s["plan"] = cm.Batch(s["pairs"], prec, graph=True, batch_angles=True)
        s["records"] = torch.zeros(24 * len(s["pairs"]), dtype=torch.uint8, device=DEVICE)
        s["status"] = torch.zeros(len(s["pairs"]), **i32)
        return s
    if kind == "volume":
        n = (case["d"], case["h"], case["w"])
        s["plan"] = cm.VolumePlan(*n, *n, case["ka"], case["kb"], prec, graph=True)
    else:
        s["plan"] = cm.Plan(case["h"], case["w"], case.get("hb", case["h"]), case.get("wb", case["w"]), case["ka"],
                            case["kb"], prec, graph=True, window=case.get("window", False),
                            nmi=case.get("nmi", False), weighted=kind == "weighted", batch_angles=kind == "rotation")
    maps = (case["angles"],) if kind == "rotation" else ()
    shape = maps + (s["plan"].R, s["plan"].C)
    s["mi"] = torch.zeros(shape, **f64)
    s["n"] = torch.zeros(shape, **(f64 if kind == "weighted" else i32))
    s["records"] = torch.zeros(24 * (min(3, case["angles"]) if kind == "rotation" else 1), dtype=torch.uint8,
                               device=DEVICE)
    return s


def _records(buf):
    """cmif_peak records as (angle index, dy, dx, n) and MI, without a copy to the host."""
    r = buf.view(-1, 24)
    return r[:, :16].contiguous().view(torch.int32), r[:, 16:].contiguous().view(torch.float64)


def run(state):
    plan, kind = state["plan"], state["kind"]
    if kind == "batch":
        plan.run(state["records"], state["status"])
        whole, mi = _records(state["records"])
        return {"peaks": whole, "peak_mi": mi, "status": state["status"]}
    mi, n, rec = state["mi"], state["n"], state["records"]
    if kind == "rotation":
        plan.align_rotations(state["a"], state["ma"], state["b"], state["mb"], state["angles"], 0.5, rec.numel() // 24,
                             rec, mi_maps=mi, n_maps=n)
    elif kind == "weighted":
        plan.compute_weighted(state["a"], state["wa"], state["b"], state["wb"], mi, n, 0.5, rec)
    else:
        plan.compute(state["a"], state.get("ma"), state["b"], state.get("mb"), mi, n, None, 0.5, rec)
    whole, best = _records(rec)
    return {"mi": mi, "n": n, "peaks": whole, "peak_mi": best}


# ---- work and tolerances ------------------------------------------------------------------------------------------

def _one(shape_a, shape_b, ka, kb, units=1):
    """Bytes and operations of one pair at `units` angles: images in, MI and N out; the level sets' transforms, a
    product and an inverse transform per label pair at 2.5 n log2 n (real data, n shifts), ten operations per count."""
    n = math.prod(x + y - 1 for x, y in zip(shape_a, shape_b))
    fft = 2.5 * n * math.log2(n)
    return (5 * (math.prod(shape_a) + math.prod(shape_b)) + 12 * n * units,
            fft * (ka + units * (kb + ka * kb)) + 10 * n * units * ka * kb)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_one((p["h"], p["w"]), (p["h"], p["w"]), p["ka"], p["kb"], case["angles"]) for p in _batch_layout(case)]
        # the maps stay inside the call: records out
        return {"bytes": sum(10 * p["h"] * p["w"] + 28 for p in _batch_layout(case)), "flops": sum(e[1] for e in each)}
    shape = ((case["d"],) if kind == "volume" else ()) + (case["h"], case["w"])
    other = (case["hb"], case["wb"]) if kind == "map" else shape
    b, f = _one(shape, other, case["ka"], case["kb"], case.get("angles", 1))
    if kind == "weighted":
        b += 7 * 2 * math.prod(shape) + 4 * math.prod(2 * x - 1 for x in shape)
    return {"bytes": b, "flops": f}


def tolerance(case):
    # N and the peaks are exact.  MI: the counts are exact, c log2 c has 23 fraction bits (about 3e-7 absolute); maps
    # of weights are FP64 sums throughout.
    if case["kind"] == "weighted":
        return {"rel": 1e-9, "max": 1e-6}
    return {"rel": 4e-6, "max": 4e-5}


# ---- the same in 64 bits, without the library ---------------------------------------------------------------------

def _fast_len(n):
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def _xlogx(c):
    return torch.where(c > 0, c * torch.log2(c.clamp_min(1e-300)), torch.zeros_like(c))


def _exact_map(a, wa, b, wb, ka, kb, nmi=False, whole=True):
    """MI (or NMI) and N at every shift, FP64: correlations of the level sets, rounded where the weights are 0/1."""
    dims = tuple(range(1, a.dim() + 1))
    out = tuple(x + y - 1 for x, y in zip(a.shape, b.shape))
    size = tuple(_fast_len(n) for n in out)

    def spectra(x, w, k):
        w = torch.ones_like(x, dtype=torch.float64) if w is None else w.to(torch.float64)
        return torch.stack([torch.fft.rfftn(torch.where(x == i, w, torch.zeros_like(w)), s=size) for i in range(k)])

    fa, fb = spectra(a, wa, ka), spectra(b, wb, kb)
    joint = torch.zeros(out, dtype=torch.float64, device=a.device)
    marg, n = torch.zeros_like(joint), torch.zeros_like(joint)
    cb = torch.zeros((kb,) + out, dtype=torch.float64, device=a.device)
    for i in range(ka):
        ca = torch.zeros_like(joint)
        for lo in range(0, kb, 4):
            c = torch.fft.irfftn(fa[i].conj() * fb[lo:lo + 4], s=size, dim=dims)
            for d, x in zip(dims, a.shape):  # shifts from -(x - 1)
                c = torch.roll(c, x - 1, d)
            c = c[(slice(None),) + tuple(slice(0, o) for o in out)]
            c = torch.round(c) if whole else c.clamp_min(0.0)
            joint += _xlogx(c).sum(0)
            ca += c.sum(0)
            cb[lo:lo + 4] += c
        marg += _xlogx(ca)
        n += ca
    for i in range(kb):
        marg += _xlogx(cb[i])
    tn = _xlogx(n)
    if nmi:
        den = tn - joint
        mi = torch.where((n > 0) & (den > 1e-9), (2 * tn - marg) / den.clamp_min(1e-9), torch.zeros_like(n))
    else:
        mi = torch.where(n > 0, (joint - marg + tn) / n.clamp_min(1e-300), torch.zeros_like(n))
    flat = (-1, out[-1])
    return mi.reshape(flat), n.reshape(flat)


def _rotated(b, mb, theta):
    h, w = b.shape
    v = torch.arange(h, dtype=torch.float64, device=b.device)[:, None] - 0.5 * (h - 1)
    u = torch.arange(w, dtype=torch.float64, device=b.device)[None, :] - 0.5 * (w - 1)
    x = torch.floor(0.5 * (w - 1) + u * math.cos(theta) - v * math.sin(theta) + 0.5).long()
    y = torch.floor(0.5 * (h - 1) + u * math.sin(theta) + v * math.cos(theta) + 0.5).long()
    inside = (x >= 0) & (x < w) & (y >= 0) & (y < h)
    x, y = x.clamp(0, w - 1), y.clamp(0, h - 1)
    if mb is not None:
        inside &= mb[y, x] != 0
    return torch.where(inside, b[y, x], torch.zeros_like(b)), inside.to(torch.uint8)


def _window(case):
    h, w = case["h"], case["w"]
    py, px = math.ceil(h * 0.5), math.ceil(w * 0.5)
    return max(0, h - 1 - py), min(2 * h - 1, h + py), max(0, w - 1 - px), min(2 * w - 1, w + px)


def _best(mi, n, r0, r1, c0, c1):
    gate = n[r0:r1, c0:c1] >= 0.5 * n[r0:r1, c0:c1].max()
    return torch.where(gate, mi[r0:r1, c0:c1], torch.full_like(mi[r0:r1, c0:c1], -math.inf)).max()


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        best = []
        for p in s["pairs"]:
            per = []
            for t in p["angles"]:
                br, mr = _rotated(p["B"], p["M_B"], float(t))
                mi, n = _exact_map(p["A"], p["M_A"], br, mr, p["K_A"], p["K_B"])
                per.append(_best(mi, n, 0, mi.shape[0], 0, mi.shape[1]))
            best.append(torch.stack(per).max())
        return {"peaks": None, "peak_mi": torch.stack(best)[:, None], "status": None}
    if kind == "rotation":
        maps, ns, best = [], [], []
        r0, r1, c0, c1 = _window(case) if case["window"] else (0, 2 * case["h"] - 1, 0, 2 * case["w"] - 1)
        for t in s["angles"]:
            br, mr = _rotated(s["b"], s["mb"], float(t))
            mi, n = _exact_map(s["a"], s["ma"], br, mr, case["ka"], case["kb"])
            best.append(_best(mi, n, r0, r1, c0, c1))
            mi[:r0], mi[r1:], n[:r0], n[r1:] = 0, 0, 0, 0  # rows outside the window are returned as 0
            maps.append(mi)
            ns.append(n)
        top = torch.stack(best).sort(descending=True).values[:min(3, case["angles"]), None]
        return {"mi": torch.stack(maps), "n": torch.stack(ns).to(torch.int32), "peaks": None, "peak_mi": top}
    if kind == "weighted":
        mi, n = _exact_map(s["a"], s["wa"], s["b"], s["wb"], case["ka"], case["kb"], whole=False)
    else:
        mi, n = _exact_map(s["a"], s.get("ma"), s["b"], s.get("mb"), case["ka"], case["kb"], case.get("nmi", False))
    best = _best(mi, n, 0, mi.shape[0], 0, mi.shape[1])
    n = n if kind == "weighted" else n.to(torch.int32)
    return {"mi": mi, "n": n, "peaks": None, "peak_mi": best.reshape(1, 1)}
