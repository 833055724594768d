"""What this library is measured on: calls of its public entry points as a user's program makes
them, with inputs made on the GPU from a seed (the tissue-like blob fields, noise fields and
seed images of paper_1605_00930_gb300/synth.py, drawn with torch's generator instead of
numpy's so that large inputs take milliseconds).

listed() names the cases, draw() gives further ones of the same ranges, prepare() / run() do
one call, work() is what a call cannot do without (every input read once, every result
written once), exact() an independent evaluation in 64 bits. In-place calls overwrite their
marker, so run() first copies the initial marker back, as a program that makes a new marker
for every image would write it.
"""
import math
import random

import torch
import torch.nn.functional as F

from paper_1605_00930_gb300 import iwpp, learned

DEV = "cuda"


def listed():
    return [
        # a small field of view, one call at a time: launches and latency
        dict(name="recon_u8_512", kind="recon", field="noise", H=512, W=512, blobs=0, u16=False, conn=8, op="dilate",
             marker="dome", h=40),
        # the ordinary call: one whole 4096 x 4096 tissue image, h-dome marker
        dict(name="recon_u8_4096", kind="recon", field="blobs", H=4096, W=4096, blobs=2000, u16=False, conn=8,
             op="dilate", marker="dome", h=30),
        # a cropped image of odd width, 4-connectivity
        dict(name="recon_u8_c4_odd", kind="recon", field="blobs", H=2777, W=3001, blobs=993, u16=False, conn=4,
             op="dilate", marker="dome", h=30),
        # fill-holes of a 16-bit image: reconstruction by erosion, values travel from the border inwards
        dict(name="fill_u16_4096", kind="recon", field="blobs", H=4096, W=4096, blobs=2000, u16=True, conn=8,
             op="erode", marker="border", h=0),
        # a whole slide with sparse seeds: the largest single image, long paths
        dict(name="seeds_u8_16384", kind="recon", field="blobs", H=16384, W=16384, blobs=2000, u16=False, conn=8,
             op="dilate", marker="seeds", h=1000),
        # an uneven batch (u8 and u16, half h-dome dilations, half fill-holes) in one call
        dict(name="batch_48", kind="batch", n=48, layout=4, conn=8, min_side=256, max_side=4096, learned=False),
        # the larger batch, with the learned schedule made inside the call
        dict(name="batch_256_learned", kind="batch", n=256, layout=5, conn=8, min_side=256, max_side=4096,
             learned=True),
        # an operator built on the reconstruction: h-maxima of a 16-bit image of odd sides
        dict(name="hmax_u16_odd", kind="hmax", H=1999, W=2501, blobs=596, u16=True, conn=8, h=20 * 257),
        # distance transform of a segmentation (tissue field above 60), with squared distances
        dict(name="edt_4096", kind="edt", H=4096, W=4096, blobs=2000, conn=8),
        # marker-controlled watershed of a 16-bit gradient image, labels and levels
        dict(name="watershed_u16_2048", kind="watershed", H=2048, W=2048, blobs=500, markers=500, u16=True, conn=8),
        # influence zones in a porous domain, with distances and label pairs
        dict(name="skiz_4096", kind="skiz", H=4096, W=4096, blobs=2000, markers=2000, conn=8),
        # an image in pinned host memory, band by band (out of core)
        dict(name="host_bands_8192", kind="host", H=8192, W=8192, blobs=1000, u16=False, conn=8, op="dilate",
             marker="seeds", h=500, band_rows=1024),
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["recon", "recon", "recon", "recon", "batch", "batch", "hmax", "edt", "watershed", "skiz",
                       "host"])
    conn = rng.choice([4, 8])
    u16 = rng.random() < 0.5
    if kind == "batch":
        return dict(kind=kind, n=rng.randrange(2, 97), layout=rng.randrange(1 << 20), conn=conn,
                    min_side=_side(rng, 64, 512), max_side=_side(rng, 1024, 4096), learned=rng.random() < 0.5)
    big = 4096 if kind in ("recon", "hmax", "edt") else 2560
    H, W = _side(rng, 200, big), _side(rng, 200, big)
    if rng.random() < 0.3:   # sides that are whole tiles are as common as odd ones
        H, W = max(64, H // 64 * 64), max(64, W // 64 * 64)
    blobs = max(1, int(2000 * H * W * rng.uniform(0.1, 1.0) / 4096 ** 2))
    if kind == "hmax":
        return dict(kind=kind, H=H, W=W, blobs=blobs, u16=u16, conn=conn, h=rng.randrange(10, 61) * (257 if u16 else 1))
    if kind == "edt":
        return dict(kind=kind, H=H, W=W, blobs=blobs, conn=conn)
    if kind in ("watershed", "skiz"):
        case = dict(kind=kind, H=H, W=W, blobs=blobs, markers=max(2, H * W // rng.randrange(4000, 40000)), conn=conn)
        return dict(case, u16=u16) if kind == "watershed" else case
    op, marker = rng.choice([("dilate", "dome"), ("dilate", "seeds"), ("erode", "border")])
    h = {"dome": rng.randrange(10, 61) * (257 if u16 else 1), "seeds": max(1, H * W // 260000), "border": 0}[marker]
    case = dict(kind=kind, H=H, W=W, blobs=blobs, u16=u16, conn=conn, op=op, marker=marker, h=h)
    if kind == "host":
        return dict(case, band_rows=rng.randrange(128, 1024))
    return dict(case, field=rng.choice(["blobs", "blobs", "noise"]))


# ---- inputs -------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _blob_field(H, W, blobs, g):
    """Uniform 0..30 background under Gaussian-profile blobs (radius 5..40, peak 80..255)."""
    out = torch.randint(0, 31, (H * W,), generator=g, device=DEV, dtype=torch.int32)
    u = torch.rand((blobs, 4), generator=g, device=DEV, dtype=torch.float64)
    d = torch.arange(-41, 42, device=DEV)
    for first in range(0, blobs, 1000):
        c = u[first:first + 1000]
        cy, cx, r = c[:, 0] * H, c[:, 1] * W, 5 + 35 * c[:, 2]
        peak = (80 + 176 * c[:, 3]).floor()
        y, x = cy.long()[:, None] + d, cx.long()[:, None] + d
        d2 = ((y + 0.5 - cy[:, None]) ** 2)[:, :, None] + ((x + 0.5 - cx[:, None]) ** 2)[:, None, :]
        r2 = (r * r)[:, None, None]
        v = torch.round(peak[:, None, None] * torch.exp(-2 * d2 / r2)).int()
        ok = (d2 <= r2) & ((y >= 0) & (y < H))[:, :, None] & ((x >= 0) & (x < W))[:, None, :]
        at = y.clamp(0, H - 1)[:, :, None] * W + x.clamp(0, W - 1)[:, None, :]
        out.scatter_reduce_(0, at.reshape(-1), torch.where(ok, v, torch.zeros_like(v)).reshape(-1), "amax")
    return out.view(H, W)


def _noise_field(H, W, g):
    """Uniform 0..255 noise, 5 x 5 box mean with replicated edges."""
    n = torch.randint(0, 256, (1, 1, H, W), generator=g, device=DEV).float()
    s = F.avg_pool2d(F.pad(n, (2, 2, 2, 2), mode="replicate"), 5, stride=1, divisor_override=1)
    return ((s[0, 0].round() + 12) / 25).floor().int()


def _pixels(v, u16):
    """An int32 field as pixels: uint8, or 16-bit pixels held in an int16 tensor."""
    return v.to(torch.int16) if u16 else v.to(torch.uint8)


def _as_image(t):
    return t.view(torch.uint16) if t.dtype == torch.int16 else t


def _marker_mask(H, W, blobs, field, u16, marker, h, g):
    """(marker, mask) as int32 fields."""
    mask = _noise_field(H, W, g) if field == "noise" else _blob_field(H, W, blobs, g)
    if u16:
        mask = mask * 257
    if marker == "dome":
        return (mask - h).clamp_(min=0), mask
    if marker == "seeds":
        m = torch.zeros_like(mask)
        at = torch.randint(0, H * W, (h,), generator=g, device=DEV)
        m.view(-1)[at] = mask.view(-1)[at]
        return m, mask
    m = torch.full_like(mask, 65535 if u16 else 255)
    m[0], m[-1] = mask[0], mask[-1]
    m[:, 0], m[:, -1] = mask[:, 0], mask[:, -1]
    return m, mask


def _batch_images(case):
    """Sides and kind of every image of a batch, from the case alone."""
    r = random.Random(case["layout"])
    out = []
    for i in range(case["n"]):
        H, W = (_side(r, case["min_side"], case["max_side"]) for _ in range(2))
        out.append((H, W, r.random() < 0.5, i < case["n"] // 2, r.randrange(10, 61)))
    return out


def _single(case, g):
    return _marker_mask(case["H"], case["W"], case["blobs"], case.get("field", "blobs"), case["u16"], case["marker"],
                        case["h"], g)


def _zone_markers(case, g):
    H, W, n = case["H"], case["W"], case["markers"]
    m = torch.zeros(H * W, dtype=torch.int32, device=DEV)
    at = torch.unique(torch.randint(0, H * W, (n,), generator=g, device=DEV))
    m[at] = torch.randint(1, n + 1, (at.numel(),), generator=g, device=DEV, dtype=torch.int32).clamp_(max=65534)
    return m.view(H, W)


def _gradient(case, g):
    """Gradient magnitude (L1) of a noisy tissue image, 8 or 16 bits."""
    f = _blob_field(case["H"], case["W"], case["blobs"], g)
    if case["u16"]:
        f = f * 256 + torch.randint(0, 256, f.shape, generator=g, device=DEV, dtype=torch.int32)
    p = F.pad(f[None, None].float(), (1, 1, 1, 1), mode="replicate")[0, 0]
    grad = (p[1:-1, 2:] - p[1:-1, :-2]).abs() + (p[2:, 1:-1] - p[:-2, 1:-1]).abs()
    return grad.clamp_(max=65535 if case["u16"] else 255).int()


def _edt_mask(case, g):
    return (_blob_field(case["H"], case["W"], case["blobs"], g) > 60).to(torch.uint8)


def _porous(case, g):
    return (_blob_field(case["H"], case["W"], case["blobs"], g) > 8).to(torch.uint8)


# ---- calls --------------------------------------------------------------------------------

def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("recon", "host"):
        m0, mask = (_pixels(t, case["u16"]) for t in _single(case, g))
        s = dict(case=case, marker0=m0)
        dtype = torch.uint16 if case["u16"] else torch.uint8
        if kind == "host":
            s["mask"] = mask.cpu().pin_memory()
            s["marker"] = torch.empty(m0.shape, dtype=m0.dtype, pin_memory=True)
            s["plan"] = iwpp.HostReconstructor(case["H"], case["W"], dtype, case["band_rows"])
        else:
            s["mask"], s["marker"] = mask, torch.empty_like(m0)
            s["plan"] = iwpp.Reconstructor(case["H"], case["W"], dtype)
        return s
    if kind == "batch":
        imgs = _batch_images(case)
        n8 = sum((H * W + 255) // 256 * 256 for H, W, u16, _, _ in imgs if not u16)
        n16 = sum((H * W + 127) // 128 * 128 for H, W, u16, _, _ in imgs if u16)
        # one arena per pixel type (images 256-byte aligned): initial markers, markers, masks
        a8 = [torch.zeros(max(n8, 1), dtype=torch.uint8, device=DEV) for _ in range(3)]
        a16 = [torch.zeros(max(n16, 1), dtype=torch.int16, device=DEV) for _ in range(3)]
        o8 = o16 = 0
        items = []
        for H, W, u16, dome, h in imgs:
            m, I = _marker_mask(H, W, max(1, 2000 * H * W // 4096 ** 2), "blobs", u16, "dome" if dome else "border",
                                h * (257 if u16 else 1), g)
            arena, at = (a16, o16) if u16 else (a8, o8)
            cut = [t[at:at + H * W].view(H, W) for t in arena]
            cut[0].copy_(_pixels(m, u16))
            cut[2].copy_(_pixels(I, u16))
            if u16:
                o16 += (H * W + 127) // 128 * 128
            else:
                o8 += (H * W + 255) // 256 * 256
            items.append((_as_image(cut[1]), _as_image(cut[2]), case["conn"], "dilate" if dome else "erode"))
        s = dict(case=case, a8=a8, a16=a16, plan=iwpp.Batch(items))
        if case["learned"]:
            # weights whose sweep output is 0 on every block, as the trained estimator's is
            p = learned.init_params(7)
            p[-130:-2].reshape(64, 2)[:, 1] = 0
            s["sched"] = learned.LearnedScheduler(p, DEV)
        return s
    if kind == "hmax":
        f = _blob_field(case["H"], case["W"], case["blobs"], g)
        return dict(case=case, image=_as_image(_pixels(f * 257 if case["u16"] else f, case["u16"])))
    if kind == "edt":
        mask = _edt_mask(case, g)
        out = [torch.empty(mask.shape, dtype=torch.int32, device=DEV) for _ in range(2)]
        return dict(case=case, mask=mask, out=out, plan=iwpp.DistanceTransform(case["H"], case["W"]))
    if kind == "watershed":
        grad = _as_image(_pixels(_gradient(case, g), case["u16"]))
        return dict(case=case, grad=grad, markers=_zone_markers(case, g))
    return dict(case=case, mask=_porous(case, g), markers=_zone_markers(case, g))


def _ok(rc):
    if rc != 0:
        raise iwpp.IwppError(rc)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("recon", "host"):
        state["marker"].copy_(state["marker0"])
        _ok(state["plan"](_as_image(state["marker"]), _as_image(state["mask"]), case["conn"], case["op"]))
        return state["marker"]
    if kind == "batch":
        for a in (state["a8"], state["a16"]):
            a[1].copy_(a[0])
        _ok(state["sched"].reconstruct(state["plan"]) if case["learned"] else state["plan"]())
        return [state["a8"][1], state["a16"][1]]
    if kind == "hmax":
        r = iwpp.hmaxima(state["image"], case["h"], case["conn"])
        return r.view(torch.int16) if case["u16"] else r
    if kind == "edt":
        _ok(state["plan"](state["mask"], state["out"][0], state["out"][1], case["conn"]))
        return state["out"]
    if kind == "watershed":
        # The levels are unique. Which marker's label a pixel gets where several reach it at its
        # level is not (2-7 % of these pixels change label from one run to the next), so the
        # labels, which the call computes and writes all the same, cannot be compared.
        return iwpp.watershed(state["markers"], state["grad"], case["conn"], with_levels=True)[1]
    return iwpp.skiz(state["markers"], state["mask"], case["conn"], with_details=True)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        px = sum(H * W * (2 if u16 else 1) for H, W, u16, _, _ in _batch_images(case))
        return {"bytes": 3 * px, "flops": 0}
    # marker and mask in, result out | image in, result out | mask in, sites and distances out |
    # markers and gradient in, labels and levels out | markers and mask in, three maps out
    per = {"recon": 3, "host": 3, "hmax": 2, "edt": 9, "watershed": 13 + case.get("u16", False), "skiz": 17}[kind]
    if kind in ("recon", "host", "hmax") and case["u16"]:
        per *= 2
    return {"bytes": per * case["H"] * case["W"], "flops": 0}


def tolerance(case):
    # A reconstruction, flooding levels, geodesic distances and zones are unique: bit for bit.
    # Which of several sites at one distance a pixel ends with depends on the order of work
    # (4e-4 of the values differ between two runs of the 4096 x 4096 case).
    return {"rel": 0.0, "differ": 0.002} if case["kind"] == "edt" else "exact"


# ---- independent evaluation (torch, 64 bits) -------------------------------------------------

def _neighbourhood_max(x, conn):
    x = x[None, None]
    if conn == 8:
        return F.max_pool2d(x, 3, 1, 1)[0, 0]
    return torch.maximum(F.max_pool2d(x, (3, 1), 1, (1, 0)), F.max_pool2d(x, (1, 3), 1, (0, 1)))[0, 0]


def _to_fixed_point(x, step):
    while True:
        y = x
        for _ in range(32):
            y = step(y)
        if torch.equal(x, y):
            return x
        x = y


def _reconstruction(m, I, conn, op):
    m, I = m.double(), I.double()
    s = 1.0 if op == "dilate" else -1.0
    return s * _to_fixed_point(s * m, lambda j: torch.minimum(_neighbourhood_max(j, conn), s * I))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch" or case["H"] * case["W"] > 1 << 24:
        return None
    g = _gen(seed)
    conn = case["conn"]
    if kind in ("recon", "host"):
        m, I = _single(case, g)
        return _reconstruction(m, I, conn, case["op"])
    if kind == "hmax":
        f = _blob_field(case["H"], case["W"], case["blobs"], g) * (257 if case["u16"] else 1)
        return _reconstruction((f - case["h"]).clamp(min=0), f, conn, "dilate")
    if kind == "edt":
        fg = (_edt_mask(case, g) != 0).double()
        far = float(case["H"] + case["W"])
        # city-block radius bounds the search; column distances first, then rows
        col = _to_fixed_point(torch.where(fg > 0, far, 0.0), lambda d: torch.minimum(
            d, 1.0 - F.max_pool2d(-d[None, None], (3, 1), 1, (1, 0))[0, 0]) * fg)
        cheb = _to_fixed_point(torch.where(fg > 0, far, 0.0), lambda d: torch.minimum(
            d, 1.0 + -_neighbourhood_max(-d, 4)) * fg)
        R, c2, best = int(cheb.max()), col * col, col * col
        p = F.pad(c2, (R, R), value=4 * far * far)
        for k in range(2 * R + 1):
            best = torch.minimum(best, p[:, k:k + case["W"]] + float((k - R) ** 2))
        return [None, best]
    if kind == "watershed":
        I, mk = _gradient(case, g), _zone_markers(case, g)
        return _reconstruction(torch.where(mk != 0, I, torch.full_like(I, 65535)), I, conn, "erode")
    dom, mk = _porous(case, g), _zone_markers(case, g)
    inside = (dom != 0) | (mk != 0)
    far = float(case["H"] * case["W"])
    d = _to_fixed_point(torch.where(mk != 0, 0.0, far).double(), lambda x: torch.where(
        inside, torch.minimum(x, 1.0 - _neighbourhood_max(-x, conn)), far))
    return [None, torch.where(d < far, d, -1.0), None]
