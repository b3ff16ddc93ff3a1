"""The calls this library is timed on: one pass of each through the C-ABI entry points (by
their binding's names), over the sizes, options and directions that users bring.

``listed()`` are the fixed cases, ``draw(rng)`` gives another one of the same ranges.  Device
frames go through ``dibr_enqueue_image`` on one context, as a program that works on a sequence
of frames calls it (the argument records are made once per buffer set); mixed batches through
``dibr_enqueue_batch``; host frames through the blocking ``dibr_synthesize_image``; video
through the serving loop (``dibr_submit_frame`` / ``dibr_poll``).

``exact(case, seed)`` restates the pipeline (luminance, smoothing, Fig. 3's shift rule, warp with
occlusion, row fill, formats) in plain torch with 64-bit integers and floats.
"""
import ctypes

import numpy as np
import torch

from paper_2009_09501_gb300 import dibr as D
from paper_2009_09501_gb300 import scenes

DEPTH = {"luma": D.DIBR_DEPTH_LUMA, "binom": D.DIBR_DEPTH_LUMA_BINOM5, "xbf": D.DIBR_DEPTH_LUMA_XBF}
STEREO = "anaglyph left right"


def _frame(name, width, height, parallax, outputs, call="device", depth="binom", rule="paper", warp="forward",
           fill="row", noise=False, radius=2):
    return {"name": name, "call": call, "width": width, "height": height, "parallax": parallax, "outputs": outputs,
            "depth": depth, "rule": rule, "warp": warp, "fill": fill, "noise": noise, "radius": radius}


def listed():
    return [
        # a small still on the device: launch and per-row latency (640x480 anaglyph, P = 16)
        _frame("vga_anaglyph", 640, 480, 16, "anaglyph"),
        # a laptop-sized picture with tight rows (3W is no multiple of 16) for a 3-D television:
        # the anamorphic half side-by-side pair
        _frame("hd_hsbs_ragged", 1366, 768, 34, "hsbs", noise=True),
        # a frame handed on to later processing: both views, their depth and holes maps, the
        # linear rule on the unsmoothed luminance
        _frame("fhd_views_maps", 1920, 1080, 48, "left right depth holes", depth="luma", rule="linear"),
        # Fig. 3's backward gather, literally
        _frame("fhd_gather", 1920, 1080, 48, "anaglyph", warp="gather"),
        # a cropped 12-megapixel camera photo: odd width, tight rows, sensor noise everywhere
        _frame("photo_odd", 4031, 3023, 100, STEREO, noise=True),
        # the 4K UHD still with both views and the anaglyph (P = 64)
        _frame("uhd_stereo", 3840, 2160, 64, STEREO),
        # the 4K frame with the cross-bilateral depth (radius 2)
        _frame("uhd_xbf", 3840, 2160, 64, "anaglyph", depth="xbf"),
        # the 4K frame with Fig. 3's iterative block inpainting (32x32 blocks)
        _frame("uhd_inpaint", 3840, 2160, 64, STEREO, fill="inpaint"),
        # an 8K UHD frame with both views and the anaglyph
        _frame("uhd8k_stereo", 7680, 4320, 192, STEREO),
        # 64 images of the mix 720p .. 8K in one call, the anaglyph of each
        {"name": "batch_mixed", "call": "batch", "images": 64, "mix": 4},
        # a 1080p frame from host memory to host memory, one blocking call
        _frame("host_fhd", 1920, 1080, 48, STEREO, call="host"),
        # one frame of each of four video streams through the serving loop (two 1080p, two 4K)
        {"name": "serve_streams", "call": "serve", "streams": 4, "mix": 0},
    ]


def draw(rng):
    kind = rng.choices(["device", "batch", "host", "serve"], [14, 3, 2, 1])[0]
    if kind == "batch":
        return {"call": "batch", "images": int(round(2 * 24 ** rng.random())), "mix": rng.randrange(100, 1 << 30)}
    if kind == "serve":
        return {"call": "serve", "streams": rng.randint(1, 6), "mix": rng.randrange(100, 1 << 30)}
    widest = 7680 if kind == "device" else 3840
    width = int(round(320 * (widest / 320) ** rng.random()))
    height = max(180, int(width * rng.choice([9 / 16, 3 / 4, 2 / 3, 1 / 2.39]) * rng.uniform(0.9, 1.05)))
    shape = rng.choice(["whole", "even", "odd"])  # rows of whole 16-byte units, or tight ragged ones
    width = width // 16 * 16 if shape == "whole" else width // 2 * 2 + (1 if shape == "odd" else 0)
    width, height = min(width, 7680), min(height, 4320)
    outputs = rng.choice(["anaglyph", "anaglyph", STEREO, STEREO, "left right", "left right depth holes", "hsbs"])
    if outputs == "hsbs" and width % 2:
        outputs = "left right"
    c = _frame("", width, height, max(4, int(width * rng.uniform(0.01, 0.04))), outputs, call=kind,
               noise=rng.random() < 0.5)
    del c["name"]
    option = rng.choices(["plain", "luma", "linear", "gather", "xbf", "inpaint"], [8, 2, 2, 2, 3, 3])[0]
    if option == "luma":
        c["depth"] = "luma"
    elif option == "linear":
        c["rule"] = "linear"
    elif option == "gather":
        c["warp"] = "gather"
    elif option == "xbf":
        c["depth"], c["radius"] = "xbf", rng.randint(1, 4 if width <= 3840 else 2)
    elif option == "inpaint":
        c["fill"] = "inpaint"
    return c


# ------------------------------------------------------------------------------- inputs
def _scene(width, height, gen, noise, n_objects=40):
    """A picture like the repository's synthetic scenes, drawn on the GPU: a vertical gradient,
    ellipses and rectangles of a random colour with a textured surface (sigma 8), and sensor
    noise (sigma 2) over the whole frame of a camera picture or video."""
    r = torch.rand((n_objects, 8), generator=gen, device="cuda").tolist()
    ends = (torch.rand((2, 3), generator=gen, device="cuda") * 255).round()
    y = torch.linspace(0, 1, height, device="cuda")[:, None, None]
    img = (ends[0] + (ends[1] - ends[0]) * y).expand(height, width, 3).contiguous()
    for kind, u, v, a, b, *colour in r:
        cx, cy = u * width, v * height
        ax, ay = (max(1.0, width / 40 + t * (width / 8 - width / 40)) for t in (a, b))
        x0, x1 = max(0, int(cx - ax)), min(width, int(cx + ax) + 1)
        y0, y1 = max(0, int(cy - ay)), min(height, int(cy + ay) + 1)
        if x0 >= x1 or y0 >= y1:
            continue
        part = img[y0:y1, x0:x1]
        paint = 8 * torch.randn(part.shape, generator=gen, device="cuda") + 255 * torch.tensor(colour, device="cuda")
        if kind < 0.5:
            px = (torch.arange(x0, x1, device="cuda") + 0.5 - cx) / ax
            py = (torch.arange(y0, y1, device="cuda") + 0.5 - cy) / ay
            paint = torch.where((px[None, :] ** 2 + py[:, None] ** 2 <= 1)[:, :, None], paint, part)
        part.copy_(paint)
    if noise:
        img += 2 * torch.randn(img.shape, generator=gen, device="cuda")
    return img.round_().clamp_(0, 255).to(torch.uint8)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _batch_sizes(case):
    if case["mix"] == 4:
        return scenes.batch_sizes(case["images"])
    r = np.random.RandomState(case["mix"])
    sizes = []
    for _ in range(case["images"]):
        w, h = scenes.BATCH_CLASSES[r.randint(len(scenes.BATCH_CLASSES))]
        if r.rand() < 0.3:  # a picture cut to some other size
            w, h = int(w * r.uniform(0.6, 1.0)), int(h * r.uniform(0.6, 1.0))
        sizes.append((w, h))
    return sizes


def _serve_sizes(case):
    if case["mix"] == 0:
        return [(1920, 1080), (3840, 2160)] * (case["streams"] // 2)
    r = np.random.RandomState(case["mix"])
    return [scenes.BATCH_CLASSES[r.randint(4)] for _ in range(case["streams"])]


def _params(case):
    return D.make_params(depth_rule=DEPTH[case["depth"]],
                         disparity_rule=D.DIBR_DISP_LINEAR if case["rule"] == "linear" else D.DIBR_DISP_PAPER,
                         warp_mode=D.DIBR_WARP_GATHER_FIG3 if case["warp"] == "gather" else D.DIBR_WARP_FORWARD,
                         max_parallax=case["parallax"], outputs=case["outputs"].split(), xbf_radius=case["radius"],
                         hole_fill=D.DIBR_FILL_INPAINT2D if case["fill"] == "inpaint" else D.DIBR_FILL_ROW)


def _image(case, seed):
    return _scene(case["width"], case["height"], _generator(seed), case["noise"])


def _batch_images(case, seed):
    gen = _generator(seed)
    return [_scene(w, h, gen, False, 24) for w, h in _batch_sizes(case)]


def _stream_images(case, seed):
    gen = _generator(seed)
    return [_scene(w, h, gen, True) for w, h in _serve_sizes(case)]


def _outputs(img, names, **where):
    h, w = img.shape[:2]
    return {n: torch.empty((h, w) if n in D.MAP_OUTPUTS else (h, w, 3), dtype=torch.uint8, **where) for n in names}


_contexts = []


def _context():
    """The program's context for frames and batches in device memory."""
    if not _contexts:
        _contexts.append(D.Context(device=0))
    return _contexts[0]


class _Streams:
    """A serving context with one open stream per video, closed with the state that holds it."""

    def __init__(self, sizes):
        self.ctx = D.Context(device=0)
        self.params = [D.make_params(max_parallax=scenes.batch_parallax(w), outputs=("anaglyph",)) for w, _ in sizes]
        self.ids = [self.ctx.open_stream(w, h, p) for (w, h), p in zip(sizes, self.params)]
        self.done = (D.dibr_completion * len(sizes))()
        self.frame = 0


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        imgs = _batch_images(case, seed)
        outs = [_outputs(i, ["anaglyph"], device="cuda") for i in imgs]
        params = [D.make_params(max_parallax=scenes.batch_parallax(i.shape[1]), outputs=("anaglyph",)) for i in imgs]
        ctx = _context()
        state = {"call": call, "ctx": ctx, "imgs": imgs, "outs": outs, "args": ctx._batch_args(imgs, params, outs)}
    elif call == "serve":
        imgs = [i.cpu().pin_memory().numpy() for i in _stream_images(case, seed)]
        outs = [{"anaglyph": _outputs(i, ["anaglyph"], pin_memory=True)["anaglyph"].numpy()} for i in imgs]
        state = {"call": call, "server": _Streams(_serve_sizes(case)), "imgs": imgs, "outs": outs,
                 "args": [(D.image_struct(i), D.outputs_struct(o)) for i, o in zip(imgs, outs)]}
    else:
        img, params = _image(case, seed), _params(case)
        names = case["outputs"].split()
        if call == "host":
            img = img.cpu().pin_memory().numpy()
            outs = {n: o.numpy() for n, o in _outputs(img, names, pin_memory=True).items()}
        else:
            outs = _outputs(img, names, device="cuda")
        state = {"call": call, "ctx": _context(), "img": img, "params": params, "outs": outs,
                 "args": (D.image_struct(img), params, D.outputs_struct(outs))}
    torch.cuda.synchronize()  # the context works on a stream of its own
    return state


def run(state):
    call = state["call"]
    if call == "device":
        ctx = state["ctx"]
        ctx.check(D.dibr_enqueue_image(ctx.handle, *state["args"]))
    elif call == "batch":
        ctx = state["ctx"]
        ctx.check(D.dibr_enqueue_batch(ctx.handle, *state["args"]))
    elif call == "host":
        ctx = state["ctx"]
        ctx.check(D.dibr_synthesize_image(ctx.handle, *state["args"]))
    else:
        s = state["server"]
        for sid, (img, out) in zip(s.ids, state["args"]):
            s.ctx.check(D.dibr_submit_frame(s.ctx.handle, sid, s.frame, img, out))
        s.frame += 1
        left, n = len(s.ids), ctypes.c_int(0)
        while left:
            s.ctx.check(D.dibr_poll(s.ctx.handle, s.done, len(s.ids), n, 1000000))
            for c in s.done[:n.value]:
                s.ctx.check(c.status)
            left -= n.value
    return state["outs"]


def _frame_work(w, h, outputs, depth="binom", radius=2):
    px = w * h
    n = sum(1 if o in D.MAP_OUTPUTS else 3 for o in outputs)
    taps = {"luma": 0, "binom": 10 * 2, "xbf": (2 * radius + 1) ** 2 * 9}[depth]
    return px * (3 + n), px * (6 + taps + 2 * 6)


def work(case):
    """Each input read once and each output written once; per pixel the luminance (6
    operations), the smoothing (a separable 5-tap filter, or the cross-bilateral taps) and one
    shift, comparison and fill per view."""
    if case["call"] in ("batch", "serve"):
        sizes = _batch_sizes(case) if case["call"] == "batch" else _serve_sizes(case)
        both = [_frame_work(w, h, ["anaglyph"]) for w, h in sizes]
    else:
        both = [_frame_work(case["width"], case["height"], case["outputs"].split(), case["depth"], case["radius"])]
    return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}


# -------------------------------------------------------------------- the values, in 64 bits
def _depth(img, depth, radius):
    c = img.to(torch.int64)
    lum = (299 * c[..., 0] + 587 * c[..., 1] + 114 * c[..., 2] + 500) // 1000
    h, w = lum.shape
    if depth == "luma":
        return lum
    if depth == "binom":
        tap = (1, 4, 6, 4, 1)
        ys, xs = torch.arange(h, device=img.device), torch.arange(w, device=img.device)
        v = sum(t * lum[(ys + k - 2).clamp(0, h - 1)] for k, t in enumerate(tap))
        return (sum(t * v[:, (xs + k - 2).clamp(0, w - 1)] for k, t in enumerate(tap)) + 128) >> 8
    num = torch.zeros((h, w), dtype=torch.float64, device=img.device)
    den = torch.zeros_like(num)
    for dy in range(-radius, radius + 1):
        for dx in range(-radius, radius + 1):
            if abs(dy) >= h or abs(dx) >= w:
                continue
            p = slice(max(0, -dy), h - max(0, dy)), slice(max(0, -dx), w - max(0, dx))
            q = slice(max(0, dy), h + min(0, dy)), slice(max(0, dx), w + min(0, dx))
            d2 = ((c[p] - c[q]) ** 2).sum(-1).double()
            wt = torch.exp(-(dx * dx + dy * dy) / (2 * 1.5 ** 2) - d2 / (2 * 16.0 ** 2))
            num[p] += wt * lum[q]
            den[p] += wt
    return torch.floor(num / den + 0.5).to(torch.int64)


def _view(img, d, shift):
    """One view of the forward warp (target x - shift) with its holes filled, and the holes."""
    h, w = d.shape
    x = torch.arange(w, device=d.device).expand(h, w)
    t = x - shift
    inside = (t >= 0) & (t < w)
    empty = 1 << 40
    key = torch.where(inside, (255 - d) << 16 | x, empty)
    z = torch.full((h, w), empty, dtype=torch.int64, device=d.device)
    z.scatter_reduce_(1, t.clamp(0, w - 1), key, "amin")
    filled = z != empty
    lo = torch.where(filled, x, -1).cummax(1).values
    hi = torch.where(filled, x, w).flip(1).cummin(1).values.flip(1)
    zl = torch.where(lo >= 0, z.gather(1, lo.clamp(min=0)), -1)
    zr = torch.where(hi < w, z.gather(1, hi.clamp(max=w - 1)), -1)
    pick = torch.where(zl < 0, zr, torch.where((zr >> 16) > (zl >> 16), zr, zl))
    src = torch.where(pick < 0, x, pick & 0xFFFF)
    return img.gather(1, src[..., None].expand(h, w, 3)), ~filled


def _synthesis(img, outputs, parallax, depth="binom", rule="paper", warp="forward", radius=2):
    d = _depth(img, depth, radius)
    h, w = d.shape
    if rule == "linear":
        num = -510 * (parallax * d // 510)
    else:
        num = torch.where(d > 150, -parallax * d, parallax * (255 - d))
    if warp == "gather":
        views, holes = [], []
        x = torch.arange(w, device=d.device).expand(h, w)
        for n in (num, -num):
            s = torch.div(510 * x + n, 510, rounding_mode="trunc")
            s = torch.where((s >= 0) & (s < w), s, x)
            views.append(img.gather(1, s[..., None].expand(h, w, 3)))
            holes.append(torch.zeros_like(d, dtype=torch.bool))
    else:
        views, holes = zip(*(_view(img, d, torch.div(n, 510, rounding_mode="floor")) for n in (num, -num)))
    left, right = views
    made = {"left": left, "right": right, "depth": d.to(torch.uint8)}
    made["holes"] = holes[0].to(torch.uint8) | holes[1].to(torch.uint8) << 1
    made["anaglyph"] = torch.cat([left[..., :1], right[..., 1:]], 2)
    if "hsbs" in outputs:
        made["hsbs"] = torch.cat([((v[:, ::2].int() + v[:, 1::2].int() + 1) >> 1).to(torch.uint8) for v in views], 1)
    return {n: made[n] for n in outputs}


def exact(case, seed):
    if case["call"] == "batch":
        return [_synthesis(i, ["anaglyph"], scenes.batch_parallax(i.shape[1])) for i in _batch_images(case, seed)]
    if case["call"] == "serve":
        return [_synthesis(i, ["anaglyph"], scenes.batch_parallax(i.shape[1])) for i in _stream_images(case, seed)]
    if case["fill"] == "inpaint" and case["warp"] == "forward":
        return None  # a sequential repair, pixel by pixel
    return _synthesis(_image(case, seed), case["outputs"].split(), case["parallax"], case["depth"], case["rule"],
                      case["warp"], case["radius"])
