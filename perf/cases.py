"""The reconstruction calls whose time is watched: what a user of the library
has it do, through its public entry points, from one small tile to a 4K frame.

A case is one pass of one entry point:

  single    ``Handle.reconstruct``: one device image
  host      ``Handle.reconstruct_host``: one image in pinned host memory
  channels  ``Handle.reconstruct_channels``: the planes of a colour image, one mask
  plan      ``fsr_batch_launch`` of a prepared batch (``fsr_batch_create``)
  reuse     the sequential form (``reuse = 0.5``): one image through
            ``Handle.reconstruct``, several through ``fsr_reconstruct_batch``

Images are 1/f noise in [0, 255] with a few step edges (natural-image
statistics), masks are quarter sampling, independent loss, or lost 16 x 16
macroblocks.  Every output is the whole reconstructed image.
"""
from __future__ import annotations

import math

import torch

from paper_2202_13926_gb300 import fsr

MB = 16                      # macroblock size of the "macroblock" masks
RHO, GAMMA = 0.7, 0.5        # the paper's parameters (Sec. IV)
SUPPORTS = {32: (2, 4, 8, 16), 24: (4, 8), 16: (2, 4, 8), 8: (2, 4), 4: (2, 4)}   # S: block sizes B
BATCH_SIZES = ((256, 256), (720, 1280), (1080, 1920), (2160, 3840))               # of a mixed batch


def _case(name, kind, height, width, support, block=4, iters=100, mask="quarter", missing=0.75, images=1, pitch=0,
          rho=RHO):
    return dict(name=name, kind=kind, height=height, width=width, support=support, block=block, iters=iters, mask=mask,
                missing=missing, images=images, pitch=pitch, rho=rho)


def listed():
    return [
        # the smallest call: one ragged tile of a picture (a lost region and its
        # surroundings), rows not 16-byte aligned; a few blocks per SM at most
        _case("tile_61x83_s32", "single", 61, 83, 32, mask="iid", missing=0.5),
        # the 128 x 128 test image of the repository: thumbnails, patches
        _case("still_128_s32", "single", 128, 128, 32, mask="iid", missing=0.5),
        # the headline workload: a 1080p frame of a quarter-sampling sensor
        _case("fhd_quarter_s32", "single", 1080, 1920, 32),
        # error concealment: a 4K frame with one macroblock in ten lost
        _case("uhd_macroblock_s32", "single", 2160, 3840, 32, iters=50, mask="macroblock", missing=0.1),
        # the paper's test-image size (Fig. 3) at its second largest support
        _case("paper_1200_s24", "single", 1200, 1200, 24),
        # the paper's frame-rate setting (Fig. 5, S = 16), end to end from host memory
        _case("fhd_s16_host", "host", 1080, 1920, 16),
        # fast previews: the small supports of Fig. 3
        _case("fhd_s8", "single", 1080, 1920, 8),
        _case("hd_s4", "single", 720, 1280, 4),
        # a colour frame with independent pixel loss, larger target blocks
        _case("rgb_hd_b8_s32", "channels", 720, 1280, 32, block=8, mask="iid", missing=0.4, images=3),
        # offline work: a prepared batch of mixed sizes, masks and iteration counts
        _case("batch_mixed_s32", "plan", 0, 0, 32, mask="mixed", images=8),
        # the original FSR's sequential form on a frame, and on a few small frames at once
        _case("reuse_fhd_s32", "reuse", 1080, 1920, 32),
        _case("reuse_6x270p_s32", "reuse", 270, 480, 32, images=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Component updates of a case (blocks x iterations x S^2), all blocks counted."""
    b = c["block"]
    return c["images"] * -(-c["height"] // b) * -(-c["width"] // b) * c["iters"] * c["support"] ** 2


def draw(rng):
    while True:
        kind = rng.choice(("single", "single", "single", "single", "host", "channels", "plan", "reuse"))
        s = 32 if kind == "reuse" else rng.choice((32, 32, 32, 24, 16, 16, 8, 4))
        b = rng.choice((4, 4, 4) + SUPPORTS[s])
        iters = _log_int(rng, 25, 200)
        px = _log_int(rng, 3000, 1920 * 1080 if kind in ("channels", "reuse") else 3840 * 2160)
        aspect = math.exp(rng.uniform(math.log(0.5), math.log(2.0)))
        h, w = max(8, int(math.sqrt(px / aspect))), max(8, int(math.sqrt(px * aspect)))
        if rng.random() < 0.5:       # frames with aligned rows; otherwise any size, rows as they come
            w = max(16, w // 16 * 16)
        mask = rng.choice(("quarter", "iid", "iid", "macroblock"))
        missing = {"quarter": 0.75, "iid": rng.choice((0.1, 0.3, 0.5, 0.7, 0.9)),
                   "macroblock": rng.choice((0.05, 0.1, 0.2))}[mask]
        n = {"channels": 3, "plan": rng.choice((2, 4, 8)), "reuse": rng.choice((1, 1, 3))}.get(kind, 1)
        pitch = -(-w // 16) * 16 if kind == "single" and rng.random() < 0.5 else 0
        c = _case("", kind, h, w, s, b, iters, mask, missing, n, pitch, rng.choice((0.6, 0.7, 0.8)))
        del c["name"]
        if kind == "reuse":          # a chain of wavefronts: at most the listed frame's, twice its work
            chain = 8 * -(-h // b) + -(-w // b)
            if chain * iters > 200_000 or _cost(c) > 2.7e10:
                continue
        if _cost(c) <= 6e10:
            return c


# ---- inputs -----------------------------------------------------------------

def _image(g, h, w):
    """1/f noise scaled to [0, 255] plus step edges, on the GPU."""
    d = torch.device("cuda")
    fy = torch.fft.fftfreq(h, device=d)[:, None]
    fx = torch.fft.rfftfreq(w, device=d)[None, :]
    f = torch.sqrt(fy * fy + fx * fx)
    f[0, 0] = 1.0
    spec = torch.complex(torch.randn(f.shape, generator=g, device=d), torch.randn(f.shape, generator=g, device=d)) / f
    spec[0, 0] = 0
    img = torch.fft.irfft2(spec, s=(h, w))
    lo, hi = img.min(), img.max()
    img = (img - lo) / (hi - lo).clamp_min(1e-12) * 255.0
    yy = torch.arange(h, device=d)[:, None] / h
    xx = torch.arange(w, device=d)[None, :] / w
    for p in torch.rand(4, 4, generator=g, device=d):
        a = p[2] * math.pi
        img = img + torch.where((xx - p[0]) * torch.sin(a) > (yy - p[1]) * torch.cos(a), p[3] * 100 - 50, 0.0)
    return img.clamp(0, 255).float()


def _mask(g, h, w, kind, missing):
    """uint8, 1 = known pixel."""
    d = torch.device("cuda")
    if kind == "iid":
        return (torch.rand(h, w, generator=g, device=d) >= missing).to(torch.uint8)
    if kind == "macroblock":
        keep = torch.rand(-(-h // MB), -(-w // MB), generator=g, device=d) >= missing
        return keep.repeat_interleave(MB, 0).repeat_interleave(MB, 1)[:h, :w].to(torch.uint8).contiguous()
    pick = torch.randint(0, 4, (-(-h // 2), -(-w // 2)), generator=g, device=d)   # quarter sampling
    m = torch.zeros(pick.shape[0] * 2, pick.shape[1] * 2, dtype=torch.uint8, device=d)
    for q in range(4):
        m[q // 2::2, q % 2::2] = pick == q
    return m[:h, :w].contiguous()


def _parts(case):
    """(height, width, mask kind, missing, iterations) of every image of a case."""
    c = case
    if c["mask"] != "mixed":
        return [(c["height"], c["width"], c["mask"], c["missing"], c["iters"])] * c["images"]
    parts = []
    for i in range(c["images"]):     # sizes in turn; masks and iteration counts as in a mixed batch
        h, w = BATCH_SIZES[i % len(BATCH_SIZES)]
        m, p = (("iid", 0.3), ("macroblock", 0.1), ("iid", 0.6), ("macroblock", 0.2))[(i + i // 4) % 4]
        parts.append((h, w, m, p, (50, 100, 200)[i % 3]))
    return parts


def _inputs(case, seed):
    """[(image, mask)] of a case, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    res, mask = [], None
    for h, w, kind, missing, _ in _parts(case):
        img = _image(g, h, w)
        if mask is None or case["kind"] != "channels":   # the planes of a colour image share one mask
            mask = _mask(g, h, w, kind, missing)
        res.append((img, mask))
    return res


_HANDLE = []


def _handle():
    """The one handle that a program keeps."""
    if not _HANDLE:
        _HANDLE.append(fsr.Handle(0))
    return _HANDLE[0]


def _pitched(t, pitch):
    if not pitch or pitch == t.shape[1]:
        return t
    r = torch.zeros(t.shape[0], pitch, dtype=t.dtype, device=t.device)[:, :t.shape[1]]
    r.copy_(t)
    return r


class _Plan:
    """A prepared batch; released with its state."""

    def __init__(self, handle, descs, params):
        self.handle, self.ptr = handle, fsr.fsr_batch_create(handle.ptr, descs, params)

    def __del__(self):
        if torch is not None and self.ptr:
            torch.cuda.synchronize()
            fsr.fsr_batch_destroy(self.ptr)


def prepare(case, seed):
    h, kind = _handle(), case["kind"]
    pairs = _inputs(case, seed)
    kw = dict(block=case["block"], border=(case["support"] - case["block"]) // 2, iters=case["iters"], rho=case["rho"],
              gamma=GAMMA)
    state = dict(kind=kind, handle=h, kw=kw)
    if kind == "channels":
        state["img"] = torch.stack([p[0] for p in pairs])
        state["mask"] = pairs[0][1]
        state["out"] = torch.zeros_like(state["img"])
        return state
    imgs = [_pitched(p[0], case["pitch"]) for p in pairs]
    masks = [_pitched(p[1], case["pitch"]) for p in pairs]
    if kind == "host":
        imgs = [t.cpu().pin_memory() for t in imgs]
        masks = [t.cpu().pin_memory() for t in masks]
        outs = [torch.zeros(t.shape, dtype=torch.float32).pin_memory() for t in imgs]
    else:
        outs = [_pitched(torch.zeros(t.shape, device="cuda"), case["pitch"]) for t in imgs]
    state.update(imgs=imgs, masks=masks, outs=outs)
    if kind in ("plan", "reuse"):
        iters = [p[4] for p in _parts(case)]
        state["descs"] = [fsr.image_desc(i, m, o, k) for i, m, o, k in zip(imgs, masks, outs, iters)]
        if kind == "plan":
            state["plan"] = _Plan(h, state["descs"], fsr.make_params(**kw))
        else:
            kw["reuse"] = 0.5
    return state


def run(state):
    h, kind, kw = state["handle"], state["kind"], state["kw"]
    if kind == "channels":
        return h.reconstruct_channels(state["img"], state["mask"], out=state["out"], **kw)
    if kind == "plan":
        fsr.fsr_batch_launch(state["plan"].ptr, handle=h.ptr)
    elif kind == "host":
        h.reconstruct_host(state["imgs"][0], state["masks"][0], out=state["outs"][0], **kw)
    elif kind == "reuse" and len(state["imgs"]) > 1:
        fsr.fsr_reconstruct_batch(h.ptr, state["descs"], fsr.make_params(**kw))
    else:
        h.reconstruct(state["imgs"][0], state["masks"][0], out=state["outs"][0], **kw)
    return state["outs"]


def work(case):
    """Image, mask and output moved once.  Per iteration of a block that has an
    unknown pixel to fill: 11 operations per component (objective 3, complex
    multiply-subtract 8); before them one complex S x S FFT."""
    s, b = case["support"], case["block"]
    nbytes = flops = 0.0
    for i, (h, w, kind, missing, iters) in enumerate(_parts(case)):
        shared = case["kind"] == "channels" and i > 0
        nbytes += h * w * (8 if shared else 9)
        filled = {"quarter": 1.0, "iid": 1.0 - (1.0 - missing) ** (b * b), "macroblock": missing}[kind]
        blocks = -(-h // b) * -(-w // b) * filled
        flops += blocks * s * s * (11.0 * iters + 10.0 * math.log2(s))
    return dict(bytes=nbytes, flops=flops)


# ---- the method in 64 bits --------------------------------------------------

def _exact_image(img, mask, s, b, iters, rho):
    """Sec. II on one image: every B x B block with an unknown pixel, in
    binary64.  Parameters as the call receives them (binary32)."""
    d = img.device
    H, W = img.shape
    border = (s - b) // 2
    rho = float(torch.tensor(rho, dtype=torch.float32))
    nby, nbx = -(-H // b), -(-W // b)
    known = mask != 0
    f = torch.where(known, img, 0.0).double()
    ph, pw = (border, nby * b - H + border), (border, nbx * b - W + border)
    fp = torch.nn.functional.pad(f, (*pw, *ph))
    kp = torch.nn.functional.pad(known.double(), (*pw, *ph))
    i = torch.arange(s, device=d, dtype=torch.float64) - (s - 1) / 2
    w0 = rho ** torch.sqrt(i[:, None] ** 2 + i[None, :] ** 2)
    t = s / 2 - (torch.arange(s, device=d, dtype=torch.float64) - s / 2).abs()
    wf = (1 - math.sqrt(2) * torch.sqrt((t[:, None] ** 2 + t[None, :] ** 2) / s ** 2)) ** 2
    g = torch.zeros(nby * b, nbx * b, device=d, dtype=torch.float64)
    ko = torch.nn.functional.pad(known, (0, nbx * b - W, 0, nby * b - H), value=True)
    todo = (~ko).view(nby, b, nbx, b).any(3).any(1).flatten().nonzero().flatten()
    si = torch.arange(s, device=d)
    px = border + torch.arange(b, device=d)
    ang = 2 * math.pi / s
    for blk in todo.split(max(1, (1 << 23) // (s * s))) if todo.numel() else ():
        n = blk.numel()
        y, x = (blk // nbx * b)[:, None, None], (blk % nbx * b)[:, None, None]
        w = kp[y + si[None, :, None], x + si[None, None, :]] * w0
        R = torch.fft.fft2(fp[y + si[None, :, None], x + si[None, None, :]] * w)
        Wf = torch.fft.fft2(w)
        W0 = Wf[:, 0, 0].real
        c0 = torch.where(W0 > 0, float(GAMMA) / torch.where(W0 > 0, W0, 1.0), 0.0)
        Rr, Ri = R.real.reshape(n, -1).contiguous(), R.imag.reshape(n, -1).contiguous()
        Wr, Wi = Wf.real.reshape(n, -1).contiguous(), Wf.imag.reshape(n, -1).contiguous()
        acc = torch.zeros(n, b, b, device=d, dtype=torch.float64)
        wfl = wf.reshape(1, -1)
        for _ in range(iters):
            pick = ((Rr * Rr + Ri * Ri) * wfl).argmax(1, keepdim=True)
            cr, ci = Rr.gather(1, pick) * c0[:, None], Ri.gather(1, pick) * c0[:, None]
            u, v = pick // s, pick % s
            th = ang * ((u[:, :, None] * px[None, :, None] + v[:, :, None] * px[None, None, :]) % s).double()
            acc += cr[:, :, None] * torch.cos(th) - ci[:, :, None] * torch.sin(th)
            at = (((si[None, :] - u) % s)[:, :, None] * s + ((si[None, :] - v) % s)[:, None, :]).reshape(n, -1)
            a, bb = Wr.gather(1, at), Wi.gather(1, at)
            Rr -= cr * a - ci * bb
            Ri -= cr * bb + ci * a
        g.view(nby, b, nbx, b)[blk // nbx, :, blk % nbx, :] = acc
    return torch.where(known, img.double(), g[:H, :W])


def exact(case, seed):
    if case["kind"] == "reuse" or _cost(dict(case, height=case["height"] or 2160, width=case["width"] or 3840)) > 4e10:
        return None   # a serial chain of blocks, or minutes in 64 bits
    res = [_exact_image(i, m, case["support"], case["block"], p[4], case["rho"])
           for (i, m), p in zip(_inputs(case, seed), _parts(case))]
    return torch.stack(res) if case["kind"] == "channels" else res
