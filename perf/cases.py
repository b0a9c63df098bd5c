"""The work that users of this codec have it do, as cases that can be timed and checked one by one.

Each case is one pass through the public binding (`paper_2607_14513_gb300.gsc`): the reorder plan of
a scene, its encoding in one of the codings, the decode to texels, the fused decode + SH evaluation,
and a rendered frame. Scenes are drawn on the GPU with the distributions of
`paper_2607_14513_gb300/synthetic.py` (clustered centres, DC ~ N(0, 0.8), band l ~ N(0, 0.15 / (l + 1)),
10% of the Gaussians with Laplace(0, 0.3) in bands 2-3); sizes are those of the repository's workloads
(4,096, 10,000, 262,144, 3,000,000), and ragged ones between.

`exact` restates what is computed in floating point in 64 bits with torch alone: the scales' order
statistics, the block decoders with the SH evaluation, and the splatting renderer (whose decisions the
paper's reading fixes in float: those are taken in float, operation by operation, and everything
else in double).
"""
import math

import torch

from paper_2607_14513_gb300 import gsc

DEV = "cuda:0"
FMT = {"bc1": gsc.FMT_BC1, "bc7": gsc.FMT_BC7, "rate": gsc.FMT_RATE, "mixed": gsc.FMT_MIXED}
LAYOUT = {"D": gsc.LAYOUT_D, "A": gsc.LAYOUT_A, "B": gsc.LAYOUT_B}
ORDER = {"views": gsc.OUT_VIEW_MAJOR, "gauss": gsc.OUT_GAUSS_MAJOR, "rows": gsc.OUT_SLOT_ROWS}
LARGEST, SMALLEST = 3_000_000, 4_096

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = gsc.Context(0)
    return _ctx


def listed():
    return [
        # the reorder plan of a small scene: what a caller waits for before its first encode (latency and launches)
        dict(name="plan_4k", kind="plan", n=4096),
        # the plan of a whole trained scene's size: order statistics over 576 MB and the two sorts
        dict(name="plan_3m", kind="plan", n=3_000_000),
        # a small served scene coded in BC7 on request: far fewer blocks than the chip has lanes for
        dict(name="encode_bc7_10k", kind="encode", n=10_000, fmt="bc7"),
        # the usual high-quality coding of an object-sized scene
        dict(name="encode_bc7_262k", kind="encode", n=262_144, fmt="bc7"),
        # the fast coding of a whole scene (4 bits per texel)
        dict(name="encode_bc1_3m", kind="encode", n=3_000_000, fmt="bc1"),
        # the offline coding of a whole scene: rate control at 6 bits per texel, every block searched in both formats
        dict(name="encode_rate_3m", kind="encode", n=3_000_000, fmt="rate", target_x4=24),
        # layout B with BC7 on the first coefficients, BC1 on the rest (10 bytes per Gaussian), a ragged size
        dict(name="encode_b4_300k", kind="encode", n=300_003, fmt="mixed", layout="B", j=4),
        # unpacking a whole scene to texels
        dict(name="decode_bc7_3m", kind="decode", n=3_000_000, fmt="bc7"),
        # colours of a small scene for shared directions (16 views): latency
        dict(name="eval_bc1_4k", kind="eval", n=4096, fmt="bc1", views=16, cams=False, order="views"),
        # colours of a rate-coded scene in the caller's own order, few cameras, ragged size, centres gathered
        dict(name="eval_rate_1m", kind="eval", n=1_000_003, fmt="rate", target_x4=24, views=3, cams=True, order="gauss"),
        # colours of a resident whole scene for 8 camera poses, in the coded scene's own order
        dict(name="eval_bc7_3m", kind="eval", n=3_000_000, fmt="bc7", views=8, cams=True, order="rows"),
        # one full-HD frame of a whole scene
        dict(name="render_3m", kind="render", n=3_000_000, fmt="bc7", width=1920, height=1080, coded=False),
    ]


def _size(rng, most=LARGEST):
    n = int(round(math.exp(rng.uniform(math.log(SMALLEST), math.log(most)))))
    how = rng.random()
    return n // 16 * 16 if how < 0.3 else n | 1 if how < 0.8 else n


def draw(rng):
    kind = rng.choice(["plan", "encode", "encode", "encode", "decode", "eval", "eval", "render"])
    n = _size(rng)
    if kind == "plan":
        return dict(kind=kind, n=n)
    target = rng.choice([12, 16, 24, 32])
    if kind == "encode":
        fmt = rng.choice(["bc1", "bc7", "rate", "mixed"])
        if fmt == "rate":
            return dict(kind=kind, n=n, fmt=fmt, target_x4=target)
        layout = rng.choice(["D", "B"]) if fmt == "mixed" else rng.choice(["D", "D", "A", "B"])
        if fmt == "mixed":
            return dict(kind=kind, n=n, fmt=fmt, layout=layout, j=rng.choice([1, 4, 9]) if layout == "D" else rng.choice([4, 8, 12]))
        return dict(kind=kind, n=n, fmt=fmt, layout=layout)
    fmt = rng.choice(["bc1", "bc7", "rate"])
    case = dict(kind=kind, n=n, fmt=fmt)
    if fmt == "rate":
        case["target_x4"] = target
    if kind == "eval":
        views = rng.choice([1, 2, 3, 5, 8, 16, 32])
        n = case["n"] = min(n, 8 * LARGEST // views // 2 if views > 8 else n)
        case.update(views=views, cams=rng.random() < 0.75, order=rng.choice(["views", "gauss", "rows", "rows"]))
    if kind == "render":
        w, h = rng.choice([(640, 480), (1280, 720), (1001, 563), (1920, 1080)])
        case.update(width=w, height=h, coded=rng.random() < 0.4)
    return case


# ---- inputs -------------------------------------------------------------------------------------
def _scene(case, g):
    n = case["n"]
    clusters = 64 if n > 300_000 else 8
    centres = 0.1 + 0.8 * torch.rand(clusters, 3, generator=g, device=DEV)
    which = torch.randint(0, clusters, (n,), generator=g, device=DEV)
    pos = (centres[which] + 0.05 * torch.randn(n, 3, generator=g, device=DEV)).clamp_(0.0, 1.0).contiguous()
    std = torch.tensor([0.8] + [0.15 / (int(math.isqrt(k)) + 1) for k in range(1, 16)], device=DEV)
    sh = torch.randn(n, 16, 3, generator=g, device=DEV) * std[None, :, None]
    if n > 300_000:  # the scene-scale workload's heavy tail
        at = (torch.rand(n, generator=g, device=DEV) < 0.1).nonzero()[:, 0]
        u = torch.rand(at.numel(), 12, 3, generator=g, device=DEV) - 0.5
        sh[at, 4:] = -0.3 * u.sign() * torch.log1p(-2.0 * u.abs().clamp_(max=0.4999999))
    return pos, sh.contiguous()


def _camera(case, g):
    """A pinhole camera on a sphere of radius 2 around the cube's centre, looking at it (50 degrees)."""
    d = torch.randn(3, generator=g, device=DEV, dtype=torch.float64).cpu()
    d = (d / d.norm()).tolist()
    eye = [0.5 + 2.0 * v for v in d]
    fwd = [-v for v in d]
    up = [0.0, 0.0, 1.0] if abs(fwd[2]) < 0.95 else [0.0, 1.0, 0.0]

    def cross(a, b):
        return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]

    right = cross(fwd, up)
    length = math.sqrt(sum(v * v for v in right))
    right = [v / length for v in right]
    rot = [*right, *cross(fwd, right), *fwd]
    t = [-sum(rot[3 * i + k] * eye[k] for k in range(3)) for i in range(3)]
    f = 0.5 * case["width"] / math.tan(math.radians(50.0) / 2)
    as32 = torch.tensor([*rot, *t, f, case["width"] / 2, case["height"] / 2, 0.2], dtype=torch.float64).float().tolist()
    return dict(R=as32[:9], t=as32[9:12], fx=as32[12], fy=as32[12], cx=as32[13], cy=as32[14], width=case["width"],
                height=case["height"], near_z=as32[15])


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    ctx, n = _context(), case["n"]
    pos, sh = _scene(case, g)
    state = dict(case=case, ctx=ctx, pos=pos, sh=sh)
    if case["kind"] == "plan":
        state["ws"] = ctx.workspace(n)
        return state
    state["perm"], state["scales"] = gsc.gsc_plan_reorder(ctx, pos, sh)
    fmt, target = FMT[case["fmt"]], case.get("target_x4", 0)
    layout, j = LAYOUT[case.get("layout", "D")], case.get("j", 0)
    state["ws"] = ctx.workspace(n, fmt, target, layout, j)
    if case["kind"] == "encode":  # the output buffer is the program's own, of the capacity that any coding may need
        state["out"] = torch.zeros((n + 15) // 16 * 256, dtype=torch.uint8, device=DEV)
        return state
    # a coded scene: its blocks, slot order and stream table are what the program keeps
    blocks, perm, table = gsc.gsc_encode(ctx, sh, state["perm"], state["scales"], fmt, target, ws=state["ws"])
    state.update(blocks=blocks.clone(), perm=perm, table=table)
    del state["sh"], state["ws"]
    if case["kind"] == "eval":
        d = torch.randn(case["views"], 3, generator=g, device=DEV, dtype=torch.float64)
        d = d / d.norm(dim=1, keepdim=True)
        state["views"] = (0.5 + 2.0 * d if case["cams"] else d).float().contiguous()
        if case["order"] == "rows" and case["cams"]:  # the coded scene keeps its centres in slot order
            state["pos_slot"] = gsc.gsc_positions_to_slots(ctx, pos, perm)
    if case["kind"] == "render":
        size = 0.004 * (LARGEST / n) ** (1.0 / 3.0)
        state["scale"] = torch.exp(math.log(size) + 0.35 * torch.randn(n, 3, generator=g, device=DEV)).contiguous()
        state["rot"] = torch.randn(n, 4, generator=g, device=DEV)
        state["logit"] = 1.5 * torch.randn(n, generator=g, device=DEV)
        state["cam"] = _camera(case, g)
        state["renderer"] = gsc.Renderer(ctx)
        if case["coded"]:
            state["geom"] = gsc.gsc_geometry_encode(ctx, pos, state["scale"], state["rot"], state["logit"], perm)
    return state


# ---- one pass -----------------------------------------------------------------------------------
def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "plan":
        perm, scales = gsc.gsc_plan_reorder(ctx, state["pos"], state["sh"], ws=state["ws"])
        return dict(perm=perm, scales=scales)
    if case["kind"] == "encode":
        fmt, ng = case["fmt"], (case["n"] + 15) // 16
        both = {}
        if fmt == "rate":  # the all-BC1 and all-BC7 codings are kept beside the streams
            both = dict(bc1_all=torch.empty(ng * 128, dtype=torch.uint8, device=DEV),
                        bc7_all=torch.empty(ng * 256, dtype=torch.uint8, device=DEV))
        _, perm, table = gsc.gsc_encode(ctx, state["sh"], state["perm"], state["scales"], FMT[fmt],
                                        case.get("target_x4", 0), ws=state["ws"], out=state["out"],
                                        layout=LAYOUT[case.get("layout", "D")], bc7_blocks=case.get("j", 0), **both)
        return dict(blocks=state["out"], perm=perm, total_bytes=int(table.total_bytes), used_bits=int(table.used_bits),
                    rate_lambda=int(table.lambda_), **both)
    if case["kind"] == "decode":
        return gsc.gsc_decode(ctx, state["table"], state["blocks"], state["perm"])
    if case["kind"] == "eval":
        view = dict(cams=state["views"]) if case["cams"] else dict(dirs=state["views"])
        if "pos_slot" in state:
            return gsc.gsc_decode_eval_sh_slots(ctx, state["table"], state["blocks"], state["perm"],
                                                pos_slot=state["pos_slot"], out_order=ORDER[case["order"]], **view)
        return gsc.gsc_decode_eval_sh(ctx, state["table"], state["blocks"], state["perm"],
                                      pos=state["pos"] if case["cams"] else None, out_order=ORDER[case["order"]], **view)
    n, cam = case["n"], state["cam"]
    trans = torch.empty((cam["height"], cam["width"]), dtype=torch.float32, device=DEV)
    if case["coded"]:
        image, trans, _, _ = state["renderer"].render_coded(state["table"], state["blocks"], state["perm"], state["geom"],
                                                            4096, cam, trans=trans)
    else:
        image, trans, _ = state["renderer"].render(state["table"], state["blocks"], state["perm"], state["pos"],
                                                   state["scale"], state["rot"], state["logit"], cam, trans=trans)
    return dict(image=image, trans=trans)


def work(case):
    """Bytes in and out once; operations where arithmetic is what the result consists of."""
    n, ng = case["n"], (case["n"] + 15) // 16
    if case["kind"] == "plan":  # centres and coefficients in, slot order and scales out
        return dict(bytes=n * (192 + 12 + 4), flops=0)
    per_group = {"bc1": 128, "bc7": 256, "rate": case.get("target_x4", 0) * 8, "mixed": 128 + 8 * case.get("j", 0)}[case["fmt"]]
    if case["kind"] == "encode":
        both = 128 + 256 if case["fmt"] == "rate" else 0
        return dict(bytes=n * 192 + ng * (64 + 64 + per_group + both), flops=0)
    if case["kind"] == "decode":
        return dict(bytes=ng * (per_group + 64) + n * 48, flops=0)
    if case["kind"] == "eval":  # 48 multiply-adds per Gaussian and view
        v = case["views"]
        return dict(bytes=ng * (per_group + 64) + n * (12 if case["cams"] else 0) + n * 12 * v, flops=96.0 * n * v)
    # a frame: colours and geometry in, image and transmittance out; per pixel of every 3-sigma ellipse the exponent,
    # its exponential and four multiply-adds (about 20 operations), for a camera 2 away from the scene's centre
    size = 0.004 * (LARGEST / n) ** (1.0 / 3.0) * 0.5 * case["width"] / math.tan(math.radians(25.0)) / 2.0
    geom = 17 if case["coded"] else 44
    return dict(bytes=ng * (per_group + 64) + n * geom + 16 * case["width"] * case["height"],
                flops=20.0 * n * 9.0 * math.pi * (size * size + 0.3))


# ---- the same in 64 bits, with torch alone --------------------------------------------------------
# BC7: two-subset partitions (bit t: texel t in subset 1), three-subset partitions (a digit per
# texel) and the anchor texels, as the format defines them
_PART2 = [
    0xCCCC, 0x8888, 0xEEEE, 0xECC8, 0xC880, 0xFEEC, 0xFEC8, 0xEC80, 0xC800, 0xFFEC, 0xFE80, 0xE800, 0xFFE8,
    0xFF00, 0xFFF0, 0xF000, 0xF710, 0x008E, 0x7100, 0x08CE, 0x008C, 0x7310, 0x3100, 0x8CCE, 0x088C, 0x3110,
    0x6666, 0x366C, 0x17E8, 0x0FF0, 0x718E, 0x399C, 0xAAAA, 0xF0F0, 0x5A5A, 0x33CC, 0x3C3C, 0x55AA, 0x9696,
    0xA55A, 0x73CE, 0x13C8, 0x324C, 0x3BDC, 0x6996, 0xC33C, 0x9966, 0x0660, 0x0272, 0x04E4, 0x4E40, 0x2720,
    0xC936, 0x936C, 0x39C6, 0x639C, 0x9336, 0x9CC6, 0x817E, 0xE718, 0xCCF0, 0x0FCC, 0x7744, 0xEE22]
_PART3 = (
    "0011001102212222 0001001122112221 0000200122112211 0222002200110111 0000000011221122 0011001100220022 "
    "0022002211111111 0011001122112211 0000000011112222 0000111111112222 0000111122222222 0012001200120012 "
    "0112011201120112 0122012201220122 0011011211221222 0011200122002220 0001001101121122 0111001120012200 "
    "0000112211221122 0022002200221111 0111011102220222 0001000122212221 0000001101220122 0000110022102210 "
    "0122012200110000 0012001211222222 0110122112210110 0000011012211221 0022110211020022 0110011020022222 "
    "0011012201220011 0000200022112221 0000000211221222 0222002200120011 0011001200220222 0120012001200120 "
    "0000111122220000 0120120120120120 0120201212010120 0011220011220011 0011112222000011 0101010122222222 "
    "0000000021212121 0022112200221122 0022001100220011 0220122102201221 0101222222220101 0000212121212121 "
    "0101010101012222 0222011102220111 0002111200021112 0000211221122112 0222011101110222 0002111211120002 "
    "0110011001102222 0000000021122112 0110011022222222 0022001100110022 0022112211220022 0000000000002112 "
    "0002000100020001 0222122202221222 0101222222222222 0111201122012220").split()
_ANCHOR2 = [15] * 17 + [2, 8, 2, 2, 8, 8, 15, 2, 8, 2, 2, 8, 8, 2, 2, 15, 15, 6, 8, 2, 8, 15, 15, 2, 8, 2, 2, 2, 15, 15,
                        6, 6, 2, 6, 8, 15, 15, 2, 2, 15, 15, 15, 15, 15, 2, 2, 15]
_ANCHOR3A = [3, 3, 15, 15, 8, 3, 15, 15, 8, 8, 6, 6, 6, 5, 3, 3, 3, 3, 8, 15, 3, 3, 6, 10, 5, 8, 8, 6, 8, 5, 15, 15, 8, 15,
             3, 5, 6, 10, 8, 15, 15, 3, 15, 5, 15, 15, 15, 15, 3, 15, 5, 5, 5, 8, 5, 10, 5, 10, 8, 13, 15, 12, 3, 3]
_ANCHOR3B = [15, 8, 8, 3, 15, 15, 3, 8, 15, 15, 15, 15, 15, 15, 15, 8, 15, 8, 15, 3, 15, 8, 15, 8, 3, 15, 6, 10, 15, 15, 10,
             8, 15, 3, 15, 10, 10, 8, 9, 10, 6, 15, 8, 15, 3, 6, 6, 8, 15, 3, 15, 15, 15, 15, 15, 15, 15, 15, 15, 15, 3, 15,
             15, 8]
# per mode: subsets, partition, rotation and selection bits, colour and alpha bits, a p-bit per
# endpoint or per subset, index bits, second index bits
_MODE = [(3, 4, 0, 0, 4, 0, 1, 0, 3, 0), (2, 6, 0, 0, 6, 0, 0, 1, 3, 0), (3, 6, 0, 0, 5, 0, 0, 0, 2, 0),
         (2, 6, 0, 0, 7, 0, 1, 0, 2, 0), (1, 0, 2, 1, 5, 6, 0, 0, 2, 3), (1, 0, 2, 0, 7, 8, 0, 0, 2, 2),
         (1, 0, 0, 0, 7, 7, 1, 0, 4, 0), (2, 6, 0, 0, 5, 5, 1, 0, 2, 0)]
_WEIGHT = {2: [0, 21, 43, 64], 3: [0, 9, 18, 27, 37, 46, 55, 64],
           4: [0, 4, 9, 13, 17, 21, 26, 30, 34, 38, 43, 47, 51, 55, 60, 64]}


def _table(v):
    return torch.tensor(v, dtype=torch.int64, device=DEV)


def _bc1(raw):
    """[m, 8] bytes -> texels [m, 16, 3] (int64), interpolated as the GPU's texture unit does."""
    w = raw.to(torch.int64)
    c = [w[:, 0] | w[:, 1] << 8, w[:, 2] | w[:, 3] << 8]
    index = w[:, 4] | w[:, 5] << 8 | w[:, 6] << 16 | w[:, 7] << 24
    wide = c[0] > c[1]
    out = []
    for shift, bits in ((11, 5), (5, 6), (0, 5)):
        a, b = ((v >> shift) & ((1 << bits) - 1) for v in c)
        a8, b8 = (((v << 3) | (v >> 2)) if bits == 5 else ((v << 2) | (v >> 4)) for v in (a, b))
        if bits == 5:
            p2, p3 = torch.where(wide, ((2 * a + b) * 11) >> 2, ((a + b) * 33) >> 3), ((2 * b + a) * 11) >> 2
        else:
            p2 = torch.where(wide, a8 + (((b8 - a8) * 321 + 512) >> 10), a8 + (((b8 - a8) * 257 + 256) >> 9))
            p3 = b8 + (((a8 - b8) * 321 + 512) >> 10)
        palette = torch.stack([a8, b8, p2, torch.where(wide, p3, torch.zeros_like(p3))], 1)
        at = torch.stack([(index >> (2 * t)) & 3 for t in range(16)], 1)
        out.append(palette.gather(1, at))
    return torch.stack(out, 2)


def _bits(lo, hi, off, count):
    """`count` bits of each 128-bit block (two int64 halves) from bit `off` (a number or a tensor)."""
    if not isinstance(off, torch.Tensor):
        off = torch.full_like(lo, off)
    mask = (1 << count) - 1
    left = 64 - off
    low = (lo >> off.clamp(max=63)) & torch.where(left >= count, torch.full_like(lo, mask), (1 << left.clamp(0, 62)) - 1)
    cross = (hi << left.clamp(0, 63)) & mask
    return torch.where(off >= 64, (hi >> (off - 64).clamp(min=0)) & mask, torch.where(left >= count, low, low | cross))


def _bc7(raw):
    """[m, 16] bytes -> texels [m, 16, 3] (int64)."""
    w = raw.to(torch.int64)
    lo = sum(w[:, k] << (8 * k) for k in range(8))
    hi = sum(w[:, 8 + k] << (8 * k) for k in range(8))
    out = torch.zeros(raw.shape[0], 16, 3, dtype=torch.int64, device=DEV)
    subset2 = _table([[(m >> t) & 1 for t in range(16)] for m in _PART2])
    subset3 = _table([[int(d) for d in row] for row in _PART3])
    for mode, (ns, pb, rb, sb, cb, ab, epb, spb, ib, ib2) in enumerate(_MODE):
        at = ((w[:, 0] & ((2 << mode) - 1)) == (1 << mode)).nonzero()[:, 0]
        if not at.numel():
            continue
        l, h = lo[at], hi[at]
        zero = torch.zeros_like(l)
        pos = mode + 1
        part = _bits(l, h, pos, pb) if pb else zero
        rot = _bits(l, h, pos + pb, rb) if rb else zero
        sel = _bits(l, h, pos + pb + rb, sb) if sb else zero
        pos += pb + rb + sb
        subset = (subset2 if ns == 2 else subset3)[part] if ns > 1 else torch.zeros(at.numel(), 16, dtype=torch.int64, device=DEV)
        pstart = pos + 2 * ns * (3 * cb + ab)
        istart = pstart + (2 * ns if epb else ns if spb else 0)
        ends = torch.zeros(at.numel(), ns, 2, 4, dtype=torch.int64, device=DEV)
        for s in range(ns):
            for e in range(2):
                for c in range(4):
                    bits = cb if c < 3 else ab
                    if not bits:
                        ends[:, s, e, c] = 255
                        continue
                    start = pos + (c * 2 * ns * cb if c < 3 else 6 * ns * cb) + (2 * s + e) * bits
                    v = _bits(l, h, start, bits)
                    if epb or (spb and c < 3):
                        v = v << 1 | _bits(l, h, pstart + (2 * s + e if epb else s), 1)
                        bits += 1
                    ends[:, s, e, c] = v << (8 - bits) | v >> (2 * bits - 8)
        anchors = [zero] + ([_table(_ANCHOR2)[part]] if ns == 2 else [_table(_ANCHOR3A)[part], _table(_ANCHOR3B)[part]] if ns == 3 else [])
        for t in range(16):
            before, here = sum((a < t).long() for a in anchors), sum((a == t).long() for a in anchors)
            first = _bits(l, h, istart + t * ib - before, ib)
            first = torch.where(here > 0, first & ((1 << (ib - 1)) - 1), first)
            wc = wa = _table(_WEIGHT[ib])[first]
            if ib2:
                second = _bits(l, h, istart + 16 * ib - 1 + t * ib2 - (t > 0), ib2 - (t == 0))
                w2 = _table(_WEIGHT[ib2])[second]
                wc, wa = torch.where(sel > 0, w2, wc), torch.where(sel > 0, wc, w2)
            e = ends.gather(1, subset[:, t].view(-1, 1, 1, 1).expand(-1, 1, 2, 4))[:, 0]
            weight = torch.stack([wc, wc, wc, wa], 1)
            px = ((64 - weight) * e[:, 0] + weight * e[:, 1] + 32) >> 6
            rgb = px[:, :3].clone()
            for c in range(3):
                rgb[:, c] = torch.where(rot == c + 1, px[:, 3], px[:, c])
            out[at, t] = rgb
    return out


def _coefficients(state):
    """Dequantised coefficients [slots, 16, 3] in double, slot order, of a coded scene (layout D)."""
    table, blocks = state["table"], state["blocks"]
    tex = torch.full((table.n_groups, 16, 16, 3), 128, dtype=torch.uint8, device=DEV)
    for s in table.streams():
        b, j, m, g0 = s["bands"], s["bc7_blocks"], s["n_groups"], s["first_group"]
        size = 16 * j + 8 * (b - j)
        if not m:
            continue
        raw = blocks[s["byte_offset"]:s["byte_offset"] + m * size].view(m, size)
        if j:
            tex[g0:g0 + m, :j] = _bc7(raw[:, :16 * j].reshape(-1, 16)).view(m, j, 16, 3).to(torch.uint8)
        if b > j:
            tex[g0:g0 + m, j:b] = _bc1(raw[:, 16 * j:].reshape(-1, 8)).view(m, b - j, 16, 3).to(torch.uint8)
    scales = torch.tensor(list(table.scales), dtype=torch.float64, device=DEV)
    # block k, texel t -> slot t, coefficient k
    return tex.transpose(1, 2).reshape(-1, 16, 3).double().sub_(128.0).mul_((scales / 255.0)[None, :, None])


def _basis(d):
    """Real SH to degree 3 (k = l*l + l + m, Condon-Shortley phase) of unit directions [..., 3] -> [..., 16]."""
    x, y, z = d.unbind(-1)
    xx, yy, zz = x * x, y * y, z * z
    p = math.pi
    c1, c2 = math.sqrt(3 / (4 * p)), math.sqrt(15 / (4 * p))
    return torch.stack([
        torch.full_like(x, math.sqrt(1 / (4 * p))), -c1 * y, c1 * z, -c1 * x, c2 * x * y, -c2 * y * z,
        math.sqrt(5 / (16 * p)) * (2 * zz - xx - yy), -c2 * x * z, math.sqrt(15 / (16 * p)) * (xx - yy),
        -math.sqrt(35 / (32 * p)) * y * (3 * xx - yy), math.sqrt(105 / (4 * p)) * x * y * z,
        -math.sqrt(21 / (32 * p)) * y * (4 * zz - xx - yy), math.sqrt(7 / (16 * p)) * z * (2 * zz - 3 * xx - 3 * yy),
        -math.sqrt(21 / (32 * p)) * x * (4 * zz - xx - yy), math.sqrt(105 / (16 * p)) * z * (xx - yy),
        -math.sqrt(35 / (32 * p)) * x * (xx - 3 * yy)], -1)


def _colours(coef, view, centres):
    """Colours [m, 3] of coefficients [m, 16, 3] seen along `view`, or from `view` when centres are given."""
    d = view.double().expand(coef.shape[0], 3)
    if centres is not None:
        d = d - centres.double()
    d = d / d.norm(dim=1, keepdim=True)
    return torch.einsum("mk,mkc->mc", _basis(d), coef)


def _exact_eval(case, state):
    coef, perm, n = _coefficients(state), state["perm"].long(), case["n"]
    centres = state["pos"][perm.clamp(min=0)] if case["cams"] else None
    real = perm >= 0
    rows = torch.zeros(perm.numel(), case["views"], 3, dtype=torch.float64, device=DEV)
    for v in range(case["views"]):
        for a in range(0, perm.numel(), 1 << 19):
            some = slice(a, a + (1 << 19))
            c = _colours(coef[some], state["views"][v], None if centres is None else centres[some])
            rows[some, v] = torch.where(real[some, None], c, torch.zeros_like(c))
    if case["order"] == "rows":
        return rows
    out = torch.zeros(n, case["views"], 3, dtype=torch.float64, device=DEV)
    out[perm[real]] = rows[real]
    return out if case["order"] == "gauss" else out.transpose(0, 1).contiguous()


def _splats(state, real):
    """Per Gaussian in type `real`: centre on screen, conic (inverse covariance), depth, and the tile rectangle's extent."""
    cam = state["cam"]
    R = [torch.tensor(v, dtype=real, device=DEV) for v in cam["R"]]
    t, fx, fy, cx, cy = cam["t"], cam["fx"], cam["fy"], cam["cx"], cam["cy"]

    def dot(a, b):
        return (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2]

    p = state["pos"].to(real).unbind(1)
    s = state["scale"].to(real).unbind(1)
    q = state["rot"].to(real).unbind(1)
    x, y, z = (dot(R[3 * i:3 * i + 3], p) + t[i] for i in range(3))
    norm = (((q[0] * q[0] + q[1] * q[1]) + q[2] * q[2]) + q[3] * q[3]).sqrt()
    w, i, j, k = (v / norm for v in q)
    rot = [[1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j)],
           [2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i)],
           [2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)]]
    m = [[rot[a][b] * s[b] for b in range(3)] for a in range(3)]
    sigma = [[dot(m[a], m[b]) for b in range(3)] for a in range(3)]
    iz = 1 / z
    J = [[fx * iz, torch.zeros_like(iz), -(fx * x) * (iz * iz)], [torch.zeros_like(iz), fy * iz, -(fy * y) * (iz * iz)]]
    T = [[dot(J[a], [R[c], R[3 + c], R[6 + c]]) for c in range(3)] for a in range(2)]
    U = [[dot(T[a], [sigma[0][c], sigma[1][c], sigma[2][c]]) for c in range(3)] for a in range(2)]
    low = torch.tensor(0.3, dtype=torch.float32, device=DEV).to(real)
    A, B, C = dot(U[0], T[0]) + low, dot(U[0], T[1]), dot(U[1], T[1]) + low
    det = A * C - B * B
    mid = 0.5 * (A + C)
    tenth = torch.tensor(0.1, dtype=torch.float32, device=DEV).to(real)
    rad = torch.ceil(3 * (mid + torch.maximum(mid * mid - det, tenth).sqrt()).sqrt())
    u, v = fx * (x / z) + cx, fy * (y / z) + cy
    return dict(z=z, norm=norm, det=det, u=u, v=v, rad=rad, conic=(C / det, -B / det, A / det))


def _exact_render(case, state):
    n, cam = case["n"], state["cam"]
    w, h = cam["width"], cam["height"]
    tx, ty = (w + 15) // 16, (h + 15) // 16
    f, d = _splats(state, torch.float32), _splats(state, torch.float64)
    R = torch.tensor(cam["R"], dtype=torch.float64, device=DEV).view(3, 3)
    eye = -(R.T @ torch.tensor(cam["t"], dtype=torch.float64, device=DEV))
    coef, perm = _coefficients(state), state["perm"].long()
    real = perm >= 0
    colour = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    for a in range(0, perm.numel(), 1 << 19):
        at = perm[a:a + (1 << 19)].clamp(min=0)
        keep = real[a:a + (1 << 19)]
        colour[at[keep]] = _colours(coef[a:a + (1 << 19)], eye, state["pos"][at])[keep]
    del coef

    def edge(v, most):
        return torch.floor(v / 16).clamp(0, most)

    x0, y0 = edge(f["u"] - f["rad"], tx), edge(f["v"] - f["rad"], ty)
    x1 = (torch.floor((f["u"] + f["rad"]) / 16) + 1).clamp(0, tx)
    y1 = (torch.floor((f["v"] + f["rad"]) / 16) + 1).clamp(0, ty)
    seen = (f["z"] > cam["near_z"]) & (f["norm"] > 0) & (f["det"] > 0) & (x1 > x0) & (y1 > y0)
    which = seen.nonzero()[:, 0]
    which = which[torch.sort(f["z"][which], stable=True).indices]  # nearest first, equal depths in index order
    x0, y0, wide, high = (v[which].long() for v in (x0, y0, x1 - x0, y1 - y0))
    tiles = wide * high
    owner = torch.repeat_interleave(torch.arange(which.numel(), device=DEV), tiles)
    k = torch.arange(owner.numel(), device=DEV) - (tiles.cumsum(0) - tiles)[owner]
    tile = (y0[owner] + k // wide[owner]) * tx + x0[owner] + k % wide[owner]
    tile, at = torch.sort(tile, stable=True)
    entry = which[owner[at]]
    count = torch.bincount(tile, minlength=tx * ty)
    first = count.cumsum(0) - count
    order = torch.argsort(count, descending=True)
    count, first = count[order], first[order]
    px = (order % tx * 16)[:, None] + torch.arange(256, device=DEV) % 16 + 0.5
    py = (torch.div(order, tx, rounding_mode="floor") * 16)[:, None] + torch.arange(256, device=DEV) // 16 + 0.5
    mu = torch.sigmoid(state["logit"].double())
    T = torch.ones(tx * ty, 256, dtype=torch.float64, device=DEV)
    image = torch.zeros(tx * ty, 256, 3, dtype=torch.float64, device=DEV)
    step, lengths = 32, count.cpu()
    for e0 in range(0, int(lengths[0]) if lengths.numel() else 0, step):
        m = int((lengths > e0).sum())
        e = e0 + torch.arange(step, device=DEV)
        live = e[None] < count[:m, None]
        i = entry[(first[:m, None] + e[None]).clamp(max=entry.numel() - 1)]
        dx = px[:m, None] - d["u"][i][..., None]
        dy = py[:m, None] - d["v"][i][..., None]
        a, b, c = (q[i][..., None] for q in d["conic"])
        g = torch.exp(-0.5 * (a * dx * dx + 2 * b * dx * dy + c * dy * dy)) * live[..., None]
        through = torch.cumprod(1 - mu[i][..., None] * g, 1)
        before = torch.cat([torch.ones_like(through[:, :1]), through[:, :-1]], 1)
        image[:m] += T[:m, :, None] * torch.einsum("mep,mec->mpc", g * before, colour[i])
        T[:m] *= through[:, -1]
    place = torch.empty_like(order)
    place[order] = torch.arange(order.numel(), device=DEV)

    def picture(v):
        v = v[place].view(ty, tx, 16, 16, -1).permute(0, 2, 1, 3, 4).reshape(ty * 16, tx * 16, -1)
        return v[:h, :w].contiguous()

    return dict(image=picture(image), trans=picture(T[..., None])[..., 0].contiguous())


def exact(case, seed):
    if case["kind"] in ("encode", "decode"):  # blocks, slot orders, texels and counts: whole numbers
        return None
    state = prepare(case, seed)
    if case["kind"] == "plan":
        n = case["n"]
        rank = -(-995 * 3 * n // 1000) - 1
        a = torch.stack([state["sh"][:, k].abs().reshape(-1).sort().values[rank].double() for k in range(16)])
        return dict(perm=None, scales=torch.where(a == 0, torch.ones_like(a), 2 * a))
    if case["kind"] == "eval":
        return _exact_eval(case, state)
    if case["coded"]:  # what is drawn is the decoded geometry: its codes are whole numbers of the encoder
        return None
    return _exact_render(case, state)
