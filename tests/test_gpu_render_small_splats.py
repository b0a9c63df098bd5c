"""Splats of a pixel's size and below, anywhere in a tile: the exponent's terms must not cancel. One opaque splat per tile at
the low-pass floor (variance 0.3 px^2) and up to 4 px^2, its centre anywhere in the tile.

Bound on the transmittance, per splat at a pixel: the exponent's error is at most 13 roundings (the conic's 5, its scaling
by log2 e 2, distances and products 6) of 2^-24 of itself, and mu g |ln g| <= 1 / e: 2.9e-7; ex2 2^-22: 2.4e-7; the
sigmoid 4 roundings: 2.4e-7; the update of T 2 roundings: 1.2e-7. 9e-7 together, and a pixel sees two splats: 2e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_14513_gb300 import synthetic as S

TR_TOL = 2e-6


@pytest.mark.parametrize("var", [0.3, 0.5, 1.0, 4.0])
def test_small_opaque_splats(O, var):
    from paper_2607_14513_gb300 import gsc
    w, h, f = 656, 640, 1000.0
    cells = [(x, y) for y in range(0, h, 16) for x in range(0, w, 16)]
    n = len(cells)
    rng = np.random.default_rng(int(10 * var))
    at = np.array(cells) + 16 * rng.random((n, 2))
    at[::4, 1] = np.floor(at[::4, 1] / 16) * 16 + 12 + 4 * rng.random(at[::4].shape[0])   # the tile's last rows
    pos = np.stack([(at[:, 0] - w / 2) / f, (at[:, 1] - h / 2) / f, np.ones(n)], axis=1).astype(np.float32)
    scale = np.full((n, 3), max(np.sqrt(var - 0.3), 1e-3) / f, np.float32)
    rot = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    logit = np.full(n, 3.0, np.float32)
    cam = dict(R=np.eye(3, dtype=np.float32).reshape(9), t=np.zeros(3, np.float32), fx=np.float32(f), fy=np.float32(f),
               cx=np.float32(w / 2), cy=np.float32(h / 2), width=w, height=h, near_z=np.float32(0.2))
    sh = S.make_scene(n, 3).sh
    cu = lambda a: torch.from_numpy(a).cuda()
    ctx = gsc.Context(0)
    perm, scales = gsc.gsc_plan_reorder(ctx, cu(pos), cu(sh))
    blk, po, tab = gsc.gsc_encode(ctx, cu(sh), perm, scales, gsc.FMT_BC1)
    tr = torch.empty((h, w), dtype=torch.float32, device="cuda")
    img, tr, pairs = gsc.Renderer(ctx).render(tab, blk, po, cu(pos), cu(scale), cu(rot), cu(logit), cam, trans=tr)
    ctx.sync()
    want = O.render(pos, scale, rot, logit, np.zeros((n, 3)), cam)[1]
    assert pairs >= n and want.min() < 0.3
    assert np.abs(tr.cpu().numpy().astype(np.float64) - want).max() <= TR_TOL
    ctx.close()
