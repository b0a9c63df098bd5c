"""Tile lists of the renderer at the sizes where its blending changes form: lists at and around the segment
length (1024) and its multiples, images of up to and beyond 65536 tiles (16- and 32-bit tile keys), against the
oracle, within the bound of FP32 blending against FP64 that the renderer's other tests use."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_14513_gb300 import synthetic as S

IMG_TOL, IMG_FLOOR, TR_TOL = 1e-4, 1e-6, 2e-5


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_14513_gb300 import gsc
    c = gsc.Context(0)
    yield c
    c.close()


def _render(ctx, O, n, scale, logit, cam, tiles=None):
    from paper_2607_14513_gb300 import gsc
    sc, geo = S.make_scene(n, 40 + n), S.make_geometry(n, 41 + n, scale=scale)
    geo.logit[:] += np.float32(logit)
    cu = lambda a: torch.from_numpy(a).cuda()
    pos, sh = cu(sc.pos), cu(sc.sh)
    perm, scales = gsc.gsc_plan_reorder(ctx, pos, sh)
    blk, po, tab = gsc.gsc_encode(ctx, sh, perm, scales, gsc.FMT_BC1)
    tr = torch.empty((cam["height"], cam["width"]), dtype=torch.float32, device="cuda")
    img, tr, pairs = gsc.Renderer(ctx).render(tab, blk, po, pos, cu(geo.scale), cu(geo.rot), cu(geo.logit), cam, trans=tr)
    ctx.sync()
    ref = O.full_encode(sc.pos, sc.sh, 1)
    tex = O.decode(ref["table"], ref["blocks"], ref["perm"])
    colour = O.eval_sh(tex, ref["scales"], pos=sc.pos, cams=O.camera_centre(cam)[None, :])[0]
    want = O.render(sc.pos, geo.scale, geo.rot, geo.logit, colour, cam, tiles=tiles, want_abs=True)
    return img.cpu().numpy().astype(np.float64), tr.cpu().numpy().astype(np.float64), pairs, want


@pytest.mark.parametrize("n", [1, 33, 1023, 1024, 1025, 2047, 2048, 2049, 5000])
@pytest.mark.parametrize("size", [(16, 16), (37, 21)])
def test_list_lengths(ctx, O, n, size):
    # every splat covers the whole image, thin enough that the far ones still count
    cam = S.look_at([0.5, 0.5, -2.0], [0.5, 0.5, 0.5], *size, fov_x_deg=20.0)
    img, tr, pairs, (want, wtr, ab) = _render(ctx, O, n, 0.6, -7.0, cam)
    assert pairs == n * ((size[0] + 15) // 16) * ((size[1] + 15) // 16)
    assert np.all(np.abs(img - want) <= IMG_TOL * ab + IMG_FLOOR)
    assert np.all(np.abs(tr - wtr) <= TR_TOL)


@pytest.mark.parametrize("size", [(4096, 4096), (4112, 4096)])
def test_many_tiles(ctx, O, size):
    cam = S.look_at([0.5, 0.5, -1.6], [0.5, 0.5, 0.5], *size)
    tx, ty = (size[0] + 15) // 16, (size[1] + 15) // 16
    rng = np.random.default_rng(5)
    tiles = np.unique(np.concatenate([rng.integers(0, tx * ty, 300), [0, tx * ty - 1, 65535]]))
    img, tr, pairs, (want, wtr, ab) = _render(ctx, O, 900, 0.01, 0.0, cam, tiles=tiles)
    assert pairs > 0
    hit = 0
    for t in tiles:
        y, x = 16 * (t // tx), 16 * (t % tx)
        part = (slice(y, y + 16), slice(x, x + 16))
        hit += bool(np.any(ab[part] > 0))
        assert np.all(np.abs(img[part] - want[part]) <= IMG_TOL * ab[part] + IMG_FLOOR)
        assert np.all(np.abs(tr[part] - wtr[part]) <= TR_TOL)
    assert hit > 20
