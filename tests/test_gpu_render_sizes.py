"""Images of every width of tile key from 1 to 13 bits, at both ends of a width: the number of tiles decides how the sort by
tile shares its key over passes. Float geometry and the coded geometry against the oracle, with more pairs than one
tile of the sort (4096), within the bound of FP32 blending against FP64 that the renderer's other tests use."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_14513_gb300 import synthetic as S
from test_gpu_geometry import _codes, _oracle_coded_render

IMG_TOL, IMG_FLOOR, TR_TOL = 1e-4, 1e-6, 2e-5


@pytest.fixture(scope="module")
def scene(O):
    from paper_2607_14513_gb300 import gsc
    c = gsc.Context(0)
    n, cs = 1501, 128
    sc, geo = S.make_scene(n, 91, clusters=3), S.make_geometry(n, 92, scale=0.02)
    geo.logit[:] -= np.float32(2.0)
    cu = lambda a: torch.from_numpy(a).cuda()
    d = dict(ctx=c, n=n, cs=cs, pos=sc.pos, geo=geo, dpos=cu(sc.pos), dgeo=[cu(a) for a in (geo.scale, geo.rot, geo.logit)])
    perm, scales = gsc.gsc_plan_reorder(c, d["dpos"], cu(sc.sh), group_size=cs)
    d["blk"], d["po"], d["tab"] = gsc.gsc_encode(c, cu(sc.sh), perm, scales, gsc.FMT_BC1)
    d["geom"] = gsc.gsc_geometry_encode(c, d["dpos"], *d["dgeo"], d["po"], cs)
    c.sync()
    d["perm"] = d["po"].cpu().numpy()
    d["codes"] = _codes(gsc, d["geom"], d["perm"].shape[0], cs)
    ref = O.full_encode(sc.pos, sc.sh, 1, group_size=cs)
    d["osc"] = ref["scales"]
    d["tex"] = O.decode(ref["table"], ref["blocks"], ref["perm"])
    yield d
    c.close()


def _check(img, tr, want, wtr, ab):
    img, tr = img.cpu().numpy().astype(np.float64), tr.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(img - want) <= IMG_TOL * ab + IMG_FLOOR)
    assert np.all(np.abs(tr - wtr) <= TR_TOL)


# tiles: 1, 2, 4, 8, 9, 16, 20, 32, 63, 64, 128, 256 and, over two passes, 260, 270, 300, 475, 512, 513, 625, 920, 1024,
# 1025, 2048, 4096
SIZES = [(16, 16), (32, 16), (32, 32), (64, 32), (48, 48), (64, 64), (80, 64), (128, 64), (144, 112), (128, 128), (256, 128),
         (256, 256), (320, 208), (480, 135), (320, 240), (400, 300), (512, 256), (432, 304), (400, 400), (640, 360),
         (512, 512), (656, 400), (1024, 512), (1024, 1024)]


@pytest.mark.parametrize("size", SIZES)
def test_image_sizes(O, scene, size):
    from paper_2607_14513_gb300 import gsc
    w, h = size
    cam = S.look_at([0.5, 0.5, -1.5], [0.5, 0.5, 0.5], w, h)
    tr = torch.empty((h, w), dtype=torch.float32, device="cuda")
    r = gsc.Renderer(scene["ctx"])
    geo = scene["geo"]
    img, tr, pairs = r.render(scene["tab"], scene["blk"], scene["po"], scene["dpos"], *scene["dgeo"], cam, trans=tr)
    scene["ctx"].sync()
    colour = O.eval_sh(scene["tex"], scene["osc"], pos=scene["pos"], cams=O.camera_centre(cam)[None, :])[0]
    _check(img, tr, *O.render(scene["pos"], geo.scale, geo.rot, geo.logit, colour, cam, want_abs=True))
    assert pairs > 4096 or w * h <= 128 * 128
    img, tr, pairs, kept = r.render_coded(scene["tab"], scene["blk"], scene["po"], scene["geom"], scene["cs"], cam, trans=tr)
    scene["ctx"].sync()
    want, wtr, ab, wkept, wpairs = _oracle_coded_render(O, scene["pos"], scene["tex"], scene["osc"], scene["perm"],
                                                        scene["codes"], cam)
    assert (kept, pairs) == (wkept, wpairs)
    _check(img, tr, want, wtr, ab)
