"""A frame of one Gaussian: one (Gaussian, depth) pair and up to one (Gaussian, tile) pair are in order as they are, so none of
the sorts' launches is made; image and transmittance against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_14513_gb300 import synthetic as S


@pytest.mark.parametrize("size,tiles", [((16, 16), 1), ((48, 40), 9)])
def test_one_gaussian(O, size, tiles):
    from paper_2607_14513_gb300 import gsc
    ctx = gsc.Context(0)
    cam = S.look_at([0.5, 0.5, -1.5], [0.5, 0.5, 0.5], *size)
    cu = lambda a: torch.from_numpy(a).cuda()
    launches = {}
    for n in (1, 2):
        sh = S.make_scene(n, 6).sh
        pos = np.tile(np.float32([0.5, 0.5, 0.5]), (n, 1))
        geo = S.make_geometry(n, 7, scale=0.5)
        perm, scales = gsc.gsc_plan_reorder(ctx, cu(pos), cu(sh))
        blk, po, tab = gsc.gsc_encode(ctx, cu(sh), perm, scales, gsc.FMT_BC1)
        tr = torch.empty((size[1], size[0]), dtype=torch.float32, device="cuda")
        before = gsc.launch_count()
        img, tr, pairs = gsc.Renderer(ctx).render(tab, blk, po, cu(pos), cu(geo.scale), cu(geo.rot), cu(geo.logit), cam, trans=tr)
        launches[n] = gsc.launch_count() - before
        ctx.sync()
        assert pairs == n * tiles
        ref = O.full_encode(pos, sh, 1)
        colour = O.eval_sh(O.decode(ref["table"], ref["blocks"], ref["perm"]), ref["scales"], pos=pos,
                           cams=O.camera_centre(cam)[None, :])[0]
        want, wtr, ab = O.render(pos, geo.scale, geo.rot, geo.logit, colour, cam, want_abs=True)
        assert np.all(np.abs(img.cpu().numpy() - want) <= 1e-4 * ab + 1e-6)
        assert np.all(np.abs(tr.cpu().numpy() - wtr) <= 2e-5)
    # four passes of three launches by depth, and one by tile where there is one pair
    assert launches[2] - launches[1] == 12 + (3 if tiles == 1 else 0)
    ctx.close()
