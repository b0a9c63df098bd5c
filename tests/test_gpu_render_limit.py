"""A frame of as many (Gaussian, tile) pairs as the renderer takes, 2^32 - 16: 4,859 Gaussians that each cover all 870 x 1016
tiles, 92 GB on the device. Every pixel's transmittance is (1 - mu)^4859 but for rounding: at most 3 roundings of 2^-24 per
splat (mu, w, T), and a weight within 2^-20 of 1 (exponents below 2e-7). One splat lost from a list would change it
by mu = 1e-3, the last segment by half."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_14513_gb300 import synthetic as S


def test_most_pairs():
    from paper_2607_14513_gb300 import gsc
    n, w, h = 4859, 870 * 16, 1016 * 16
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 110e9:
        pytest.skip("needs 110 GB free")
    f = np.float32(1000.0)
    cam = dict(R=np.eye(3, dtype=np.float32).reshape(9), t=np.zeros(3, np.float32), fx=f, fy=f, cx=np.float32(w / 2),
               cy=np.float32(h / 2), width=w, height=h, near_z=np.float32(0.2))
    pos = np.tile(np.float32([0, 0, 1]), (n, 1))
    rot = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    logit = np.full(n, -6.9, np.float32)
    cu = lambda a: torch.from_numpy(a).cuda()
    ctx = gsc.Context(0)
    sh = cu(S.make_scene(n, 3).sh)
    perm, scales = gsc.gsc_plan_reorder(ctx, cu(pos), sh)
    blk, po, tab = gsc.gsc_encode(ctx, sh, perm, scales, gsc.FMT_BC1)
    tr = torch.full((h, w), -1.0, dtype=torch.float32, device="cuda")
    # a standard deviation of 2e7 pixels
    img, tr, pairs = gsc.Renderer(ctx).render(tab, blk, po, cu(pos), torch.full((n, 3), 2e4, device="cuda"), cu(rot),
                                              cu(logit), cam, trans=tr)
    ctx.sync()
    assert pairs == 2 ** 32 - 16
    mu = 1.0 / (1.0 + np.exp(-np.float64(logit[0])))
    want = (1.0 - mu) ** n
    tol = n * (3 * 2.0 ** -24 + mu * 2.0 ** -20)
    assert tol < mu
    assert abs(tr.min().item() / want - 1) <= tol and abs(tr.max().item() / want - 1) <= tol
    assert bool(torch.isfinite(img).all())
    del img, tr
    ctx.close()
    torch.cuda.empty_cache()
