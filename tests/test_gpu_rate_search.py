"""The lambda search by one CTA (up to 2048 groups) and by a grid whose last CTA narrows, on both sides of the line
between them, against the sharded search, which counts and narrows in kernels of their own: the same lambda, streams
and bytes, at a target that is nearly free, in between, and hardly feasible (Sec. IV-B)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2607_14513_gb300 import synthetic as S


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_14513_gb300 import gsc
    c = gsc.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("t4", [3, 17, 63])
@pytest.mark.parametrize("n", [16, 257, 16 * 1024 + 1, 16 * 2048, 16 * 2048 + 1])
def test_search_is_the_sharded_one(ctx, n, t4):
    from paper_2607_14513_gb300 import gsc, shard
    sc = S.make_scene(n, n + t4)
    pos, sh = torch.from_numpy(sc.pos).cuda(), torch.from_numpy(sc.sh).cuda()
    perm, scales = gsc.gsc_plan_reorder(ctx, pos, sh, group_size=256)
    blocks, order, tab = gsc.gsc_encode(ctx, sh, perm, scales, gsc.FMT_RATE, t4)
    _, tab2, blocks2, order2 = shard.encode_scene_sharded(ctx, [pos], [sh], t4, group_size=256)
    ctx.sync()
    assert (tab.lambda_, tab.used_bits, tab.total_bytes) == (tab2.lambda_, tab2.used_bits, tab2.total_bytes)
    assert torch.equal(blocks[:tab.total_bytes], blocks2[:tab.total_bytes])
    assert torch.equal(order, order2)
