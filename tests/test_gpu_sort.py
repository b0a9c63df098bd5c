"""Edges of the plan's sorts against the oracle's: the slot order at sizes around a sort tile (4096 pairs), its
multiples and the small-scene limits, whole-scene and small chunks, ragged sizes, equal positions and equal
colours (stability), each bit-exact (Sec. III-C)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2607_14513_gb300 import gsc
    c = gsc.Context(0)
    yield c
    c.close()


def _scene(n, kind, seed):
    from paper_2607_14513_gb300 import synthetic as S
    sc = S.make_scene(n, seed)
    if kind == "grid":       # many equal positions and equal colours: ties everywhere
        sc.pos[:] = np.round(sc.pos * 4) / 4
        sc.sh[:] = np.round(sc.sh * 4) / 4
    if kind == "one":        # one position, one colour
        sc.pos[:] = sc.pos[0]
        sc.sh[:, 0] = sc.sh[0, 0]
    if kind == "zeros":      # bands that are not used
        sc.sh[:, 4:] = 0.0
    return sc


SIZES = [1, 17, 4096, 4097, 8192, 8193, 12289, 40001, 70007]
CASES = [(n, "random", g) for n in SIZES + [15, 255, 4095] for g in (0, 16, 256, 4096, 8192)]
CASES += [(n, kind, g) for kind in ("grid", "one", "zeros") for n in SIZES for g in (0, 256, 4096)]


@pytest.mark.parametrize("n,kind,group", CASES)
def test_slot_order_and_scales(ctx, O, n, kind, group):
    from paper_2607_14513_gb300 import gsc
    sc = _scene(n, kind, n % 97 + group)
    perm, scales = gsc.gsc_plan_reorder(ctx, torch.from_numpy(sc.pos).cuda(), torch.from_numpy(sc.sh).cuda(), group_size=group)
    ctx.sync()
    want = O.scales(sc.sh)
    assert np.array_equal(scales.cpu().numpy(), want)
    assert np.array_equal(perm.cpu().numpy(), O.plan(sc.pos, O.quantise(sc.sh, want), group, 1))


@pytest.mark.parametrize("permille", [1, 500, 994, 1000])
@pytest.mark.parametrize("n", [1, 4096, 8193, 50021])
def test_scales_at_other_quantiles(ctx, O, n, permille):
    from paper_2607_14513_gb300 import gsc
    rng = np.random.default_rng(n + permille)
    sh = rng.standard_normal((n, 16, 3)).astype(np.float32)
    sh[:, 1] = np.round(sh[:, 1] * 2) / 2                      # few distinct magnitudes
    sh[:, 2] = np.where(rng.random((n, 3)) < 0.996, 0.0, sh[:, 2])   # almost all zero
    sh[:, 3] *= np.float32(1e-30)
    sh[:, 4, :] = 3.5                                          # one magnitude
    sh[:, 5] *= np.exp(8 * rng.standard_normal((n, 3))).astype(np.float32)
    sh[: n // 2, 6] = 0.25                                     # half the values equal, in one half of the scene
    _, scales = gsc.gsc_plan_reorder(ctx, None, torch.from_numpy(sh).cuda(), sort=0, permille=permille)
    ctx.sync()
    assert np.array_equal(scales.cpu().numpy(), O.scales(sh, permille))


@pytest.mark.parametrize("n", [4096, 20_001])
def test_plan_captured_and_eager_agree(ctx, n):
    """A captured plan (one stream) replays to what the eager plan (two streams) gives, also with an eager plan of the
    same context enqueued while the capture is open."""
    from paper_2607_14513_gb300 import gsc
    sc = _scene(n, "random", 5)
    pos, sh = torch.from_numpy(sc.pos).cuda(), torch.from_numpy(sc.sh).cuda()
    ws = [ctx.workspace(n) for _ in range(2)]
    want = gsc.gsc_plan_reorder(ctx, pos, sh, ws=ws[0])
    torch.cuda.synchronize()
    other, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        got = gsc.gsc_plan_reorder(ctx, pos, sh, ws=ws[1])
        eager = gsc.gsc_plan_reorder(ctx, pos, sh, ws=ws[0], stream=other)
    other.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    for k in range(2):
        assert torch.equal(got[k], want[k])
    del eager
