"""The BC1 encoder with its per-warp queue of neighbourhood steps, and the staging that quantises without a divide,
against the oracle. Bit-exact (Sec. III-B, V-A)."""
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


def _content(n, rng):
    """Of each kind a share: noise, two far colours, ramps, nearly constant blocks at the ends of the range, one
    varying channel, points on a line, constant blocks (queues of unequal length in one warp)."""
    y, x = np.divmod(np.arange(16), 4)
    g = rng.integers(-40, 41, size=(n, 2, 3))
    kinds = [
        rng.integers(0, 256, size=(n, 16, 3)),
        255 * rng.integers(0, 2, size=(n, 16, 3)),
        rng.integers(0, 256, size=(n, 1, 3)) + y[None, :, None] * g[:, :1] + x[None, :, None] * g[:, 1:],
        rng.choice([0, 1, 4, 128, 250, 255], size=(n, 1, 3)) + rng.integers(-3, 4, size=(n, 16, 3)),
        np.where(np.arange(3) == 1, rng.integers(0, 256, size=(n, 16, 1)), rng.integers(0, 256, size=(n, 1, 3))),
        np.rint(rng.integers(0, 256, size=(n, 1, 3)) + rng.integers(-255, 256, size=(n, 1, 3)) * rng.random((n, 16, 1))),
        np.repeat(rng.integers(0, 256, size=(n, 1, 3)), 16, axis=1),
    ]
    which = rng.integers(0, len(kinds), size=n)
    v = np.stack(kinds)[which, np.arange(n)]
    return np.clip(v, 0, 255).astype(np.uint8)


# 420,000 blocks are past the line where a warp takes 128 blocks instead of 32; the last warp has 32 of them
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 129, 3000, 420_000])
def test_queued_search_is_the_plain_one(ctx, O, n):
    from paper_2607_14513_gb300 import gsc
    rng = np.random.default_rng(n)
    tex = _content(min(n, 3001), rng)
    ob, osse = O.encode_blocks(tex, 1)
    at = np.arange(n) % tex.shape[0]
    gb, gsse = gsc.gsc_encode_blocks(ctx, torch.from_numpy(tex).cuda()[torch.from_numpy(at).cuda()].contiguous(), gsc.FMT_BC1)
    torch.cuda.synchronize()
    assert np.array_equal(gsse.cpu().numpy().astype(np.uint64), osse[at])
    assert np.array_equal(gb.cpu().numpy(), ob[at])


# scales inside the range of the correction, at its ends, and (the last two) outside, where the divide is used
SCALES = [[0.3, 1.0, 1e-3, 7.77, 2.0 ** -60, 2.0 ** 60, 1 + 2.0 ** -23, 2 - 2.0 ** -23, 1e9, 3e-9, 0.1, 5.0, 0.7, 1 / 3, 1.1, 255.0],
          [0.3] * 15 + [2.0 ** -61], [2.0 ** 61] + [1e-3] * 15]


@pytest.mark.parametrize("scales", SCALES, ids=["inside", "below", "above"])
@pytest.mark.parametrize("n", [1, 16, 33, 16 * 500 + 7])
def test_staged_texels_are_the_quantised_ones(ctx, O, scales, n):
    """The rows of a group are equal, so every block is constant and its BC7 coding exact: the decoded texels are the
    quantised values. They lie on and beside the ties of the rounding, beyond the ends of the range, and anywhere."""
    from paper_2607_14513_gb300 import gsc
    rng = np.random.default_rng([n, len(set(scales))])
    ng = (n + 15) // 16
    sc = np.asarray(scales, np.float32)
    u = (rng.integers(-131, 132, size=(ng, 16, 3)) + 0.5) / 255.0
    x = (u * sc[None, :, None].astype(np.float64)).astype(np.float32)
    for _ in range(2):
        x = np.where(rng.random(x.shape) < 0.4, np.nextafter(x, rng.choice([-np.inf, np.inf], size=x.shape).astype(np.float32)), x)
    x = np.where(rng.random(x.shape) < 0.2, (0.2 * rng.standard_normal(x.shape) * sc[None, :, None]).astype(np.float32), x)
    odd = rng.choice(np.asarray([0.0, -0.0, 1e-45, -1e-40, 3e38, -3e38, np.inf, -np.inf], np.float32), size=x.shape)
    x = np.where(rng.random(x.shape) < 0.05, odd, x).astype(np.float32)
    rows = np.repeat(x, 16, axis=0)[:n]
    perm = np.full(ng * 16, -1, np.int32)
    perm[:n] = np.arange(n)
    blocks, _, _ = gsc.gsc_encode(ctx, torch.from_numpy(rows).cuda(), torch.from_numpy(perm).cuda(),
                                  torch.from_numpy(sc).cuda(), gsc.FMT_BC7)
    torch.cuda.synchronize()
    got = O.decode_blocks(blocks.cpu().numpy().reshape(-1, 16), 7).reshape(ng, 16, 16, 4)[..., :3]
    with np.errstate(over="ignore"):
        want = O.quantise(x.reshape(ng, 48), sc).reshape(ng, 1, 16, 3).transpose(0, 2, 1, 3)
    assert np.array_equal(got, np.broadcast_to(want, got.shape))
