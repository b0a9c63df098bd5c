"""The pruned BC7 search against the oracle's exhaustive one, block for block and error for error, at the
edges of a warp's 32 blocks and of a CTA's 128, on contents that stress the pruning bound: blocks where
most candidates survive (smooth ramps, nearly constant blocks, points on a line), where few do (noise,
noise with outliers), full-range values and ties between candidates. Bit-exact (Sec. III-B)."""
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


def _content(kind, n, rng):
    if kind == "ramp":       # a plane over the 4x4 block per channel, one level of noise
        y, x = np.divmod(np.arange(16), 4)
        g = rng.integers(-12, 13, size=(n, 2, 3))
        v = rng.integers(60, 196, size=(n, 1, 3)) + y[None, :, None] * g[:, :1] + x[None, :, None] * g[:, 1:]
        return v + rng.integers(-1, 2, size=v.shape)
    if kind == "near":       # a few levels around one colour, at the ends of the range too
        return rng.choice([0, 2, 128, 253, 255], size=(n, 1, 3)) + rng.integers(-2, 3, size=(n, 16, 3))
    if kind == "line":       # texels on one line in colour space
        a, b = rng.integers(0, 256, size=(2, n, 1, 3))
        return np.rint(a + (b - a) * rng.random((n, 16, 1)))
    if kind == "noise":
        return rng.integers(0, 256, size=(n, 16, 3))
    if kind == "outliers":   # a narrow distribution with a few far texels
        v = 128 + 8 * rng.standard_normal((n, 16, 3))
        return np.where(rng.random((n, 16, 1)) < 0.1, rng.integers(0, 256, size=(n, 16, 3)), v)
    if kind == "extreme":    # every channel 0 or 255
        return 255 * rng.integers(0, 2, size=(n, 16, 3))
    # one channel varies, the others constant; and grey: ties between rotations and modes
    v = np.repeat(rng.integers(0, 256, size=(n, 1, 3)), 16, axis=1)
    v[:, :, n % 3] = rng.integers(0, 256, size=(n, 16))
    v[::2] = v[::2, :, n % 3:n % 3 + 1]
    return v


@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 129, 300])
@pytest.mark.parametrize("kind", ["ramp", "near", "line", "noise", "outliers", "extreme", "ties"])
def test_pruned_search_is_the_exhaustive_one(ctx, O, kind, n):
    from paper_2607_14513_gb300 import gsc
    rng = np.random.default_rng([n, len(kind)])
    tex = np.clip(_content(kind, n, rng), 0, 255).astype(np.uint8)
    ob, osse = O.encode_blocks(tex, 7)
    gb, gsse = gsc.gsc_encode_blocks(ctx, torch.from_numpy(tex).cuda(), gsc.FMT_BC7)
    torch.cuda.synchronize()
    assert np.array_equal(gsse.cpu().numpy().astype(np.uint64), osse)
    assert np.array_equal(gb.cpu().numpy(), ob)


@pytest.mark.parametrize("n", [20_001, 200_003])
def test_pruned_search_in_wider_launches(ctx, O, n):
    """A warp per 32 blocks, in CTAs of four warps and (beyond 1280 blocks per SM) of ten, the last CTA partly empty:
    repeated blocks of every kind, against the oracle's coding of each."""
    from paper_2607_14513_gb300 import gsc
    rng = np.random.default_rng(n)
    kinds = ["ramp", "near", "line", "noise", "outliers", "extreme", "ties"]
    tex = np.clip(np.concatenate([_content(k, 101, rng) for k in kinds]), 0, 255).astype(np.uint8)
    ob, osse = O.encode_blocks(tex, 7)
    at = rng.integers(0, tex.shape[0], size=n)
    gb, gsse = gsc.gsc_encode_blocks(ctx, torch.from_numpy(tex[at]).cuda(), gsc.FMT_BC7)
    torch.cuda.synchronize()
    assert np.array_equal(gsse.cpu().numpy().astype(np.uint64), osse[at])
    assert np.array_equal(gb.cpu().numpy(), ob[at])
