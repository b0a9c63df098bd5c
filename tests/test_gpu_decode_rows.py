"""Scene decode of arbitrary BC7 blocks (every mode, rotation, index selection, partition and the reserved mode) against
the oracle, texel for texel, through the whole-block path and, with blocks that are only 8-byte aligned, the stream path;
with empty slots and a last pair of groups that is half missing. Bit-exact (Sec. III-B)."""
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


@pytest.mark.parametrize("offset", [0, 8])
@pytest.mark.parametrize("n", [1, 16, 17, 48, 5000])
def test_decode_scene_of_arbitrary_blocks(ctx, O, n, offset):
    from paper_2607_14513_gb300 import gsc
    rng = np.random.default_rng([n, offset])
    ng = (n + 15) // 16
    perm = np.full(ng * 16, -1, np.int32)
    perm[np.sort(rng.choice(ng * 16, size=n, replace=False))] = rng.permutation(n)
    _, _, table = gsc.gsc_encode(ctx, torch.zeros(n, 48, device="cuda"), torch.from_numpy(perm).cuda(),
                                 torch.ones(16, device="cuda"), gsc.FMT_BC7)
    blk = rng.integers(0, 256, size=(ng * 16, 16)).astype(np.uint8)
    mode = np.arange(ng * 16) % 9
    blk[:, 0] = np.where(mode == 8, 0, (blk[:, 0] & ~((2 << mode) - 1)) | (1 << mode))
    buf = torch.zeros(ng * 256 + 16, dtype=torch.uint8, device="cuda")
    at = buf[offset:offset + ng * 256]
    at.copy_(torch.from_numpy(blk.reshape(-1)))
    got = gsc.gsc_decode(ctx, table, at, torch.from_numpy(perm).cuda())
    torch.cuda.synchronize()
    ref = O.decode_blocks(blk, 7)[..., :3].reshape(ng, 16, 16, 3).transpose(0, 2, 1, 3).reshape(ng * 16, 16, 3)
    want = np.zeros((n, 16, 3), np.uint8)
    want[perm[perm >= 0]] = ref[perm >= 0]
    assert np.array_equal(got.cpu().numpy().reshape(n, 16, 3), want)
