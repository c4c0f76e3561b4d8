"""The distance transform on bit tiles at the limits of its near stage:
distances around 31 and 32, tiles filled to about three quarters with little
background, tiles without any, images without background, and images of few
and of many tiles (another number of threads per tile)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def same(rt, m):
    got = rt.edt(torch.from_numpy(np.ascontiguousarray(m)).cuda())
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), oracle.edt(m))


@pytest.mark.parametrize("gap", [30, 31, 32, 33, 64])
def test_distances_around_the_reach(rt, gap):
    m = np.ones((3 * gap + 5, 4 * gap + 9), np.uint8)
    m[gap, :: 2 * gap + 1] = 0
    m[::gap, 2 * gap] = 0
    same(rt, m)
    m = np.ones((200, 230), np.uint8)
    m[100, 115] = 0
    same(rt, m)


@pytest.mark.parametrize("fill", [0.70, 0.7499, 0.7501, 0.80, 0.97])
def test_tiles_filled_to_three_quarters(rt, fill):
    rng = np.random.default_rng(int(fill * 1e4))
    m = np.ones((192, 256), np.uint8)
    cut = int(round(64 * 64 * (1 - fill)))
    for ty in range(3):
        for tx in range(4):
            t = np.ones(64 * 64, np.uint8)
            t[:cut] = 0                          # the background in the tile's first rows
            if (ty + tx) % 3 == 2:
                rng.shuffle(t)                   # or all over it
            m[64 * ty:64 * ty + 64, 64 * tx:64 * tx + 64] = t.reshape(64, 64)
    same(rt, m)


def test_no_background_and_many_tiles(rt):
    same(rt, np.ones((70, 130), np.uint8))
    rng = np.random.default_rng(3)
    m = (rng.random((4200, 4161)) < 0.3).astype(np.uint8)   # 66 x 66 tiles
    m[1000:1400, 700:1900] = 1
    same(rt, m)


def test_a_bound_on_propagations_leaves_the_transform_alone(rt):
    """A stripe of foreground 256 columns wide and 32768 rows high: the far
    stage's walk over its empty segments takes some of the blocks milliseconds
    while the others wait at the barrier. rt_set_limits bounds propagations
    only, so the distances are exact and the status is RT_OK."""
    H, W, c0, n = 32768, 4096, 1024, 256
    fg = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    fg[:, c0:c0 + n] = 1
    c = torch.arange(n, device="cuda", dtype=torch.int32)
    want = torch.minimum(c + 1, n - c) ** 2
    st = torch.full((1,), 99, dtype=torch.int32, device="cuda")
    ctx = rt.Context()
    ctx.set_limits(timeout_ms=1)
    d = rt.edt(fg, status=st, ctx=ctx)
    assert int(st.item()) == rt.RT_OK
    assert bool((d[:, c0:c0 + n] == want).all())
    assert int(d.sum(dtype=torch.int64).item()) == H * int(want.sum().item())
    ctx.close()
