"""GPU tests of hole filling and labeling on runs of bit rows (and of the pixel
union-find that labels small images): sizes around
their 64 x 64 tiles, both connectivities, images with the most runs and pairs
a tile can hold, holes and components across many tiles, against the CPU
oracle (whole numbers: no tolerance)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(1, 1), (1, 130), (130, 1), (63, 65), (64, 64), (65, 64), (128, 129), (191, 193), (300, 517)]


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def masks(H, W):
    r, c = np.mgrid[0:H, 0:W]
    out = {"empty": np.zeros((H, W)), "full": np.ones((H, W)), "checkerboard": (r + c) & 1, "columns": c & 1,
           "rows": r & 1, "combs": ((c & 1) | (r % 16 == 0)), "dots": (r & 1) & (c & 1),
           "rings": (np.maximum(abs(r - H // 2), abs(c - W // 2)) // 3) & 1,
           "frame": (r == 0) | (c == 0) | (r == H - 1) | (c == W - 1),
           "inner frame": ((abs(r - H // 2) == max(H // 2 - 2, 0)) | (abs(c - W // 2) == max(W // 2 - 2, 0))) &
                          (abs(r - H // 2) <= H // 2 - 2) & (abs(c - W // 2) <= W // 2 - 2),
           "spiral": synth.spiral(max(H, W), low=0, high=1)[:H, :W], "diagonals": ((r - c) % 5 == 0)}
    for p in (100, 300, 500, 600, 850):
        out[f"random {p}"] = synth.random_binary(H, W, H * 31 + W + p, p)
    return {k: np.asarray(v).astype(np.uint8) for k, v in out.items()}


def test_chain_labels_of_dense_masks(rt):
    """The chain labels bit planes at every size: masks with the most runs,
    thresholded from two grey values (dark = foreground)."""
    for H, W in ((1, 130), (64, 65), (191, 193)):
        for name, m in masks(H, W).items():
            I = np.where(m > 0, 20, 220).astype(np.uint8)
            out = rt.segment_batch([dev(I)], rt.SegParams(min_area=2, max_area=10 ** 6))[0]
            want = oracle.chain(I, min_area=2, max_area=10 ** 6)
            for k in ("F", "L", "D"):
                assert np.array_equal(host(out[k]), want[k]), (name, k)


@pytest.mark.parametrize("conn", [4, 8])
@pytest.mark.parametrize("H,W", SIZES)
def test_fill_and_label_equal_the_oracle(rt, H, W, conn):
    n = torch.zeros(1, dtype=torch.int32, device="cuda")
    for name, m in masks(H, W).items():
        for b in (m, 1 - m):
            d = dev(b * 255)
            assert np.array_equal(host(rt.fill_holes(d, conn=conn)), oracle.fill_holes(b, conn)), name
            for lo, hi in ((0, 2 ** 31 - 1), (2, 60)):
                want, kept = oracle.label_area(b, lo, hi, conn, return_count=True)
                assert np.array_equal(host(rt.label_area(d, lo, hi, conn=conn, n_kept=n)), want), (name, lo)
                assert int(host(n)[0]) == kept


def test_unaligned_views(rt):
    m = synth.random_binary(150, 201, 3, 550)
    for off in (1, 2, 3):
        src = torch.full((150, 230), 9, dtype=torch.uint8, device="cuda")[:, off:off + 201]
        src.copy_(dev(m))
        F = torch.full((150, 219), 7, dtype=torch.uint8, device="cuda")
        L = torch.full((150, 219), 7, dtype=torch.int32, device="cuda")
        rt.fill_holes(src, conn=4, out=F[:, off:off + 201])
        rt.label_area(src, 1, 500, out=L[:, off:off + 201])
        assert np.array_equal(host(F)[:, off:off + 201], oracle.fill_holes(m, 4))
        assert np.array_equal(host(L)[:, off:off + 201], oracle.label_area(m, 1, 500, 8))
        for x in (host(F), host(L)):
            assert (x[:, :off] == 7).all() and (x[:, off + 201:] == 7).all()


def test_many_tiles(rt):
    """Thousands of tiles: one background and one component across all of
    them, and the tiles' order must not matter."""
    r, c = np.mgrid[0:3000, 0:3301]
    grid = ((r % 97 < 2) | (c % 89 < 2)).astype(np.uint8)          # meshes: every cell a hole
    grid[1500:, 1550] = 0                                            # some of them open
    for m in (grid, 1 - grid, synth.random_binary(3000, 3301, 8, 420)):
        assert np.array_equal(host(rt.fill_holes(dev(m))), oracle.fill_holes(m, 4))
        for conn in (4, 8):   # large enough for the union-find over runs
            got = host(rt.label_area(dev(m), 2, 2 ** 31 - 1, conn=conn))
            assert np.array_equal(got, oracle.label_area(m, 2, 2 ** 31 - 1, conn)), conn


def test_tiles_around_a_warps_share_of_memory(rt):
    """Tiles of 100 to 1000 runs side by side in an image large enough for
    several tiles per block: 384 runs (local stages) and 640 (labels) fit a
    warp's share, the others take another way."""
    rng = np.random.default_rng(5)
    p = np.kron(rng.uniform(0.03, 0.5, (47, 48)), np.ones((64, 64)))[:3000, :3070]
    m = (rng.random(p.shape) < p).astype(np.uint8)
    for conn in (4, 8):
        assert np.array_equal(host(rt.fill_holes(dev(m), conn=conn)), oracle.fill_holes(m, conn)), conn
        assert np.array_equal(host(rt.fill_holes(dev(1 - m), conn=conn)), oracle.fill_holes(1 - m, conn)), conn
        got = host(rt.label_area(dev(m), 2, 400, conn=conn))
        assert np.array_equal(got, oracle.label_area(m, 2, 400, conn)), conn
