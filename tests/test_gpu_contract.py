"""GPU tests of the reconstruction by contraction (RT_AUTO, 8-connected):
sizes around its 64 x 64 tiles, markers given and derived, images that make
its clusters, chains and ties extreme, unaligned views, and batches, against
the CPU oracle and the directional sweeps (whole numbers: no tolerance)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(1, 1), (1, 200), (200, 1), (2, 2), (63, 64), (64, 64), (64, 65), (65, 63), (128, 128), (127, 193), (300, 500)]


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def images(H, W, rng):
    """name -> mask"""
    r, c = np.mgrid[0:H, 0:W]
    return {
        "noise": rng.integers(0, 256, (H, W)),
        "two values": rng.integers(0, 2, (H, W)) * 255,
        "few values": rng.integers(0, 4, (H, W)) * 3,
        "flat": np.full((H, W), 200),
        "zero": np.zeros((H, W)),
        "checkerboard": ((r + c) & 1) * 255,
        "dots": ((r & 1) & (c & 1)) * 250 + 3,
        "falling": 255 - np.minimum(r + c, 255),
        "rows": np.where(r % 2 == 0, 250 - (c % 200), 5),
        "nuclei": synth.config2_tile(H * 7 + W, H=H, W=W),
    }


@pytest.mark.parametrize("H,W", SIZES)
def test_contraction_equals_the_oracle(rt, H, W):
    rng = np.random.default_rng(H * 1000 + W)
    for name, I in images(H, W, rng).items():
        I = I.astype(np.uint8)
        d = dev(I)
        point = np.zeros_like(I)
        point[rng.integers(0, H), rng.integers(0, W)] = 255
        for J in (np.minimum(I, rng.integers(0, 256, (H, W))).astype(np.uint8), np.minimum(point, I)):
            assert np.array_equal(host(rt.reconstruct(d, dev(J))), oracle.recon(J, I, 8)), name
        for h in (0, 30, 255):
            J = host(rt.marker(d, h))
            assert np.array_equal(host(rt.reconstruct(d, h_offset=h)), oracle.recon(J, I, 8)), (name, h)


@pytest.mark.parametrize("n", [65, 130, 257])
def test_corridors(rt, n):
    """One long path through every tile many times over."""
    for I in (synth.spiral(n, low=0), synth.serpentine(n, n), synth.serpentine(n, n).T.copy()):
        J = np.zeros_like(I)
        J[0, 0] = I[0, 0]
        assert np.array_equal(host(rt.reconstruct(dev(I), dev(J))), oracle.recon(J, I, 8))


def test_marker_above_the_mask_and_views(rt):
    """EMARKER is raised as by the sweeps; odd strides and offsets."""
    rng = np.random.default_rng(3)
    I = rng.integers(0, 200, (140, 260)).astype(np.uint8)
    J = I.copy()
    J[100, 200] = 255
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    for off in (0, 1, 2, 3):
        wide = torch.zeros((140, 271), dtype=torch.uint8, device="cuda")
        mask = wide[:, off:off + 260]
        mask.copy_(dev(I))
        out = torch.full((140, 283), 77, dtype=torch.uint8, device="cuda")
        got = rt.reconstruct(mask, dev(J), out=out[:, off:off + 260], status=st)
        assert int(host(st)[0]) == rt.RT_EMARKER
        assert np.array_equal(host(got), oracle.recon(np.minimum(I, J), I, 8))
        rest = host(out)
        assert (rest[:, :off] == 77).all() and (rest[:, off + 260:] == 77).all()
        rt.reconstruct(mask, status=st)
        assert int(host(st)[0]) == rt.RT_OK


def test_in_place_marker_and_repeats(rt):
    I = synth.config2_tile(9, H=333, W=470)
    J = np.where(np.random.default_rng(1).random(I.shape) < 0.01, I, 0).astype(np.uint8)
    want = oracle.recon(J, I, 8)
    d = dev(I)
    for _ in range(3):
        j = dev(J)
        rt.reconstruct(d, j, out=j)
        assert np.array_equal(host(j), want)


@pytest.mark.parametrize("seed", [1, 2])
def test_large_random_tiles_equal_the_sweeps(rt, seed):
    """Against the directional sweeps, at sizes with thousands of tiles."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    for H, W in ((1500, 2111), (4096, 1024)):
        for hi in (2, 16, 256):
            I = torch.randint(0, hi, (H, W), generator=g, device="cuda").to(torch.uint8)
            J = torch.minimum(I, torch.randint(0, hi, (H, W), generator=g, device="cuda").to(torch.uint8))
            J = torch.where(torch.rand((H, W), generator=g, device="cuda") < 1e-4, J, torch.zeros_like(J))
            assert torch.equal(rt.reconstruct(I, J), rt.reconstruct(I, J, variant=rt.RT_RASTER))
    I = rt.config2_tile(seed, H=2900, W=3001)
    assert torch.equal(rt.reconstruct(I), rt.reconstruct(I, variant=rt.RT_RASTER))


def test_batch_of_uneven_tiles_equals_the_sweeps(rt):
    shapes = [(1, 70), (64, 64), (700, 1031), (65, 129), (333, 64), (1024, 900)]
    imgs = [rt.synth_tile(H, W, 70 + i, 1 + H * W // 5000) for i, (H, W) in enumerate(shapes)]
    for a, b in zip(rt.segment_batch(imgs), rt.segment_batch(imgs, rt.SegParams(variant=rt.RT_RASTER))):
        for k in ("R", "F", "L", "D", "n_kept", "status"):
            assert torch.equal(a[k], b[k]), k
