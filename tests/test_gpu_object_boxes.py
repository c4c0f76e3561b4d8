"""GPU parity of the per-object steps at the limits of their box sizes: the
watershed of one warp (up to 640 cells of the box with its border), of four
warps (2944) and of a block (6968; sweeps in shared memory up to 4096 pixels
of the box, in global memory above), the features of one warp (8192 pixels, sides of 1024)
and of a block; distance maps with wide levels, with few, with values that
no distance map of the object has, and images whose rows are not aligned.
Labels, basins and integer-valued features are compared exactly; the other
features within 1e-12 relative, as for the chain's outputs."""
import numpy as np
import pytest

import oracle
from test_gpu_objects import check_features, check_watershed, dev, host, rt  # noqa: F401  (rt: fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def boxes(shapes, W, holes=0.0, seed=0):
    """Objects with the given bounding boxes, below one another; `holes` of
    their inner pixels taken out (still one object each: rows stay joined
    by the first column, the box by its last row and column)."""
    rng = np.random.default_rng(seed)
    H = sum(h + 1 for h, _ in shapes)
    m = np.zeros((H, W), np.uint8)
    r = 0
    for k, (h, w) in enumerate(shapes):
        c = (7 * k) % (W - w + 1)
        box = (rng.random((h, w)) >= holes).astype(np.uint8)
        box[:, 0] = 1
        box[-1, :] = 1
        box[0, -1] = 1
        m[r:r + h, c:c + w] = box
        r += h + 1
    L = oracle.label_area(m, 1, 10 ** 9)
    return L


def distances(L, kind, seed=1):
    rng = np.random.default_rng(seed)
    if kind == "edt":
        D = oracle.edt((L >= 0).astype(np.uint8))
    elif kind == "flat":
        D = np.full(L.shape, 3, np.int32)
    elif kind == "noise":
        D = rng.integers(0, 6, L.shape)
    elif kind == "ramp":
        D = np.add.outer(np.arange(L.shape[0]), 2 * np.arange(L.shape[1])) % 97
    else:   # values beyond what the small boxes sort
        D = rng.integers(0, 2 ** 31 - 1, L.shape)
    return np.where(L >= 0, D, 0).astype(np.int32)


# (h + 2) (w + 2) = 640, 2944, 6960 and next to them; h w = 4096 and next to it
SHAPES = [(18, 30), (30, 18), (14, 38), (19, 30), (1, 211), (1, 212), (62, 44), (44, 62), (21, 126), (63, 44), (1, 979),
          (64, 64), (64, 65), (1, 1), (2, 2), (126, 3), (78, 85), (79, 85), (5, 960)]


@pytest.mark.parametrize("kind", ["edt", "flat", "noise", "ramp", "large"])
@pytest.mark.parametrize("h", [0, 2, 40])
def test_watershed_box_limits(rt, kind, h):  # noqa: F811
    L = boxes(SHAPES, 1000, holes=0.3, seed=h)
    check_watershed(rt, L, distances(L, kind), h)


@pytest.mark.parametrize("kind", ["flat", "noise", "edt"])
def test_watershed_full_boxes(rt, kind):  # noqa: F811
    L = boxes(SHAPES, 1001)
    check_watershed(rt, L, distances(L, kind), 1)


@pytest.mark.parametrize("W", [1024, 1027])
def test_feature_box_limits(rt, W):  # noqa: F811
    shapes = [(8, 1024), (8, 1023), (9, 1000), (9, 911), (1, 1024), (90, 91), (91, 91), (256, 32), (256, 33), (31, 31),
              (5, 32), (5, 62), (5, 63), (1, 1), (2, 1), (1024, 8), (1025, 2)]
    L = boxes(shapes, W, holes=0.2, seed=W)
    I = np.random.default_rng(W).integers(0, 256, L.shape).astype(np.uint8)
    check_features(rt, L, I)


@pytest.mark.parametrize("W", [1, 2, 3, 5, 127, 129, 260, 1023, 1025, 2050])
def test_enumeration_of_ragged_rows(rt, W):  # noqa: F811
    """Many small objects, rows that wrap inside a lane's four pixels."""
    rng = np.random.default_rng(W)
    H = min(20000, max(7, 40000 // W))
    L = oracle.label_area((rng.random((H, W)) < 0.35).astype(np.uint8), 1, 10 ** 9)
    I = rng.integers(0, 256, (H, W)).astype(np.uint8)
    check_features(rt, L, I)
    check_watershed(rt, L, distances(L, "edt"), 0)
    # the same labels in rows of another stride, off the 16-byte alignment
    for stride, first in ((W + 5, 1), (W + 4 + -W % 4, 0)):
        B = torch.full((H, stride), 7, dtype=torch.int32, device="cuda")
        B[:, first:first + W] = dev(L)
        D = distances(L, "noise")
        out = torch.full((H, stride), -7, dtype=torch.int32, device="cuda")
        rt.watershed(B[:, first:first + W], dev(D), 1, out=out[:, first:first + W])
        assert np.array_equal(host(out)[:, first:first + W], oracle.watershed(L, D, 1))
        rest = np.delete(host(out), np.s_[first:first + W], axis=1)
        assert (rest == -7).all()
