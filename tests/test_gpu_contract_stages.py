"""The global stage of the contraction on either side of its limits: one CTA
for up to 128 tiles while 4096 nodes and 16384 edges hold the batch, one
cluster for 128 tiles with more, the cooperative grid above, and 304 tiles,
where the local stage's threads change. Nuclei tiles have about 40 nodes a
tile and noise about 60, so the heights below cross the node limit between
64 and 112 tiles. Against the directional sweeps, and the oracle at two
sizes (whole numbers: no tolerance)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def images(rt, H, W):
    g = torch.Generator(device="cuda").manual_seed(H + W)
    r, c = torch.arange(H, device="cuda")[:, None], torch.arange(W, device="cuda")[None]
    rnd = lambda hi: torch.randint(0, hi, (H, W), generator=g, device="cuda")
    yield "nuclei", rt.config2_tile(H + W, H=H, W=W)
    yield "noise", rnd(256).to(torch.uint8)
    yield "few values", (rnd(5) * 50).to(torch.uint8)
    yield "dots", (((r & 1) & (c & 1)) * (200 + rnd(50)) + 3).to(torch.uint8)
    yield "smooth", ((r * 5 + c * 3) % 251 // 3 + rnd(6)).to(torch.uint8)


def check(rt, H, W, exact=False):
    g = torch.Generator(device="cuda").manual_seed(7)
    for name, I in images(rt, H, W):
        marks = [torch.where(torch.rand((H, W), generator=g, device="cuda") < q, I, torch.zeros_like(I))
                 for q in (1e-2, 1e-4)]
        for h in (0, 30):
            assert torch.equal(rt.reconstruct(I, h_offset=h), rt.reconstruct(I, h_offset=h, variant=rt.RT_RASTER)), (name, h)
        for J in marks:
            got = rt.reconstruct(I, J)
            assert torch.equal(got, rt.reconstruct(I, J, variant=rt.RT_RASTER)), name
            if exact:
                assert np.array_equal(got.cpu().numpy(), oracle.recon(J.cpu().numpy(), I.cpu().numpy(), 8)), name


@pytest.mark.parametrize("rows", range(7, 17))
def test_up_to_128_tiles(rt, rows):
    check(rt, 64 * rows, 512, exact=rows == 13)


@pytest.mark.parametrize("H,W", [(512, 1088), (1024, 513), (640, 704), (1088, 1088), (1150, 1100), (1152, 1152)])
def test_around_128_and_304_tiles(rt, H, W):
    check(rt, H, W, exact=(H, W) == (640, 704))
