"""The picker beside the chain: a lone tile under the learned policy with the
default (raster) classes, whose picks are computed on the context's own stream
while the chain runs. The picks and outputs are those of the same call where
nothing overlaps."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def dark_picker(rt, ctx):
    """A hand-set network on the fraction f of pixels below 80 alone: logits
    (0.5, f, -1), so class 1 where more than half of the image is dark (all
    weights exact in bf16)."""
    pk = rt.Picker(seed=0)
    w = torch.zeros(pk.NPARAM, dtype=torch.float32)
    w[16] = 1.0                      # W1[0][16]
    w[1600] = 1.0                    # W2[0][0]
    w[5760 + 64] = 1.0               # W3[1][0]
    w[5952:5955] = torch.tensor([0.5, 0.0, -1.0])
    pk.master.copy_(w)
    pk.wb = pk.master.to(torch.bfloat16).view(torch.int16).contiguous()
    pk.norm = torch.cat([torch.zeros(24), torch.ones(24)]).cuda()
    pk.attach(ctx)
    return pk


def tile(rt, dark, H=1500, W=1300):
    img = rt.config2_tile(5, H=H, W=W)
    if dark:
        img[: 3 * H // 4] = img[: 3 * H // 4] // 4
    return img


@pytest.mark.parametrize("name", ["F", "R"])
@pytest.mark.parametrize("dark", [False, True])
def test_output_over_the_image(rt, name, dark):
    """F over the image is 0 and 1, all dark: the picks are the image's all
    the same, and the outputs those of the call with buffers of their own."""
    img = tile(rt, dark)
    ctx = rt.Context()
    pk = dark_picker(rt, ctx)
    p = rt.SegParams(policy=1)
    for _ in range(3):
        want = rt.segment_batch([img], p, ctx=ctx, want_recon=name == "R")
        assert rt.last_picks(ctx) == [1 if dark else 0]
        buf = img.clone()
        outs = rt.segment_batch([img], p, ctx=ctx, want_recon=name == "R")
        outs[0][name] = buf
        rt.segment_batch([buf], p, outputs=outs, ctx=ctx)
        assert rt.last_picks(ctx) == [1 if dark else 0]
        torch.cuda.synchronize()
        for k in want[0]:
            assert torch.equal(want[0][k], outs[0][k]), k
    ctx.close()


@pytest.mark.parametrize("want_recon", [False, True])
def test_captured_call_captures_both_streams(rt, want_recon):
    """Two inputs through one graph: picks and outputs of the eager calls."""
    ctx = rt.Context()
    pk = dark_picker(rt, ctx)
    p = rt.SegParams(policy=1)
    imgs = [tile(rt, False), tile(rt, True)]
    want = [rt.segment_batch([i], p, ctx=ctx, want_recon=want_recon)[0] for i in imgs]
    img = imgs[0].clone()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        outs = rt.segment_batch([img], p, ctx=ctx, want_recon=want_recon)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        rt.segment_batch([img], p, outputs=outs, ctx=ctx)
    for k in (1, 0, 1):
        img.copy_(imgs[k])
        for o in outs[0].values():
            o.fill_(77)
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert rt.last_picks(ctx) == [k]
        for name, t in want[k].items():
            assert torch.equal(t, outs[0][name]), name
    ctx.close()


@pytest.mark.parametrize("want_recon", [False, True])
def test_last_tile_of_33_is_a_chunk_of_its_own(rt, want_recon):
    """32 tiles run the plain schedule; the 33rd forks, in the same
    workspace. Plain calls of one tile each give the same outputs."""
    shapes = [(150 + 17 * (i % 7), 130 + 29 * (i % 5)) for i in range(32)] + [(1500, 1300)]
    for dark in (False, True):
        imgs = [rt.config2_tile(100 + i, H=H, W=W) for i, (H, W) in enumerate(shapes[:32])] + [tile(rt, dark)]
        ctx = rt.Context()
        pk = dark_picker(rt, ctx)
        for _ in range(2):
            outs = rt.segment_batch(imgs, rt.SegParams(policy=1), ctx=ctx, want_recon=want_recon)
            assert rt.last_picks(ctx) == [1 if dark else 0]
        for i, o in zip(imgs, outs):
            w = rt.segment_batch([i], want_recon=want_recon)[0]
            torch.cuda.synchronize()
            for name, t in w.items():
                assert torch.equal(t, o[name]), name
        ctx.close()
