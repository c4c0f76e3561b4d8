"""The context's workspace and CUDA graphs: a call captured on a context that
was reserved with less than it needs grows the workspace without ending the
capture, and a graph captured before the workspace grew still replays on the
block that it was captured with. Outputs against an eager call on a context of
its own (whole numbers: no tolerance)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def operations(rt, H, W):
    """name -> (call on a context that returns its outputs, bytes per pixel
    that the operation once needed)"""
    img = rt.config2_tile(11, H=H, W=W)
    o = rt.segment_batch([img])[0]
    binary = (o["R"] < 80).to(torch.uint8)
    u8, i32 = torch.empty_like(img), torch.empty_like(o["L"])
    return {
        "reconstruct": (lambda c: [rt.reconstruct(img, out=u8, ctx=c)], 2.2),
        "fill_holes": (lambda c: [rt.fill_holes(binary, out=u8, ctx=c)], 0.3),
        "watershed": (lambda c: [rt.watershed(o["L"], o["D"], out=i32, ctx=c)], 37.1),
    }


def captured(call, ctx):
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        outs = call(ctx)
    return g, outs


@pytest.mark.parametrize("name", ["reconstruct", "fill_holes", "watershed"])
@pytest.mark.parametrize("H,W", [(1024, 1024), (1500, 2111)])
def test_capture_on_a_small_reservation(rt, name, H, W):
    call, per_px = operations(rt, H, W)[name]
    own = rt.Context()
    want = [t.clone() for t in call(own)]
    torch.cuda.synchronize()
    ctx = rt.Context(workspace_bytes=int(per_px * H * W))
    g, outs = captured(call, ctx)
    for t in outs:
        t.fill_(7)
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
    ctx.close()
    own.close()


def test_graph_outlives_the_growth_of_its_workspace(rt):
    small, big = rt.config2_tile(1, H=512, W=640), rt.config2_tile(2, H=3000, W=2900)
    want, want_big = rt.segment_batch([small])[0], rt.segment_batch([big])[0]
    ctx = rt.Context()
    rt.segment_batch([small], ctx=ctx)                     # eager: allocates the workspace
    outs = rt.segment_batch([small], ctx=ctx)
    g, _ = captured(lambda c: rt.segment_batch([small], outputs=outs, ctx=c), ctx)
    for k in range(3):
        ctx_bytes = ctx.workspace_bytes()
        got = rt.segment_batch([big[:1000 + 1000 * k]], ctx=ctx)[0]   # eager: grows it
        assert ctx.workspace_bytes() > ctx_bytes
        junk = torch.full((ctx.workspace_bytes(),), 255, dtype=torch.uint8, device="cuda")
        for o in outs:
            o["L"].fill_(-7)
        g.replay()
        torch.cuda.synchronize()
        for name in ("R", "F", "L", "D", "n_kept"):
            assert torch.equal(outs[0][name], want[name]), name
        del junk
    assert all(torch.equal(got[k], want_big[k]) for k in ("R", "F", "L", "D", "n_kept"))
    ctx.close()


def test_growth_between_two_calls_of_one_capture(rt):
    a, b = rt.config2_tile(3, H=200, W=333), rt.config2_tile(4, H=1100, W=1300)
    want = [rt.reconstruct(a), rt.reconstruct(b), rt.reconstruct(a, h_offset=60)]
    ctx = rt.Context()
    g, outs = captured(lambda c: [rt.reconstruct(a, ctx=c), rt.reconstruct(b, ctx=c),
                                  rt.reconstruct(a, h_offset=60, ctx=c)], ctx)
    for _ in range(2):
        for t in outs:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for x, y in zip(outs, want))
    ctx.close()
