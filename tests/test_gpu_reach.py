"""The chain without R among its outputs: R is then not computed, only where
it is below the threshold (connectivity to seeds inside {I >= threshold}).
Same labels, distances, filled masks and counts as the oracle's and as the
call that returns R, at the ends of the threshold's and the offset's ranges,
on ragged tiles, noise of many runs per tile, flat images, batches, an image
of many tiles, and with unaligned rows."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def rt():
    import paper_1405_7958_gb300 as rt
    return rt


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def same_as_with_R(rt, images, **kw):
    p = rt.SegParams(**kw)
    d = [dev(i) for i in images]
    want = rt.segment_batch(d, p)
    got = rt.segment_batch(d, p, want_recon=False)
    for w, g in zip(want, got):
        assert "R" not in g
        for k in ("F", "L", "D", "n_kept", "status"):
            assert np.array_equal(host(w[k]), host(g[k])), (k, kw)
    return got


def images(H, W, rng):
    yield synth.config2_tile(17 + H, H=H, W=W)
    yield rng.integers(0, 256, (H, W)).astype(np.uint8)
    yield np.clip(rng.normal(80, 12, (H, W)), 0, 255).astype(np.uint8)   # specks around the threshold
    yield np.full((H, W), 79, np.uint8)
    yield np.full((H, W), 200, np.uint8)
    rr, cc = np.mgrid[0:H, 0:W]
    yield (((rr % 9 < 2) | (cc % 11 < 2)) * 90 + (rr + cc) % 40).astype(np.uint8)   # a mesh, its cells dark


@pytest.mark.parametrize("H,W", [(1, 1), (1, 130), (64, 64), (65, 63), (127, 200), (300, 333)])
def test_chain_without_R_equals_the_oracle(rt, H, W):
    rng = np.random.default_rng(H + W)
    for I in images(H, W, rng):
        I = I.astype(np.uint8)
        o = rt.segment_batch([dev(I)], want_recon=False)[0]
        c = oracle.chain(I)
        for k in ("F", "L", "D"):
            assert np.array_equal(host(o[k]), c[k]), k
        assert int(host(o["n_kept"])[0]) == c["n_kept"]


@pytest.mark.parametrize("threshold", [0, 1, 80, 127, 128, 129, 255, 256])
@pytest.mark.parametrize("h", [0, 1, 30, 255])
def test_thresholds_and_offsets(rt, threshold, h):
    rng = np.random.default_rng(threshold + h)
    ims = [i.astype(np.uint8) for i in images(150, 171, rng)]
    same_as_with_R(rt, ims, threshold=threshold, h_offset=h, conn_fill=8 if h == 1 else 4)


def test_many_tiles_and_unaligned_rows(rt):
    rng = np.random.default_rng(9)
    big = np.clip(rng.normal(85, 15, (3000, 3301)), 0, 255).astype(np.uint8)
    big[:, 1700:] = synth.config2_tile(3, H=3000, W=1601)
    same_as_with_R(rt, [big])
    buf = torch.zeros((500, 701), dtype=torch.uint8, device="cuda")
    buf[:, 3:650] = dev(synth.config2_tile(8, H=500, W=647))
    view = buf[:, 3:650]
    a = rt.segment_batch([view])[0]
    b = rt.segment_batch([view], want_recon=False)[0]
    assert all(np.array_equal(host(a[k]), host(b[k])) for k in ("F", "L", "D", "n_kept"))


def test_learned_call_and_mixed_outputs(rt):
    """A tile that asks for R beside one that does not; a captured call."""
    ims = [dev(synth.config2_tile(60 + k, H=400 + 64 * k, W=500)) for k in range(2)]
    want = rt.segment_batch(ims)
    outs = rt.segment_batch(ims, want_recon=False)
    outs[0]["R"] = torch.empty_like(ims[0])
    rt.segment_batch(ims, outputs=outs)
    assert np.array_equal(host(outs[0]["R"]), host(want[0]["R"]))
    for w, g in zip(want, outs):
        assert all(np.array_equal(host(w[k]), host(g[k])) for k in ("F", "L", "D", "n_kept"))
    outs = rt.segment_batch(ims, want_recon=False)
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        rt.segment_batch(ims, outputs=outs)
    s.synchronize()
    with torch.cuda.graph(g, stream=s):
        rt.segment_batch(ims, outputs=outs)
    for o in outs:
        o["L"].fill_(-7)
    g.replay()
    for w, o in zip(want, outs):
        assert np.array_equal(host(w["L"]), host(o["L"]))
