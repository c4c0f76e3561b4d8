"""The picker's tensor-core backward on large batches: a batch four times as
large takes at most four times as long (the kernel that adds up the gradients
lost its cache to the kernel before it from about 5000 samples on: 40 us for
4096, 205 for 16384)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_backward_grows_no_faster_than_the_batch():
    import paper_1405_7958_gb300 as rt
    pk = rt.Picker(seed=1)
    us = {}
    for B in (4096, 16384):
        g = torch.Generator().manual_seed(B)
        x = (torch.randn(B, 24, generator=g) * 50).cuda()
        y = torch.randint(0, 3, (B,), generator=g).to(torch.int32).cuda()
        logits, act, _ = pk.forward(x, with_act=True, tensor_cores=True)
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                pk.backward(x, act, logits, y, tensor_cores=True)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) / 20 * 1e3)
        us[B] = min(times[1:])
    assert us[16384] < 4 * us[4096], us
