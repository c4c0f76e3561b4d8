"""The tensor-core forward and backward of the picker on inputs that are not
16-byte aligned give the bits of the aligned ones, at batches that fill no,
some and all rows of a block of 128 samples."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def off_by(t, k):
    """The same values, k elements into a longer buffer."""
    buf = torch.empty(t.numel() + k, dtype=t.dtype, device="cuda")
    buf[k:] = t.reshape(-1)
    return buf[k:].view(t.shape)


@pytest.mark.parametrize("B", [1, 7, 127, 128, 129, 300])
def test_unaligned_inputs_give_the_same_bits(B):
    import paper_1405_7958_gb300 as rt
    g = torch.Generator().manual_seed(B)
    x = torch.randn(B, 24, generator=g).cuda()
    y = torch.randint(0, 3, (B,), generator=g).to(torch.int32).cuda()
    pk = rt.Picker(seed=3)
    want = []
    for k in (0, 1):
        pk.wb = off_by(pk.wb, k)
        xk = off_by(x, k)
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        logits, act, pick = pk.forward(xk, with_act=True, tensor_cores=True, status=st)
        pk.grad.zero_()
        grad, loss = pk.backward(xk, off_by(act, k), off_by(logits, k), off_by(y, k), tensor_cores=True, status=st)
        torch.cuda.synchronize()
        assert int(st[0]) == 0
        got = [v.clone() for v in (logits, act, pick, grad, loss)]
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(got, want))
