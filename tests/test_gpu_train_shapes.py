"""The training step at the edges of its tiles (32 samples; more tiles than
CTAs) and with parameters, inputs and gradients off the alignment its vector
loads and stores need.  The summed gradient stays within 1e-4 of the largest
FP64 component, the loss within 1e-5 (BF16 operands split into two terms, FP32
sums: a few units of 2^-16 of FP32 arithmetic)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _fp64(w, x, y):
    w = w.double().requires_grad_()
    at, h = 0, x.double()
    for k, (i, o) in enumerate(((48, 64), (64, 64), (64, 112))):
        h = h @ w[at:at + i * o].reshape(o, i).T + w[at + i * o:at + i * o + o]
        h = torch.relu(h) if k < 2 else h
        at += i * o + o
    cls = (y.long() >> 5) * 28 + (y.long() & 31)
    ok = (y & 31) < 28
    loss = torch.nn.functional.cross_entropy(h[ok], cls[ok], reduction="sum")
    loss.backward()
    return float(loss.detach()), w.grad


@pytest.mark.parametrize("n", [1, 31, 32, 33, 200, 5000])
@pytest.mark.parametrize("shift", [0, 1])
def test_loss_and_gradient_at_tile_edges(n, shift):
    import ctypes

    from paper_1805_06019_gb300 import rlfc

    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    P = 14576
    w = (torch.randn(P, generator=g, device="cuda") * 0.15).to(torch.bfloat16)
    x = torch.randn((n + 7, 48), generator=g, device="cuda").to(torch.bfloat16)
    y = (torch.randint(0, 28, (n + 7,), generator=g, device="cuda") + 32 * torch.randint(0, 4, (n + 7,), generator=g, device="cuda")).to(torch.uint8)
    y[n // 2] = 31    # not a mode: skipped
    order = torch.randperm(n + 7, generator=g, device="cuda")[:n].to(torch.int32)

    def moved(t):   # the same values, `shift` elements past an aligned address
        b = torch.empty(t.numel() + 8, dtype=t.dtype, device="cuda")
        b[shift:shift + t.numel()] = t.reshape(-1)
        return b[shift:shift + t.numel()]

    wm, xm, gm = moved(w), moved(x), moved(torch.zeros(P, device="cuda"))
    loss = torch.zeros(1, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    rlfc._check(rlfc.lib().rlfc_mlp_loss_grad(p(wm), p(xm), p(y), p(order), n, p(gm), p(loss),
                                              torch.cuda.current_stream().cuda_stream))
    want_loss, want = _fp64(w, x[order.long()], y[order.long()])
    assert float((gm.double() - want).abs().max()) <= 1e-4 * max(float(want.abs().max()), 1e-30)
    assert abs(float(loss) - want_loss) <= 1e-5 * abs(want_loss) + 1e-6
