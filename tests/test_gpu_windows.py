"""Batches of cameras blended from decoded views: groups cut by the shared
memory their shift spreads need, window rows wider than the compile-time
pitch, rows of every alignment.  A view's pixels are the same bits whatever
batch, group or store path rendered it, and meet the oracle's bound (1e-3 on
the [0, 1] scale, FP32 against FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,spread", [(64, 32, 0.5), (61, 37, 3.0), (130, 18, 12.0), (70, 33, 90.0)])
def test_batches_do_not_change_a_view(W, H, spread):
    from paper_1805_06019_gb300 import rlfc

    U, V, n = 4, 3, 90
    lf = lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=60 + W)
    data = oracle.encode(lf, U, V, B=4, L=2, c=[0, 4], tau_p=2, tau_b=16)
    ref = oracle.Stream(data).decode_all()
    rng = np.random.default_rng(W)
    uv = np.stack([rng.uniform(-0.2, 1.4, n), rng.uniform(0.8, V - 0.8, n)], 1).astype(np.float32)
    uv[:6] = [[0, 0], [3, 2], [1, 1.5], [2.5, 1], [0, 2], [1, 1]]
    d = rng.uniform(-spread, spread, n).astype(np.float32)
    st = rlfc.Stream(data)
    duv, dd = torch.from_numpy(uv).cuda(), torch.from_numpy(d).cuda()
    whole = st.render(duv, dd, W, H)
    u8 = st.render(duv, dd, W, H, u8=True)
    parts = torch.cat([st.render(duv[i:i + 5].contiguous(), dd[i:i + 5].contiguous(), W, H) for i in range(0, n, 5)])
    assert torch.equal(whole, parts)
    # decoded on demand, one camera and two at a time (footprints apart when
    # the shifts are large)
    ones = torch.cat([st.render(duv[i:i + 1].contiguous(), dd[i:i + 1].contiguous(), W, H) for i in range(20)])
    twos = torch.cat([st.render(duv[i:i + 2].contiguous(), dd[i:i + 2].contiguous(), W, H) for i in range(0, 20, 2)])
    assert torch.equal(whole[:20], ones) and torch.equal(whole[:20], twos)
    # other sizes: the same from decoded views (as a large batch) and on demand
    for w, h in ((W // 2 + 3, H // 3 + 1), (W + 17, 2 * H)):
        reps = 1 + 450_000 // (n * W * H)
        many = st.render(duv.repeat(reps, 1), dd.repeat(reps), w, h)
        few = torch.cat([st.render(duv[i:i + 2].contiguous(), dd[i:i + 2].contiguous(), w, h) for i in range(0, 20, 2)])
        assert torch.equal(many[:20], few)
        want = oracle.render_view(ref, U, V, float(uv[7, 0]), float(uv[7, 1]), float(d[7]), w, h)
        assert np.abs(few[7].cpu().numpy() - want).max() <= 1e-3
    # an output off the 16-byte boundary, in both formats
    buf = torch.full((whole.numel() + 8,), -1.0, device="cuda")
    st.render(duv, dd, W, H, out=buf[1:1 + whole.numel()].view(whole.shape))
    assert torch.equal(buf[1:1 + whole.numel()].view(whole.shape), whole)
    assert (buf[:1] == -1).all() and (buf[1 + whole.numel():] == -1).all()
    b8 = torch.full((u8.numel() + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    st.render(duv, dd, W, H, out=b8[7:7 + u8.numel()].view(u8.shape))
    assert torch.equal(b8[7:7 + u8.numel()].view(u8.shape), u8)
    assert (b8[:7] == 0xA5).all() and (b8[7 + u8.numel():] == 0xA5).all()
    got = whole.cpu().numpy()
    assert np.array_equal(u8.cpu().numpy(), np.floor(np.clip(got, 0, 1) * np.float32(255) + np.float32(0.5)).astype(np.uint8))
    for r in range(0, n, 9):
        want = oracle.render_view(ref, U, V, float(uv[r, 0]), float(uv[r, 1]), float(d[r]), W, H)
        assert np.abs(got[r] - want).max() <= 1e-3, r
