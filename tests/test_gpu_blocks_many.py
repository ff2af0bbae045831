"""Request lists long enough for the thread-per-channel decoder: every ancestor
depth, bad requests among good ones, a last partial CTA, outputs on and off
4-byte boundaries.  Bit-exact against the oracle's full decode."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U,V,L,c,tp,tb,q", [(3, 3, 2, [0, 3], 1, 8, 0), (13, 12, 3, [0, 4, 4], 2, 16, 0),
                                             (9, 8, 6, [0, 2, 2, 2, 2, 2], 1, 4, 1)])
@pytest.mark.parametrize("n", [16384, 20001])
def test_many_requests(U, V, L, c, tp, tb, q, n):
    from paper_1805_06019_gb300 import rlfc

    W, H = 24, 16
    lf = lf_synth.make_lightfield(U, V, W, H, [0.0, 1.3], 4.0, preset_id=90 + U)
    data = oracle.encode(lf, U, V, B=4, L=L, c=c, tau_p=tp, tau_b=tb, q=q)
    ref = oracle.Stream(data).decode_all().reshape(U * V, H // 4, 4, W // 4, 4, 3).swapaxes(2, 3).reshape(U * V, -1, 4, 4, 3)
    st = rlfc.Stream(data)
    rng = np.random.default_rng(n)
    views, locs = rng.integers(0, U * V, n), rng.integers(0, st.nloc, n)
    views[::97] = U * V + 3
    locs[5::89] = st.nloc
    bad = np.where(views >= U * V, 1, np.where(locs >= st.nloc, 2, 0))
    want = np.where((bad == 0)[:, None, None, None], ref[views % (U * V), locs % st.nloc], 0).astype(np.uint8)
    dv, dl = torch.from_numpy(views.astype(np.int32)).cuda(), torch.from_numpy(locs.astype(np.int32)).cuda()
    for offset in (0, 3):
        buf = torch.full((want.size + 16,), 0xA5, dtype=torch.uint8, device="cuda")
        _, status = st.decode_blocks(dv, dl, buf[offset:offset + want.size].view(want.shape))
        b = buf.cpu().numpy()
        assert np.array_equal(status.cpu().numpy(), bad)
        assert np.array_equal(b[offset:offset + want.size].reshape(want.shape), want)
        assert (b[:offset] == 0xA5).all() and (b[offset + want.size:] == 0xA5).all()
