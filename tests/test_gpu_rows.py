"""Output rows of any alignment and length: the full decode writes the rows of
a strip as the destination's aligned 16-byte chunks, with partial chunks at
both ends.  Bit-exact against the oracle, nothing written around the output."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [1, 5, 31, 33, 37, 48, 66])
def test_rows_of_any_length_and_alignment(W):
    from paper_1805_06019_gb300 import rlfc

    U, V, H = 3, 2, 7
    lf = lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=40 + W)
    data = oracle.encode(lf, U, V, B=4, L=2, c=[0, 3], tau_p=1, tau_b=8)
    ref = oracle.Stream(data).decode_all()
    st = rlfc.Stream(data)
    for offset in (0, 2, 3, 7, 12, 13, 15):
        buf = torch.full((ref.size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        st.decode_all(buf[16 + offset:16 + offset + ref.size].view(ref.shape))
        b = buf.cpu().numpy()
        assert np.array_equal(b[16 + offset:16 + offset + ref.size].reshape(ref.shape), ref), (W, offset)
        assert (b[:16 + offset] == 0xA5).all() and (b[16 + offset + ref.size:] == 0xA5).all()
    # the packed views behind a batch of cameras: an integer camera gives the view back
    cams = torch.tensor([[0.0, 0.0], [1.0, 1.0], [2.0, 0.0], [2.0, 1.0]], device="cuda")
    img = st.render(cams, torch.zeros(4, device="cuda"), W, H, u8=True).cpu().numpy()
    assert np.array_equal(img, ref[[0, 4, 2, 5]])
