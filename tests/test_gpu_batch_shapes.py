"""The binned decode over the forms its parse and its rounds branch on: masks of
the three records in one warp step or several, records of 2^16 bits and more
(32-bit payload offsets), deep trees, bins around a round's requests, and
outputs on 16-, 4- and 1-byte boundaries.  Bit-exact against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [  # U, V, L, cluster sides, thresholds
    (3, 3, 2, [0, 3], 1, 8),            # one mask word per record
    (19, 19, 3, [0, 4, 5], 2, 16),      # 36 mask words in all
    (24, 21, 2, [0, 24], 0, 0),         # lossless: records past 2^16 bits
    (9, 8, 6, [0, 2, 2, 2, 2, 2], 1, 4),
]


@pytest.mark.parametrize("U,V,L,c,tp,tb", SHAPES)
@pytest.mark.parametrize("warps", [4, 16])
def test_binned_decode_shapes(U, V, L, c, tp, tb, warps):
    from paper_1805_06019_gb300 import rlfc

    W, H = 14, 9
    lf = lf_synth.make_lightfield(U, V, W, H, [0.0, 1.3], 30.0 if tp == 0 else 4.0, preset_id=80 + U)
    data = oracle.encode(lf, U, V, B=4, L=L, c=c, tau_p=tp, tau_b=tb)
    ost = oracle.Stream(data)
    st = rlfc.Stream(data)
    rng = np.random.default_rng(U)
    # bins of 1, 12, 13, 16, 17, 33 requests and an empty one, shuffled
    counts = [1, 12, 13, 16, 17, 33, 0, 40]
    locs = np.concatenate([np.full(k, i % st.nloc) for i, k in enumerate(counts)])
    views = rng.integers(0, U * V, locs.size)
    order = rng.permutation(locs.size)
    views, locs = views[order].astype(np.int32), locs[order].astype(np.int32)
    want = np.stack([ost.decode_block(int(v), int(l)) for v, l in zip(views, locs)])
    dv, dl = torch.from_numpy(views).cuda(), torch.from_numpy(locs).cuda()
    b = rlfc.Batch(st, locs.size)
    b.config = {"warps_per_cta": warps, "graph": 0}
    n = want.size
    for offset in (0, 4, 9):
        buf = torch.full((n + 32,), 0xA5, dtype=torch.uint8, device="cuda")
        b.decode(dv, dl, buf[offset:offset + n].view(want.shape))
        got = buf.cpu().numpy()
        assert np.array_equal(got[offset:offset + n].reshape(want.shape), want), offset
        assert (got[:offset] == 0xA5).all() and (got[offset + n:] == 0xA5).all()
