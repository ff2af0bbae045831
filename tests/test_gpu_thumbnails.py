"""Renders much smaller than the views, the list of an album: a few cameras of
a large light field sample its pixels one by one instead of decoding whole
views; many cameras, or a small light field, do not.  The same bits by every
path, and the oracle's bound (1e-3 on the [0, 1] scale)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

U, V = 3, 2


def _field(rlfc, W, H):
    lf = torch.from_numpy(lf_synth.make_lightfield(U, V, W, H, [0.0, 1.5], 1.0, preset_id=540)).cuda()
    return rlfc.Stream(rlfc.encode(lf, U, V, 2, [0, 3], tau_p=3, tau_b=48))


def _cameras(n):
    rng = np.random.default_rng(n)
    uv = np.stack([rng.uniform(-0.2, U - 0.8, n), rng.uniform(-0.2, V - 0.8, n)], 1).astype(np.float32)
    uv[0] = [1, 0]                                   # one neighbour of weight 1
    return uv, rng.choice([0.0, 1.5, -40.0], n).astype(np.float32)


def _traced(rlfc, call):
    rlfc.trace_enable(True)
    try:
        rlfc.trace_read(reset=True)
        out = call()
        return out, set(rlfc.trace_read(reset=True))
    finally:
        rlfc.trace_enable(False)


@pytest.mark.parametrize("w,h", [(40, 31), (1, 1), (129, 7)])
def test_thumbnails_of_a_large_field(w, h):
    from paper_1805_06019_gb300 import rlfc

    st = _field(rlfc, 2051, 1537)
    ref = st.decode_all().cpu().numpy()
    n = 2000 if w * h < 4000 else 1400
    uv, d = _cameras(n)
    duv, dd = torch.from_numpy(uv).cuda(), torch.from_numpy(d).cuda()
    one, k1 = _traced(rlfc, lambda: st.render(duv[:1], dd[:1], w, h))
    few, k7 = _traced(rlfc, lambda: st.render(duv[:7], dd[:7], w, h))
    few8, _ = _traced(rlfc, lambda: st.render(duv[:7], dd[:7], w, h, u8=True))
    many, kn = _traced(rlfc, lambda: st.render(duv, dd, w, h))
    assert k1 == k7 == {"render_direct_kernel"}
    if w * h > 1:
        assert "render_sampled_kernel" in kn
    assert torch.equal(one, many[:1]) and torch.equal(few, many[:7])
    got = few.cpu().numpy()
    assert np.array_equal(few8.cpu().numpy(), np.floor(np.clip(got, 0, 1) * np.float32(255) + np.float32(0.5)).astype(np.uint8))
    for r in range(7):
        want = oracle.render_view(ref, U, V, float(uv[r, 0]), float(uv[r, 1]), float(d[r]), w, h)
        assert np.abs(got[r] - want).max() <= 1e-3, r


def test_small_fields_and_larger_outputs_keep_their_paths():
    from paper_1805_06019_gb300 import rlfc

    uv, d = (torch.from_numpy(x).cuda() for x in _cameras(64))
    small = _field(rlfc, 200, 150)
    for n, w, h, kernel in ((1, 100, 75, "render_demand_kernel"), (1, 12, 9, "render_sampled_kernel"),
                            (64, 12, 9, "render_sampled_kernel"), (64, 230, 150, "render_sampled_kernel")):
        _, kernels = _traced(rlfc, lambda: small.render(uv[:n], d[:n], w, h))
        assert kernel in kernels and "render_direct_kernel" not in kernels, (n, w, h, kernels)
    large = _field(rlfc, 2051, 1537)
    for n, w, h, kernel in ((1, 1025, 768, "render_demand_kernel"), (1, 2051, 1537, "render_demand_kernel"),
                            (8, 1025, 768, "render_sampled_kernel")):
        _, kernels = _traced(rlfc, lambda: large.render(uv[:n], d[:n], w, h))
        assert kernel in kernels and "render_direct_kernel" not in kernels, (n, w, h, kernels)
