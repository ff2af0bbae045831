"""Batches large enough to decode their views first (three or more cameras over
400 000 or more source pixels), at the views' own size: rows and tiles that end
inside the image, every alignment of the output, shifts wider than a window,
grids of one row, both formats.  The trace names the kernels, so that the batch
is known to be blended from decoded views and its reference decoded on demand;
the two give the same bits, and meet the oracle's bound (1e-3 on the [0, 1]
scale, FP32 against FP64)."""
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIRST = {"render_plan_kernel", "decode_all_kernel<packed>", "render_native_kernel"}
DEMAND = {"render_demand_kernel"}

# (U, V, W, H, L, cluster sides, largest |disparity|)
CASES = [(4, 3, 64, 32, 2, [0, 4], 0.5), (4, 3, 61, 37, 2, [0, 4], 3.0), (4, 3, 130, 18, 2, [0, 4], 12.0),
         (4, 3, 70, 33, 2, [0, 4], 90.0), (5, 5, 68, 15, 3, [0, 2, 3], 2.0), (5, 1, 81, 34, 2, [0, 5], 1.5),
         (1, 4, 144, 17, 2, [0, 4], 2.5), (8, 8, 30, 21, 4, [0, 2, 2, 2], 1.0), (3, 3, 5, 6, 2, [0, 3], 4.0)]


def _traced(rlfc, call):
    rlfc.trace_enable(True)
    try:
        rlfc.trace_read(reset=True)
        return call(), set(rlfc.trace_read(reset=True))
    finally:
        rlfc.trace_enable(False)


def check(U, V, W, H, L, c, spread):
    from paper_1805_06019_gb300 import rlfc

    lf = lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=600 + W)
    data = oracle.encode(lf, U, V, B=4, L=L, c=c, tau_p=2, tau_b=16)
    ref = oracle.Stream(data).decode_all()
    st = rlfc.Stream(data)
    n = 1 + -(-400_000 // (W * H))
    rng = np.random.default_rng(W)
    uv = np.stack([rng.uniform(-0.2, U - 0.8, n), rng.uniform(-0.2, V - 0.8, n)], 1).astype(np.float32)
    uv[:3] = [[0, 0], [U - 1, V - 1], [U - 1, 0]]        # neighbours of weight zero
    d = rng.uniform(-spread, spread, n).astype(np.float32)
    d[n // 2:] = rng.choice([0.0, 0.7, -1.0], n - n // 2)
    duv, dd = torch.from_numpy(uv).cuda(), torch.from_numpy(d).cuda()
    whole, kernels = _traced(rlfc, lambda: st.render(duv, dd, W, H))
    assert kernels == FIRST
    u8, kernels = _traced(rlfc, lambda: st.render(duv, dd, W, H, u8=True))
    assert kernels == FIRST
    some = sorted({int(r) for r in rng.integers(0, n, 24)} | {0, 1, 2, n - 1})
    for r in some:
        one, kernels = _traced(rlfc, lambda: st.render(duv[r:r + 1].contiguous(), dd[r:r + 1].contiguous(), W, H))
        assert kernels == DEMAND
        assert torch.equal(one[0], whole[r]), r
    two = torch.tensor([some[3], some[4]], device="cuda")
    pair, kernels = _traced(rlfc, lambda: st.render(duv[two].contiguous(), dd[two].contiguous(), W, H, u8=True))
    assert kernels == DEMAND and torch.equal(pair, u8[two])
    # outputs off the 16-byte boundary, nothing written around them
    for off in (1, 2, 3):
        buf = torch.full((whole.numel() + 8,), -1.0, device="cuda")
        st.render(duv, dd, W, H, out=buf[off:off + whole.numel()].view(whole.shape))
        assert torch.equal(buf[off:off + whole.numel()].view(whole.shape), whole), off
        assert (buf[:off] == -1).all() and (buf[off + whole.numel():] == -1).all()
    for off in (1, 4, 7, 14):
        b8 = torch.full((u8.numel() + 32,), 0xA5, dtype=torch.uint8, device="cuda")
        st.render(duv, dd, W, H, out=b8[off:off + u8.numel()].view(u8.shape))
        assert torch.equal(b8[off:off + u8.numel()].view(u8.shape), u8), off
        assert (b8[:off] == 0xA5).all() and (b8[off + u8.numel():] == 0xA5).all()
    got = whole[torch.tensor(some, device="cuda")].cpu().numpy()
    g8 = u8[torch.tensor(some, device="cuda")].cpu().numpy()
    assert np.array_equal(g8, np.floor(np.clip(got, 0, 1) * np.float32(255) + np.float32(0.5)).astype(np.uint8))
    for k, r in enumerate(some):
        want = oracle.render_view(ref, U, V, float(uv[r, 0]), float(uv[r, 1]), float(d[r]), W, H)
        assert np.abs(got[k] - want).max() <= 1e-3, r
    return st


@pytest.mark.parametrize("case", range(len(CASES)))
def test_decode_first_batches(case):
    check(*CASES[case])


def test_debug_build_raises_no_flag_on_these_batches():
    import __graft_entry__
    import paper_1805_06019_gb300 as pkg

    __graft_entry__.build()
    pkg.build(debug=True)
    child = ("import os, sys; sys.path[:0] = [%r, %r]; os.environ['RLFC_DEBUG_LIBRARY'] = '1'\n"
             "import test_gpu_decode_first as t\n"
             "from paper_1805_06019_gb300 import rlfc\n"
             "assert '_build_debug' in rlfc.library_path()\n"
             "for k in (1, 4, 7):\n"
             "    st = t.check(*t.CASES[k]); assert st.debug_flags() == 0, k\n"
             "print('OK')" % (ROOT, os.path.dirname(os.path.abspath(__file__))))
    r = subprocess.run([sys.executable, "-c", child], capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout[-3000:] + r.stderr[-3000:]
