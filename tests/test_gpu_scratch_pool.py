"""Scratch memory that render calls keep: one bounded pool per device, however
many light fields are loaded, given back when they are freed."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_scratch_is_bounded_and_given_back():
    from paper_1805_06019_gb300 import rlfc

    U, V, W, H, n = 5, 5, 352, 352, 24
    lf = torch.from_numpy(lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=560)).cuda()
    data = rlfc.encode(lf, U, V, 2, [0, 5], tau_p=2, tau_b=32)
    rng = np.random.default_rng(5)
    uv = torch.from_numpy(rng.uniform(0, 4, (n, 2)).astype(np.float32)).cuda()
    disp = torch.zeros(n, device="cuda")
    out = torch.empty((n, H, W, 3), device="cuda")
    warm = rlfc.Stream(data)
    warm.render(uv, disp, W, H, out)     # the kernels are loaded
    want = out.clone()
    warm.close()
    fields = [rlfc.Stream(data) for _ in range(24)]
    before = _free()
    for st in fields:
        st.render(uv, disp, W, H, out)
        assert torch.equal(out, want)
    # a call's scratch is 12 MB; blocks are mapped 32 MiB at a time
    assert before - _free() <= 64 * MB
    # half of them freed, the rest still render
    for st in fields[::2]:
        st.close()
    out.zero_()
    fields[1].render(uv, disp, W, H, out)
    assert torch.equal(out, want)
    held = _free()
    for st in fields:
        st.close()
    own = sum(st.info.device_bytes for st in fields[1::2])
    assert _free() - held >= own          # their data, and no less for a pool left behind
    again = rlfc.Stream(data)
    out.zero_()
    again.render(uv, disp, W, H, out)
    assert torch.equal(out, want)
    again.close()


def test_threads_load_render_and_free():
    import threading

    from paper_1805_06019_gb300 import rlfc

    U, V, W, H, n = 4, 4, 160, 128, 24
    lf = torch.from_numpy(lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=561)).cuda()
    data = rlfc.encode(lf, U, V, 2, [0, 4], tau_p=2, tau_b=32)
    uv = torch.full((n, 2), 1.4, device="cuda")
    disp = torch.full((n,), 0.7, device="cuda")
    st = rlfc.Stream(data)
    want = st.render(uv, disp, W, H)
    st.close()
    torch.cuda.synchronize()
    errors = []

    def loop(k):
        try:
            stream = torch.cuda.Stream()
            out = torch.empty_like(want)
            torch.cuda.synchronize()
            for _ in range(20):
                s = rlfc.Stream(data, stream=stream)
                for _ in range(3):
                    s.render(uv, disp, W, H, out, stream=stream)
                stream.synchronize()
                assert torch.equal(out.cpu(), host)
                s.close()
        except Exception as e:
            errors.append((k, repr(e)))

    host = want.cpu()
    threads = [threading.Thread(target=loop, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
