"""Calls of several host threads on light fields of different trees: each call
must run with the shared memory that it asked for, whatever another thread's
call asked for in between."""
import threading

import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _load(rlfc, U, V, W, H, L, c, tau, preset):
    lf = torch.from_numpy(lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=preset)).cuda()
    return rlfc.Stream(rlfc.encode(lf, U, V, L, c, tau_p=tau, tau_b=16 * tau))


def _calls(st, what):
    uv = torch.tensor([[0.4, 0.6]], device="cuda")
    disp = torch.tensor([0.5], device="cuda")
    if what == "decode_all":
        out = torch.empty((st.n_views, st.H, st.W, 3), dtype=torch.uint8, device="cuda")
        return out, lambda stream: st.decode_all(out, stream=stream)
    w, h = (st.W, st.H) if what == "view" else (st.W // 2 * 3, st.H // 2 * 3)
    out = torch.empty((1, h, w, 3), device="cuda")
    return out, lambda stream: st.render(uv, disp, w, h, out, stream=stream)


@pytest.mark.parametrize("what", ["view", "scaled_view", "decode_all"])
def test_threads_do_not_change_each_others_launches(what):
    from paper_1805_06019_gb300 import rlfc

    # four, three and two levels: 50.7, 41.5 and fewer KB for a tile of one
    # view; records of very different lengths for the full decode.  Two threads
    # on each field, queueing without a wait.
    fields = [_load(rlfc, 3, 3, 512, 320, 4, [0, 2, 2, 2], 0, 501),
              _load(rlfc, 3, 3, 512, 320, 3, [0, 2, 2], 4, 502),
              _load(rlfc, 2, 2, 512, 320, 2, [0, 2], 40, 503)] * 2
    work = [_calls(st, what) for st in fields]
    streams = [torch.cuda.Stream() for _ in fields]
    for (_, call), s in zip(work, streams):
        call(s)
    torch.cuda.synchronize()
    want = [out.clone() for out, _ in work]
    for out, _ in work:
        out.zero_()
    torch.cuda.synchronize()
    errors = []
    start = threading.Barrier(len(fields))

    def loop(k):
        try:
            start.wait()
            for _ in range(3000):
                work[k][1](streams[k])
        except Exception as e:
            errors.append((k, repr(e)))

    threads = [threading.Thread(target=loop, args=(k,)) for k in range(len(fields))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for (out, _), w in zip(work, want):
        assert torch.equal(out, w)
