"""Blocks whose minimum lies far below every value they hold.  The format and
the loader bound a block's decoded values, (min + u) * 2^(q + shift), not its
minimum: an encoder that does not choose the smallest minimum writes min = -600
with u = 590 .. 610.  Every decoder must give the oracle's bytes (exact), and
so must a request list at any length."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import lf_synth  # noqa: E402
import oracle  # noqa: E402

pytestmark = pytest.mark.gpu

U, V, W, H = 5, 5, 26, 18
MOST = 300   # largest |value| of a block: top + 2 levels stay far inside the loader's bound


def _bits(value, width):
    return [(value >> k) & 1 for k in range(width)]


def _record(rng, S, q):
    """One record of random blocks (presence mask, headers, payloads), as bytes."""
    modes = oracle.mode_table()
    present = rng.random(S) < 0.5
    head, body = [], []
    for _ in range(int(present.sum())):
        shift = int(rng.integers(0, 4))
        most = MOST >> (q + shift)
        k = int(rng.choice([k for k, m in enumerate(modes) if m[0] > 2 * most + 1]))
        lo = int(rng.integers(-most, most + 1))
        hi = int(rng.integers(lo, most + 1))
        # the minimum anywhere from the smallest that reaches hi up to lo
        mn = int(rng.integers(max(-1024, hi - (modes[k][0] - 1)), lo + 1))
        u = rng.integers(lo - mn, hi - mn + 1, 16)
        head += _bits(k, 5) + _bits(shift, 2) + _bits(mn & 0x7FF, 11)
        pay = int.from_bytes(oracle.bise_pack(u, k), "little")
        body += _bits(pay, oracle.bise_bits(16, k))
    mask = np.zeros((S + 31) // 32 * 32, np.uint8)
    mask[:S] = present
    bits = mask.tolist() + head + body
    bits += [0] * (-len(bits) % 32)
    return np.packbits(np.array(bits, np.uint8), bitorder="little").tobytes()


def _stream(seed, q):
    """An encoded light field with every record replaced by random blocks."""
    lf = lf_synth.make_lightfield(U, V, W, H, [0.0, 0.7], 1.0, preset_id=400 + seed)
    s = oracle.encode(lf, U, V, B=4, L=3, c=[0, 2, 3], tau_p=2, tau_b=32, q=q)
    rng = np.random.default_rng(seed)
    S, off_offsets, off_records = (int.from_bytes(s[a:a + 4], "little") for a in (40, 48, 52))
    n = 3 * ((W + 3) // 4) * ((H + 3) // 4)
    recs = [_record(rng, S, q) for _ in range(n)]
    offs = np.concatenate([[0], np.cumsum([len(r) // 4 for r in recs])]).astype("<u4")
    return (s[:56] + int(offs[-1]).to_bytes(4, "little") + s[60:off_offsets] + offs.tobytes() +
            b"\0" * (off_records - off_offsets - offs.nbytes) + b"".join(recs))


@pytest.mark.parametrize("q", [0, 2, 4, 7])
def test_every_decoder_takes_a_minimum_far_below_the_values(q):
    from paper_1805_06019_gb300 import rlfc

    data = _stream(q, q)
    ost = oracle.Stream(data)
    ref = ost.decode_all()
    st = rlfc.Stream(data)
    assert np.array_equal(st.decode_all().cpu().numpy(), ref)
    # every block: a short request list, a long one (the same requests again),
    # the binned decode
    pairs = [(v, l) for v in range(U * V) for l in range(st.nloc)]
    want = np.stack([ost.decode_block(v, l) for v, l in pairs])
    views, locs = (torch.tensor([p[k] for p in pairs], dtype=torch.int32, device="cuda") for k in (0, 1))
    assert np.array_equal(st.decode_blocks(views, locs)[0].cpu().numpy(), want)
    reps = 1 + 40000 // len(pairs)
    long, _ = st.decode_blocks(views.repeat(reps), locs.repeat(reps))
    assert np.array_equal(long.cpu().numpy().reshape(reps, *want.shape), np.broadcast_to(want, (reps, *want.shape)))
    batch = rlfc.Batch(st, len(pairs))
    assert np.array_equal(batch.decode(views, locs)[0].cpu().numpy(), want)
    # cameras on the grid at disparity 0 show the views themselves: one at a
    # time (decoded on demand) and as a batch (views decoded first)
    uv = torch.tensor([[v % U, v // U] for v in range(U * V)], dtype=torch.float32, device="cuda")
    disp = torch.zeros(U * V, device="cuda")
    ones = torch.cat([st.render(uv[v:v + 1], disp[v:v + 1], W, H, u8=True) for v in range(0, U * V, 4)])
    assert np.array_equal(ones.cpu().numpy(), ref[::4])
    reps = 1 + 400_000 // (U * V * W * H)
    many = st.render(uv.repeat(reps, 1), disp.repeat(reps), W, H, u8=True).cpu().numpy()
    assert np.array_equal(many.reshape(reps, *ref.shape), np.broadcast_to(ref, (reps, *ref.shape)))
