"""The encoder's device scratch: the bound that rlfc_encode allocates and
rlfc_encode_no_alloc admits by is the sum of the buffers that the encoder
carves, and no more.  The no-alloc entry point reports it, before any device
work, for a light field beyond its 32 MiB."""
import ctypes
import re

import pytest

from paper_1805_06019_gb300 import buildlib, rlfc

E_RANGE = 6


def _carved(U, V, W, H, L, c):
    """Bytes of every buffer (an item more than 16 bytes of slack, on a 256-byte boundary)."""
    cnt, gu, gv = [U * V], U, V
    for l in range(1, L):
        gu, gv = -(-gu // c[l]), -(-gv // c[l])
        cnt.append(gu * gv)
    wp, hp = -(-W // 4) * 4, -(-H // 4) * 4
    nloc, npix, S = wp * hp // 16, 3 * wp * hp, sum(cnt[:-1])
    sizes = [2 * npix * n for n in cnt]                      # images of every level
    sizes += [2 * npix * n for n in cnt[1:-1]]               # reconstructions between top and views
    sizes += [3 * nloc * n for n in cnt[:-1]]                # (shift, mode) of every block
    sizes += [4]                                             # error word
    for l in range(1, L):                                    # filter members and weights, parents
        sizes += [4 * (cnt[l] + 1), 4 * cnt[l - 1], 4 * cnt[l], 8 * cnt[l - 1], 4 * cnt[l - 1]]
    sizes += [4 * S, 4 * S, 4 * 3 * nloc, 4 * (3 * nloc + 1), 8 * L, 8 * L]
    sizes += [4 * (3 * nloc * (-(-S // 32) + -(-S * (18 + 160) // 32)) + 1)]   # records, every block stored at its longest
    return sum(-(-(s + 16) // 256) * 256 for s in sizes)


@pytest.mark.parametrize("U,V,W,H,L,c", [(9, 9, 512, 512, 3, [0, 3, 3]), (17, 17, 1024, 1024, 3, [0, 5, 4]),
                                         (5, 5, 640, 301, 2, [0, 5]), (8, 8, 333, 250, 4, [0, 2, 2, 2])])
def test_the_bound_is_what_the_encoder_carves(U, V, W, H, L, c):
    lib = ctypes.CDLL(buildlib.build())
    lib.rlfc_last_error.restype = ctypes.c_char_p
    p = rlfc.EncParams()
    p.U, p.V, p.W, p.H, p.B, p.L, p.tau_p, p.tau_b = U, V, W, H, 4, L, 4, 64
    for l in range(1, L):
        p.c[l] = c[l]
    n = ctypes.c_size_t()
    rc = lib.rlfc_encode_no_alloc(ctypes.byref(p), ctypes.c_void_p(256), None, None, ctypes.c_size_t(0), ctypes.byref(n))
    assert rc == E_RANGE
    need = int(re.search(r"needs (\d+) bytes", lib.rlfc_last_error().decode()).group(1))
    assert need == _carved(U, V, W, H, L, c)
