"""Size rules that split work over the SMs, called in the built library (no GPU needed).  The
C++ functions are not part of the C ABI and go by their exported names."""
import ctypes as C

import pytest

I, L = C.c_int, C.c_int64


@pytest.fixture(scope="module")
def rule():
    import __graft_entry__ as g
    g.build()
    from paper_1610_02121_gb300 import LIB_PATH
    lib = C.CDLL(LIB_PATH)

    def get(name, *args):
        f = getattr(lib, name)
        f.restype, f.argtypes = L, list(args)
        return f

    return get


# Gram product of a tall block (559,625 rows) on 152 SMs: 256-row groups of the CTA that ends
# last.  The figures are those of the segments that an array of four 48 x 48 blocks an SM allowed;
# fewer segments leave most SMs idle.
@pytest.mark.parametrize("N,groups", [(16, 32), (65, 32), (80, 32), (100, 33), (135, 67), (160, 58), (200, 88),
                                      (300, 169), (400, 274), (512, 365), (640, 547)])
def test_gram_segments_fill_the_sms(rule, N, groups):
    n_sm, total = 152, (559625 + 255) // 256
    pairs = rule("_ZN3efe13oz_gram_pairsEiibP4int2", I, I, C.c_bool, C.c_void_p)
    pairs.restype = I
    np_ = pairs(N, N, True, None)
    work = rule("_ZN3efe18oz_gram_work_elemsEiii", I, I, I)(N, N, n_sm)
    seg = rule("_ZN3efe18oz_gram_seg_groupsEliil", L, I, I, L)(total, np_, n_sm, work // (N * N))
    items = -(-total // seg) * np_
    assert -(-items // n_sm) * seg <= groups
    assert items >= 0.9 * n_sm or N > 300
    assert -(-total // seg) * N * N <= work
    # a narrower block's partials fit the array of a wider one
    assert rule("_ZN3efe18oz_gram_work_elemsEiii", I, I, I)(N, N // 2, n_sm) <= work


# DFMA A^T A of a tall block: of a symmetric product only the tiles on and above the diagonal
# are formed.  Work of the busiest SM over the average, for the widths that take 16- and 32-wide
# tiles: 1.25 at most (153 tiles on 152 SMs are the worst), 1.69 by a rule that counts all tiles.
def test_symmetric_splits_count_the_tiles_they_form(rule):
    n_sm, rows = 152, 559625
    splits = rule("_ZN3efe14gemm_tn_splitsEliibi", L, I, I, C.c_bool, I)
    for N in range(1, 1200):
        pad = {t: -(-N // t) * t for t in (48, 32, 16)}
        t = min(pad, key=lambda k: (pad[k], -k))
        n = pad[t] // t
        s, formed = splits(rows, N, N, True, n_sm), n * (n + 1) // 2
        assert s >= splits(rows, N, N, False, n_sm)
        if t < 48:
            assert -(-formed * s // n_sm) / s <= 1.25 * formed / n_sm, N
        assert splits(100, N, N, True, n_sm) <= 2          # no split is shorter than 64 rows
