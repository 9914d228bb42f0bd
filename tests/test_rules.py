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
