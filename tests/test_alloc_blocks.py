"""Blocks from a caller's allocator, which may start at any multiple of 16: the
library uses each from a multiple of 32 (its widest loads and stores), inside
what it asked for, and frees exactly what it was given.  Host code alone, with
made-up addresses."""
import ctypes as C

import pytest


class Arena:
    """Hands out the given addresses in turn (None: refuses) and keeps what was asked and freed."""

    def __init__(self, *addresses):
        from paper_1212_1639_gb300 import build
        build.build()
        from paper_1212_1639_gb300 import pf
        self.pf, self.give, self.live, self.asked = pf, list(addresses), {}, []

        def _alloc(nbytes, stream, ctx):
            p = self.give.pop(0)
            self.asked.append(nbytes)
            if p is not None:
                assert p not in self.live
                self.live[p] = nbytes
            return p

        def _free(p, stream, ctx):
            del self.live[p]

        self.alloc, self.free = pf.ALLOC_FN(_alloc), pf.FREE_FN(_free)

    def block(self, nbytes):
        raw, start = C.c_void_p(), C.c_void_p()
        st = self.pf._lib.pf_diag_block(self.alloc, self.free, None, nbytes, C.byref(raw), C.byref(start))
        return st, raw.value, start.value


@pytest.mark.parametrize("nbytes", [1, 16, 240, 241, 255, 256, 257, 4096, 12345, 1 << 30])
@pytest.mark.parametrize("first", [0x10000, 0x10010, 0x10020, 0x10030, 0x100f0])
@pytest.mark.parametrize("second", [0x70000000, 0x70000010, 0x700000f0])
def test_block_starts_at_a_multiple_of_32(first, second, nbytes):
    a = Arena(first, second)
    st, raw, start = a.block(nbytes)
    assert st == a.pf.PF_OK
    assert list(a.live) == [raw]  # one block in use: the one to be freed
    assert start % 32 == 0 and raw <= start and start + nbytes <= raw + a.live[raw]
    if first % 32 == 0:  # nothing changes for an allocator that aligns to 32
        assert raw == start == first and a.asked == [(nbytes + 255) // 256 * 256]


@pytest.mark.parametrize("addresses,want", [([None], 2), ([0x10010, None], 2), ([0x10008], 1),
                                            ([0x10001], 1), ([0x10010, 0x20008], 1)])
def test_refusals_leave_nothing_in_use(addresses, want):
    a = Arena(*addresses)
    assert a.block(1000)[0] == want  # 1: PF_ERR_INVALID, 2: PF_ERR_OOM
    assert not a.live
