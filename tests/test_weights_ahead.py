"""The lists of gate/up weights that are asked into L2 ahead of their phase, from the functions the kernels walk: a request
changes no value, so only the list shows whether the intended rows, and nothing else, are asked for."""
import pytest

from paper_2509_18362_b200 import binding as Bd

L2 = 132644864           # what the driver reports for a B200
HUGE = 1 << 40           # no bound that any shape here meets
SHARE = {False: (4, 16), True: (32, 128)}      # rows asked for of a tile's rows


def _requests(batched, ffn, d, grid, l2):
    return [Bd.fmtp_selftest_ahead(batched, ffn, d, grid, l2, cta) for cta in range(grid)]


def _tiles(batched, ffn, grid, cta):
    """First and end row of the tiles a CTA asks for, in order."""
    take, cap = SHARE[batched]
    if batched:
        return [(t * cap, min(ffn, t * cap + cap)) for t in range(cta, -(-ffn // cap), grid)]
    v0, v1 = cta * ffn // grid, (cta + 1) * ffn // grid
    return [(r, min(v1, r + cap)) for r in range(v0, v1, cap)][1:]         # the first tile is in the ring already


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("d,grid", [(64, 148), (256, 2), (3584, 148), (3584, 140), (8256, 97)])
@pytest.mark.parametrize("ffn", [
    16, 128, 144,      # fewer rows than CTAs; one tile of 128, and 16 rows more
    2352, 2384,        # one tile of 16 per CTA, and a few CTAs with a second one of one row
    7168, 9520,        # the last tile of 16 has a few rows; the last one of 128 all, and 48
    18944, 19040,      # as many tiles of 128 as CTAs, and one more
])
def test_every_tile_is_asked_for_once_and_nothing_else(ffn, d, grid, batched):
    take, _ = SHARE[batched]
    for cta, got in enumerate(_requests(batched, ffn, d, grid, HUGE)):
        want = [(m, lo, min(hi, lo + take)) for lo, hi in _tiles(batched, ffn, grid, cta) for m in (0, 1)]
        rows = []                                    # pieces joined to what they make up: matrix, first and end row
        for m, at, size in got:
            assert at >= 0 and size > 0 and size % 16 == 0 and at * 2 % 16 == 0 and at + size // 2 <= ffn * d
            assert not batched or size <= 16384
            if rows and rows[-1][0] == m and rows[-1][2] == at:
                rows[-1][2] = at + size // 2
            else:
                rows.append([m, at, at + size // 2])
        assert [(m, lo * d, hi * d) for m, lo, hi in want] == [tuple(r) for r in rows], cta


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("d,ffn", [(3584, 18944), (5120, 27648), (8192, 28672), (16384, 53248), (64, 1 << 20)])
def test_requests_stay_within_their_share_of_l2(d, ffn, batched):
    bounded, free = _requests(batched, ffn, d, 148, L2), _requests(batched, ffn, d, 148, HUGE)
    total = sum(size for got in bounded for _, _, size in got)
    assert total <= L2 * 9 // 16
    # unused: less than a pair of requests per CTA; what rounding to 16 bytes takes from a tile
    unused = 16 * (ffn // 128 + 1) if batched else 148 * 2 * 4 * d * 2
    assert total >= min(L2 * 9 // 16 - unused, 0.999 * sum(size for got in free for _, _, size in got))
    for got, all_of_them in zip(bounded, free):      # nothing but what is asked for without the bound, or the beginning of it
        sizes = {(m, at): size for m, at, size in all_of_them}
        assert len(set((m, at) for m, at, _ in got)) == len(got)
        assert all(0 < size <= sizes[m, at] and size % 16 == 0 for m, at, size in got)


@pytest.mark.parametrize("batched,total", [(False, 148 * 7 * 2 * 4 * 7168), (True, 148 * 2 * 32 * 7168)])
def test_the_7b_shape_keeps_all_requests(batched, total):
    got = _requests(batched, 18944, 3584, 148, L2)
    assert got == _requests(batched, 18944, 3584, 148, HUGE)
    assert sum(size for one in got for _, _, size in one) == total
    few = _requests(batched, 18944, 3584, 140, L2)             # W_o's GEMM has 140 CTAs: eight of them ask for two tiles
    assert not batched or sum(size for one in few for _, _, size in one) == total


def test_any_size_of_l2_gives_a_list():
    for l2 in (1, 15, 1 << 31, 1 << 40, (1 << 63) - 1):
        for batched in (0, 1):
            total = sum(size for _, _, size in Bd.fmtp_selftest_ahead(batched, 1 << 22, 64, 1, l2, 0))
            assert total <= max(l2 * 9 // 16, 0)
            assert l2 < 1 << 31 or total == (1 << 22) * 64 * 2 * 2 // 4 - (0 if batched else 2 * 4 * 64 * 2)


def test_no_room_and_bad_arguments():
    assert Bd.fmtp_selftest_ahead(0, 18944, 3584, 148, 0, 3) == [] and Bd.fmtp_selftest_ahead(1, 18944, 3584, 148, 0, 3) == []
    for args in ((0, 0, 64, 1, L2, 0), (0, 64, 64, 0, L2, 0), (1, 64, 64, 4, L2, 4), (1, 64, 64, 4, L2, -1), (0, 64, 64, 4, -1, 0),
                 (0, 64, 1 << 29, 1, L2, 0), (1, (1 << 31) - 1, 64, 1, L2, 0)):
        with pytest.raises(Bd.FastMTPError):
            Bd.fmtp_selftest_ahead(*args)
