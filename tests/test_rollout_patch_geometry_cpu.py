"""Host-side check of the whole-rollout kernel's smaller patches (8 latitudes x 8
or 4 longitudes; the 16-longitude patch has its own test): for every admitted
width, a slab of the patch's longitudes and two on each side holds no longitude
twice and every window; the wrapping ones split into a two-column box and the
others, both inside the grid; the query groups of 4 x 4 and the head groups
cover every (query, head) once; the columns of a row's copies cover it once."""
import pytest

TH = 8


@pytest.mark.parametrize("TW", [4, 8, 16])
def test_longitude_slabs(TW):
    SW = TW + 4
    for W in range(32, 385, 16):
        for w0 in range(0, W, TW):
            slab = [(w0 - 2 + c) % W for c in range(SW)]
            assert len(set(slab)) == SW
            wrap = -1 if w0 == 0 else (1 if w0 + TW + 2 > W else 0)
            if wrap == 0:
                assert slab == list(range(w0 - 2, w0 - 2 + SW)) and w0 - 2 >= 0 and w0 - 2 + SW <= W
            elif wrap < 0:
                assert slab == [W - 2, W - 1] + list(range(SW - 2))
            else:
                assert w0 == W - TW and slab == list(range(W - (SW - 2), W)) + [0, 1]
            for gc in range(TW // 4):
                rect = slab[4 * gc:4 * gc + 8]
                assert len(rect) == 8
                for qc in range(4):
                    for kw in (1, 3, 5):
                        q = w0 + 4 * gc + qc
                        window = {(q + d) % W for d in range(-(kw // 2), kw // 2 + 1)}
                        assert {rect[j] for j in range(8) if abs(j - 2 - qc) <= kw // 2} == window


@pytest.mark.parametrize("TW", [4, 8, 16])
def test_warps_cover_queries_and_heads_once(TW):
    TP = TH * TW
    NCP = 128 // TP
    NH = 4 // NCP
    seen = []
    for warp in range(8):
        grp, hs = (warp, 0) if NCP == 1 else (warp % (TP // 16), warp // (TP // 16))
        gr, gc = grp // (TW // 4), grp % (TW // 4)
        for head in range(hs * NH, hs * NH + NH):
            for g8 in range(8):
                row = 4 * gr + (g8 >> 2)
                for r in (row, row + 2):
                    seen.append((r * TW + 4 * gc + (g8 & 3), head))
    assert sorted(seen) == sorted((q, h) for q in range(TP) for h in range(4))


@pytest.mark.parametrize("TW", [4, 8, 16])
def test_copies_cover_a_rows_columns_once(TW):
    TP = TH * TW
    NCP = 128 // TP
    NC = 64 // NCP
    seen = []
    for warp in range(8):
        for lane in range(32):
            mr = 32 * (warp & 3) + lane
            copy, tr, hf = mr // TP, mr % TP, warp >> 2
            seen += [(tr, 64 * hf + NC * copy + j) for j in range(NC)]
    assert sorted(seen) == [(t, c) for t in range(TP) for c in range(128)]


@pytest.mark.parametrize("TW", [4, 8, 16])
def test_swizzled_boxes_start_on_their_pattern(TW):
    """A 64-byte swizzle repeats every 512 bytes: the second box of a wrapping slab starts on a multiple."""
    SW, rows, key = TW + 4, 12, 64
    for first in (2, SW - 2):
        assert rows * first * key % 512 == 0
    assert rows * SW * key % 512 == 0
