"""Launch shapes of the monotone search's row blocks on the host: windows that a
block of at least weff - 1 rows holds by divide and conquer are taken, whatever
the register-tile searches would need; blocks sized for those are searched by
them; long lines that fit one CTA are launched whole when there are enough."""
import pytest

from paper_1210_4090_gb300 import hjlo

SMEM = 232448


@pytest.fixture(autouse=True)
def _no_overrides(monkeypatch):
    for k in ("HJLO_LANES_PER_LINE", "HJLO_LINES_PER_TILE", "HJLO_OFFLOAD", "HJLO_BLOCK_ROWS"):
        monkeypatch.delenv(k, raising=False)


def _holds(weff, esize):
    """Whether divide and conquer holds weff - 1 rows: their span of 2 (weff - 1) points at esize + 6 bytes
    each (value, screened value, argmin offset) and 16 a displacement, less 1 KB of padding."""
    return 2 * (weff - 1) <= (SMEM - 1024 - 16 * weff) // (esize + 6)


@pytest.mark.parametrize("esize", [8, 4])
@pytest.mark.parametrize("lines", [1, 40, 1024])
def test_wide_windows_are_taken(lines, esize):
    taken = []
    for weff in range(3001, 6602, 100):
        N = 4 * weff + 7
        if not _holds(weff, esize):
            with pytest.raises(hjlo.HjloError):
                hjlo.shape_query(1 << 18, 1, weff, esize)
            continue
        s = hjlo.shape_query(max(N, 1 << 16), lines, weff, esize)
        assert s["row_blocks"] > 1 and s["block_rows"] >= weff - 1, (weff, s)
        taken.append(weff)
    assert max(taken) >= (5200 if esize == 8 else 6300)


@pytest.mark.parametrize("N,lines,weff", [(10000, 1024, 2401), (12000, 300, 1601), (14000, 200, 881)])
def test_long_lines_that_fit_are_whole(N, lines, weff):
    assert hjlo.shape_query(N, lines, weff)["row_blocks"] == 1


@pytest.mark.parametrize("N,weff,rows,seg", [
    (1 << 18, 3271, 3270, 11), (65536, 1601, 1600, 11),    # weff - 1 rows, searched in segments of 11
    (1 << 18, 201, 1725, 9), (65536, 291, 432, None),      # one SM's share; few lanes: divide and conquer
    (20000, 2401, 2400, 11), (1 << 18, 3801, 7600, None),      # divide and conquer: 2 (weff - 1) rows
    (8192, 291, 290, None)])
def test_block_rows(N, weff, rows, seg):
    s = hjlo.shape_query(N, 1, weff)
    assert s["block_rows"] == rows, s
    if seg:
        assert s["segment_rows"] == seg, s
    assert s["threads"] >= (128 if weff > 512 else 32), s


@pytest.mark.parametrize("N,lines,weff,seg", [
    (65536, 1, 291, 0), (80000, 1, 201, 0), (320, 320, 129, 0),   # 64 and 32 lanes a line: divide and conquer
    (80000, 1, 501, 9), (180000, 1, 201, 13), (1 << 18, 1, 201, 9), (448, 448, 129, 9)])
def test_few_lanes_go_to_divide_and_conquer(N, lines, weff, seg):
    s = hjlo.shape_query(N, lines, weff)
    assert (s["segment_rows"] == seg) if seg else s["segment_rows"] < 9, s
    assert s["threads"] >= 64, s


def test_wide_windows_have_four_warps():
    for N, weff in [(65536, 521), (50000, 601), (100000, 601)]:
        s = hjlo.shape_query(N, 1, weff)
        assert s["segment_rows"] == 11 and s["threads"] >= 128, (N, weff, s)


def test_short_lines_of_few_lanes():
    """Contiguous lines of 105 to 208 points (16 lanes each): divide and conquer up to 160 lanes an SM."""
    assert hjlo.shape_query(166, 1000, 99)["segment_rows"] < 9
    assert hjlo.shape_query(166, 2500, 99)["segment_rows"] in (11, 13)


# the flat search's blocks are of a power of two of rows, divide and conquer's hold an SM's share
@pytest.mark.parametrize("N,lines,weff,rows", [
    (4096, 1, 61, 128), (9600, 1, 95, 128), (30000, 1, 95, 198),      # a few rows an SM; too few to fill it
    (78000, 1, 95, 256), (1 << 18, 1, 95, 512), (500000, 1, 25, 1024),   # four blocks an SM at most
    (1 << 20, 1, 95, 6899), (100000, 1, 9, 658),          # the whole window's cost; a few displacements
    (900, 60, 91, 128), (20000, 16, 81, 1024)])           # several lines
def test_flat_row_blocks(N, lines, weff, rows):
    s = hjlo.shape_query(N, lines, weff)
    assert s["block_rows"] == rows and s["row_blocks"] > 1, s


@pytest.mark.parametrize("esize", [8, 4])
def test_lines_of_32_lanes(esize):
    """Contiguous lines of 209 to 383 points (32 lanes each): divide and conquer up to 250 lanes an SM."""
    assert hjlo.shape_query(250, 752, 153, esize)["segment_rows"] < 9
    assert hjlo.shape_query(250, 1400, 153, esize)["segment_rows"] in (9, 13)
    assert hjlo.shape_query(414, 1000, 99, esize)["segment_rows"] in (9, 13)
