"""Band tiles of the boundary strips, 8, 16 or 32 nodes long: every column that a tile's output nodes and face terms read
lies in the window that the tile stages, for every remainder of the block's length and both ends (the extents of the
operators' rows are those that test_strip_extents pins against the oracle)."""
import os
import re

import pytest

TABLES = os.path.join(os.path.dirname(__file__), "..", "paper_2003_12811_gb300", "csrc", "sbp_tables.inc")
MIN_NODES = {2: 5, 4: 18, 6: 27}


def _consts(order):
    txt = open(TABLES).read()
    return {m.group(1): int(m.group(2)) for m in re.finditer(r"#define SBP%d_(\w+) (-?\d+)" % order, txt)}


def _narrow(c, n, i):
    """Columns of row i of D_xx^FC, through u and b."""
    if i < c["NCLOS"]:
        return 0, c["NCLOSJ"] - 1
    if i >= n - c["NCLOS"]:
        return n - c["NCLOSJ"], n - 1
    return i - (c["Q"] - c["ELO"]), i + max(c["Q"], c["EHI"])


def _first(c, n, i):
    """Columns of row i of D."""
    if i < c["NB"]:
        return 0, c["NCOL"] - 1
    if i >= n - c["NB"]:
        return n - c["NCOL"], n - 1
    return i - c["Q"], i + c["Q"]


def _transpose(c, n, s):
    """Rows of D with a non-zero in column s (the tangential transpose of a face term)."""
    lo, hi = s - c["Q"], s + c["Q"]
    if s < c["NCOL"]:
        lo, hi = 0, max(hi, c["NB"] - 1)
    if s >= n - c["NCOL"]:
        lo, hi = min(lo, n - c["NB"]), n - 1
    return max(lo, 0), min(hi, n - 1)


@pytest.mark.parametrize("order", (2, 4, 6))
@pytest.mark.parametrize("tl", (8, 16, 32))
def test_band_tiles_read_inside_their_window(order, tl):
    c = _consts(order)
    ht = (c["Q"] - c["ELO"] + 3) // 4 * 4
    width = tl + 2 * ht + 4
    for n in range(MIN_NODES[order], MIN_NODES[order] + 3 * tl + 9):
        seen = set()
        for x0 in range(0, n, tl):
            w = min(tl, n - x0)
            xs = (min(x0, max(0, n - tl)) & ~3) - ht
            assert xs % 4 == 0                              # a copy starts on a 16-byte boundary
            reads = []
            for i in range(x0, x0 + w):
                seen.add(i)
                reads += [_narrow(c, n, i), _first(c, n, i), _transpose(c, n, i)]
            if x0 < c["NCOL"]:                              # terms of the faces across the band's ends
                reads.append((0, c["NCOL"] - 1))
            if x0 + w > n - c["NCOL"]:
                reads.append((n - c["NCOL"], n - 1))
            for lo, hi in reads:
                assert 0 <= lo and hi < n and xs <= lo and hi < xs + width, (n, x0, lo, hi, xs)
        assert seen == set(range(n))
