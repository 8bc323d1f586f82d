"""Bank conflicts of the partial tiles that grass_fim's blocks exchange, from the index arithmetic of the source (no GPU)."""
import pathlib
import re

import pytest

SRC = (pathlib.Path(__file__).resolve().parent.parent / "paper_2505_18976_b200" / "csrc" / "grass_fim_gram.cu").read_text()
EXPR = re.search(r"int slice_offset\(int row, int c\)\s*\{\s*return ([^;]*);", SRC).group(1)
TILE = int(re.search(r"constexpr int TILE = (\d+);", SRC).group(1))


def _offset(row, c):
    return eval(EXPR, {"row": row, "c": c, "TILE": TILE})


def _ways(words):
    """Largest number of different words of one bank among the lanes' words."""
    banks = {}
    for w in words:
        banks.setdefault(w % 32, set()).add(w)
    return max(len(b) for b in banks.values())


def test_offsets_are_a_permutation_of_whole_chunks():
    assert sorted(_offset(r, c) for r in range(TILE) for c in range(TILE)) == list(range(TILE * TILE))
    assert all(_offset(r, c) % 4 == c % 4 for r in range(TILE) for c in range(TILE))


# 16-byte accesses are served eight lanes at a time
def test_writers_and_readers_of_rows():
    for first in range(0, TILE, 8):
        for c in range(0, TILE, 4):
            assert _ways([_offset(first + lane, c) + e for lane in range(8) for e in range(4)]) == 1
    for row in range(TILE):
        for c in range(0, TILE, 32):
            assert _ways([_offset(row, c + 4 * lane) + e for lane in range(8) for e in range(4)]) == 1


# consecutive threads take four rows each of a column, then of the next column
@pytest.mark.parametrize("rows,ways", [(16, 1), (32, 1), (64, 2), (128, 4)])
def test_readers_of_four_rows_of_a_column(rows, ways):
    for first in range(0, rows * TILE // 4, 32):
        for part in range(4):
            lanes = [(e % (rows // 4) * 4 + part, e // (rows // 4)) for e in range(first, first + 32)]
            assert _ways([_offset(r, c) for r, c in lanes]) <= ways
