"""The resident PCG kernel's split of the rows, restated on the CPU: its items (tiles of falling
size, whole or cut into chunks) and the shares of its workers cover every row exactly once."""
from math import comb

import pytest

from test_tile_layout import _rank, _unrank


def _items(L, n_up, B, chunk):
    H = L - B
    classes = sorted(range(max(0, n_up - H), min(B, n_up) + 1), key=lambda p: -comb(B, p))
    out = []
    for p in classes:
        rows = comb(B, p)
        for i in range(comb(H, n_up - p)):
            t = _unrank(H, n_up - p, i)
            off = _rank((t << B) | ((1 << p) - 1))
            out += [(off + jb, off + min(rows, jb + chunk)) for jb in range(0, rows, chunk)]
    return out


def _there_and_back(items, workers):
    shares = []
    for w in range(workers):
        full, left = divmod(items, workers)
        count = full + (1 if left > (workers - 1 - w if full & 1 else w) else 0)
        shares.append([i * workers + (workers - 1 - w if i & 1 else w) for i in range(count)])
    return shares


def _even(items, blocks, warps=24):
    shares = []
    for b in range(blocks):
        b0, b1 = items * b // blocks, items * (b + 1) // blocks
        for w in range(warps):
            first = b0 + w
            count = (b1 - first + warps - 1) // warps if first < b1 else 0
            shares.append([first + i * warps for i in range(count)])
    return shares


@pytest.mark.parametrize("L,n_up,B,chunk,blocks", [
    (8, 4, 6, 32, 1), (10, 3, 8, 16, 3), (12, 6, 10, 252, 152), (12, 6, 10, 8, 11), (13, 5, 11, 24, 152),
    (14, 7, 9, 126, 7), (16, 8, 13, 48, 152), (16, 0, 13, 32, 2), (16, 16, 13, 32, 2)])
def test_every_row_has_one_worker(L, n_up, B, chunk, blocks):
    items = _items(L, n_up, B, chunk)
    whole_tiles = chunk >= comb(B, B // 2)
    shares = _there_and_back(len(items), 3 * blocks) if whole_tiles else _even(len(items), blocks)
    taken = sorted(i for s in shares for i in s)
    assert taken == list(range(len(items)))
    rows = sorted(items[i] for i in taken)
    assert rows[0][0] == 0 and rows[-1][1] == comb(L, n_up)
    assert all(a[1] == b[0] for a, b in zip(rows, rows[1:]))
