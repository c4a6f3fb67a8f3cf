"""Host-side check of the digit planes' storage image (no GPU).

Planes are stored as the image that the MMA's 32-byte-swizzle operand has in shared memory, and
copied in box rows of 512 bytes (16 stored rows).  This test restates the storage position of a value
(its row's 16-byte halves swap with bit 2 of the row), checks it against the swizzle of the operand
(16-byte chunk index, exclusive or, address bit 7) for boxes read along the rows and MN-major, and
checks the starting rows of a product and the padded ragged rows of the packed layout."""
import numpy as np
import pytest

BK, BM, GRAN = 16, 128, 16


def _pos(r, k):
    """Position of value k (0..15) of row r inside a K block, in values of 2 bytes."""
    return r * BK + (k ^ ((r & 4) << 1))


def _swizzled(byte):
    """Address of a byte of a 32-byte-swizzled operand tile: bit 4 ^= bit 7."""
    return byte ^ ((byte >> 3) & 16)


@pytest.mark.parametrize("row0", [0, 16, 48, 368])
def test_image_is_the_swizzled_tile(row0):
    """A box of whole 512-byte rows lands at a 256-byte-aligned address: what the operand reads for
    (row, k) there is the stored value, for every row of the tile."""
    R = row0 + BM
    plane = np.empty(R * BK, dtype=np.int64)
    for r in range(R):
        for k in range(BK):
            plane[_pos(r, k)] = 1000 * r + k
    smem = plane[row0 * BK:(row0 + BM) * BK]           # plain copy
    for r in range(BM):
        for k in range(BK):
            assert smem[_swizzled(2 * (r * BK + k)) // 2] == 1000 * (row0 + r) + k


def test_image_read_mn_major():
    """An MN-major box is 16 stored rows (values of K) of 8 consecutive K blocks (values of M), 512
    bytes each: within one, the same swizzle holds."""
    rows, nkb, row0 = 64, 8, 32
    planes = np.empty((nkb, rows * BK), dtype=np.int64)
    for b in range(nkb):
        for r in range(rows):
            for k in range(BK):
                planes[b, _pos(r, k)] = 1000 * r + 16 * b + k
    smem = planes[:, row0 * BK:(row0 + 16) * BK].reshape(-1)
    for m in range(BM):
        for k in range(16):
            byte = 512 * (m // 16) + 2 * (k * BK + m % 16)
            assert smem[_swizzled(byte) // 2] == 1000 * (row0 + k) + m


@pytest.mark.parametrize("n", [16, 37, 100, 300])
def test_products_start_at_box_rows(n):
    """A chunk's rows (L, mu) from l0 n on: the product starts row_skip rows early at a multiple of 16,
    and the rows it drops and the tiles it adds leave exactly the chunk's rows."""
    for l0, nL in ((0, 5), (7, 5), (12, 1)):
        a_row0, M = l0 * n, nL * n
        skip = a_row0 % GRAN
        start, tiles = a_row0 - skip, (M + skip + BM - 1) // BM
        assert start % GRAN == 0 and 0 <= skip < GRAN
        rows = [start + t for t in range(tiles * BM) if 0 <= t - skip < M]
        assert rows == list(range(a_row0, a_row0 + M))


@pytest.mark.parametrize("n", [129, 300, 383, 400, 1200])
def test_ragged_rows_start_at_box_rows(n):
    """The ragged rows of every b^L take rp rows, a multiple of 16, so that the box of K block kb =
    8 J + kk (J past the last whole block) starts at row L rp + 16 (kb - 8 nb1); rows j >= r are
    zero padding that no product stores."""
    nb1, r = n // BM, n % BM
    rp = (r + GRAN - 1) // GRAN * GRAN
    for L in (0, 1, 5, 311):
        base = L * rp - 8 * nb1 * BK
        for kb in range(8 * nb1, (n + BK - 1) // BK):
            y = base + kb * BK
            assert y % GRAN == 0 and L * rp <= y and y + BK <= (L + 1) * rp
    live = [(row // rp, row % rp) for row in range(4 * rp) if row % rp < r]
    assert live == [(L, j) for L in range(4) for j in range(r)]
