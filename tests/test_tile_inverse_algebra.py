"""The column-tile inverse restated in numpy: panels of TW columns, rows that stay where they are and keep
the position they would hold after the interchanges, tiles that take a panel as y_r + C_r y_K (a
pivot row: C_r y_K), the next panel factored on its tile alone, and X[i][c] = W[row at position
i][position of row c] at the end."""
import numpy as np
import pytest


def tile_inverse(M, TW):
    n = len(M)
    W = M.astype(complex).copy()
    pos = np.arange(n)                       # position of each row
    singular = False
    tiles = [slice(t, min(t + TW, n)) for t in range(0, n, TW)]

    def factor(t):                           # the pivot steps of tile t's columns, on that tile
        nonlocal singular
        a = W[:, tiles[t]]
        for j in range(a.shape[1]):
            k = tiles[t].start + j
            cand = [(-abs(a[r, j]) ** 2, pos[r], r) for r in range(n) if pos[r] >= k]
            _, p, win = min(cand)            # the largest, first in position order
            d = a[win, j]
            singular |= d == 0
            di = 0.0 if d == 0 else 1.0 / d
            row = a[win].copy()
            h = -a[:, j] * di
            new = a + np.outer(h, row)
            new[win] = row * di
            new[:, j] = h
            new[win, j] = di
            a[:] = new
            at_k = int(np.nonzero(pos == k)[0][0])
            pos[at_k], pos[win] = p, k

    factor(0)
    for panel in range(len(tiles)):
        K = tiles[panel]
        C = W[:, K]
        pivots = [int(np.nonzero(pos == k)[0][0]) for k in range(K.start, K.stop)]
        for t in range(len(tiles)):
            if t == panel:
                continue
            y = W[:, tiles[t]]
            yk = y[pivots].copy()
            y[pivots] = 0.0
            y += C @ yk
        if panel + 1 < len(tiles):
            factor(panel + 1)
    row_at = np.argsort(pos)
    return W[np.ix_(row_at, pos)], singular


@pytest.mark.parametrize("TW", [8, 16])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 31, 40, 57])
def test_inverse(n, TW):
    rng = np.random.default_rng(100 * n + TW)
    M = rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n))
    M /= np.sqrt(n)
    M[np.arange(n), rng.permutation(n)] += 2.0
    X, singular = tile_inverse(M, TW)
    assert not singular
    ref = np.linalg.inv(M)
    assert np.abs(X - ref).max() <= 64 * n * 2.0 ** -53 * np.linalg.norm(M) * np.linalg.norm(ref) * np.abs(ref).max()


def test_equal_candidates_take_the_first_position():
    M = np.array([[0, 1, 0], [1, 0, 0], [1, 0, 1]], dtype=complex)
    X, singular = tile_inverse(M, 8)
    assert not singular and np.array_equal(X, np.linalg.inv(M))


def test_zero_column_is_seen():
    M = np.eye(12, dtype=complex)
    M[:, 10] = 0.0
    assert tile_inverse(M, 8)[1]
