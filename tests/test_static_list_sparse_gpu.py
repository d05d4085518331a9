"""GPU test of hd_nlist_static where cells hold few atoms and a warp takes a
row by itself: just below and at six atoms a cell, a gas, dense blobs in an
empty box (stencils of several hundred candidates, rows at their capacity), a
film on an open axis, more rows than warps.  Rows are whole numbers and must
equal a brute-force search (the same FP64 operations)."""
import numpy as np
import pytest

from test_static_list_gpu import RL, build, hd  # noqa: F401

pytestmark = pytest.mark.gpu
CUBE = (21.0, 21.0, 21.0)        # seven cells along every axis


def uniform(n, box, periodic, seed, high=8.0):
    rng = np.random.default_rng(seed)
    return rng.uniform(-0.5, 0.5, size=(n, 3)) * [b if p else high for b, p in zip(box, periodic)]


def blobs(n, seed):
    rng = np.random.default_rng(seed)
    at = np.array([[0.0, 0.0, 0.0], [10.4, -10.4, 3.0], [-4.2, 6.1, 9.9]])
    return at[np.arange(n) % 3] + rng.uniform(-1.35, 1.35, size=(n, 3))


@pytest.mark.parametrize("x,box,periodic", [
    (uniform(2057, CUBE, (1, 1, 1), 1), CUBE, (1, 1, 1)),
    (uniform(2058, CUBE, (1, 1, 1), 2), CUBE, (1, 1, 1)),
    (uniform(40, CUBE, (1, 1, 1), 3), CUBE, (1, 1, 1)),
    (uniform(9, (9.0, 200.0, 9.0), (1, 1, 1), 4), (9.0, 200.0, 9.0), (1, 1, 1)),
    (blobs(300, 5), CUBE, (1, 1, 1)),
    (uniform(900, (60.0, 45.0, 0.0), (1, 1, 0), 6, 2.0), (60.0, 45.0, 0.0), (1, 1, 0)),
    (uniform(700, (0.0, 0.0, 0.0), (0, 0, 0), 7, 30.0), (0.0, 0.0, 0.0), (0, 0, 0)),
    (uniform(6500, (64.0, 64.0, 64.0), (1, 1, 1), 8), (64.0, 64.0, 64.0), (1, 1, 1))])
def test_rows_equal_brute_force(hd, x, box, periodic):  # noqa: F811
    rows = [r for k in range(0, len(x), 500) for r in brute_part(x, k, box, periodic)]
    most = max(1, max(len(r) for r in rows))
    assert most <= 160
    st, nbr, nnb = build(hd, x, box, periodic, most)
    assert st == hd.HD_OK
    for i, r in enumerate(rows):
        assert nnb[i] == len(r)
        assert np.array_equal(nbr[i, :len(r)], r) and (nbr[i, len(r):] == -1).all()
    if most > 1:
        assert build(hd, x, box, periodic, most - 1)[0] == hd.HD_ERR_OVERFLOW
    assert build(hd, x, box, periodic, most)[0] == hd.HD_OK


def brute_part(x, k, box, periodic):
    """Rows k .. k + 499 of the brute-force search (all pairs of 6,500 atoms at once would take 1 GB)."""
    d = x[k:k + 500, None, :] - x[None, :, :]
    for a in range(3):
        if periodic[a]:
            d[..., a] -= box[a] * np.rint(d[..., a] / box[a])
    r2 = (d[..., 0] ** 2 + d[..., 1] ** 2) + d[..., 2] ** 2
    r2[np.arange(len(r2)), k + np.arange(len(r2))] = np.inf
    return [np.flatnonzero(r < RL * RL) for r in r2]
