"""GPU test of hd_nlist_static at the sizes where its staged row build can go
wrong: rows that do not fill a group of four or a warp, one cell per axis, a
capacity that a row just fills, atoms in no particular order.  Rows are whole
numbers and must equal a brute-force search (the same FP64 operations)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
RL = 2.8


@pytest.fixture(scope="module")
def hd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd as H
    _build.build()
    return H


def brute(x, box, periodic, rl):
    d = x[:, None, :] - x[None, :, :]
    for a in range(3):
        if periodic[a]:
            d[..., a] -= box[a] * np.rint(d[..., a] / box[a])
    r2 = (d[..., 0] ** 2 + d[..., 1] ** 2) + d[..., 2] ** 2
    np.fill_diagonal(r2, np.inf)
    return [np.flatnonzero(r < rl * rl) for r in r2]


def build(hd, x, box, periodic, maxnb, rl=RL):
    import torch
    n = len(x)
    pos = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    nbr = torch.full((n, maxnb), -7, dtype=torch.int32, device="cuda")
    nnb = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    st = hd.hd_nlist_static(pos.data_ptr(), n, box, periodic, rl, maxnb, nbr.data_ptr(), nnb.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    return st, nbr.cpu().numpy(), nnb.cpu().numpy()


@pytest.mark.parametrize("n,box,periodic,seed", [
    (1, (0.0, 0.0, 0.0), (0, 0, 0), 1),            # a single atom: no extent on any axis
    (2, (6.0, 6.0, 6.0), (1, 1, 1), 2),            # one cell on every axis
    (33, (6.0, 0.0, 0.0), (1, 0, 0), 3),           # one cell along x, open y and z
    (129, (40.0, 0.0, 0.0), (1, 0, 0), 4),         # a strip
    (700, (9.0, 9.0, 9.0), (1, 1, 1), 5),          # three cells on every axis: the stencil is the box
    (1500, (17.0, 11.3, 0.0), (1, 1, 0), 6)])      # slab, five by four cells
def test_rows_equal_brute_force(hd, n, box, periodic, seed):
    rng = np.random.default_rng(seed)
    ext = [box[a] if periodic[a] else (8.0 if n > 1 else 0.0) for a in range(3)]
    x = rng.uniform(-0.5, 0.5, size=(n, 3)) * ext + 3.0
    rows = brute(x, box, periodic, RL)
    most = max(1, max(len(r) for r in rows))
    st, nbr, nnb = build(hd, x, box, periodic, most)
    assert st == hd.HD_OK
    for i, r in enumerate(rows):
        assert nnb[i] == len(r)
        assert np.array_equal(nbr[i, :len(r)], r) and (nbr[i, len(r):] == -1).all()
    if most > 1:
        assert build(hd, x, box, periodic, most - 1)[0] == hd.HD_ERR_OVERFLOW


def test_refused_inputs(hd):
    x = np.random.default_rng(7).uniform(0, 5, size=(40, 3))
    assert build(hd, x, (0.0, 5.0, 0.0), (1, 1, 0), 64)[0] == hd.HD_ERR_ARG        # periodic axis without a length
    assert build(hd, x, (5.0, 5.0, 0.0), (1, 1, 0), 161)[0] == hd.HD_ERR_ARG
    far = x.copy()
    far[0, 2] = 5000.0                                                             # over 1,023 cells on the open axis
    assert build(hd, far, (5.0, 5.0, 0.0), (1, 1, 0), 64)[0] == hd.HD_ERR_ARG
    bad = x.copy()
    bad[3, 2] = np.nan
    assert build(hd, bad, (5.0, 5.0, 0.0), (1, 1, 0), 64)[0] == hd.HD_ERR_NUMERIC
    assert build(hd, x, (5.0, 5.0, 0.0), (1, 1, 0), 64)[0] == hd.HD_OK             # an earlier error leaves no trace
