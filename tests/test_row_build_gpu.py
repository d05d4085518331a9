"""GPU test of the Verlet-row build where its staging changes form: one cell,
three cells and four cells along a periodic axis (offsets from the cell's
centre are used from four on), replicas of both kinds in one batch, stencils
that do not fill the last 64 candidates, and rows at their capacity.  Rows are
whole numbers and must equal the oracle's brute-force rows, at the start and
after steps with rebuilds."""
import numpy as np
import pytest

from conftest import small2d, thermalise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd as H
    _build.build()
    return H


def replicas():
    from paper_0909_5215_gb300 import model as M
    out = [thermalise(M.afm3d(nx=nx, ny=ny, nz=nz, tip_radius=2.5, kT=0.15, eps=M.PAPER_EPS_3D), amp=0.05, seed=nx + ny)
           for nx, ny, nz in ((4, 4, 3), (6, 6, 3), (6, 9, 4), (8, 8, 3), (13, 4, 3))]
    out += [thermalise(small2d(cols=c, rows=6, n_tip=13, kT=0.15), amp=0.05, seed=c) for c in (7, 9, 11, 64)]
    for k, r in enumerate(out):
        r.rep_id = k
    return out


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("driver", ["kernels", "persistent"])
def test_rows_equal_oracle(hd, oracle_mod, prec, driver):
    from paper_0909_5215_gb300 import model as M
    reps, p = replicas(), M.Params(prec=prec, bias_on=0)
    drv = hd.HD_DRIVER_KERNELS if driver == "kernels" else hd.HD_DRIVER_PERSISTENT
    b = hd.Batch(reps, p, driver=drv, block=64)
    rebuilt = 0
    for steps in (0, 40):
        b.step(steps)
        for k, r in enumerate(reps):
            o = oracle_mod.OracleReplica(r, p)
            # the list belongs to the positions of its last build: the initial ones until one is rebuilt
            if steps:
                rebuilt += int(b.obs(k)["n_rebuild"])
                continue
            o.nlist_brute()
            assert all(np.array_equal(g, e) for g, e in zip(b.rows(k), o.rows()))
    assert rebuilt > 0
    # a zero-iteration quench relists at the current positions
    b.quench(max_iter=0)
    for k, r in enumerate(reps):
        o = oracle_mod.OracleReplica(r, p)
        o.set_positions(b.positions(k))
        o.nlist_brute()
        assert all(np.array_equal(g, e) for g, e in zip(b.rows(k), o.rows()))
    b.close()


def test_row_capacity(hd, oracle_mod):
    from paper_0909_5215_gb300 import model as M
    r, p = replicas()[3], M.Params(prec=1, bias_on=0)
    o = oracle_mod.OracleReplica(r, p)
    o.nlist_brute()
    most = max(len(x) for x in o.rows())
    b = hd.Batch([r], p, maxnb=most)
    assert all(np.array_equal(g, e) for g, e in zip(b.rows(0), o.rows()))
    b.close()
    with pytest.raises(hd.HdError) as e:
        hd.Batch([r], p, maxnb=most - 1)
    assert e.value.status == hd.HD_ERR_OVERFLOW
