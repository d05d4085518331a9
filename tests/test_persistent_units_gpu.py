"""GPU test of the persistent launch's units (8 or 16 atoms, or a whole tile):
replicas whose last unit is ragged or empty, tiles smaller than a unit's share,
and replicas that one CTA steps alone (several units each, no barrier).  The
per-phase kernels take the same atoms in tiles; both hold FP64 sums over the
same FP32 rows, so observables agree as in the driver comparison (1e-10) and
both count the same list rebuilds."""
import numpy as np
import pytest

from conftest import small2d, small3d, thermalise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd as H
    _build.build()
    return H


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("block,many", [(32, 1), (64, 1), (128, 1), (128, 60), (64, 60)])
def test_units_match_per_phase_kernels(hd, prec, block, many):
    from paper_0909_5215_gb300 import model as M
    base = [thermalise(small2d(cols=7, rows=4, n_tip=5, kT=0.15), seed=1), thermalise(small3d(kT=0.15), seed=2),
            thermalise(small2d(cols=13, rows=5, n_tip=13, kT=0.15), seed=3)]
    base[1].nhc_len = 2
    reps = []
    for q in range(many):
        for r in base:
            c = r.copy()
            c.rep_id, c.dvmax, c.sig_lo, c.sig_hi = len(reps), 0.3, 0.0, 60.0
            reps.append(c)
    p = M.Params(prec=prec, bias_on=1)
    a = hd.Batch(reps, p, driver=hd.HD_DRIVER_KERNELS, block=block)
    b = hd.Batch(reps, p, driver=hd.HD_DRIVER_PERSISTENT, block=block)
    assert b.info()["driver"] == hd.HD_DRIVER_PERSISTENT
    for n in (1, 9, 30):
        a.step(n)
        b.step(n)
    oa, ob = a.obs(), b.obs()
    assert oa[:, 12].max() > 0 and np.array_equal(oa[:, 12], ob[:, 12])
    assert np.allclose(oa, ob, rtol=1e-10, atol=1e-11)
    a.close()
    b.close()
