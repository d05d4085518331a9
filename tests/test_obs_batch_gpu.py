"""GPU test: the observables of all replicas in one read equal those read one
replica at a time, after stepping, after a quench, and after an error (the
record can still be read then)."""
import numpy as np
import pytest

from conftest import small2d, small3d, thermalise

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
def test_all_observables_equal_single_reads(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import hd as H, model as M
    reps = [thermalise(small2d(), seed=1), thermalise(small3d(), seed=2), thermalise(small2d(cols=14), seed=3)]
    for k, r in enumerate(reps):
        r.rep_id, r.dvmax, r.sig_lo, r.sig_hi = k, 0.2, 1.0, 30.0
    reps[2].nhc_len = 2
    b = H.Batch(reps, M.Params(prec=prec, bias_on=1))
    for go in (lambda: b.step(7), lambda: b.quench(max_iter=20)):
        go()
        got = b.obs()
        assert np.array_equal(got, np.array([[b.obs(r)[f] for f in H.OBS_FIELDS] for r in range(3)]))
        assert np.isfinite(got).all() and (got[:, 0] == 7).all()
    with pytest.raises(H.HdError):
        b.step(-1)
    assert np.array_equal(b.obs(), got)
    b.close()
