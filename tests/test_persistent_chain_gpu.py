"""GPU test of the Nose-Hoover chain in the persistent launch where a replica
spans many CTAs: on a call's last step the closing scale rewrites the kinetic
sums that every CTA has just read, so no CTA may scale before all have read
them.  Calls of one step end that way each time.  A CTA that mixed old and new
sums would scale its atoms by another factor and, as the leader, keep another
chain state, so two runs must give the same words, both drivers must agree to
rounding (1e-10, as in the driver comparison), and K must be that of the
velocities (FP64 sums of the same terms in another order: 1e-12)."""
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
def test_last_step_of_a_call(hd, prec):
    from paper_0909_5215_gb300 import model as M
    reps = [thermalise(M.paper3d(kT=0.1), amp=0.02, seed=1), thermalise(small3d(kT=0.15), amp=0.04, seed=2),
            thermalise(small2d(cols=40, rows=6, n_tip=13), amp=0.04, seed=3)]
    rng = np.random.default_rng(4)
    for k, r in enumerate(reps):
        r.rep_id, r.nhc_len, r.nhc_tau = k, 3, 0.5
        on = np.array([1.0, 1.0, 1.0 if r.dim == 3 else 0.0]) * (r.role == 1)[:, None]
        r.vel = on * rng.normal(0.0, r.kT ** 0.5, r.pos.shape)
    p = M.Params(prec=prec, bias_on=0)
    runs = []
    for drv in (hd.HD_DRIVER_PERSISTENT, hd.HD_DRIVER_PERSISTENT, hd.HD_DRIVER_KERNELS):
        b = hd.Batch(reps, p, driver=drv)
        if drv == hd.HD_DRIVER_PERSISTENT:
            assert b.info()["persistent_ctas"] > 100
        for n in [1] * 40 + [2, 7]:
            b.step(n)
        ob = b.obs()
        for k, r in enumerate(reps):
            v = b.velocities(k)
            body = ob[k, hd.OBS_FIELDS.index("vbody_x"):][:3]
            kin = 0.5 * (v[r.role == 1] ** 2).sum() + 0.5 * (r.role == 2).sum() * (body ** 2).sum()
            assert prec == 1 or ob[k, hd.OBS_FIELDS.index("K")] == pytest.approx(kin, rel=1e-12)
        runs.append((ob, [b.positions(k) for k in range(3)], [b.velocities(k) for k in range(3)]))
        b.close()
    for x, y in zip(runs[0], runs[1]):
        assert all(np.array_equal(u, v) for u, v in zip(x, y))
    assert np.allclose(runs[0][0], runs[2][0], rtol=1e-10, atol=1e-12)
    for k in range(3):
        assert np.abs(runs[0][1][k] - runs[2][1][k]).max() < 1e-10
        assert np.abs(runs[0][2][k] - runs[2][2][k]).max() < 1e-9
