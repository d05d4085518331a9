"""GPU tests of routes that only some batches take: the rebuild plan of more
than 4,000 replicas, the put-off evaluation of the split form, a chain in a
batch that forms H.(r - r_O) on demand, and rows built inside the persistent
launch.  The same replicas in a batch on another route are the reference, at
rounding (1e-9 in positions, FP64 form); rows are whole numbers and must equal
the oracle's brute-force rows."""
import numpy as np
import pytest

from conftest import small2d, small3d, thermalise

pytestmark = pytest.mark.gpu
NREB = 12


@pytest.fixture(scope="module")
def hd():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd as H
    _build.build()
    return H


def test_plan_of_more_than_4000_replicas(hd, oracle_mod):
    from paper_0909_5215_gb300 import model as M
    kinds = [thermalise(small2d(cols=7, rows=4, n_tip=5, kT=0.15), amp=0.06, seed=s) for s in range(8)]
    reps = []
    for k in range(4100):
        r = kinds[k % 8].copy()
        r.rep_id = k
        reps.append(r)
    some = [0, 5, 31, 32, 2049, 3999, 4000, 4098, 4099]
    p = M.Params(prec=0, bias_on=0)
    a = hd.Batch(reps, p, driver=hd.HD_DRIVER_KERNELS)
    b = hd.Batch([reps[k] for k in some], p, driver=hd.HD_DRIVER_KERNELS)
    at = a.info()["launches"], b.info()["launches"]
    for n in (1, 40):
        a.step(n)
        b.step(n)
    # the plan is a kernel of its own
    assert b.info()["launches"] - at[1] == 2 * 2 + 6 * 41 and a.info()["launches"] - at[0] == 2 * 2 + 7 * 41
    oa, ob = a.obs(), b.obs()
    assert ob[:, NREB].max() > 0 and (oa[:, NREB] > 0).sum() > 100
    for q, k in enumerate(some):
        assert oa[k, NREB] == ob[q, NREB]
        assert np.abs(a.positions(k) - b.positions(q)).max() < 1e-9
        assert all(np.array_equal(x, y) for x, y in zip(a.rows(k), b.rows(q)))
    a.quench(max_iter=6)
    b.quench(max_iter=6)
    for q, k in enumerate(some):
        assert np.abs(a.qpos(k) - b.qpos(q)).max() < 1e-9
        o = oracle_mod.OracleReplica(reps[k], p)
        o.set_positions(a.positions(k))
        o.nlist_brute()
        assert all(np.array_equal(g, e) for g, e in zip(a.rows(k), o.rows()))
    a.close()
    b.close()


def test_unexpected_entry_in_the_split_form(hd):
    """At rest at r_O the slope is zero and the band lies where it is a step later: over 200,000 atoms the
    evaluation is put off and made up for; the same replicas in a smaller batch always form the Hessian
    term.  Both walk a row with one lane, so their forces are the same words."""
    from paper_0909_5215_gb300 import model as M
    base = thermalise(M.afm3d(nx=20, ny=20, nz=6, tip_radius=3.0, kT=0.1, eps=M.PAPER_EPS_3D), amp=0.0, seed=9)
    reps = []
    for k in range(22):
        r = base.copy()
        r.rep_id, r.dvmax, r.pos_ref = k, 0.4, base.pos.copy()
        reps.append(r)
    assert sum(r.n for r in reps) >= 200000 and 5 * base.n >= 152 * 8 * 32
    first = hd.Batch(reps[:5], M.Params(prec=1, bias_on=0))
    assert (first.obs()[:, 6] == 0.0).all()
    first.step(1)
    s1 = first.obs()[:, 6]
    first.close()
    for k, r in enumerate(reps):
        s = s1[k % 5]
        w = 0.3 * abs(s)
        r.sig_lo, r.sig_hi = (s - w, s + w) if k % 5 != 2 else (s + 1e3, s + 2e3)
        assert not (r.sig_lo <= 0.0 <= r.sig_hi)
    p = M.Params(prec=1, bias_on=1)
    a, b = hd.Batch(reps, p), hd.Batch(reps[:5], p)
    a.step(3)
    b.step(3)
    oa, ob = a.obs(), b.obs()
    assert (oa[[0, 1, 3, 4], 25] >= 1).all()
    assert np.array_equal(oa[:5, 24:27], ob[:, 24:27])
    assert np.allclose(oa[:5, :12], ob[:, :12], rtol=1e-12, atol=1e-12)
    for k in range(5):
        assert np.abs(a.positions(k) - b.positions(k)).max() < 1e-12
        assert np.array_equal(a.forces(k), b.forces(k)) and np.array_equal(a.hdr(k), b.hdr(k))
    a.close()
    b.close()


def test_chain_with_the_hessian_on_demand(hd):
    from paper_0909_5215_gb300 import model as M
    base = thermalise(small3d(nx=8, nz=4, radius=3.0), amp=0.04, seed=7)
    rng = np.random.default_rng(8)
    reps = []
    for k in range(9):
        r = base.copy()
        r.pos_ref = base.pos - 0.02 * (base.role == 1)[:, None] * rng.normal(size=base.pos.shape)
        r.vel = (base.role == 1)[:, None] * rng.normal(0.0, 0.3, base.pos.shape)
        r.rep_id, r.dvmax, r.nhc_len, r.nhc_tau = k, 0.4, 3, 0.5
        reps.append(r)
    probe = hd.Batch(reps, M.Params(prec=0, bias_on=0))
    s = [probe.obs()[:, 6]]
    for _ in range(3):
        probe.step(10)
        s.append(probe.obs()[:, 6])
    probe.close()
    for k, r in enumerate(reps):
        a, z = min(v[k] for v in s), max(v[k] for v in s)
        # about its band throughout; crossing it; below it
        r.sig_lo, r.sig_hi = [(a - 0.5 * abs(a), z + 0.5 * abs(z)), (0.5 * (a + z), 0.5 * (a + z) + 0.1 * (z - a)),
                              (z + 1e4, z + 2e4)][k % 3]
    p = M.Params(prec=0, bias_on=1)
    assert sum(r.n for r in reps) >= 8192 > 3 * base.n
    a, b = hd.Batch(reps, p), hd.Batch(reps[:3], p)
    for n in (1, 2, 30):
        a.step(n)
        b.step(n)
    oa, ob = a.obs(), b.obs()
    assert oa[0, 25] > 0 and oa[2, 24] == 33            # in the band at some time; never
    assert np.array_equal(oa[:3, 24:27], ob[:, 24:27])
    assert np.allclose(oa[:3], ob, rtol=1e-9, atol=1e-11)
    for k in range(3):
        assert np.abs(a.positions(k) - b.positions(k)).max() < 1e-9
    a.close()
    b.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_rows_built_inside_the_persistent_launch(hd, oracle_mod, prec):
    """A one-step call whose step rebuilds leaves the rows of the positions it returns."""
    from paper_0909_5215_gb300 import model as M
    reps = [thermalise(M.afm3d(nx=nx, ny=ny, nz=3, tip_radius=2.5, kT=0.15, eps=M.PAPER_EPS_3D), amp=0.05, seed=nx)
            for nx, ny in ((4, 4), (6, 6), (8, 5))]
    reps += [thermalise(small2d(cols=c, rows=6, n_tip=13, kT=0.15), amp=0.05, seed=c) for c in (9, 64)]
    rng = np.random.default_rng(3)
    for k, r in enumerate(reps):
        on = np.array([1.0, 1.0, 1.0 if r.dim == 3 else 0.0]) * (r.role == 1)[:, None]
        r.rep_id, r.vel = k, on * rng.normal(0.0, 0.6, r.pos.shape)
    p = M.Params(prec=prec, bias_on=0)
    b = hd.Batch(reps, p, driver=hd.HD_DRIVER_PERSISTENT, block=64)
    assert b.info()["driver"] == hd.HD_DRIVER_PERSISTENT
    seen, done = b.obs()[:, NREB], np.zeros(len(reps), dtype=int)
    for _ in range(200):
        b.step(1)
        now = b.obs()[:, NREB]
        for k in np.flatnonzero(now > seen):
            if done[k] >= 2:
                continue
            o = oracle_mod.OracleReplica(reps[k], p)
            o.set_positions(b.positions(k))
            o.nlist_brute()
            assert all(np.array_equal(g, e) for g, e in zip(b.rows(k), o.rows()))
            done[k] += 1
        seen = now
        if (done >= 2).all():
            break
    assert (done >= 1).all()
    b.close()
