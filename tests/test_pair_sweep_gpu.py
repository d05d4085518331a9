"""GPU tests of the pair sweep's dispatch, at the sizes where it can go wrong.

Forces, energies and H.(r - r_O) against the FP64 oracle where a row is shared
by four lanes (small batches) and where it is not (over 38,912 atoms), with
axes that share one fixed-point unit and with axes that do not, rows that do
not fill a group of four, and rows with and without tip atoms.  Tolerances are
the project's: 1e-5 (split form) and 1e-12 (FP64 form), RMS relative.

A large batch takes H.(r - r_O) only for replicas expected in their bias band
(and sweeps one again that got there unexpectedly); the same replicas in small
batches take it always.  The two routes hold the same sums, so they agree to
the rounding of the sums' order: 1e-9 in positions after 60 steps in the FP64
form.
"""
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


def slab(nx, ny, nz, radius, seed, amp=0.04):
    from paper_0909_5215_gb300 import model as M
    return thermalise(M.afm3d(nx=nx, ny=ny, nz=nz, tip_radius=radius, kT=0.1, eps=M.PAPER_EPS_3D), amp=amp, seed=seed)


def shifted(r, seed):
    """r_O apart from the positions, so that H.(r - r_O) is not zero."""
    r.pos_ref = r.pos + np.random.default_rng(seed).normal(0.0, 0.05, r.pos.shape) * (r.role == 1)[:, None] * \
        np.array([1.0, 1.0, 1.0 if r.dim == 3 else 0.0])
    return r


def rms(a, b):
    return np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum())


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("block", [32, 64, 256])
@pytest.mark.parametrize("many", [False, True])
def test_sweep_matches_oracle(hd, oracle_mod, prec, block, many):
    from paper_0909_5215_gb300 import model as M
    reps = [shifted(r, k) for k, r in enumerate([
        thermalise(small2d(cols=8, rows=4, n_tip=5), amp=0.04, seed=1),        # fewer atoms than a tile
        slab(5, 5, 3, 2.5, 2), slab(5, 7, 3, 2.5, 3),                          # a common unit, and none
        thermalise(small2d(cols=23, rows=7, n_tip=30), amp=0.04, seed=4)])]
    reps[3].sig = ((1.0, 0.95), (0.95, 0.9))                                   # r_0 differs by type
    n_checked = len(reps)
    if many:
        big = shifted(slab(9, 9, 6, 3.0, 5), 6)
        reps += [big.copy() for _ in range(20)]
        assert sum(r.n for r in reps) > 152 * 8 * 32
        n_checked += 1
    for k, r in enumerate(reps):
        r.rep_id = k
    p = M.Params(prec=prec, bias_on=0)
    b = hd.Batch(reps, p, block=block)
    tol = 1e-12 if prec == 0 else 1e-5
    for k in range(n_checked):
        o = oracle_mod.OracleReplica(reps[k], p)
        o.nlist_brute()
        o.forces()
        assert rms(b.forces(k), o.f_lj) < tol
        assert rms(b.hdr(k), o.hdr) < tol
        assert rms(b.energies(k), o.e_atom) < tol
    b.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_hessian_only_where_needed_changes_nothing(hd, prec):
    from paper_0909_5215_gb300 import model as M
    nx, n = (10, 4) if prec == 0 else (20, 22)                                 # over 8,192 and 200,000 atoms
    base = slab(nx, nx, 6, 3.0, 8, amp=0.03)
    reps = []
    for k in range(n):
        r = base.copy()
        r.pos_ref = base.pos - 0.0
        r.pos = base.pos + np.random.default_rng(k).normal(0.0, 0.01, base.pos.shape) * (base.role == 1)[:, None]
        r.rep_id, r.dvmax = k, 0.4
        reps.append(r)
    # no band reached at first: read the slope that each replica starts from and the one a step later
    probe = hd.Batch(reps[:4], M.Params(prec=prec, bias_on=0))
    s = [probe.obs()[:, 6]]
    for _ in range(3):
        probe.step(10)
        s.append(probe.obs()[:, 6])
    probe.close()
    for k in range(4):
        a, z = min(v[k] for v in s), max(v[k] for v in s)
        # in its band throughout; crossing into and out of it; above it; below it
        lo, hi = [(a - 0.5 * abs(a), z + 0.5 * abs(z)), (0.5 * (a + z), 0.5 * (a + z) + 0.1 * (z - a)),
                  (-3.0, -2.0), (z + 1e4, z + 2e4)][k]
        for q in range(k, n, 4):
            reps[q].sig_lo, reps[q].sig_hi = lo, hi
    p = M.Params(prec=prec, bias_on=1)
    assert sum(r.n for r in reps) >= (8192 if prec == 0 else 200000)
    b = hd.Batch(reps, p)
    b.step(30)
    b.step(30)
    ob = b.obs()
    counts = ob[:4, 24:27]
    assert counts[0, 1] == 60 and counts[2, 2] == 60 and counts[3, 0] == 60 and (counts[1] > 0).sum() >= 2
    for k in range(4):
        one = hd.Batch([reps[k]], p)
        one.step(60)
        o1 = one.obs()[0]
        assert np.array_equal(o1[24:27], ob[k, 24:27])
        # split form: the trajectory tolerance of the other tests (1e-4).  Its sums
        # meet in another order when four lanes share a row, positions part by
        # ~1e-8, and a pair within that of rc, where the force jumps by 0.04, is
        # then cut a step sooner in one of them (~1e-6 in x a step from there on)
        assert np.abs(one.positions(0) - b.positions(k)).max() < (1e-9 if prec == 0 else 1e-4)
        tol = 1e-9 if prec == 0 else 1e-6
        assert abs(o1[2] - ob[k, 2]) < tol * abs(o1[2]) and abs(o1[6] - ob[k, 6]) < tol * abs(o1[6])
        assert rms(b.hdr(k), one.hdr(0)) < (1e-9 if prec == 0 else 1e-5)
        one.close()
    b.close()


def test_unexpected_entry_into_the_band(hd):
    """At rest at r_O the slope is zero; one step later it is not, and the band
    lies there: the sweep without the Hessian term is made up for."""
    from paper_0909_5215_gb300 import model as M
    base = slab(10, 10, 6, 3.0, 9, amp=0.0)
    reps = []
    for k in range(4):
        r = base.copy()
        r.rep_id, r.dvmax, r.pos_ref = k, 0.4, base.pos.copy()
        reps.append(r)
    first = hd.Batch(reps, M.Params(prec=0, bias_on=0))
    assert (first.obs()[:, 6] == 0.0).all()
    first.step(1)
    s1 = first.obs()[:, 6]
    first.close()
    for k, r in enumerate(reps):
        w = 0.3 * abs(s1[k])
        r.sig_lo, r.sig_hi = (s1[k] - w, s1[k] + w) if k != 2 else (s1[k] + 1e3, s1[k] + 2e3)
        assert not (r.sig_lo <= 0.0 <= r.sig_hi)
    p = M.Params(prec=0, bias_on=1)
    b = hd.Batch(reps, p)
    b.step(3)
    ob = b.obs()
    assert (ob[[0, 1, 3], 25] >= 1).all()
    for k in range(4):
        one = hd.Batch([reps[k]], p)
        one.step(3)
        assert np.abs(one.positions(0) - b.positions(k)).max() < 1e-12
        assert np.allclose(one.obs()[0, :12], ob[k, :12], rtol=1e-9, atol=1e-12)
        one.close()
    b.close()
