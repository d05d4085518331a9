"""GPU test of H.(r - r_O) on demand with replicas by the hundred about their
band: more of them than one pass over the list takes, ragged tiles, neighbours
in the list that are far apart in the batch.  The same replicas in a batch that
always forms the term are the reference: the same words in the split form (one
lane walks a row in both), rounding (1e-9 in positions) in the FP64 form."""
import numpy as np
import pytest

from conftest import small2d, thermalise

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
def test_hundreds_of_listed_replicas(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd
    from paper_0909_5215_gb300 import model as M
    _build.build()
    kinds = [thermalise(small2d(cols=cols, rows=5, n_tip=13, kT=0.15), amp=0.05, seed=cols) for cols in (12, 27, 40)]
    count = int((210000 if prec else 40000) / (sum(r.n for r in kinds) / 3))
    rng = np.random.default_rng(2)
    for r in kinds:
        r.pos_ref = r.pos - 0.02 * (r.role == 1)[:, None] * [1.0, 1.0, 0.0] * rng.normal(size=r.pos.shape)
    probe = hd.Batch(kinds, M.Params(prec=prec, bias_on=0))
    sig = [probe.obs()[:, 6]]
    probe.step(10)
    sig.append(probe.obs()[:, 6])
    probe.close()
    reps = []
    for k in range(count):
        r = kinds[k % 3].copy()
        lo, hi = min(s[k % 3] for s in sig), max(s[k % 3] for s in sig)
        w = 0.5 * (abs(lo) + abs(hi))
        r.rep_id, r.dvmax = k, 0.4
        # a third of each kind stays far from its band
        r.sig_lo, r.sig_hi = (lo - w, hi + w) if k % 9 < 6 else (1e5, 2e5)
        reps.append(r)
    some = sorted(rng.permutation(count)[:50 if prec == 0 else 110].tolist())
    sub = [reps[k] for k in some]
    total, part = sum(r.n for r in reps), sum(r.n for r in sub)
    assert total >= (200000 if prec else 38912) and (part < 8192 if prec == 0 else 9728 < part < 200000)
    p = M.Params(prec=prec, bias_on=1)
    a, b = hd.Batch(reps, p), hd.Batch(sub, p)
    for n in (1, 2, 20):
        a.step(n)
        b.step(n)
    oa, ob = a.obs(), b.obs()
    assert (oa[:, 25] > 0).sum() > 64                          # in their band at some time
    assert np.array_equal(oa[some][:, 24:27], ob[:, 24:27])
    for q, k in enumerate(some):
        if prec == 1:
            assert np.array_equal(a.forces(k), b.forces(q)) and np.array_equal(a.hdr(k), b.hdr(q))
        assert np.abs(a.positions(k) - b.positions(q)).max() < (1e-9 if prec == 0 else 1e-12)
    a.close()
    b.close()
