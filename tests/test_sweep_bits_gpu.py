"""GPU test of the split pair sweep to the last bit.

The LJ force is cut at rc, where it jumps, so trajectories that part by
rounding part by far more once a pair is cut a step sooner in one of them: a
force must not change in its last bits from one build to the next, nor with
the tile size.  Where a lane walks a row (batches from 38,912 atoms on) the
FP32 sums are taken entry by entry in the row's order, and what they give is
kept here as hashes of the FP32 words, made with the sweep that took one entry
at a time.  Cases: fewer atoms than a tile, a common fixed-point unit and none,
r_0 that differs by type, bonds, rows near their capacity, atoms far from the
lattice (cores that overlap).
"""
import hashlib
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "pair_sweep_fp32_bits.txt")
FIELDS = ("forces", "hdr", "energies")


def jittered(rep, seed, amp=0.04):
    """Uniform displacements (exact on every machine) of the mobile atoms and of their r_O."""
    rng = np.random.default_rng(seed)
    on = np.array([1.0, 1.0, 1.0 if rep.dim == 3 else 0.0]) * (rep.role == 1)[:, None]
    base = rep.pos.copy()
    rep.pos = base + on * rng.uniform(-amp, amp, base.shape)
    rep.pos_ref = base + on * rng.uniform(-amp, amp, base.shape)
    return rep


def replicas():
    from paper_0909_5215_gb300 import model as M
    two = lambda cols, rows, tip: M.afm2d(n_cols=cols, n_rows=rows, n_tip=tip, eps=M.PAPER_EPS_2D, kT=0.05)  # noqa: E731
    slab = lambda nx, ny, nz, rad: M.afm3d(nx=nx, ny=ny, nz=nz, tip_radius=rad, eps=M.PAPER_EPS_3D, kT=0.1)  # noqa: E731
    reps = [jittered(two(8, 4, 5), 1), jittered(slab(5, 5, 3, 2.5), 2), jittered(slab(5, 7, 3, 2.5), 3),
            jittered(two(23, 7, 30), 4), jittered(M.paper3d(), 5, 0.02), jittered(slab(16, 16, 4, 4.0), 8, 0.1)]
    reps[3].sig = ((1.0, 0.95), (0.95, 0.9))
    reps += [jittered(slab(13, 13, 6, 4.0), 100 + q) for q in range(10)]     # company, and one lane to a row
    assert sum(r.n for r in reps) > 152 * 8 * 32
    for k, r in enumerate(reps):
        r.rep_id = k
    return reps


def words(hd, block):
    """(replica, field) -> hash of its FP32 words, for the first six replicas."""
    from paper_0909_5215_gb300 import model as M
    b = hd.Batch(replicas(), M.Params(prec=1, bias_on=0), driver=hd.HD_DRIVER_KERNELS, block=block)
    out = {}
    for k in range(6):
        for f in FIELDS:
            v = np.asarray(getattr(b, f)(k), dtype="<f4") + np.float32(0)     # -0 and 0 are the same
            out["%d %s" % (k, f)] = hashlib.sha256(v.tobytes()).hexdigest()
    b.close()
    return out


@pytest.mark.parametrize("block", [64, 128, 256])
def test_forces_keep_their_bits(block):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd
    _build.build()
    with open(GOLDEN) as f:
        want = {" ".join(w[:2]): w[2] for w in (line.split() for line in f if not line.startswith("#"))}
    assert words(hd, block) == want
