"""GPU test of contexts of different size side by side: the shared memory that
a kernel may ask for belongs to the process, so a batch created later, with
smaller cells and rows, must not lower it under an earlier one.  The earlier
one has not launched anything yet when the later one is created, so that all
its launches are queued (and captured) afterwards."""
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
@pytest.mark.parametrize("driver", [1, 2])
def test_small_batch_after_a_large_one(hd, prec, driver):
    from paper_0909_5215_gb300 import model as M
    large = thermalise(small3d(nx=6, nz=3, radius=3.0), amp=0.05, seed=1)
    small = thermalise(small2d(), amp=0.05, seed=2)
    p = M.Params(prec=prec, bias_on=0)

    def go(b):
        b.step(30)
        b.quench(max_iter=5)
        b.step(2)
        return b.positions(0), b.obs(0)["n_rebuild"]

    alone = hd.Batch([large], p, driver=driver)
    want = go(alone)
    alone.close()
    a = hd.Batch([large], p, driver=driver)
    b = hd.Batch([small], p, driver=driver)
    got = go(a)
    go(b)
    assert np.array_equal(got[0], want[0]) and got[1] == want[1]
    b.step(1)
    b.sync()
    a.close()
    b.close()
