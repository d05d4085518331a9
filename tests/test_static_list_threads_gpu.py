"""GPU test of hd_nlist_static called from several threads at once, each with
its own stream and number of atoms: the calls share one scratch array and take
turns on it, so every call's rows must be those of its own atoms (brute force,
whole numbers) and nothing is written past its own buffers."""
import threading

import numpy as np
import pytest

from test_static_list_gpu import RL, brute

pytestmark = pytest.mark.gpu


def test_threads_take_turns():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0909_5215_gb300 import _build, hd
    _build.build()
    hd.lib()
    rng = np.random.default_rng(1)
    jobs = []
    for n, box, per in ((40, (7.0, 7.0, 0.0), (1, 1, 0)), (900, (11.0, 12.0, 0.0), (1, 1, 0)), (2000, (16.0, 16.0, 16.0), (1, 1, 1))):
        x = rng.uniform(0.0, 1.0, size=(n, 3)) * [b if p else 6.0 for b, p in zip(box, per)]
        rows = brute(x, box, per, RL)
        most = max(len(r) for r in rows)
        # eight rows of guard behind the caller's own
        nbr = torch.full((n + 8, most), -7, dtype=torch.int32, device="cuda")
        nnb = torch.full((n + 8,), -7, dtype=torch.int32, device="cuda")
        jobs.append((n, box, per, most, rows, torch.from_numpy(x).cuda(), nbr, nnb, torch.cuda.Stream()))
    torch.cuda.synchronize()
    bad = []

    def work(job):
        n, box, per, most, _, pos, nbr, nnb, s = job
        for _ in range(200):
            st = hd.hd_nlist_static(pos.data_ptr(), n, box, per, RL, most, nbr.data_ptr(), nnb.data_ptr(), s.cuda_stream)
            if st != hd.HD_OK:
                bad.append((n, st))

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for n, _, _, _, rows, _, nbr, nnb, _ in jobs:
        a, c = nbr.cpu().numpy(), nnb.cpu().numpy()
        assert (a[n:] == -7).all() and (c[n:] == -7).all()
        for i, r in enumerate(rows):
            assert c[i] == len(r) and np.array_equal(a[i, :len(r)], r) and (a[i, len(r):] == -1).all()
