"""The library's scratch pool: calls of different sizes from several host
threads on their own streams give the results of serial calls, and what the
pool keeps after a large call stays within its bound."""
from __future__ import annotations

import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_threads_and_streams_share_the_pool():
    import torch
    from paper_1606_08281_gb300 import pf
    from paper_1606_08281_gb300 import workloads as W
    w = W.telegraph()
    th = w.thetas(96)
    y = torch.from_numpy(w.observations()).cuda()

    def call(i):
        t = torch.from_numpy(th[: 1 + 9 * (i % 10)].copy()).cuda()
        return pf.pf_loglik(w.net, t, w.x0, w.obs_times, y, w.C, w.sigma, 32 + 13 * (i % 7), 100 + i)["loglik"]

    want = [call(i).cpu().numpy() for i in range(40)]
    got, errors = {}, []

    def worker(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(k, 40, 4):
                    r = call(i)
                    torch.cuda.current_stream().synchronize()
                    got[i] = r.cpu().numpy()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=worker, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i in range(40):
        assert np.array_equal(got[i], want[i])


def test_what_the_pool_keeps_is_bounded():
    import torch
    from paper_1606_08281_gb300 import pf
    from paper_1606_08281_gb300 import workloads as W
    w = W.cascade().subset(T=4, K=1)
    args = (w.net, w.thetas(80), w.x0, w.obs_times, w.observations(), w.C, w.sigma)
    pf.pf_loglik(*args, 32, 1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    pf.pf_loglik(*args, 16384, 1)          # 304 slabs of 852 KB
    torch.cuda.synchronize()
    pf.pf_loglik(*args, 32, 1)
    torch.cuda.synchronize()
    # 64 MiB, and one granule of the driver's either way
    assert before - torch.cuda.mem_get_info()[0] <= (64 + 32) << 20
