"""Query labels from several threads at once, each on its own stream with its own numbers
of queries and channels: the kernels' shared-memory requests differ, and no thread's
call may refuse or change another's.
"""
import threading

import numpy as np
import pytest
import torch

from paper_2604_10951_gb300 import scenes
from paper_2604_10951_gb300.raster import query_labels
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu


def test_threads_with_different_requests():
    means = scenes.room_scene(n=5000, C=4, seed=1).means[:1000]
    jobs = []
    for nq, dim in ((96, 16), (256, 128), (144, 64), (192, 112)):
        f_ins, f_q, p_q, prec = scenes.room_queries(means, nq, dim, seed=nq)
        jobs.append((dev(f_ins, torch.bfloat16), dev(means), dev(f_q, torch.bfloat16), dev(p_q), dev(prec)))
    want = [query_labels(*j) for j in jobs]
    torch.cuda.synchronize()
    failed, start = [], threading.Barrier(len(jobs))

    def work(k):
        try:
            stream = torch.cuda.Stream()
            err = torch.zeros(1, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            start.wait()
            with torch.cuda.stream(stream):
                for _ in range(1500):
                    out = query_labels(*jobs[k], err=err)
                stream.synchronize()
            assert int(err.item()) == 0 and torch.equal(out, want[k])
        except Exception as e:
            failed.append(f"{k}: {e}")

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
