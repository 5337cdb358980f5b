"""Query labels from several threads at once, each on its own stream with its own numbers
of queries and channels.  The kernels' shared-memory requests differ, and no thread's
call may refuse or change another's.  The calls are made in a row from a compiled loop:
between two of them the interpreter would let only one thread run.
"""
import ctypes
import subprocess
import threading

import pytest
import torch

from paper_2604_10951_gb300 import _lib as L
from paper_2604_10951_gb300 import scenes
from paper_2604_10951_gb300.raster import query_labels
from tests.gpu_util import dev

pytestmark = pytest.mark.gpu

LOOP = """
#include <stdint.h>
typedef int (*labels_fn)(int64_t, int32_t, int32_t, const void *, const float *, const void *, const float *,
                         const float *, void *, int32_t, int32_t *, void *);
int refused(labels_fn f, int64_t n, int32_t nq, int32_t dim, const void *fi, const float *m, const void *fq,
            const float *p, const float *s, void *out, int32_t *err, void *stream, int times)
{
    int bad = 0;
    for (int i = 0; i < times; ++i) bad += f(n, nq, dim, fi, m, fq, p, s, out, 0, err, stream) != 0;
    return bad;
}
"""


def test_threads_with_different_requests(tmp_path):
    src, so = tmp_path / "loop.c", tmp_path / "loop.so"
    src.write_text(LOOP)
    subprocess.run(["gcc", "-O2", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    refused = ctypes.CDLL(str(so)).refused
    P, i32 = ctypes.c_void_p, ctypes.c_int32
    refused.argtypes = [P, ctypes.c_int64, i32, i32, P, P, P, P, P, P, P, P, ctypes.c_int]
    f = ctypes.cast(L.lib().fss_query_labels, P)

    means = scenes.room_scene(n=5000, C=4, seed=1).means[:1000]
    jobs, want = [], []
    for nq, dim in ((96, 16), (256, 128), (144, 64), (192, 112)):
        f_ins, f_q, p_q, prec = scenes.room_queries(means, nq, dim, seed=nq)
        jobs.append((dev(f_ins, torch.bfloat16), dev(means), dev(f_q, torch.bfloat16), dev(p_q), dev(prec)))
        want.append(query_labels(*jobs[-1]))
    outs, err = [torch.zeros_like(w) for w in want], torch.zeros(1, dtype=torch.int32, device="cuda")
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()
    bad, start = [None] * len(jobs), threading.Barrier(len(jobs))

    def work(k):
        torch.cuda.set_device(0)
        nq, dim = jobs[k][2].shape
        start.wait()
        bad[k] = refused(f, len(means), nq, dim, *(x.data_ptr() for x in jobs[k]), outs[k].data_ptr(), err.data_ptr(),
                         streams[k].cuda_stream, 5000)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert bad == [0] * len(jobs) and int(err.item()) == 0
    assert all(torch.equal(o, w) for o, w in zip(outs, want))
