"""GPU parity of the query-label kernel for many queries (query_wide.cu) at
the edges of its tiles: one Gaussian, one more and one less than a block of
128 and a tile of 256, the last query pieces (8, 16 and 24 columns), the
largest operands, and enough Gaussians for two per thread, in both label
types.  Tolerances as in test_gpu_queries.py: FP32 labels within 5e-5 of
themselves (plus 1e-7), BF16 storage adds 2^-8.
"""
import numpy as np
import pytest
import torch

from paper_2604_10951_gb300 import scenes
from tests.test_gpu_queries import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,dim,dtype", [
    (1, 96, 16, torch.float32), (127, 96, 48, torch.float32), (129, 96, 128, torch.float32),
    (255, 112, 64, torch.float32), (257, 176, 112, torch.float32), (1000, 256, 128, torch.float32),
    (78_001, 112, 32, torch.float32), (78_080, 144, 80, torch.float32), (200_003, 96, 64, torch.bfloat16),
    (200_000, 144, 96, torch.bfloat16)])
def test_wide_labels_against_oracle(n, nq, dim, dtype):
    means = scenes.room_scene(n=max(n, 5000), C=4, seed=n).means[:n]
    f_ins, f_q, p_q, prec = scenes.room_queries(means, nq, dim, seed=nq + dim)
    got, ref = _run(means, f_ins, f_q, p_q, prec, dtype)
    rel = 5e-5 + (2.0 ** -8 if dtype == torch.bfloat16 else 0.0)
    assert (np.abs(got - ref) <= rel * ref + 1e-7).all()
