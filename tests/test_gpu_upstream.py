"""GPU parity of the gradient that arrives through the top-k weights where its spread over a
token's thread group can go wrong: more slots than lanes of the group (k = 16 on 8 and 4 lanes),
one slot, a single bin per lane and bins that end inside a lane's eight experts."""
import numpy as np
import pytest
import torch

from paper_2604_23996_gb300.workloads import random_router_case

from .parity import compare, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_23996_gb300 import binding
    return binding


@pytest.mark.parametrize("T,d,E,k,K,renorm,dtype", [
    (300, 64, 64, 16, 8, 1, torch.bfloat16),
    (200, 72, 128, 16, 32, 0, torch.bfloat16),
    (130, 64, 24, 1, 2, 1, torch.bfloat16),       # N_B = 12: bins end inside a lane's experts
    (200, 64, 64, 16, 4, 1, torch.float32),
    (65, 40, 8, 5, 2, 0, torch.float32),
])
def test_upstream_gradient(bd, T, d, E, k, K, renorm, dtype):
    wl = random_router_case(E + k, T, d, E, k, K, [T // 3, T - T // 3], dtype=dtype, aligned=True)
    wl.renorm_topk = renorm
    dtw = 1e-3 * np.random.default_rng(T).standard_normal((T, k)).astype(np.float32)
    g = run_gpu(wl, bd, d_topk_w=dtw)
    ref = run_oracle(wl, d_topk_w=dtw.astype(np.float64), topk_idx_for_up=g["topk_idx"])
    compare(wl, g, ref)
