"""GPU parity of the tensor-core router where its hand-offs between warps and its staging change:
every length of the top-k networks, one tile per CTA at the widest gate, CTAs that hand many
samples to their reducer warp, two tiles per CTA with the permutation in the same launch, and
backward slices whose last 64-column box starts past the hidden size."""
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


def _lengths(T, n):
    return [T // n] * (n - 1) + [T - (n - 1) * (T // n)]


@pytest.mark.parametrize("T,d,E,k,K,samples", [
    (300, 128, 64, 1, 8, 2),
    (300, 128, 64, 3, 8, 2),
    (300, 128, 64, 5, 8, 2),
    (300, 128, 64, 9, 8, 2),
    (300, 512, 128, 16, 16, 3),          # one tile per CTA, E = 128
    (20001, 64, 64, 2, 8, 7),            # up to two tiles per CTA, ragged last tile
    (45000, 64, 16, 2, 4, 900),          # several tiles per CTA, each with three samples
    (200, 136, 64, 4, 8, 2),             # 8 columns past a 128-column block
    (200, 1416, 48, 4, 6, 2),            # several slices, the last one partly filled
])
def test_router_pipeline(bd, T, d, E, k, K, samples):
    wl = random_router_case(T + k, T, d, E, k, K, _lengths(T, samples), aligned=True)
    g = run_gpu(wl, bd, fused=True)
    compare(wl, g, run_oracle(wl))
