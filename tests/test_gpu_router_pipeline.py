"""GPU parity of the tensor-core router where its hand-offs between warps and its staging change:
every length of the top-k networks, one tile per CTA at the widest gate, CTAs that hand many
samples to their reducer warp, two tiles per CTA with the permutation in the same launch, and
backward slices whose last 64-column box starts past the hidden size."""
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


@pytest.mark.parametrize("T,d,E,k,K", [(65536, 2048, 64, 6, 8), (65536, 1280, 48, 4, 6), (131072, 512, 32, 4, 8)])
def test_dw_error_of_the_accumulators(bd, T, d, E, k, K):
    # dW against the 64-bit product of the operands that the tensor cores get: dz as bf16 hi + lo and X.
    # What is left is the truncation of the fp32 accumulators, half an ulp (2^-25 .. 2^-24 of the
    # accumulator) per instruction on average. A sum over random tokens grows like the square root, 2/3
    # of its final size on average, so n instructions leave at most n 2^-25. A CTA's tiles (64 tokens,
    # four K steps, hi and lo) go to two accumulators in turn; with one the error is twice as large.
    g = torch.Generator(device="cuda").manual_seed(T + d)
    X = torch.randn((T, d), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.02 * torch.randn((E, d), generator=g, device="cuda")).to(torch.bfloat16)
    r = bd.Router(T, d, E, k, K, [0, T], np.arange(E) // (E // K))
    r.forward(X, W, mu=0.05 * torch.randn((2, d), generator=g, device="cuda"), var=torch.ones((2, d), device="cuda"))
    dW, dz = torch.empty((E, d), device="cuda"), torch.empty((T, E), device="cuda")
    r.backward(X, W, r.M, dW, dlogits=dz, d_topk_w=1e-3 * torch.randn((T, k), generator=g, device="cuda"))
    assert r.device_status()[0] == 0
    hi = dz.to(torch.bfloat16)
    lo = (dz - hi.float()).to(torch.bfloat16)
    ref = torch.zeros((E, d), dtype=torch.float64, device="cuda")
    for s in range(0, T, 8192):
        ref += (hi[s:s + 8192].double() + lo[s:s + 8192].double()).T @ X[s:s + 8192].double()
    groups = torch.cuda.get_device_properties(0).multi_processor_count // -(-d // 256)
    tiles = -(-(T // 64) // groups)
    n = -(-tiles // 2) * 4 * 2
    err = float((dW.double() - ref).norm() / ref.norm())
    assert err <= n * 2.0 ** -25, f"{err:.3g} > {n * 2.0 ** -25:.3g}"
    print(f"{T} x {d}, E = {E}: {err:.2e}, {n} instructions per accumulator: at most {n * 2.0 ** -25:.2e}")


@pytest.mark.parametrize("E,K,dtype", [(64, 8, torch.bfloat16), (128, 16, torch.bfloat16), (72, 8, torch.bfloat16), (32, 4, torch.float32)])
def test_scores_far_below_the_row_maximum_are_kept(bd, E, K, dtype):
    # logits of 0, -60, -88 and -98 by bin: the last two bins' scores lie at 2^-127 and 2^-141, below
    # the normal range, where fp32 still has steps of 2^-149. Scores, sums and products are each off by
    # at most a step: bin sums of N_B scores by N_B / 2 steps and the rounding of the product.
    T, d, k = 160, 64, 2
    X = torch.zeros((T, d), dtype=dtype, device="cuda")
    X[:, 0] = 1.0
    eb = np.arange(E) // (E // K)
    depth = torch.tensor([0.0, -60.0, -88.0, -98.0])[torch.from_numpy(eb % 4)]
    W = torch.zeros((E, d), dtype=dtype, device="cuda")
    W[:, 0] = depth.to(dtype).cuda()
    r = bd.Router(T, d, E, k, K, [0, T], eb, bd.SMOES_F32 if dtype == torch.float32 else bd.SMOES_BF16)
    M = torch.full((T, 2), 0.5, device="cuda")
    r.forward(X, W, M_in=M)
    g = torch.softmax(depth.double(), dim=0).numpy()
    ref = np.array([g[eb == b].sum() for b in range(K)])
    got = r.bin_prob.cpu().numpy()
    step = 2.0 ** -149
    np.testing.assert_allclose(got, np.tile(ref, (T, 1)), rtol=2e-5, atol=(E // K / 2 + 1) * step)
    assert (got[:, eb[::E // K] % 4 == 3] > 0).all()
