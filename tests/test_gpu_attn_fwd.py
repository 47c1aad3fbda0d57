"""GPU parity of the attention forward with the vision score as one more value column (Sec. 3.2.1,
eqs. 2-4) against the fp64 oracle: O = softmax(s Q K^T + bias) V per head and the head-averaged
vision mass, causal and not, grouped-query heads (H / H_kv = 1, 2, 4), hard labels and a carried
float score with the eq. (4) blend.

Tolerance of O (stored in bf16): the softmax weights reach the tensor cores in bf16 (relative
error 2^-9 each), which moves an output by at most 2^-9 max|V|, and the output's own rounding adds
half a bf16 ulp; the bar is one ulp of the exact value + 2^-8 max|V| per element, and 2e-3 + 2^-8
in norm. The score M (fp32 softmax weights) meets the 2e-3 bar of every floating-point output.
"""
import numpy as np
import pytest
import torch

from oracle import smoes_oracle as O
from paper_2604_23996_gb300.workloads import attn_workload

from .parity import assert_tensor_close, bf16_ulp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_23996_gb300 import binding
    return binding


def _case(B, H, Hkv, S, seed, n_image):
    aw = attn_workload(B=B, H=H, S=S, hd=128, n_image=n_image, seed=seed)
    rng = np.random.default_rng(seed + 7)
    # keys and values with H_kv heads (the query heads of a group share them)
    K = torch.from_numpy(rng.standard_normal((B, Hkv, S, 128), dtype=np.float32)).to(torch.bfloat16)
    V = torch.from_numpy(rng.standard_normal((B, Hkv, S, 128), dtype=np.float32)).to(torch.bfloat16)
    return aw, K, V


def _run(bd, aw, K, V, Hkv, causal=1, m_prev=None, norms=None):
    T = aw.B * aw.S
    r = bd.Router(T, 64, 16, 2, 4, [0, T], np.arange(16) // 4, attn_max_heads=aw.H)
    M = torch.empty((T, 2), device="cuda")
    Ot = torch.empty((aw.B, aw.H, aw.S, 128), dtype=torch.bfloat16, device="cuda")
    attn = dict(Q=aw.Q.cuda(), K=K.cuda(), B=aw.B, H=aw.H, S=aw.S, hd=128, sm_scale=aw.sm_scale,
                causal=causal, key_bias=torch.from_numpy(aw.key_bias).cuda())
    if m_prev is None:
        attn["is_vision"] = torch.from_numpy(aw.is_vision).cuda()
    else:
        attn["m_prev"] = torch.from_numpy(m_prev).cuda()
    if norms is not None:
        attn["xattn_norm"] = torch.from_numpy(norms[0]).cuda()
        attn["x_norm"] = torch.from_numpy(norms[1]).cuda()
    code = bd.smoes_attention_fwd(r.plan, attn, V.cuda(), Hkv, Ot, M, r.ws)
    assert code == 0, bd.smoes_status_string(code)
    assert r.device_status()[0] == 0
    torch.cuda.synchronize()
    return r, attn, Ot.float().cpu().numpy(), M.cpu().numpy()


def _check_O(got, ref, Vmax, what):
    err = np.abs(got - ref)
    bad = err > bf16_ulp(ref) + 2.0 ** -8 * Vmax
    assert not np.any(bad), f"{what}: {int(bad.sum())} elements off; worst {err.max():.3e}"
    rel = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert rel <= 2e-3 + 2.0 ** -8, f"{what}: rel L2 {rel:.3e}"
    return rel


@pytest.mark.parametrize("B,H,Hkv,S,causal", [(2, 4, 4, 256, 1), (1, 4, 2, 384, 1), (2, 8, 2, 256, 1),
                                              (1, 4, 1, 128, 1), (1, 2, 2, 256, 0)])
def test_attention_forward_with_mass(bd, B, H, Hkv, S, causal):
    aw, K, V = _case(B, H, Hkv, S, seed=200 + S + H, n_image=S // 4)
    _, _, Og, Mg = _run(bd, aw, K, V, Hkv, causal=causal)
    m = aw.is_vision.reshape(B, S).astype(np.float64)
    Oref, mass = O.attention_forward_with_mass(aw.Q.double().numpy(), K.double().numpy(), V.double().numpy(),
                                               m, aw.sm_scale, bool(causal), aw.key_bias.reshape(B, S))
    e = _check_O(Og, Oref, float(V.float().abs().max()), "O")
    assert_tensor_close(Mg[:, 0], mass.reshape(-1), "vision mass")
    np.testing.assert_array_equal(Mg[:, 1], (1.0 - Mg[:, 0]).astype(np.float32))
    print(f"B{B} H{H} Hkv{Hkv} S{S} causal{causal}: O rel L2 {e:.2e}")


def test_carried_float_score_and_residual_blend(bd):
    B, H, Hkv, S = 2, 4, 2, 256
    aw, K, V = _case(B, H, Hkv, S, seed=301, n_image=64)
    rng = np.random.default_rng(3)
    m_prev = rng.uniform(0.0, 1.0, B * S).astype(np.float32)
    an = rng.uniform(0.5, 2.0, B * S).astype(np.float32)
    xn = rng.uniform(0.5, 2.0, B * S).astype(np.float32)
    _, _, Og, Mg = _run(bd, aw, K, V, Hkv, m_prev=m_prev, norms=(an, xn))
    Oref, mass = O.attention_forward_with_mass(aw.Q.double().numpy(), K.double().numpy(), V.double().numpy(),
                                               m_prev.reshape(B, S).astype(np.float64), aw.sm_scale, True,
                                               aw.key_bias.reshape(B, S))
    _check_O(Og, Oref, float(V.float().abs().max()), "O")
    ref = O.residual_score_update(mass.reshape(-1), m_prev, an, xn)
    assert_tensor_close(Mg[:, 0], ref, "blended score (eq. 4)")


def test_score_equals_the_mass_only_kernel(bd):
    # with H_kv = H the score of the forward and of smoes_modality_score(ATTN) are the same quantity
    B, H, S = 2, 4, 512
    aw, _, V = _case(B, H, H, S, seed=302, n_image=128)
    r, attn, _, Mg = _run(bd, aw, aw.K, V, H)
    M2 = torch.empty((B * S, 2), device="cuda")
    r.modality_score(bd.SMOES_SCORE_ATTN, M2, attn=attn)
    torch.cuda.synchronize()
    assert_tensor_close(Mg[:, 0], M2.cpu().numpy()[:, 0], "forward vs mass-only score")


def test_attention_forward_limits(bd):
    aw, K, V = _case(1, 4, 4, 128, seed=303, n_image=32)
    T = aw.S
    r = bd.Router(T, 64, 16, 2, 4, [0, T], np.arange(16) // 4, attn_max_heads=4)
    M = torch.empty((T, 2), device="cuda")
    Ot = torch.empty((1, 4, 128, 128), dtype=torch.bfloat16, device="cuda")
    attn = dict(Q=aw.Q.cuda(), K=K.cuda(), B=1, H=4, S=128, hd=128, sm_scale=aw.sm_scale, causal=1,
                is_vision=torch.from_numpy(aw.is_vision).cuda())
    assert bd.smoes_attention_fwd(r.plan, attn, V.cuda(), 3, Ot, M, r.ws) == -1     # H % H_kv != 0
    assert bd.smoes_attention_fwd(r.plan, dict(attn, hd=64), V.cuda(), 4, Ot, M, r.ws) == -2


@pytest.mark.parametrize("B,H,Hkv,S,case", [(1, 2, 1, 640, "rising"), (3, 8, 8, 128, "padded"), (20, 16, 16, 256, "runs"),
                                            (1, 4, 4, 384, "scattered"), (1, 2, 2, 256, "negative"),
                                            (4, 16, 4, 384, "rising"), (10, 16, 16, 128, "padded"), (5, 16, 8, 384, "scattered"),
                                            (6, 16, 16, 256, "negative")])
def test_forward_key_chunks_and_rescale(bd, B, H, Hkv, S, case):
    # up to 152 query tiles take the kernel of one tile per item, more that of two (there with an odd
    # number of tiles, so a pair of one, and many short items per CTA): keys whose bias and score
    # change inside a 32-key chunk or are -inf, logits that grow by far more than 2^8 along the keys
    # (the running maximum is raised, O rescaled), and a logit scale whose maximum is not the products'
    aw, K, V = _case(B, H, Hkv, S, seed=900 + S + H, n_image=S // 4)
    rng = np.random.default_rng(S)
    if case == "rising":
        aw.key_bias = np.tile(np.linspace(0.0, 60.0, S, dtype=np.float32), B)
    elif case == "padded":                                # every query keeps key 0
        aw.key_bias = np.where(np.arange(B * S) % S > 90, -np.inf, 0.0).astype(np.float32)
    elif case == "scattered":
        aw.is_vision = (rng.random(B * S) < 0.5).astype(np.uint8)
        aw.key_bias = rng.standard_normal(B * S).astype(np.float32)
    elif case == "negative":
        aw.sm_scale = -aw.sm_scale
    _, _, Og, Mg = _run(bd, aw, K, V, Hkv)
    Oref, mass = O.attention_forward_with_mass(aw.Q.double().numpy(), K.double().numpy(), V.double().numpy(),
                                               aw.is_vision.reshape(B, S).astype(np.float64), aw.sm_scale, True,
                                               aw.key_bias.reshape(B, S))
    _check_O(Og, Oref, float(V.float().abs().max()), "O")
    assert_tensor_close(Mg[:, 0], mass.reshape(-1), "vision mass")


@pytest.mark.parametrize("B,H,S", [(1, 8, 128), (3, 8, 384), (19, 8, 128), (10, 8, 256)])
def test_forward_heads_averaged_on_repeated_calls(bd, B, H, S):
    # up to 152 query tiles the tile's last head averages the heads (a ticket that every call leaves
    # at zero, shared with the attention score's), with more a kernel of its own: one launch of each
    # kind at the line (152 and 160 tiles), repeated on one workspace with the score in between
    aw, K, V = _case(B, H, H, S, seed=40 + B, n_image=S // 4)
    rng = np.random.default_rng(B)
    m_prev = rng.random(B * S).astype(np.float32)
    norms = [(0.5 + rng.random(B * S)).astype(np.float32) for _ in range(2)]
    r, attn, _, M0 = _run(bd, aw, K, V, H, m_prev=m_prev, norms=norms)
    _, mass = O.attention_forward_with_mass(aw.Q.double().numpy(), K.double().numpy(), V.double().numpy(),
                                            m_prev.reshape(B, S).astype(np.float64), aw.sm_scale, True,
                                            aw.key_bias.reshape(B, S))
    an, xn = (n.astype(np.float64) for n in norms)
    assert_tensor_close(M0[:, 0], (an * mass.reshape(-1) + xn * m_prev) / (an + xn), "blended score")
    Vg, Ot = V.cuda(), torch.empty((B, H, S, 128), dtype=torch.bfloat16, device="cuda")
    M, Ms = (torch.empty((B * S, 2), device="cuda") for _ in range(2))
    for _ in range(3):
        M.fill_(float("nan"))
        assert bd.smoes_attention_fwd(r.plan, attn, Vg, H, Ot, M, r.ws) == 0
        r.modality_score(bd.SMOES_SCORE_ATTN, Ms, attn=attn)
        assert r.device_status()[0] == 0
        np.testing.assert_array_equal(M.cpu().numpy(), M0)
        assert_tensor_close(Ms.cpu().numpy(), M0, "score kernel")


@pytest.mark.parametrize("B,H,S", [(1, 2, 640), (4, 16, 640), (3, 28, 256)])
@pytest.mark.parametrize("rows", ["all", "some", "even_tiles", "odd_tiles"])
def test_forward_rescales_before_either_halfs_products(bd, B, H, S, rows):
    # logits that grow by more than 2^8 with every key block, so that O is rescaled at every block: in
    # every row, in every third row, or in one tile of each pair only. 10 query tiles take the kernel
    # of one tile per item, 320 (with a pair of one) and 168 that of two. Each key half rescales its
    # columns of O and both halves' products add to all of them: a product that came before the other
    # half's rescale would differ from the oracle, or from call to call.
    aw, K, V = _case(B, H, H, S, seed=500 + S + H, n_image=S // 4)
    pos = np.arange(S)
    on = {"all": pos >= 0, "some": pos % 3 == 1, "even_tiles": pos // 128 % 2 == 0, "odd_tiles": pos // 128 % 2 == 1}[rows]
    aw.Q[..., 0] = torch.from_numpy(np.where(on, 16.0, 0.0)).to(torch.bfloat16)
    K[..., 0] = torch.from_numpy(pos * (14.0 / 128) / (16.0 * aw.sm_scale)).to(torch.bfloat16)   # 14 nats a block
    r, attn, Og, Mg = _run(bd, aw, K, V, H)
    Oref, mass = O.attention_forward_with_mass(aw.Q.double().numpy(), K.double().numpy(), V.double().numpy(),
                                               aw.is_vision.reshape(B, S).astype(np.float64), aw.sm_scale, True,
                                               aw.key_bias.reshape(B, S))
    _check_O(Og, Oref, float(V.float().abs().max()), "O")
    assert_tensor_close(Mg[:, 0], mass.reshape(-1), "vision mass")
    Vg = V.cuda()
    first = torch.empty((B, H, S, 128), dtype=torch.bfloat16, device="cuda")
    again, M1, M2 = torch.empty_like(first), torch.empty((B * S, 2), device="cuda"), torch.empty((B * S, 2), device="cuda")
    assert bd.smoes_attention_fwd(r.plan, attn, Vg, H, first, M1, r.ws) == 0
    for _ in range(50):
        assert bd.smoes_attention_fwd(r.plan, attn, Vg, H, again, M2, r.ws) == 0
        assert torch.equal(again.view(torch.int16), first.view(torch.int16)) and torch.equal(M1, M2)
    assert r.device_status()[0] == 0


@pytest.mark.parametrize("B,S,bias", [(1, 256, -1e30), (11, 256, -1e30), (1, 256, 1e30), (1, 256, 3e9), (11, 256, -1.4e9), (1, 256, -1e9)])
@pytest.mark.parametrize("scale", [1.0, 30.0])
def test_forward_one_bias_of_any_size_on_every_key(bd, B, S, bias, scale):
    # left-padded prompts: every key that a padded query sees is masked by the same large finite bias.
    # Past 2^53 the bias swallows the scores in 64 bits too and the row is a plain mean; a bias that the
    # kernel keeps out of the scores (below 2^31 in log2 units) leaves the softmax of the scores. In
    # between fp32 rounds the scores at the bias's size: the outputs then only have to be finite and
    # within the values' range. Scores of up to 120 nats: none of it may overflow.
    aw, K, V = _case(B, 8, 8, S, seed=77, n_image=S // 4)
    aw.key_bias[:] = bias
    aw.sm_scale *= scale
    _, _, Og, Mg = _run(bd, aw, K, V, 8)
    assert np.isfinite(Og).all() and np.isfinite(Mg).all()
    Vmax = float(V.float().abs().max())
    if 1.4e9 < abs(bias) < 1e16:
        assert np.abs(Og).max() <= Vmax * (1 + 2.0 ** -7)
        return
    Oref, mass = O.attention_forward_with_mass(aw.Q.double().numpy(), K.double().numpy(), V.double().numpy(),
                                               aw.is_vision.reshape(B, S).astype(np.float64), aw.sm_scale, True,
                                               aw.key_bias.reshape(B, S))
    _check_O(Og, Oref, Vmax, "O")
    assert_tensor_close(Mg[:, 0], mass.reshape(-1), "vision mass")
