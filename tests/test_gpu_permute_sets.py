"""The standalone bin permutation where its 128-bit selection sets can go wrong: bins of 32 experts, bins
that straddle the words of the set, one expert, sixteen selections, expert-to-bin maps in any order,
and batches of one token, of one block and a token, and of several rounds per block."""
import numpy as np
import pytest
import torch

from oracle import smoes_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,E,k,K,shuffle", [(1, 1, 1, 1, False), (257, 128, 16, 4, False), (1000, 120, 7, 5, True),
                                             (777, 96, 8, 8, False), (600, 128, 2, 32, True), (400000, 32, 4, 8, False)])
def test_permutation_of_given_selections(T, E, k, K, shuffle):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_23996_gb300 import binding as bd

    rng = np.random.default_rng(T + E)
    eb = np.arange(E) // (E // K)
    if shuffle:
        eb = rng.permutation(eb)
    idx = np.argsort(rng.random((T, E), dtype=np.float32), axis=1)[:, :k].astype(np.int32)
    vis = (rng.random(T) < 0.4).astype(np.uint8)
    r = bd.Router(T, 8, E, k, K, [0, T], eb.astype(np.int32))
    r.permute(is_vision=torch.from_numpy(vis).cuda(), topk_idx=torch.from_numpy(np.ascontiguousarray(idx)).cuda())
    assert r.device_status()[0] == 0
    ref = O.bin_permute(idx, eb, K, is_vision=vis)
    P = int(r.bin_offsets[-1])
    np.testing.assert_array_equal(r.bin_offsets.cpu().numpy(), ref["offsets"])
    np.testing.assert_array_equal(r.perm_token[:P].cpu().numpy(), ref["perm"])
    np.testing.assert_array_equal(r.perm_mask[:P].cpu().numpy().view(np.uint32).astype(np.uint64), ref["mask"])
    np.testing.assert_array_equal(r.dispatch.cpu().numpy(), ref["dispatch"])
    np.testing.assert_array_equal(r.expert_counts.cpu().numpy(), ref["expert_counts"])
