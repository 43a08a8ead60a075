"""Requests that share chunks are launched in another order: the results are those of each request by itself, bit for bit."""
import numpy as np
import pytest

from paper_2608_11231_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_req", [2, 3, 9, 17])
def test_shared_chunks_equal_single_requests(n_req):
    import torch
    H, d, n_pool = 32, 128, 5
    # more chunk loads than L2 holds, spread unevenly over the requests (one of them empty)
    rng = np.random.default_rng(n_req)
    ks = rng.multinomial(40, np.ones(n_req - 1) / (n_req - 1)).tolist() + [0]
    cu_k = np.concatenate([[0], np.cumsum(ks)]).astype(np.int32)
    ids = rng.integers(0, n_pool, cu_k[-1]).astype(np.int32)
    g = torch.Generator(device="cuda").manual_seed(n_req)
    states = torch.randn((n_pool, H, d, d), generator=g, device="cuda")
    trans = torch.randn((n_pool, H, d, d), generator=g, device="cuda") * (0.45 / d ** 0.5)
    got = b.lkv_init_state_batched(states, trans, ids, cu_k, n_req, b.LKV_INIT_EXACT, family=b.LKV_FAMILY_GDN)
    for r in range(n_req):
        own = ids[cu_k[r]:cu_k[r + 1]]
        # (as one chain: with room for it a single request is composed in two halves)
        ref = b.lkv_init_state(states, trans, len(own), b.LKV_INIT_EXACT, family=b.LKV_FAMILY_GDN, chunk_ids=own,
                               workspace_t=torch.zeros(256, dtype=torch.uint8, device="cuda"))
        assert torch.equal(got[r], ref), r
