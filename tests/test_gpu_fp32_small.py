"""The fp32 GDN kernels of small calls at the edges of their tiles: head sizes around the row and channel tiles, rings with more and with
fewer stages than chunks, requests of no and of one chunk."""
import numpy as np
import pytest

from helpers import dev, host
from paper_2608_11231_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_k, d_v", [(8, 8), (64, 64), (72, 40), (120, 16), (128, 24)])
@pytest.mark.parametrize("bf16", [False, True])
def test_small_composition(d_k, d_v, bf16):
    import torch
    rng = np.random.default_rng(d_k + d_v)
    H, n_pool, ks = 2, 9, [0, 1, 2, 3, 9]
    states = rng.standard_normal((n_pool, H, d_k, d_v)).astype(np.float32)
    pool = dev(states, torch.bfloat16) if bf16 else dev(states)
    states = host(pool.float()).astype(np.float64)
    trans = (rng.standard_normal((n_pool, H, d_k, d_k)) / d_k ** 0.5).astype(np.float32)
    cu_k = np.concatenate([[0], np.cumsum(ks)]).astype(np.int32)
    ids = rng.integers(0, n_pool, cu_k[-1]).astype(np.int32)
    out = host(b.lkv_init_state_batched(pool, dev(trans), ids, cu_k, len(ks), b.LKV_INIT_EXACT, family=b.LKV_FAMILY_GDN, compute=b.LKV_COMPUTE_FP32))
    for r, K in enumerate(ks):
        S, size = np.zeros((H, d_k, d_v)), np.zeros((H, d_k, d_v))
        for j in range(K):
            c = ids[cu_k[r] + j]
            T = trans[c].astype(np.float64)
            S, size = (T @ S + states[c], np.abs(T) @ size + np.abs(states[c])) if j else (states[c], np.abs(states[c]))
        # a step is d_k / 2 + 2 roundings of sums of absolute value `size` at most
        assert np.all(np.abs(out[r] - S) <= max(K - 1, 0) * (d_k / 2 + 2) * 2.0 ** -24 * size), (r, K)
