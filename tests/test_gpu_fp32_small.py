"""The fp32 GDN kernels of small calls at the edges of their tiles: head sizes around the row and channel tiles, rings with more and with
fewer stages than chunks, requests of no and of one chunk, lengths around the 32-token block with the next block's copies in flight."""
import numpy as np
import pytest

import oracle
from helpers import dev, host
from paper_2608_11231_b200 import binding as b
from paper_2608_11231_b200 import workloads as wl

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


@pytest.mark.parametrize("H_k, H_v, d_k, d_v, lens, io", [
    (1, 2, 64, 64, [1, 31, 32, 33, 96, 0], "f32"),
    (2, 2, 64, 16, [100], "bf16"),
    (1, 2, 63, 32, [65, 2], "f32"),        # rows that are copied channel by channel
    (1, 1, 66, 32, [40], "f32"),
    (1, 2, 256, 16, [70], "f32"),
    (1, 1, 4, 16, [33], "bf16"),
    (1, 1, 80, 128, [64, 40], "f32"),      # two clusters a head
])
@pytest.mark.parametrize("init", [True, False])
def test_small_scan(H_k, H_v, d_k, d_v, lens, io, init):
    import torch
    rng = np.random.default_rng(d_k * 1000 + d_v)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    tok = wl.gdn_tokens(rng, int(cu[-1]), H_k, H_v, d_k, d_v, io=io)
    S0 = rng.standard_normal((len(lens), H_v, d_k, d_v)).astype(np.float32)
    t = torch.bfloat16 if io == "bf16" else None
    o, ST = b.lkv_gdn_fwd(*(dev(tok[n], t) for n in ("q", "k", "v")), dev(tok["g"]), dev(tok["beta"]), dev(S0) if init else None, cu_seqlens=cu,
                          compute=b.LKV_COMPUTE_FP32)
    for s in range(len(lens)):
        sl = slice(cu[s], cu[s + 1])
        o_ref, ST_ref = oracle.gdn_seq(tok["q"][sl], tok["k"][sl], tok["v"][sl], tok["g"][sl], tok["beta"][sl], S0[s] if init else None)
        if lens[s]:   # outputs in bf16 round by 2^-9 of themselves
            assert np.abs(host(o.float())[sl] - o_ref).max() <= (4e-3 if t else 1e-5) * max(1.0, np.abs(o_ref).max())
        assert np.abs(host(ST)[s] - ST_ref).max() <= 1e-5 * max(1.0, np.abs(ST_ref).max())


@pytest.mark.parametrize("H, d_k, d_v", [(15, 176, 64), (16, 176, 64), (33, 168, 32), (34, 168, 32), (18, 64, 64), (74, 16, 16), (18, 160, 64),
                                         (15, 20, 64), (60, 130, 16), (17, 130, 64)])
@pytest.mark.parametrize("T, io", [(40, "f32"), (256, "f32"), (70, "bf16")])   # clusters that share SMs are taken from 256 tokens up
def test_scan_around_the_calls_that_go_to_clusters(H, d_k, d_v, T, io):
    import torch
    rng = np.random.default_rng(H + T)
    tok = wl.gdn_tokens(rng, T, H, H, d_k, d_v, io=io)
    S0 = rng.standard_normal((1, H, d_k, d_v)).astype(np.float32)
    t = torch.bfloat16 if io == "bf16" else None
    o, ST = b.lkv_gdn_fwd(*(dev(tok[n], t) for n in ("q", "k", "v")), dev(tok["g"]), dev(tok["beta"]), dev(S0), compute=b.LKV_COMPUTE_FP32)
    o_ref, ST_ref = oracle.gdn_seq(tok["q"], tok["k"], tok["v"], tok["g"], tok["beta"], S0[0])
    # outputs in bf16 round by 2^-9 of themselves
    assert np.abs(host(o.float()) - o_ref).max() <= (4e-3 if t else 1e-5) * max(1.0, np.abs(o_ref).max())
    assert np.abs(host(ST)[0] - ST_ref).max() <= 1e-5 * max(1.0, np.abs(ST_ref).max())
