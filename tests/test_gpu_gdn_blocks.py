"""Gated DeltaNet scan at the edges of its blocks: lengths around the 64-token tile and the depth of its rings, decays that
switch between the two forms of a block, the state's scale going back to one, and one sequence long enough for segments."""
import numpy as np
import pytest

import oracle
from helpers import TOL_BF16, dev, host, maxrel_per_head
from paper_2608_11231_b200 import binding as b
from paper_2608_11231_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _decays(kind, rng, T, H):
    g = -rng.uniform(0.0, 0.02, (T, H))
    blk = np.arange(T) // 64
    if kind == "violent":        # whole heads, then every third block: per-block factors leave their range
        g[:, 0] *= 300.0
        g[blk % 3 == 1] *= 200.0
    elif kind == "reset":        # the running scale passes its limit every few blocks
        g *= 40.0
    elif kind == "edge":         # blocks on either side of the limit of the exact form, in turn and within a block
        g *= 85.0 * (1.0 + 0.1 * np.sin(blk))[:, None]
        g[:, 1] *= 3.0
    return g.astype(np.float32)


@pytest.mark.parametrize("lens, kind", [
    ([1, 63, 64, 65, 127, 128, 129, 191, 193], "mild"),
    ([257, 320, 321, 640], "violent"),
    ([1000, 64], "reset"),
    ([1000, 65, 130], "edge"),
    ([3000], "mild"),                                            # one long sequence: segments
    ([2943], "reset"),
])
@pytest.mark.parametrize("outputs", [True, False])
def test_gdn_scan_block_edges(lens, kind, outputs):
    import torch
    rng = np.random.default_rng(len(lens) * 1000 + lens[0])
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    T = int(cu[-1])
    tok = wl.gdn_tokens(rng, T, 2, 4, 128, 128, io="bf16", live_chunk_len=128)
    tok["g"] = _decays(kind, rng, T, 4)
    S0 = rng.standard_normal((len(lens), 4, 128, 128)).astype(np.float32)
    bf = torch.bfloat16
    o, ST = b.lkv_gdn_fwd(dev(tok["q"], bf), dev(tok["k"], bf), dev(tok["v"], bf), dev(tok["g"]), dev(tok["beta"]), dev(S0),
                          cu_seqlens=cu if len(lens) > 1 else None, want_outputs=outputs)
    o = host(o) if outputs else None
    ST = host(ST)
    for s in range(len(lens)):
        sl = slice(cu[s], cu[s + 1])
        o_ref, ST_ref = oracle.gdn_seq(tok["q"][sl], tok["k"][sl], tok["v"][sl], tok["g"][sl], tok["beta"][sl], S0[s])
        assert maxrel_per_head(ST[s], ST_ref, 0) <= TOL_BF16
        if outputs:
            assert maxrel_per_head(o[sl], o_ref, 1) <= TOL_BF16


@pytest.mark.parametrize("decay", [0.01, 0.6, 1.0, 3.0])
def test_gdn_scan_is_homogeneous(decay):
    """Values and states times a power of two: the results times that power, bit for bit.  (A held state times 2^100 became infinite
    from 2^27 on.)"""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(7)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    T = 1000
    bf = torch.bfloat16
    unit = lambda x: torch.nn.functional.normalize(x, dim=-1).to(bf)
    q, k, v, S0 = unit(rn(T, 2, 128)), unit(rn(T, 2, 128)), rn(T, 4, 128).to(bf), rn(1, 4, 128, 128)
    beta, g = torch.rand(T, 4, generator=gen, device="cuda"), -2 * decay * torch.rand(T, 4, generator=gen, device="cuda")
    o, S = b.lkv_gdn_fwd(q, k, v, g, beta, S0)
    for f in (2.0 ** 42, 2.0 ** -80):
        of, Sf = b.lkv_gdn_fwd(q, k, v * f, g, beta, S0 * f)
        assert torch.equal(of, o * f) and torch.equal(Sf, S * f)


def test_gdn_scan_time_bends_with_the_decays_but_does_not_break():
    """Decays of 250 log2 units a block (the exact form, whose mask takes an exponential per element) against mild ones: it took three
    times as long while that form was written for rare use."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    n, L = 16, 2048
    T = n * L
    bf = torch.bfloat16
    unit = lambda x: torch.nn.functional.normalize(x, dim=-1).to(bf)
    q, k, v, beta = unit(rn(T, 16, 128)), unit(rn(T, 16, 128)), rn(T, 32, 128).to(bf), torch.rand(T, 32, generator=gen, device="cuda")
    cu = (np.arange(n + 1) * L).astype(np.int32)

    def us(scale):
        g = -scale * torch.rand(T, 32, generator=gen, device="cuda")
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            b.lkv_gdn_fwd(q, k, v, g, beta, cu_seqlens=cu)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    assert us(5.4) < 2.2 * us(0.1)


@pytest.mark.parametrize("outputs", [True, False])
def test_gdn_scan_results_repeat_on_a_full_gpu(outputs):
    """Every SM busy, loads from DRAM: the same inputs give the same bits (a tile released before it is read does not)."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    n, L = 16, 1500
    T = n * L
    bf = torch.bfloat16
    args = (torch.nn.functional.normalize(rn(T, 16, 128), dim=-1).to(bf), torch.nn.functional.normalize(rn(T, 16, 128), dim=-1).to(bf),
            rn(T, 32, 128).to(bf), -0.1 * torch.rand(T, 32, generator=gen, device="cuda"), torch.rand(T, 32, generator=gen, device="cuda"))
    cu = (np.arange(n + 1) * L).astype(np.int32)
    o0, S0 = b.lkv_gdn_fwd(*args, cu_seqlens=cu, want_outputs=outputs)
    for _ in range(10):
        o, S = b.lkv_gdn_fwd(*args, cu_seqlens=cu, want_outputs=outputs)
        assert torch.equal(S, S0) and (not outputs or torch.equal(o, o0))
