"""Mamba-2 scan at the edges of its blocks: lengths around the 64- and 128-token tiles, groups with an odd number of heads,
decays that end blocks early in one head of a pair, and one sequence long enough to be scanned in segments."""
import numpy as np
import pytest

import oracle
from helpers import TOL_BF16, dev, host, maxrel_per_head
from paper_2608_11231_b200 import binding as b
from paper_2608_11231_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H, G, lens, decay", [
    (3, 1, [1, 63, 64, 65, 127, 128, 129, 255, 257], 1.0),       # odd head count, every remainder that matters
    (6, 2, [200, 128, 640], 1.0),                                # odd heads per group: pairs do not straddle groups
    (4, 1, [700, 130], np.array([0.05, 20.0, 1.0, 200.0])),      # mild and violent heads in one CTA: blocks end early
    (80, 1, [300], 0.02),                                        # benchmark shape, weak decay
    (4, 1, [3333], 0.3),                                         # one long sequence: segments
    (4, 1, [700, 130, 128, 1], np.array([2.0, 3.0, 5.0, 9.0])),  # tiles of several blocks
    (3, 1, [257, 384], np.array([6.0, 0.1, 12.0])),              # the same beside a mild head, and the last head alone
    (4, 1, [3333], np.array([3.0, 8.0, 20.0, 0.5])),             # the same in segments
])
@pytest.mark.parametrize("outputs", [True, False])
def test_ssd_scan_block_edges(H, G, lens, decay, outputs):
    import torch
    rng = np.random.default_rng(H * 1000 + lens[0])
    P, N = 64, 128
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    A = (wl.ssd_A(rng, H) * decay).astype(np.float32)
    tok = wl.ssd_tokens(rng, int(cu[-1]), H, P, N, G)
    S0 = rng.standard_normal((len(lens), H, N, P)).astype(np.float32)
    bf = torch.bfloat16
    y, ST = b.lkv_ssd_fwd(dev(tok["x"], bf), dev(tok["dt"]), dev(A), dev(tok["B"], bf), dev(tok["C"], bf), dev(S0),
                          cu_seqlens=cu if len(lens) > 1 else None, want_outputs=outputs)
    y = host(y) if outputs else None
    ST = host(ST)
    for s in range(len(lens)):
        sl = slice(cu[s], cu[s + 1])
        y_ref, ST_ref = oracle.ssd_seq(tok["x"][sl], tok["dt"][sl], A, tok["B"][sl], tok["C"][sl], S0[s])
        assert maxrel_per_head(ST[s], ST_ref, 0) <= TOL_BF16
        if outputs:
            assert maxrel_per_head(y[sl], y_ref, 1) <= TOL_BF16


@pytest.mark.parametrize("A, power", [(-0.2, 50), (-3.0, 50), (-5.0, 24), (-60.0, 24)])
def test_ssd_scan_is_homogeneous(A, power):
    """Inputs and states times a power of two: the results times that power, upwards bit for bit.  (A held state times 2^100 became
    infinite from 2^27 on.)  Downwards the low halves of the factors of x leave the range first: one more rounding to bf16."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(7)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    T, H = 1000, 4
    bf = torch.bfloat16
    x, B, C = rn(T, H, 64).to(bf), (rn(T, 1, 128) / 128 ** 0.5).to(bf), (rn(T, 1, 128) / 128 ** 0.5).to(bf)
    dt, S0 = torch.nn.functional.softplus(-2.0 + 0.5 * rn(T, H)), rn(1, H, 128, 64)
    a = torch.full((H,), A, device="cuda")
    y, S = b.lkv_ssd_fwd(x, dt, a, B, C, S0)
    f = 2.0 ** power
    yf, Sf = b.lkv_ssd_fwd(x * f, dt, a, B, C, S0 * f)
    assert torch.equal(yf, y * f) and torch.equal(Sf, S * f)
    yf, Sf = b.lkv_ssd_fwd(x / f, dt, a, B, C, S0 / f)
    assert maxrel_per_head(host(yf * f), host(y), 1) <= 2.0 ** -8 and maxrel_per_head(host(Sf * f), host(S), 1) <= 2.0 ** -8
    yf, Sf = b.lkv_ssd_fwd(x * 0.0, dt, a, B, C, S0 * 2.0 ** 110)   # a state that is only carried on
    y0, S1 = b.lkv_ssd_fwd(x * 0.0, dt, a, B, C, S0)
    assert torch.isfinite(yf).all() and torch.equal(yf[:8], y0[:8] * 2.0 ** 110)


@pytest.mark.parametrize("every, dt", [(37, 60.0), (16, 1000.0), (5, 30.0)])
def test_ssd_scan_with_tokens_that_forget_everything(every, dt):
    """Single tokens whose own decay is beyond the range of a block's scale, among mild ones: they cut tiles at any offset."""
    import torch
    rng = np.random.default_rng(every)
    H, T = 4, 500
    A = wl.ssd_A(rng, H).astype(np.float32)
    tok = wl.ssd_tokens(rng, T, H, 64, 128, 1)
    tok["dt"][every - 1::every, ::2] = dt
    S0 = rng.standard_normal((1, H, 128, 64)).astype(np.float32)
    bf = torch.bfloat16
    y, ST = b.lkv_ssd_fwd(dev(tok["x"], bf), dev(tok["dt"]), dev(A), dev(tok["B"], bf), dev(tok["C"], bf), dev(S0))
    y_ref, ST_ref = oracle.ssd_seq(tok["x"], tok["dt"], A, tok["B"], tok["C"], S0[0])
    assert maxrel_per_head(host(ST)[0], ST_ref, 0) <= TOL_BF16
    y = host(y)
    forget = np.arange(T) % every == every - 1   # their outputs are as large as dt: scored apart
    for rows in (forget, ~forget):
        assert maxrel_per_head(y[rows], y_ref[rows], 1) <= TOL_BF16


def test_ssd_scan_time_bends_with_the_decays_but_does_not_break():
    """Decays of 600 log2 units a tile: the chain runs several times per tile, everything else once (every block a tile of its own
    took four times as long as mild decays)."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    H, n, L = 80, 16, 2048
    T = n * L
    bf = torch.bfloat16
    x, B, C = rn(T, H, 64).to(bf), (rn(T, 1, 128) / 128 ** 0.5).to(bf), (rn(T, 1, 128) / 128 ** 0.5).to(bf)
    dt = torch.nn.functional.softplus(0.2 + 0.3 * rn(T, H))
    cu = (np.arange(n + 1) * L).astype(np.int32)

    def us(A):
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            b.lkv_ssd_fwd(x, dt, A, B, C, cu_seqlens=cu)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    mild, strong = us(torch.full((H,), -0.05, device="cuda")), us(torch.full((H,), -4.0, device="cuda"))
    assert strong < 3 * mild


@pytest.mark.parametrize("decay, outputs", [(1.0, True), (40.0, True), (40.0, False)])
def test_ssd_scan_results_repeat_on_a_full_gpu(decay, outputs):
    """Every SM busy, loads from DRAM: the same inputs give the same bits (a tile released before it is read does not).  Strong
    decays make blocks of a few tokens, so that the ring of block descriptors turns fastest."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    H, n, L = 80, 16, 2000
    T = n * L
    bf = torch.bfloat16
    args = (rn(T, H, 64).to(bf), torch.nn.functional.softplus(-2.0 + 0.5 * rn(T, H)), -decay * torch.exp(2.0 * torch.rand(H, generator=gen, device="cuda")),
            (rn(T, 1, 128) / 128 ** 0.5).to(bf), (rn(T, 1, 128) / 128 ** 0.5).to(bf))
    cu = (np.arange(n + 1) * L).astype(np.int32)
    y0, S0 = b.lkv_ssd_fwd(*args, cu_seqlens=cu, want_outputs=outputs)
    for _ in range(10):
        y, S = b.lkv_ssd_fwd(*args, cu_seqlens=cu, want_outputs=outputs)
        assert torch.equal(S, S0) and (not outputs or torch.equal(y, y0))
