"""The log-decay reduction at the edges of its split: eight warps of every eighth token up to 512 tokens, eight parts of that beyond, side by side
in a cluster of CTAs or one after the other in one CTA."""
import numpy as np
import pytest

import oracle
from helpers import dev, host
from paper_2608_11231_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [1, 32, 33, 80])
def test_logdecay_of_ragged_lengths(H):
    lens = [1, 7, 8, 0, 9, 63, 64, 65, 511, 512, 513, 4097]
    rng = np.random.default_rng(H)
    A = (-np.exp(rng.uniform(0, 2, H))).astype(np.float32)
    dts = [rng.uniform(0.01, 1.0, (L, H)).astype(np.float32) for L in lens]
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    lam = host(b.lkv_mamba_chunk_logdecay(dev(np.concatenate(dts)), dev(A), cu_seqlens=cu))
    for c, d in enumerate(dts):
        ref = oracle.mamba_logdecay(d, A) if len(d) else np.zeros(H)
        # positive terms: each of at most L / 64 + 22 additions on a term's way to the sum rounds by 2^-24, and one product
        assert np.all(np.abs(lam[c] - ref) <= (len(d) / 64 + 24) * 2.0 ** -24 * np.abs(ref)), c


def test_bits_of_a_chunk_do_not_depend_on_the_call():
    """Alone, a long chunk is a cluster; among many it is one CTA."""
    import torch
    lens = [5, 64, 511, 512, 513, 2050] + [3] * 200
    rng = np.random.default_rng(7)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    dt, A = dev(rng.uniform(0.01, 1.0, (cu[-1], 80)).astype(np.float32)), dev((-np.exp(rng.uniform(0, 2, 80))).astype(np.float32))
    many = b.lkv_mamba_chunk_logdecay(dt, A, cu_seqlens=cu)
    few = b.lkv_mamba_chunk_logdecay(dt[:cu[6]], A, cu_seqlens=cu[:7])
    assert torch.equal(many[:6], few)
    for c in range(7):
        assert torch.equal(b.lkv_mamba_chunk_logdecay(dt[cu[c]:cu[c + 1]], A)[0], many[c])
        ref = oracle.mamba_logdecay(host(dt[cu[c]:cu[c + 1]]), host(A))
        assert np.all(np.abs(host(many[c]) - ref) <= (lens[c] / 64 + 24) * 2.0 ** -24 * np.abs(ref))
