"""The log-decay reduction at the edges of its split: a cluster of eight CTAs per sequence and 32 heads, eight warps of eight tokens."""
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
