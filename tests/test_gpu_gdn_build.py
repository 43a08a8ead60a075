"""States and transitions of chunks in one pass: the bits of the two scans that give them one by one, at the edges of blocks, of the block ring
and of the scaling."""
import numpy as np
import pytest

from paper_2608_11231_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H_k,H_v", [(1, 75), (16, 80), (2, 6)])   # one CTA for both from 75 heads a chunk on 148 SMs; two
@pytest.mark.parametrize("lens", [[1], [65], [0, 63, 65, 0, 128], [257, 2, 320, 641, 1000]])
@pytest.mark.parametrize("decay", [0.01, 1.0, 5.0])   # plain blocks; states rescaled and both forms in turn; exact blocks
def test_build_equals_the_two_scans(H_k, H_v, lens, decay):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(len(lens) + H_v)
    F, T, cu = torch.nn.functional, sum(lens), np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    k, v = F.normalize(rn(T, H_k, 128), dim=-1).bfloat16(), rn(T, H_v, 128).bfloat16()
    g, beta = -decay * F.softplus(rn(T, H_v)), torch.sigmoid(rn(T, H_v))
    S, P = b.lkv_gdn_chunk_artifacts(k, v, g, beta, cu_seqlens=cu)
    _, S1 = b.lkv_gdn_fwd(k, k, v, g, beta, cu_seqlens=cu, want_outputs=False)
    P1 = b.lkv_gdn_chunk_transition(k, g, beta, cu_seqlens=cu)
    assert torch.equal(S, S1) and torch.equal(P, P1)
