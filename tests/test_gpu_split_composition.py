"""One request's composition in two halves: around the length from which it is cut, odd and even halves, both pool types, and the chain in one for a
caller whose workspace has no room for the halves."""
import numpy as np
import pytest

from paper_2608_11231_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [9, 10, 11, 33])
@pytest.mark.parametrize("H, bf16", [(1, False), (49, True), (50, False)])   # 50 heads: three CTAs a head no longer find an SM each
def test_composition_in_halves(K, H, bf16):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(K + H)
    states = torch.randn((K + 2, H, 128, 128), generator=gen, device="cuda")
    pool = states.bfloat16() if bf16 else states
    trans = torch.linalg.qr(torch.randn((K + 2, H, 128, 128), generator=gen, device="cuda"))[0].contiguous() * 0.97   # every chunk counts
    ids = np.random.default_rng(K).permutation(K + 2)[:K].astype(np.int32)
    ref = pool[ids[0]].double()
    for j in ids[1:]:
        ref = trans[j].double() @ ref + pool[j].double()
    kw = dict(family=b.LKV_FAMILY_GDN, chunk_ids=ids)
    err = lambda x: float((x.double() - ref).norm() / ref.norm())
    cut = err(b.lkv_init_state(pool, trans, K, b.LKV_INIT_EXACT, **kw))
    chain = err(b.lkv_init_state(pool, trans, K, b.LKV_INIT_EXACT, workspace_t=torch.zeros(256, dtype=torch.uint8, device="cuda"), **kw))
    # tf32 operands, rounded to nearest: 2^-12 a step and operand at most, added in squares
    assert chain <= 2 ** -12 * (2 * K) ** 0.5 and cut <= 1.02 * chain, (cut, chain)
