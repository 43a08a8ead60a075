"""The fp32 GDN kernels at the edges of their tiles: head sizes that are not multiples of four or of the row tile, column splits
for few and for many heads, lengths around the 32-token block, rows so long that the ring has few stages."""
import numpy as np
import pytest

import oracle
from helpers import dev, host
from paper_2608_11231_b200 import binding as b
from paper_2608_11231_b200 import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-4


def _close(x, ref):
    assert np.abs(x - ref).max() <= TOL * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("H_k, H_v, d_k, d_v, lens", [
    (1, 2, 64, 64, [1, 31, 32, 33, 65]),
    (2, 2, 7, 16, [40]),              # rows of an odd length
    (1, 1, 130, 32, [70]),
    (1, 1, 64, 256, [33]),
    (2, 80, 66, 64, [37, 5]),         # every column of a head in one CTA
])
def test_gdn_fp32_scan_shapes(H_k, H_v, d_k, d_v, lens):
    rng = np.random.default_rng(d_k * 1000 + d_v)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    tok = wl.gdn_tokens(rng, int(cu[-1]), H_k, H_v, d_k, d_v, io="f32")
    S0 = rng.standard_normal((len(lens), H_v, d_k, d_v)).astype(np.float32)
    o, ST = b.lkv_gdn_fwd(*(dev(tok[n]) for n in ("q", "k", "v", "g", "beta")), dev(S0), cu_seqlens=cu, compute=b.LKV_COMPUTE_FP32)
    for s in range(len(lens)):
        sl = slice(cu[s], cu[s + 1])
        o_ref, ST_ref = oracle.gdn_seq(tok["q"][sl], tok["k"][sl], tok["v"][sl], tok["g"][sl], tok["beta"][sl], S0[s])
        _close(host(o)[sl], o_ref)
        _close(host(ST)[s], ST_ref)


@pytest.mark.parametrize("K, H, d_k, d_v", [(1, 2, 64, 64), (5, 2, 64, 64), (3, 1, 7, 8), (4, 2, 130, 36), (3, 1, 256, 64), (3, 1, 600, 32), (2, 90, 64, 64)])
def test_gdn_fp32_composition_shapes(K, H, d_k, d_v):
    rng = np.random.default_rng(K * 1000 + d_k)
    states = rng.standard_normal((K, H, d_k, d_v)).astype(np.float32)
    trans = (rng.standard_normal((K, H, d_k, d_k)) / d_k ** 0.5).astype(np.float32)
    S = states[0].astype(np.float64)
    for j in range(1, K):
        S = trans[j].astype(np.float64) @ S + states[j]
    out = b.lkv_init_state(dev(states), dev(trans), K=K, mode=b.LKV_INIT_EXACT, family=b.LKV_FAMILY_GDN, compute=b.LKV_COMPUTE_FP32)
    _close(host(out).reshape(S.shape), S)
