"""Timed cases of the library's public calls: what a serving engine has this path do for one recurrent layer.

A layer serves requests in passes: build the initial state of every request from cached chunk states
(``lkv_init_state*``), then scan the tokens to recompute from it (``lkv_gdn_fwd`` / ``lkv_ssd_fwd``).  Beside that it
prefills requests that have no cache entry and turns new chunks into cache entries.  Layer shapes are those of
``workloads.CONFIGS``; inputs are drawn as ``workloads`` draws them, on the device.

Kinds of case
  tiny     fp32 GDN layer, d = 64, one request: exact composition and the scan of its suffix (fp32 arithmetic)
  request  one request: exact composition of its K cached chunks, then the scan of its recompute tokens (bf16)
  suffix   requests whose cached state (bf16 pool) is taken as it is, then the scan of a short ragged suffix
  batch    concurrent requests over one shared pool, each with its own chunk order, equal recompute lengths
  mix      ragged serving mix: every request with its own chunks, number of chunks and recompute length
  prefill  one request with no cache entry: the plain scan from the empty state
  build    new chunks (ragged) to cache entries: final states and transitions, no outputs
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2608_11231_b200 import binding as b
from paper_2608_11231_b200 import workloads as wl

GDN = {k: wl.CONFIGS[2][k] for k in ("H_k", "H_v", "d_k", "d_v")}
SSD = {k: wl.CONFIGS[1][k] for k in ("H", "P", "N", "G")}
TINY = {k: wl.CONFIGS[0][k] for k in ("H_k", "H_v", "d_k", "d_v")}


def listed():
    return [
        # configuration 0: the smallest layer, fp32 throughout; latency of two small calls
        dict(name="gdn_tiny_f32", kind="tiny", family="gdn", K=4, T=64),
        # configuration 1: one 8K request of a Mamba-2 layer, 1024 tokens to recompute
        dict(name="mamba_request_8k", kind="request", family="mamba2", K=8, T=1024),
        # configuration 2: one 16K request of a GDN layer, a fifth of its tokens to recompute
        dict(name="gdn_request_16k", kind="request", family="gdn", K=16, T=3276),
        # the shortest pass in serving: one request continues from its last cached state with a query of a few tokens
        dict(name="mamba_suffix_1", kind="suffix", family="mamba2", n_req=1, len_lo=37, len_hi=37, seed=0),
        # the same for a batch, every query of another length
        dict(name="gdn_suffix_16", kind="suffix", family="gdn", n_req=16, len_lo=1, len_hi=128, seed=1),
        # configuration 3: eight 32K requests that share their cached chunks
        dict(name="gdn_batch_32k", kind="batch", family="gdn", n_req=8, K=32, T=2048),
        # configuration 4, both halves: the ragged mix
        dict(name="mamba_mix_32", kind="mix", family="mamba2", n_req=32, seed=4),
        dict(name="gdn_mix_32", kind="mix", family="gdn", n_req=32, seed=4),
        # nothing cached: full prefill of the single requests of configurations 1 and 2
        dict(name="mamba_prefill_8k", kind="prefill", family="mamba2", T=8192),
        dict(name="gdn_prefill_16k", kind="prefill", family="gdn", T=16384),
        # filling the cache: chunks of the mix's lengths
        dict(name="mamba_build_32", kind="build", family="mamba2", n_req=32, len_lo=256, len_hi=2048, seed=2),
        dict(name="gdn_build_16", kind="build", family="gdn", n_req=16, len_lo=256, len_hi=2048, seed=3),
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], its logarithm uniform."""
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["tiny", "request", "suffix", "batch", "mix", "prefill", "build"])
    case = dict(kind=kind, family="gdn" if kind == "tiny" else rng.choice(["mamba2", "gdn"]))
    if kind == "tiny":
        case.update(K=_spread(rng, 1, 16), T=_spread(rng, 16, 512))
    elif kind == "request":
        case.update(K=_spread(rng, 2, 64), T=_spread(rng, 64, 6554))
    elif kind == "suffix":
        case.update(n_req=_spread(rng, 1, 64), len_lo=1, len_hi=_spread(rng, 8, 256), seed=rng.randrange(1 << 20))
    elif kind == "batch":
        case.update(n_req=_spread(rng, 2, 16), K=_spread(rng, 4, 32), T=_spread(rng, 128, 2048))
    elif kind == "mix":
        case.update(n_req=_spread(rng, 4, 31), seed=rng.randrange(1 << 20))
    elif kind == "prefill":
        case.update(T=_spread(rng, 1024, 24576))
    else:
        case.update(n_req=_spread(rng, 1, 24), len_lo=256, len_hi=2048, seed=rng.randrange(1 << 20))
    return case


def _layout(case):
    """(pool size, chunk ids, cu_k, lengths of the scanned sequences) of a case; the ids are None where nothing is composed."""
    kind = case["kind"]
    if kind == "mix":
        reqs = wl.ragged_mix(seed=case["seed"], n_req=2 * case["n_req"])
        reqs = [r for r in reqs if r["family"] == case["family"]]
        ks, lens = [r["K"] for r in reqs], [r["recompute"] for r in reqs]
        return sum(ks), np.arange(sum(ks), dtype=np.int32), _cu(ks), lens
    if kind == "batch":
        n, K = case["n_req"], case["K"]
        ids = np.concatenate([wl.request_permutation(3, r, K) for r in range(n)]).astype(np.int32)
        return K, ids, _cu([K] * n), [case["T"]] * n
    if kind in ("suffix", "build"):
        rng = random.Random(case["seed"])
        lens = [rng.randint(case["len_lo"], case["len_hi"]) for _ in range(case["n_req"])]
        if kind == "build":
            return 0, None, None, lens
        n = case["n_req"]
        ids = np.array(rng.sample(range(2 * n), n), dtype=np.int32)  # one matched chunk of each request, in a pool of twice as many
        return 2 * n, ids, np.arange(n + 1, dtype=np.int32), lens
    if kind == "prefill":
        return 0, None, None, [case["T"]]
    return case["K"], np.random.default_rng(case["K"]).permutation(case["K"]).astype(np.int32), None, [case["T"]]


def _cu(lens):
    return np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)


def _gdn_tokens(rn, T, s, io, live=None):
    """As workloads.gdn_tokens."""
    F = torch.nn.functional
    q = F.normalize(rn(T, s["H_k"], s["d_k"]), dim=-1).to(io)
    k = F.normalize(rn(T, s["H_k"], s["d_k"]), dim=-1).to(io)
    v = rn(T, s["H_v"], s["d_v"]).to(io)
    beta, g = torch.sigmoid(rn(T, s["H_v"])), -0.1 * F.softplus(rn(T, s["H_v"]))
    if live is not None:
        g, beta = g * (4.0 / live), beta / 8.0
    return dict(q=q, k=k, v=v, g=g, beta=beta)


def _ssd_tokens(rn, T, s, io):
    """As workloads.ssd_tokens."""
    return dict(x=rn(T, s["H"], s["P"]).to(io), dt=torch.nn.functional.softplus(-2.0 + 0.5 * rn(T, s["H"])),
                B=(rn(T, s["G"], s["N"]) / s["N"] ** 0.5).to(io), C=(rn(T, s["G"], s["N"]) / s["N"] ** 0.5).to(io))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def rn(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    kind, gdn = case["kind"], case["family"] == "gdn"
    n_pool, ids, cu_k, lens = _layout(case)
    T = int(sum(lens))
    io = torch.float32 if kind == "tiny" else torch.bfloat16
    # chunks that become cache entries have the weak decays with which a carried state matters
    live = 1024 if kind == "build" else None
    st = dict(case=case, gdn=gdn, ids=ids, cu_k=cu_k, cu=_cu(lens) if len(lens) > 1 else None)
    if gdn:
        s = TINY if kind == "tiny" else GDN
        st["tok"] = _gdn_tokens(rn, T, s, io, live)
        H, dk, dv = s["H_v"], s["d_k"], s["d_v"]
    else:
        st["tok"] = _ssd_tokens(rn, T, SSD, io)
        H, dk, dv = SSD["H"], SSD["N"], SSD["P"]
        st["A"] = -torch.exp(2.0 * torch.rand(H, generator=gen, device="cuda")) * (4.0 / live if live else 1.0)
    if n_pool:
        st["states"] = rn(n_pool, H, dk, dv)
        if kind == "suffix":
            st["states"] = st["states"].to(torch.bfloat16)
        elif gdn:
            st["trans"] = rn(n_pool, H, dk, dk) * (0.45 / dk ** 0.5)
        else:
            st["trans"] = -2.0 * torch.rand((n_pool, H), generator=gen, device="cuda")
    return st


def run(st):
    case, t, gdn = st["case"], st["tok"], st["gdn"]
    kind, family = case["kind"], b.LKV_FAMILY_GDN if gdn else b.LKV_FAMILY_MAMBA2
    if kind == "build":
        if gdn:
            return b.lkv_gdn_chunk_artifacts(t["k"], t["v"], t["g"], t["beta"], cu_seqlens=st["cu"])
        # Mamba-2 states are cached in bf16
        _, S = b.lkv_ssd_fwd(t["x"], t["dt"], st["A"], t["B"], t["C"], cu_seqlens=st["cu"], want_outputs=False,
                             state_dtype=torch.bfloat16)
        return S, b.lkv_mamba_chunk_logdecay(t["dt"], st["A"], cu_seqlens=st["cu"])
    S0 = None
    if kind in ("tiny", "request"):
        S0 = b.lkv_init_state(st["states"], st["trans"], case["K"], b.LKV_INIT_EXACT, family=family, chunk_ids=st["ids"])[None]
    elif kind == "suffix":
        S0 = b.lkv_init_state_batched(st["states"], None, st["ids"], st["cu_k"], case["n_req"], b.LKV_INIT_LAST, family=family)
    elif kind in ("batch", "mix"):
        S0 = b.lkv_init_state_batched(st["states"], st["trans"], st["ids"], st["cu_k"], case["n_req"], b.LKV_INIT_EXACT,
                                      family=family)
    if gdn:
        o, S_T = b.lkv_gdn_fwd(t["q"], t["k"], t["v"], t["g"], t["beta"], S0, cu_seqlens=st["cu"])
    else:
        o, S_T = b.lkv_ssd_fwd(t["x"], t["dt"], st["A"], t["B"], t["C"], S0, cu_seqlens=st["cu"])
    return S0, o, S_T


def work(case):
    """Every input read once, every output written once; operations of the token recurrence (update and read-out)."""
    kind, gdn = case["kind"], case["family"] == "gdn"
    n_pool, ids, cu_k, lens = _layout(case)
    T, n = sum(lens), len(lens)
    io = 4 if kind == "tiny" else 2
    if gdn:
        s = TINY if kind == "tiny" else GDN
        H, dk, dv = s["H_v"], s["d_k"], s["d_v"]
        q_bytes = T * s["H_k"] * dk * io
        token_bytes = 2 * q_bytes + 2 * T * H * dv * io + 2 * T * H * 4
        flops = 6.0 * T * H * dk * dv
    else:
        H, dk, dv = SSD["H"], SSD["N"], SSD["P"]
        q_bytes = 0
        token_bytes = 2 * T * H * dv * io + 2 * T * SSD["G"] * dk * io + T * H * 4 + H * 4
        flops = 4.0 * T * H * dk * dv
    out_bytes, state = T * H * dv * io, H * dk * dv * 4
    trans = H * (dk * dk if gdn else 1) * 4
    if kind == "build":
        if gdn:  # keys, values and gates in, states and transitions out
            return dict(bytes=token_bytes - q_bytes - out_bytes + n * (state + trans), flops=2.0 * T * H * dk * (2 * dv + 2 * dk))
        C_bytes = T * SSD["G"] * dk * io
        return dict(bytes=token_bytes - C_bytes - out_bytes + n * (state // 2 + trans), flops=2.0 * T * H * dk * dv)
    total = token_bytes + n * state
    if kind == "suffix":
        total += n * (state // 2 + state)
    elif n_pool:
        cu = _cu([len(ids)]) if cu_k is None else cu_k
        first = {int(ids[cu[r]]) for r in range(n)}
        later = {int(i) for r in range(n) for i in ids[cu[r] + 1:cu[r + 1]]}
        total += len(first | later) * state + len(later) * trans + n * state
        flops += (len(ids) - n) * 2.0 * H * dk * dv * (dk if gdn else 1)
    return dict(bytes=total, flops=flops)


def tolerance(case):
    if case["kind"] == "tiny":
        return {"rel": 1e-5, "max": 1e-4}  # fp32 sums over a few hundred tokens
    if case["kind"] == "build" and case["family"] == "gdn":
        return {"rel": 2e-2, "max": 0.2}  # products over up to 2048 tokens with bf16 operands
    return {"rel": 1e-2, "max": 0.15}  # bf16 tensors and operands, fp32 sums
