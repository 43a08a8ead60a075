"""The binding among several Python threads: the interpreter lock is free during a call, and calls that share a stream (and with it
a workspace) do not mix."""
import threading
import time
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2608_11231_b200 import binding as b

pytestmark = pytest.mark.gpu


def test_other_threads_run_during_a_call():
    """A long index list whose last entry is out of range keeps the host in the argument checks (nothing is launched)."""
    import torch
    states = torch.zeros((1, 1, 64, 64), device="cuda")
    S0 = torch.empty((1, 1, 64, 64), device="cuda")
    ids = np.zeros(200_000_000, dtype=np.int32)
    ids[-1] = 1
    cu = np.array([0, ids.size], dtype=np.int32)
    ws = torch.zeros(4096, dtype=torch.uint8, device="cuda")
    stop, ticks = threading.Event(), []

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.0005)

    t = threading.Thread(target=tick)
    t.start()
    time.sleep(0.05)
    t0 = time.perf_counter()
    with pytest.raises(b.LkvError):
        b.lkv_init_state_batched(states, None, ids, cu, 1, b.LKV_INIT_LAST, S0=S0, family=b.LKV_FAMILY_GDN, workspace_t=ws)
    t1 = time.perf_counter()
    stop.set()
    t.join()
    assert t1 - t0 > 0.02, "the call is too short to tell"
    inside = [x for x in ticks if t0 < x < t1]
    assert max(np.diff([t0, *inside, t1])) < 0.5 * (t1 - t0)


def test_threads_that_share_a_stream():
    """One sequence in segments is three launches that hand states through the workspace of the stream."""
    import torch
    bf = torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(3)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    T = 4096
    unit = lambda x: torch.nn.functional.normalize(x, dim=-1).to(bf)
    gdn = [(unit(rn(T, 4, 128)), unit(rn(T, 4, 128)), rn(T, 8, 128).to(bf), -0.01 * torch.rand(T, 8, generator=gen, device="cuda"),
            torch.rand(T, 8, generator=gen, device="cuda")) for _ in range(2)]
    ssd = [(rn(T, 8, 64).to(bf), 0.01 * torch.rand(T, 8, generator=gen, device="cuda"), -torch.rand(8, generator=gen, device="cuda"),
            rn(T, 1, 128).to(bf), rn(T, 1, 128).to(bf)) for _ in range(2)]
    work = [(b.lkv_gdn_fwd, a) for a in gdn] + [(b.lkv_ssd_fwd, a) for a in ssd]
    alone = [f(*a) for f, a in work]
    torch.cuda.synchronize()

    def engine(i):
        f, a = work[i]
        for _ in range(20):
            o, S = f(*a)   # the thread's first CUDA call
            assert torch.equal(o, alone[i][0]) and torch.equal(S, alone[i][1])

    with ThreadPoolExecutor(len(work)) as pool:
        for r in [pool.submit(engine, i) for i in range(len(work))]:
            r.result()


def test_calls_on_streams_passed_explicitly():
    """The segments' states travel through the workspace: calls that may overlap have one each, whatever stream is current."""
    import torch
    bf = torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(4)
    rn = lambda *s: torch.randn(s, generator=gen, device="cuda")
    T = 8192
    unit = lambda x: torch.nn.functional.normalize(x, dim=-1).to(bf)
    work = [(unit(rn(T, 2, 128)), unit(rn(T, 2, 128)), rn(T, 2, 128).to(bf), -0.01 * torch.rand(T, 2, generator=gen, device="cuda"),
             torch.rand(T, 2, generator=gen, device="cuda")) for _ in range(2)]
    alone = [b.lkv_gdn_fwd(*a) for a in work]
    streams = [torch.cuda.Stream() for _ in work]
    outs = [[(torch.empty_like(a[2]), torch.empty((1, 2, 128, 128), device="cuda")) for _ in range(10)] for a in work]
    torch.cuda.synchronize()
    for i in range(10):
        for s, a, o in zip(streams, work, outs):
            b.lkv_gdn_fwd(*a, None, *o[i], stream=s)
    torch.cuda.synchronize()
    for ref, o in zip(alone, outs):
        assert all(torch.equal(x, ref[0]) and torch.equal(S, ref[1]) for x, S in o)
