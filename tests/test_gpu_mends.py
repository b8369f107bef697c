"""Results that single paths once got wrong: each test fails on the form it names."""
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

import oracle
from paper_2102_05613_gb300 import inputs, sk

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("figures", [True, False])
@pytest.mark.parametrize("N,chains", [(64, 3), (130, 300), (1000, 129)])
def test_pm1_resync_sets_integer_fields(N, chains, figures):
    # the product's float bits went into the int32 fields, so that every later
    # step, record and energy was wrong; here the fields are stale first (other
    # couplings), the resync sets J s, and the chain goes on as the oracle's
    need_gpu()
    J = inputs.couplings_pm1(N, N)
    init = inputs.initial_spins(chains, N, 92)
    inst = sk.Instance(inputs.couplings_pm1(N, N + 1))
    run = sk.Run(inst, chains=chains, K=24, beta=0.7, seed=93, init=init, record_every=20, max_records=2)
    inst.set_couplings(J)
    if figures:
        h0 = run.state(fields=True)[1].astype(np.int64)
        st, _ = run.recompute(sk.SK_RECOMPUTE_RESYNC)
        d = h0 - init.astype(np.int64) @ J.astype(np.int64)
        assert st["mismatches"] == np.count_nonzero(d) and st["max_field_drift"] == np.abs(d).max()
    else:
        run.recompute(sk.SK_RECOMPUTE_RESYNC, sync=False)
    s, h, _ = run.state(fields=True)
    assert np.array_equal(s, init) and np.array_equal(h, init.astype(np.int64) @ J.astype(np.int64))
    st, _ = run.recompute(sk.SK_RECOMPUTE_CHECK)
    assert st["mismatches"] == 0 and st["max_field_drift"] == 0.0 and st["max_energy_drift"] == 0.0
    run.advance(40)
    E, _, acc = run.observables()
    o = oracle.run(J, K=24, beta=0.7, seed=93, chains=chains, init=init, steps=40, record_every=20)
    assert np.array_equal(E, o["E"]) and np.array_equal(acc, o["acc"]) and np.array_equal(run.state()[0], o["spins"])
    run.close(); inst.close()


# Gaussian, N = 64, couplings seed 81, starts seed 82, beta = 1: (K, run seed, chain, step) where the
# draw lies between the last slot's prefix and the rounded total.
GAPS = [(40, 144, 300, 859), (40, 24, 1746, 72), (100, 119, 919, 917), (100, 98, 1729, 448), (200, 58, 902, 838),
        (200, 64, 2170, 398)]


@pytest.mark.parametrize("K,seed,chain,step", GAPS)
def test_search_never_leaves_the_slots(K, seed, chain, step):
    # the search took slot 4 L + 4 (past K) with site 0 there, unproposed; now
    # the last slot with a positive weight, alike in every layout
    need_gpu()
    N, steps = 64, step + 20
    J = inputs.couplings(N, sk.SK_J_GAUSS, 81)
    init = inputs.initial_spins(4900, N, 82)

    def go(chains, warps=0, lanes=0, staging=0, cluster=0, fused=0):
        inst = sk.Instance(J)
        run = sk.Run(inst, chains=chains, K=K, beta=1.0, seed=seed, init=init[:chains], trace_chains=chains,
                     trace_steps=steps)
        b = sk.Batch([run], warps_per_cta=warps)
        if lanes or staging:
            b.set_layout(lanes=lanes, staging=staging)
        if cluster:
            b.set_cluster(cluster)
        if fused:
            b.set_fused(fused)
        b.advance(steps)
        out = run.trace(), run.state(fields=True)
        b.close(); run.close(); inst.close()
        return out

    few = chain + 1
    forms = [dict(chains=4900), dict(chains=few), dict(chains=few, warps=4, lanes=32, staging=2),
             dict(chains=few, warps=24, lanes=32, staging=2), dict(chains=few, warps=4, lanes=32, staging=1),
             dict(chains=few, cluster=1), dict(chains=few, cluster=2), dict(chains=few, fused=8)]
    if K <= 128:
        forms.append(dict(chains=few, lanes=128))
    if K <= 64:
        forms += [dict(chains=few, lanes=64), dict(chains=few, lanes=16, staging=2)]
    tr0, (s0, h0, _) = go(**forms[0])
    assert tr0.max() <= K and tr0[chain, step] == K
    r = oracle.replay(J, tr0[chain], K=K, beta=1.0, seed=seed, chain=chain, init=init[chain], tol=1e-4)
    assert r["bad"] == 0 and np.array_equal(r["spins"], s0[chain])
    for f in forms[1:]:
        tr, (s, h, _) = go(**f)
        n = f["chains"]
        assert np.array_equal(tr, tr0[:n]) and np.array_equal(s, s0[:n]) and np.array_equal(h, h0[:n]), f
    # layouts with sums of their own
    for lanes in (8, 16):
        if K <= 16 * lanes:
            assert go(few, lanes=lanes, staging=2)[0].max() <= K


def test_energy_without_host_memory_is_an_error():
    # the host copy of the energies threw through the C entry and ended the
    # process; in a process of its own whose data size is limited meanwhile
    need_gpu()
    code = """
import ctypes as C, resource, sys
import numpy as np, torch
from paper_2102_05613_gb300 import inputs, sk
count = 1 << 25
s = torch.ones((count, 2), dtype=torch.int8, device="cuda")
out = np.zeros(count)
inst = sk.Instance(inputs.couplings_pm1(2, 1))
def call(n):
    return sk.lib().sk_energy(inst.handle, C.c_void_p(s.data_ptr()), n, sk.SK_MEM_DEVICE,
                              out.ctypes.data_as(C.c_void_p))
assert call(1000) == sk.SK_OK
data = [int(x.split()[1]) for x in open("/proc/self/status") if x.startswith("VmData")][0] << 10
soft, hard = resource.getrlimit(resource.RLIMIT_DATA)
resource.setrlimit(resource.RLIMIT_DATA, (data + (100 << 20), hard))
st = call(count)
resource.setrlimit(resource.RLIMIT_DATA, (soft, hard))
assert st == sk.SK_ERR_OOM and not out[1000:].any(), st
assert call(count) == sk.SK_OK and np.all(out == out[0]) and abs(out[0]) == 1.0
inst.close()
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("N,chains,K,rule,lanes", [
    (128, 1, 33, 0, 32), (512, 304, 64, 0, 32), (768, 600, 48, 0, 32), (1024, 304, 48, 0, 128), (1024, 600, 48, 0, 32),
    (2048, 600, 64, 0, 64), (512, 1, 100, 0, 128), (512, 304, 1, 1, 64), (1024, 304, 1, 1, 128), (1024, 600, 1, 1, 32)])
def test_default_of_few_pm1_chains(N, chains, K, rule, lanes):
    # +-J chains whose weight table is short got teams where their one-warp
    # loop is the faster one; either layout gives the oracle's chain
    need_gpu()
    J = inputs.couplings_pm1(N, 95)
    init = inputs.initial_spins(chains, N, 96)
    inst = sk.Instance(J)
    run = sk.Run(inst, chains=chains, K=K, rule=rule, beta=1.0, seed=97, init=init)
    b = sk.Batch([run])
    assert b.classes()[0][1] == lanes, b.classes()
    b.advance(30)
    o = oracle.run(J, K=K, rule=rule, beta=1.0, seed=97, chains=chains, init=init, steps=30)
    assert np.array_equal(run.state()[0], o["spins"])
    b.close(); run.close(); inst.close()


@pytest.mark.parametrize("spare", [2 << 20, 80 << 20])
def test_server_keeps_no_workspace_beyond_its_budget(spare):
    # the pool of the operands of retiring jobs' energies stayed with the process
    # on top of budget_bytes
    torch = need_gpu()
    N, chains = 1024, 2048
    job = dict(couplings_id=1, N=N, kind=sk.SK_J_GAUSS, chains=chains, steps=20, K=8, seed=4)

    def go(budget):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        srv = sk.Server(budget_bytes=budget, quantum_steps=20)
        srv.add_couplings(1, inputs.couplings(N, sk.SK_J_GAUSS, 98))
        t = srv.submit(**job)
        srv.wait_all()
        held = free - torch.cuda.mem_get_info()[0]
        footprint = srv.poll(t)["footprint_bytes"]
        out = srv.result(t, chains, N)
        srv.close()
        return held, footprint, out

    _, footprint, first = go(1 << 30)  # (loads the kernels)
    held, _, out = go(footprint + spare)
    assert held <= footprint + spare, (held, footprint, spare)
    assert all(np.array_equal(x, y) for x, y in zip(out, first))


def test_wait_without_a_limit_does_not_hold_a_core():
    # the wait for a long run polled or synchronised without a pause
    need_gpu()
    inst = sk.Instance(inputs.couplings_pm1(64, 1))
    run = sk.Run(inst, chains=1, K=8, beta=1.0, seed=2)
    run.advance(100)
    run.wait()
    run.advance(1_000_000)
    w0, c0 = time.perf_counter(), time.thread_time()
    run.wait()
    wall, cpu = time.perf_counter() - w0, time.thread_time() - c0
    assert wall > 0.2 and cpu < 0.5 * wall, (wall, cpu)
    assert run.state()[1] == 1_000_100
    run.close(); inst.close()


@pytest.mark.parametrize("N,arity,depth,chains,nw", [(300, 2, 2, 3000, 1), (300, 2, 2, 12000, 1), (1024, 2, 3, 3000, 1),
                                                     (1024, 2, 7, 32, 8), (1024, 2, 7, 6000, 2)])
def test_default_warps_of_graph_chains(N, arity, depth, chains, nw):
    # thousands of chains on small trees got 4 and 8 warps per chain, 1.6 to 2.9
    # times the time of one; results are the oracle's either way
    need_gpu()
    J = inputs.couplings_pm1(N, 101)
    init = inputs.initial_spins(chains, N, 102)
    inst = sk.Instance(J)
    run = sk.Run(inst, chains=chains, K=1, beta=0.05, seed=103, init=init, graph=sk.SK_GRAPH_TREE, arity=arity,
                 depth=depth, trace_chains=chains, trace_steps=6)
    b = sk.Batch([run])
    got = b.classes()[0][1] // 32
    assert got == 1 if nw == 1 else got >= nw, b.classes()
    b.advance(6)
    tr, s = run.trace(), run.state()[0]
    n = min(chains, 40)
    o = oracle.run_graph(J, graph=oracle.TREE, arity=arity, depth=depth, beta=0.05, seed=103, chains=n, init=init[:n],
                         steps=6, trace=True)
    assert np.array_equal(tr[:n], o["trace"]) and np.array_equal(s[:n], o["spins"])
    b.close(); run.close(); inst.close()


def test_wait_all_wakes_up():
    # a waiter that took the lock between the last job's retirement and its
    # leaving the active list waited for ever; several waiters, many bursts
    need_gpu()
    srv = sk.Server(budget_bytes=1 << 30, quantum_steps=8)
    srv.add_couplings(1, inputs.couplings_pm1(64, 1))
    for burst in range(250):
        t = [srv.submit(couplings_id=1, N=64, kind=sk.SK_J_PM1, chains=2, steps=8, K=4, seed=1, stream_id=k)
             for k in range(2)]
        # (the condition holds when the limit is reached, so that a lost wake-up shows as a late return)
        ws = [threading.Thread(target=srv.wait_all, args=(4_000_000_000,)) for _ in range(8)]
        t0 = time.perf_counter()
        for w in ws:
            w.start()
        for w in ws:
            w.join()
        assert time.perf_counter() - t0 < 3.0, burst
        for x in t:
            srv.result(x, 2, 64)
    srv.close()


@pytest.mark.parametrize("arity,depth,lanes", [(2, 10, 512), (2, 10, 64), (2, 11, 0), (2, 9, 256), (3, 6, 512)])
def test_graph_scan_of_large_trees(arity, depth, lanes):
    # trees of 1024 nodes and more whose words per lane are even scan them in turned
    # order (all lanes on one bank before: 1.5 times the step): same results as
    # on one warp per chain, and the oracle's decisions
    need_gpu()
    N, chains, steps = 96, 3, 12
    J = inputs.couplings_gauss(N, 111)
    init = inputs.initial_spins(chains, N, 112)
    outs = []
    for lay in (32, lanes):
        inst = sk.Instance(J)
        run = sk.Run(inst, chains=chains, K=1, beta=0.8, seed=113, init=init, graph=sk.SK_GRAPH_TREE, arity=arity,
                     depth=depth, trace_chains=chains, trace_steps=steps)
        b = sk.Batch([run])
        if lay:
            b.set_layout(lanes=lay)
        b.advance(steps)
        outs.append((run.trace(),) + run.state(fields=True))
        b.close(); run.close(); inst.close()
    assert all(np.array_equal(x, y) for x, y in zip(*outs))
    for c in range(chains):
        r = oracle.replay_graph(J, outs[1][0][c], graph=oracle.TREE, arity=arity, depth=depth, line_nodes=2, beta=0.8,
                                seed=113, chain=c, init=init[c], tol=1e-4)
        assert r["bad"] == 0, (c, r)
