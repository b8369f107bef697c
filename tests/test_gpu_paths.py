"""Edges of single kernels and of the layouts a run gets by default: alignment
remainders, tile edges and the smallest and largest sizes of each path."""
import ctypes as C

import numpy as np
import pytest

import oracle
from paper_2102_05613_gb300 import inputs, sk

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1, 7, 15])
@pytest.mark.parametrize("chains,N", [(1, 5), (3, 17), (64, 100), (40, 4099)])
def test_start_spin_check_finds_the_first_bad_spin(offset, chains, N):
    # spins in device memory at any alignment: the bytes before the first
    # 16-byte boundary, the body and the remainder are all checked, and the
    # smallest offending index is named
    torch = need_gpu()
    n = chains * N
    inst = sk.Instance(inputs.couplings_pm1(N, 3))
    good = torch.from_numpy(inputs.initial_spins(chains, N, 4).reshape(-1))
    buf = torch.ones(n + 16, dtype=torch.int8, device="cuda")
    run = sk.Run(inst, chains=chains, K=4, seed=2)
    view = buf[offset:offset + n]
    head = min(n, (16 - view.data_ptr() % 16) % 16)
    for at in sorted({0, max(0, head - 1), min(head, n - 1), n // 2, min(n - 1, max(head, n - (n - head) % 16 - 1)), n - 1}):
        for bad in (0, 2, -2, -128, 127):
            view.copy_(good)
            view[at] = bad
            if at + 3 < n:
                view[at + 3] = 5  # a later one must not be reported instead
            with pytest.raises(sk.SKError) as e:
                run.reset(view)
            assert e.value.status == sk.SK_ERR_INVALID_ARG and f"spin {at} " in str(e.value), (at, bad, str(e.value))
    buf.fill_(3)  # what lies around the spins is not looked at
    view.copy_(good)
    run.reset(view)
    assert np.array_equal(run.state()[0].reshape(-1), good.numpy())
    run.close(); inst.close()


def _exact_energy(J, s, scale):
    # correctly rounded sum of the couplings' signed values
    import math
    i, j = np.triu_indices(J.shape[0], 1)
    return -scale * math.fsum((J[i, j].astype(np.float64) * s[i] * s[j]).tolist())


def _sym(upper):
    upper = np.triu(upper, 1)
    return np.ascontiguousarray((upper + upper.T).astype(np.float32))


@pytest.mark.parametrize("N,count", [(2, 1), (33, 127), (96, 128), (256, 129), (257, 40), (300, 700)])
def test_energies_are_exact_products(N, count):
    # tile edges of 128 configurations and 256 columns; +-J exact, Gaussian
    # rounded once (and once more by the scale)
    torch = need_gpu()
    S = inputs.initial_spins(count, N, 5)
    some = sorted({0, count // 2, count - 1})
    for J in (inputs.couplings_pm1(N, 6), inputs.couplings_gauss(N, 7)):
        inst = sk.Instance(J, scale=0.75)
        E = inst.energy(S)
        odd = torch.zeros(count * N + 3, dtype=torch.int8, device="cuda")[3:]  # device spins at an odd address
        odd.copy_(torch.from_numpy(S.reshape(-1)))
        assert np.array_equal(inst.energy(odd), E)
        for c in some:
            want = _exact_energy(J, S[c], 0.75)
            assert abs(E[c] - want) <= 4 * 2.0 ** -53 * abs(want), (N, c)
        bad = S.copy()
        bad[-1, -1] = 3
        with pytest.raises(sk.SKError) as e:
            inst.energy(bad)
        assert e.value.status == sk.SK_ERR_INVALID_ARG and f"spin {count * N - 1} " in str(e.value)
        inst.close()


@pytest.mark.parametrize("low,span_fits", [(-1, True), (-45, True), (-61, True), (-62, False), (-140, False)])
def test_energies_of_couplings_of_any_range(low, span_fits):
    # couplings of 1 and 2^low: up to 62 bits as digits, else the direct
    # double-precision sum (N^2/2 terms, each rounded)
    need_gpu()
    N, count = 70, 150
    rng = np.random.Generator(np.random.PCG64(8))
    J = _sym(np.where(rng.random((N, N)) < 0.5, 1.0, 2.0 ** low) * rng.choice([-1.0, 1.0], (N, N)))
    S = inputs.initial_spins(count, N, 9)
    inst = sk.Instance(J)
    E = inst.energy(S)
    inst.close()
    total = float(np.abs(np.triu(J.astype(np.float64), 1)).sum())
    for c in (0, count - 1):
        want = _exact_energy(J, S[c], 1.0)
        assert abs(E[c] - want) <= (4 * 2.0 ** -53 * abs(want) if span_fits else N * N * 2.0 ** -53 * total), c
    zero = sk.Instance(np.zeros((N, N), dtype=np.float32))
    assert np.array_equal(zero.energy(S), np.zeros(count))
    zero.close()


def test_energies_in_blocks_of_couplings_and_configurations():
    # N = 4128: the digit slices of Gaussian couplings come in several blocks
    # of rows, and 8200 configurations in two blocks
    torch = need_gpu()
    N, count = 4128, 8200
    g = torch.Generator(device="cuda").manual_seed(3)
    J = torch.triu(torch.randn((N, N), generator=g, device="cuda"), 1)
    J = (J + J.T).contiguous()
    S = (2 * torch.randint(0, 2, (count, N), generator=g, device="cuda", dtype=torch.int8) - 1).contiguous()
    inst = sk.Instance(J)
    E = inst.energy(S)
    inst.close()
    pick = [0, 127, 8063, 8064, 8199]
    want = -0.5 * ((S[pick].double() @ J.double()) * S[pick].double()).sum(1).cpu().numpy()
    # the reference's own rounding: ~N sums of N terms, each 2^-53 of |J| sqrt(N)
    assert np.abs(E[pick] - want).max() <= N * np.sqrt(N) * 64 * 2.0 ** -53


@pytest.mark.parametrize("n", [1, 2, 5, 6, 7, 10, 13, 21])
def test_set_generation_block_form(n):
    # below, at and above the six low elements of a block; every sum has at
    # most 28 positive terms of relative error 2^-53 and n levels build on it
    need_gpu()
    rng = np.random.Generator(np.random.PCG64(n))
    P = rng.random((n, n)) * 10.0 ** rng.integers(-3, 1, (n, n))
    got, want = sk.set_generation(P), sk.set_generation(P, method=sk.SK_SETGEN_DIRECT)
    assert np.all(np.abs(got - want) <= 64 * n * 2.0 ** -53 * want)
    P[:, 0] = 0.0
    P[0, :] = 0.0  # an element that is never generated
    got, want = sk.set_generation(P), sk.set_generation(P, method=sk.SK_SETGEN_DIRECT)
    assert np.all(np.abs(got - want) <= 64 * n * 2.0 ** -53 * want)
    huge = np.full((n, n), 1e200)  # overflows to infinity, never to NaN
    got, want = sk.set_generation(huge), sk.set_generation(huge, method=sk.SK_SETGEN_DIRECT)
    assert np.array_equal(np.isinf(got), np.isinf(want)) and not np.isnan(got).any()


@pytest.mark.parametrize("graph,arity,depth,L,N,chains", [
    (sk.SK_GRAPH_TREE, 2, 7, 0, 200, 5),     # 255 nodes: chunks of 8, ragged last lane
    (sk.SK_GRAPH_TREE, 3, 2, 0, 64, 3),      # 13 nodes: fewer than lanes
    (sk.SK_GRAPH_TREE, 16, 2, 0, 1000, 2),   # 273 nodes, odd chunks
    (sk.SK_GRAPH_LINE, 0, 0, 128, 130, 4),   # nodes of factor 0
    (sk.SK_GRAPH_LINE, 0, 0, 33, 40, 1),
])
def test_graph_results_do_not_depend_on_the_warps_per_chain(graph, arity, depth, L, N, chains):
    # Gaussian couplings: the weights are summed in one order whatever the team
    # (and the default picks a team by the number of chains)
    need_gpu()
    J = inputs.couplings_gauss(N, 31)
    init = inputs.initial_spins(chains, N, 32)
    outs = []
    for lanes in (0, 32, 64, 128, 256, 512):
        inst = sk.Instance(J)
        run = sk.Run(inst, chains=chains, K=1, beta=1.3, seed=33, record_every=40, max_records=3, init=init,
                     trace_chains=chains, trace_steps=120, graph=graph, arity=arity, depth=depth, line_nodes=L)
        b = sk.Batch([run])
        b.set_layout(lanes=lanes)
        b.advance(41)
        b.advance(79)
        E, q, acc = run.observables()
        outs.append((run.trace(), E, q, acc) + run.state(fields=True))
        b.close(); run.close(); inst.close()
    for o in outs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(outs[0], o))
    for c in range(chains):
        r = oracle.replay_graph(J, outs[0][0][c], graph=oracle.TREE if graph == sk.SK_GRAPH_TREE else oracle.LINE,
                                arity=arity, depth=depth, line_nodes=L, beta=1.3, seed=33, chain=c, init=init[c],
                                tol=1e-4)
        assert r["bad"] == 0, (c, r)


@pytest.mark.parametrize("K,rule,p_center,lanes", [(1, 0, 0.0, 64), (5, 0, 0.0, 128), (32, 0, 0.2, 64), (33, 0, 0.0, 64),
                                                   (64, 0, 0.0, 64), (65, 0, 0.0, 128), (100, 0, 0.05, 128),
                                                   (128, 0, 0.0, 128), (1, 1, 0.0, 64), (1, 1, 0.0, 128)])
@pytest.mark.parametrize("N,chains", [(96, 3), (515, 1)])
def test_team_results_are_those_of_one_warp_per_chain(K, rule, p_center, lanes, N, chains):
    # Gaussian couplings: a team sums the weights in the one-warp order, so the
    # layouts (and the default, which picks one by the number of chains) agree
    # bit for bit; advances of ragged lengths cross the draws' batches
    need_gpu()
    J = inputs.couplings_gauss(N, 41)
    init = inputs.initial_spins(chains, N, 42)
    outs = []
    for lay in (32, lanes, 0):
        inst = sk.Instance(J)
        run = sk.Run(inst, chains=chains, K=K, rule=rule, beta=1.2, seed=43, record_every=50, max_records=6, init=init,
                     trace_chains=chains, trace_steps=300, p_center=p_center)
        b = sk.Batch([run])
        b.set_layout(lanes=lay)
        if lay != 0:
            assert b.classes()[0][1] == lay
        for n in (1, 32, 67, 200):
            b.advance(n)
        E, q, acc = run.observables()
        outs.append((run.trace(), E, q, acc) + run.state(fields=True) + run.counters())
        b.close(); run.close(); inst.close()
    for o in outs[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(outs[0], o))


@pytest.mark.parametrize("K", [33, 36, 47, 63, 64])
@pytest.mark.parametrize("warps", [4, 24, 32])
def test_two_slots_per_lane(K, warps):
    # whole-warp chains with K of 33 to 64 hold two slots per lane: +-J against
    # the oracle (short and long weight tables, traced and not, a non-uniform
    # root); Gaussian bit for bit against 16 lanes with four slots each
    need_gpu()
    N, chains, steps = 77, 2 * warps + 1, 151
    init = inputs.initial_spins(chains, N, 52)

    def go(J, lanes, scale, trace, p_center):
        inst = sk.Instance(J, scale=scale)
        run = sk.Run(inst, chains=chains, K=K, beta=1.1, seed=53, record_every=50, max_records=3, init=init,
                     trace_chains=chains if trace else 0, trace_steps=steps if trace else 0, p_center=p_center)
        b = sk.Batch([run], warps_per_cta=warps)
        b.set_layout(lanes=lanes, staging=2)
        for n in (1, 50, 100):
            b.advance(n)
        E, q, acc = run.observables()
        out = (run.trace() if trace else None, E, q, acc) + run.state(fields=True)
        b.close(); run.close(); inst.close()
        return out

    J = inputs.couplings_pm1(N, 51)
    for scale, trace, pc in ((1.0, False, 0.0), (1.0, True, 0.3), (0.1, False, 0.0)):
        g = go(J, 32, scale, trace, pc)
        o = oracle.run(J, K=K, beta=1.1, seed=53, chains=chains, init=init, steps=steps, record_every=50, trace=True,
                       scale=scale, p_center=pc)
        assert np.array_equal(g[1], o["E"]) and np.array_equal(g[3], o["acc"]) and np.array_equal(g[4], o["spins"])
        if trace:
            assert np.array_equal(g[0], o["trace"])
    Jg = inputs.couplings_gauss(N, 54)
    for pc in (0.0, 0.1):
        a, b = go(Jg, 32, 1.0, True, pc), go(Jg, 16, 1.0, True, pc)
        for k in (0, 2, 3, 4, 5, 6):  # (record energies, entry 1, are summed in the order of the lanes)
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("N,chains", [(1024, 16301), (2000, 4100)])
def test_recompute_on_256_row_tiles(N, chains):
    # enough rows and terms for the 256-row tiles: last tiles with 173 rows and
    # with 4 (no row in the second half), ragged columns; start fields, drift
    # figures, both forms of the resync
    torch = need_gpu()
    J = torch.from_numpy(inputs.couplings(N, sk.SK_J_GAUSS, 61)).cuda()
    g = torch.Generator(device="cuda").manual_seed(62)
    S = (2 * torch.randint(0, 2, (chains, N), generator=g, device="cuda", dtype=torch.int8) - 1).contiguous()
    inst = sk.Instance(J)
    run = sk.Run(inst, chains=chains, K=4, beta=1.0, seed=3, init=S)

    def state():
        s = torch.empty_like(S)
        h = torch.empty((chains, N), dtype=torch.float32, device="cuda")
        assert sk.lib().mcmcmc_state(run.handle, C.c_void_p(s.data_ptr()), C.c_void_p(h.data_ptr()), None,
                                     sk.SK_MEM_DEVICE) == sk.SK_OK
        return s, h
    # the tensor core's FP32 accumulator rounds once per MMA step of 16 products
    tol = max(3e-5, 3 * N / 16 * 2.0 ** -23 * 4)
    s, h = state()
    assert torch.equal(s, S) and (h.double() - S.double() @ J.double()).abs().max().item() <= tol
    run.advance(20)
    exact = state()[0].double() @ J.double()
    st, _ = run.recompute(sk.SK_RECOMPUTE_CHECK)
    assert st["max_field_drift"] <= 2 * tol + 1e-4
    run.recompute(sk.SK_RECOMPUTE_RESYNC, sync=False)  # enqueued only: sets the fields
    h1 = state()[1].clone()
    st, _ = run.recompute(sk.SK_RECOMPUTE_RESYNC)      # with figures: they are the same fields
    h2 = state()[1]
    assert torch.equal(h1, h2) and st["max_field_drift"] == 0.0 and (h2.double() - exact).abs().max().item() <= tol
    run.close(); inst.close()


@pytest.mark.parametrize("rule,K,N", [(0, 33, 77), (0, 64, 640), (0, 65, 33), (0, 100, 512), (0, 128, 130), (1, 1, 250)])
def test_default_layout_of_many_chains(rule, K, N):
    # Gaussian chains beyond 32 per SM default to 16 lanes with the whole-warp
    # form's sums: every result (trace, records with their energies, state)
    # bit for bit that of forced whole warps; ragged N, K and last item
    torch = need_gpu()
    chains = 33 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    J = inputs.couplings(N, sk.SK_J_GAUSS, 71)
    init = inputs.initial_spins(chains, N, 72)
    outs = []
    for lanes in (0, 32):
        inst = sk.Instance(J)
        run = sk.Run(inst, chains=chains, K=K, rule=rule, beta=1.2, seed=73, record_every=16, max_records=3, init=init,
                     trace_chains=chains, trace_steps=48, p_center=0.2 if K == 100 else 0.0)
        b = sk.Batch([run])
        b.set_layout(lanes=lanes)
        assert b.classes()[0][1] == (lanes or 16)
        for n in (1, 16, 31):
            b.advance(n)
        outs.append((run.trace(),) + run.observables() + run.state(fields=True) + run.counters())
        b.close(); run.close(); inst.close()
    assert all(np.array_equal(x, y) for x, y in zip(*outs))


def test_reset_many_by_stream_and_kind():
    # runs of both coupling kinds, uneven sizes and two streams restarted in one
    # call (grouped by stream and kind, one run alone) against single restarts
    torch = need_gpu()
    sts = [torch.cuda.Stream(), torch.cuda.Stream()]
    specs = [(33, 0, 6, 0), (700, 1, 300, 0), (200, 0, 258, 0), (64, 1, 1, 0), (1024, 1, 130, 0), (96, 0, 10, 1)]
    insts = [sk.Instance(inputs.couplings(N, k, 600 + i), stream=sts[s]) for i, (N, k, _, s) in enumerate(specs)]
    inits = [inputs.initial_spins(c, N, 700 + i) for i, (N, _, c, _) in enumerate(specs)]
    inits[2] = None
    runs = [sk.Run(x, chains=c, K=8, seed=2, stream_id=i, record_every=10, max_records=2)
            for i, (x, (_, _, c, _)) in enumerate(zip(insts, specs))]
    for r in runs:
        r.advance(20)
    sk.reset_many(runs, inits)
    got = [r.state(fields=True) + r.observables() + r.counters() for r in runs]
    for i, r in enumerate(runs):
        r.advance(10)
        r.reset(inits[i])
        one = r.state(fields=True) + r.observables() + r.counters()
        assert one[2] == 0 and all(np.array_equal(x, y) for x, y in zip(got[i], one)), i
        r.close()
    for x in insts:
        x.close()


def test_reset_many_of_long_gaussian_runs():
    # restarts of one stream together, sized for the 256-row tiles of the field
    # launch (two rounds of 128-row tiles on 152 SMs, one of 256-row ones): uneven N,
    # last tiles with 100 rows (none in the second half), with 130 and with 2
    torch = need_gpu()
    specs = [(1024, 2660), (1500, 1410), (1100, 130), (1030, 258)]
    runs, insts, inits = [], [], []
    for i, (N, chains) in enumerate(specs):
        insts.append(sk.Instance(inputs.couplings(N, sk.SK_J_GAUSS, 800 + i)))
        runs.append(sk.Run(insts[-1], chains=chains, K=8, seed=3, stream_id=i))
        inits.append(inputs.initial_spins(chains, N, 810 + i))
    for r in runs:
        r.advance(3)
    sk.reset_many(runs, inits)
    for i, ((N, chains), r) in enumerate(zip(specs, runs)):
        s, h, step = r.state(fields=True)
        exact = torch.from_numpy(inits[i]).cuda().double() @ torch.from_numpy(inputs.couplings(N, sk.SK_J_GAUSS, 800 + i)).cuda().double()
        err = (torch.from_numpy(h).cuda().double() - exact).abs().max().item()
        # the tensor core's FP32 accumulator rounds once per MMA step of 16 products
        assert step == 0 and np.array_equal(s, inits[i]) and err <= max(3e-5, 3 * N / 16 * 2.0 ** -23 * 4), (N, err)
    for x in runs + insts:
        x.close()


@pytest.mark.parametrize("scale", [1.0, 0.1])
@pytest.mark.parametrize("rule,K,N,chains,lanes", [
    (0, 5, 33, 9001, 8), (0, 32, 250, 9001, 8), (0, 33, 130, 9001, 16), (0, 64, 256, 9001, 16), (0, 65, 77, 5017, 16),
    (0, 128, 130, 20001, 16), (1, 1, 250, 9001, 16), (0, 48, 128, 20001, 32), (0, 20, 300, 5017, 32)])
def test_default_layout_of_many_pm1_chains(rule, K, N, chains, lanes, scale):
    # the lanes +-J chains get by default beyond 32 per SM (short and long weight
    # tables), against the oracle; ragged N, K and last item
    need_gpu()
    steps = 24
    J = inputs.couplings_pm1(N, 75)
    init = inputs.initial_spins(chains, N, 76)
    inst = sk.Instance(J, scale=scale)
    run = sk.Run(inst, chains=chains, K=K, rule=rule, beta=1.2, seed=77, record_every=8, max_records=3, init=init)
    b = sk.Batch([run])
    assert b.classes()[0][1] == lanes, b.classes()
    for n in (1, 16, 7):
        b.advance(n)
    E, q, acc = run.observables()
    o = oracle.run(J, K=K, rule=rule, beta=1.2, seed=77, chains=chains, init=init, steps=steps, record_every=8,
                   scale=scale)
    assert np.array_equal(E, o["E"]) and np.array_equal(q, o["q"]) and np.array_equal(acc, o["acc"])
    assert np.array_equal(run.state()[0], o["spins"])
    b.close(); run.close(); inst.close()
