"""The work a user of the sampler has it do, as cases that can be timed and compared.

Each case is one call pattern through the public entry points (the classes and
functions of paper_2102_05613_gb300.sk and the C ABI behind them), at sizes of
the repository's own workloads: the single +-J chain of N = 64, the Gaussian
N = 512 and N = 2048 batches, the uneven batch, the request server, the deeper
graphs of the thermalisation study, the field recompute, energies and the
set-generation probabilities.  `listed()` gives the cases, `draw()` more of
the same ranges.  `prepare` makes what a program holds before the call (inputs
on the GPU from the seed alone, the instances, runs and batch); `run` makes
one pass and returns its outputs.  A sampling pass restarts the chains from
the given spins, advances them and reads records and state, so it can be
repeated on the same state.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2102_05613_gb300 import inputs, sk

PM1, GAUSS = sk.SK_J_PM1, sk.SK_J_GAUSS


def listed():
    return [
        # The smallest use: one +-J chain of 64 spins, 8 proposals per step, as
        # in the repository's first workload.  Latency of a lone chain, and of
        # the restart and the read-back around a short run.
        dict(name="lone_chain_pm1", family="star", kind=PM1, N=64, chains=1, K=8, rule=0, beta=1.0, p_center=0.0,
             steps=2000, records=20, recompute=0),
        # The thermalisation study's chain: Gaussian N = 1024 at T_c, K = 128, one
        # chain on the whole GPU (the time to a given number of steps).
        dict(name="lone_chain_gauss", family="star", kind=GAUSS, N=1024, chains=1, K=128, rule=0, beta=1.0,
             p_center=0.0, steps=1000, records=10, recompute=0),
        # The Metropolis comparator with one chain per core, as the paper runs
        # it: 152 chains, a third of the steps accepted at beta = 1.
        dict(name="few_chains_metropolis", family="star", kind=GAUSS, N=512, chains=152, K=1, rule=1, beta=1.0,
             p_center=0.0, steps=4000, records=40, recompute=0),
        # The headline workload at the layout a long measurement pins (16 lanes
        # per chain, 24 warps per CTA): Gaussian N = 512, K = 128, many chains.
        dict(name="pinned_batch_gauss", family="batch", kind=GAUSS, N=512, instances=8, chains=8192, K=128, beta=1.0,
             steps=100, lanes=16, warps=24),
        # The same model run once per disorder realisation, without tuning: new
        # couplings and starts from pinned host memory, 100 steps, records back.
        dict(name="fresh_disorder_gauss", family="fresh", kind=GAUSS, N=512, instances=16, chains=4096, K=128,
             beta=1.0, steps=100),
        # The precision workload's sampling: +-J at beta = 2 with the tensor-core
        # field check every 256 steps, 8192 chains; a ragged N.
        dict(name="checked_run_pm1", family="star", kind=PM1, N=2000, chains=8192, K=64, rule=0, beta=2.0,
             p_center=0.0, steps=256, records=2, recompute=256),
        # Instances of uneven N, K and chains, half +-J and half Gaussian, in one
        # persistent launch.
        dict(name="uneven_batch", family="uneven", instances=32, mix=1, steps=100),
        # The thermalisation study's binary tree of depth 7 with a few chains.
        dict(name="tree_gauss", family="graph", kind=GAUSS, N=1024, chains=32, graph=1, arity=2, depth=7, nodes=0,
             beta=1.0, steps=50),
        # Energies of a set of configurations of one instance, e.g. of stored
        # samples or of replicas exchanged from elsewhere.
        dict(name="energies_gauss", family="energy", kind=GAUSS, N=2048, count=2048),
        # The resynchronisation of maintained Gaussian fields on the tensor cores
        # at the precision workload's size, and the fields read back.
        dict(name="resync_gauss", family="recompute", kind=GAUSS, N=2048, chains=8192),
        # Generation probabilities of every subset of a 22-element set.
        dict(name="set_generation", family="setgen", n=22),
        # The request server: a burst of jobs of mixed size, both coupling kinds
        # and K of the serving workload, until every result is back.
        dict(name="server_burst", family="server", jobs=10, mix=3, n_max=1024, chains_max=1024, steps_max=2000),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    family = rng.choice(["star", "star", "star", "batch", "fresh", "uneven", "graph", "energy", "recompute",
                         "setgen", "server"])
    kind = rng.choice([PM1, GAUSS])
    beta = round(rng.uniform(0.4, 3.0), 3)
    if family == "star":
        N = _log(rng, 48, 4096)
        rule = 1 if rng.random() < 0.25 else 0
        K = 1 if rule else _log(rng, 1, 256)
        chains = _log(rng, 1, max(1, min(16384, (1 << 26) // N)))
        us = max(2.0, chains * (N + 4 * K) * 1e-6)  # a step, roughly
        steps = max(20, min(2000, int(5000 / us)))
        pc = round(rng.uniform(0.05, 0.6), 2) if rule == 0 and rng.random() < 0.15 else 0.0
        return dict(family="star", kind=kind, N=N, chains=chains, K=K, rule=rule, beta=beta, p_center=pc,
                    steps=steps, records=rng.choice([1, 2, 5]), recompute=rng.choice([0, 0, max(10, steps // 2)]))
    if family == "batch":
        N = rng.randint(256, 768)
        chains = _log(rng, 1024, 8192)
        return dict(family="batch", kind=kind, N=N, instances=rng.randint(1, 6), chains=chains,
                    K=rng.randint(33, 128), beta=beta, steps=rng.randint(30, 80), lanes=16, warps=24)
    if family == "fresh":
        return dict(family="fresh", kind=kind, N=_log(rng, 128, 768), instances=rng.randint(2, 12),
                    chains=_log(rng, 64, 4096), K=_log(rng, 2, 128), beta=beta, steps=rng.randint(20, 100))
    if family == "uneven":
        return dict(family="uneven", instances=rng.randint(6, 28), mix=rng.randint(2, 1 << 20),
                    steps=rng.randint(20, 60))
    if family == "graph":
        chains = _log(rng, 1, 512)
        if rng.random() < 0.4:
            arity, depth, nodes = 0, 0, rng.randint(8, 128)
            V = nodes
        else:
            arity = rng.choice([2, 2, 3, 4, 8])
            depth = rng.randint(2, {2: 8, 3: 5, 4: 4, 8: 3}[arity])
            nodes = 0
            V = sum(arity ** d for d in range(depth + 1))
        us = (8 + 0.15 * V) * max(1.0, chains * V / 1e5)
        return dict(family="graph", kind=kind, N=_log(rng, 64, 1024), chains=chains, graph=1 if arity else 2,
                    arity=arity, depth=depth, nodes=nodes, beta=beta, steps=max(10, min(200, int(2500 / us))))
    if family == "energy":
        N = _log(rng, 32, 4096)
        most = max(1, int(8e9) // (N * N))
        return dict(family="energy", kind=kind, N=N, count=_log(rng, 1, min(8192, most)))
    if family == "recompute":
        return dict(family="recompute", kind=kind, N=_log(rng, 200, 2048), chains=_log(rng, 200, 8192))
    if family == "setgen":
        return dict(family="setgen", n=rng.randint(5, 21))
    return dict(family="server", jobs=rng.randint(3, 10), mix=rng.randint(4, 1 << 20), n_max=_log(rng, 128, 1024),
                chains_max=_log(rng, 64, 1024), steps_max=_log(rng, 400, 2000))


# ---------------------------------------------------------------------------
# inputs from the seed
# ---------------------------------------------------------------------------
def _gen(seed, tag=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 7919 * int(tag) + 1)


def _couplings(N, kind, g):
    """Symmetric, zero diagonal: +-1 equiprobable (int8) or N(0, 1/N) (float32), on the GPU."""
    if kind == PM1:
        J = (2 * torch.randint(0, 2, (N, N), generator=g, device="cuda") - 1).to(torch.int8)
    else:
        J = torch.randn((N, N), generator=g, device="cuda") / math.sqrt(N)
    J = torch.triu(J, 1)
    return (J + J.T).contiguous()


def _spins(count, N, g):
    return (2 * torch.randint(0, 2, (count, N), generator=g, device="cuda", dtype=torch.int8) - 1).contiguous()


def _records(R, chains, device="cuda", pin=False):
    mk = lambda shape, dt: torch.zeros(shape, dtype=dt, device=device, pin_memory=pin)  # noqa: E731
    return (mk((R, chains), torch.float64), mk((R, chains // 2), torch.float64), mk((R, chains), torch.int32))


def _state(run, spins, fields=None):
    """mcmcmc_state into device buffers."""
    status = sk.lib().mcmcmc_state(run.handle, ctypes.c_void_p(spins.data_ptr()),
                                   None if fields is None else ctypes.c_void_p(fields.data_ptr()), None,
                                   sk.SK_MEM_DEVICE)
    if status != sk.SK_OK:
        raise sk.SKError(status, sk.lib().sk_last_error().decode())
    return spins


def _fields(chains, N, kind):
    return torch.zeros((chains, N), dtype=torch.int32 if kind == PM1 else torch.float32, device="cuda")


# ---------------------------------------------------------------------------
# the families
# ---------------------------------------------------------------------------
def _prepare_star(c, seed):
    g = _gen(seed)
    inst = sk.Instance(_couplings(c["N"], c["kind"], g))
    start = _spins(c["chains"], c["N"], g)
    every = c["steps"] // c["records"]
    run = sk.Run(inst, chains=c["chains"], K=c["K"], rule=c["rule"], beta=c["beta"], seed=seed + 1,
                 record_every=every, max_records=c["records"], init=start, recompute_every=c["recompute"],
                 p_center=c["p_center"])
    return dict(c=c, run=run, start=start, rec=_records(c["records"], c["chains"]),
                spins=torch.empty_like(start), fields=_fields(c["chains"], c["N"], c["kind"]))


def _run_star(s):
    run, c = s["run"], s["c"]
    run.reset(s["start"])
    run.advance(c["steps"])
    E, q, acc = run.observables(0, c["records"], out=s["rec"])
    return dict(energy=E, overlap=q, accepted=acc, spins=_state(run, s["spins"], s["fields"]), fields=s["fields"])


def _prepare_graph(c, seed):
    g = _gen(seed)
    inst = sk.Instance(_couplings(c["N"], c["kind"], g))
    start = _spins(c["chains"], c["N"], g)
    run = sk.Run(inst, chains=c["chains"], K=1, beta=c["beta"] / (1.0 if c["kind"] == GAUSS else math.sqrt(c["N"])),
                 seed=seed + 1, record_every=c["steps"], max_records=1, init=start, graph=c["graph"],
                 arity=c["arity"], depth=c["depth"], line_nodes=c["nodes"])
    return dict(c=dict(c, records=1), run=run, start=start, rec=_records(1, c["chains"]),
                spins=torch.empty_like(start), fields=_fields(c["chains"], c["N"], c["kind"]))


def _prepare_many(c, seed, host):
    """Instances, runs and starts of one shape; host: the inputs in pinned host memory."""
    insts, runs, Js, starts, recs = [], [], [], [], []
    for i in range(c["instances"]):
        g = _gen(seed, i + 1)
        J, s0 = _couplings(c["N"], c["kind"], g), _spins(c["chains"], c["N"], g)
        insts.append(sk.Instance(J))
        runs.append(sk.Run(insts[i], chains=c["chains"], K=c["K"], beta=c["beta"], seed=seed + 1, stream_id=i,
                           record_every=c["steps"], max_records=1, init=s0))
        Js.append(J.cpu().pin_memory() if host else J)
        starts.append(s0.cpu().pin_memory() if host else s0)
        recs.append(_records(1, c["chains"], "cpu" if host else "cuda", host))
    return dict(c=c, insts=insts, runs=runs, J=Js, start=starts, rec=recs,
                spins=torch.empty((c["instances"], c["chains"], c["N"]), dtype=torch.int8, device="cuda"))


def _prepare_batch(c, seed):
    s = _prepare_many(c, seed, False)
    s["batch"] = sk.Batch(s["runs"], warps_per_cta=c["warps"])
    s["batch"].set_layout(c["lanes"], 2)
    return s


def _run_batch(s):
    sk.reset_many(s["runs"], s["start"])
    s["batch"].advance(s["c"]["steps"])
    sk.observables_many(s["runs"], 0, 1, s["rec"])
    for r, x in zip(s["runs"], s["spins"]):
        _state(r, x)
    return dict(records=s["rec"], spins=s["spins"])


def _prepare_fresh(c, seed):
    s = _prepare_many(c, seed, True)
    s["batch"] = sk.Batch(s["runs"])
    return s


def _run_fresh(s):
    sk.set_couplings_many(s["insts"], s["J"])
    sk.reset_many(s["runs"], s["start"])
    s["batch"].advance(s["c"]["steps"])
    sk.observables_many(s["runs"], 0, 1, s["rec"])
    return dict(records=s["rec"])


def _uneven(c):
    return inputs.uneven_batch(c["instances"], seed=c["mix"])


def _prepare_uneven(c, seed):
    st = torch.cuda.Stream()
    specs = _uneven(c)
    total = sum(sp["chains"] for sp in specs)
    # records and states of all runs in one buffer each, a slice per run
    flat = _records(1, total)
    spins = torch.empty(sum(sp["chains"] * sp["N"] for sp in specs), dtype=torch.int8, device="cuda")
    runs, starts, recs, states = [], [], [], []
    at = at_s = 0
    for i, sp in enumerate(specs):
        g = _gen(seed, i + 1)
        J, s0 = _couplings(sp["N"], sp["kind"], g), _spins(sp["chains"], sp["N"], g)
        torch.cuda.synchronize()
        runs.append(sk.Run(sk.Instance(J, stream=st), chains=sp["chains"], K=sp["K"], beta=sp["beta"], seed=seed + 1,
                           stream_id=i, record_every=c["steps"], max_records=1, init=s0))
        starts.append(s0)
        n, m = sp["chains"], sp["chains"] * sp["N"]
        recs.append((flat[0][0, at:at + n], flat[1][0, at // 2:(at + n) // 2], flat[2][0, at:at + n]))
        states.append(spins[at_s:at_s + m])
        at, at_s = at + n, at_s + m
    batch = sk.Batch(runs)
    batch.set_fused(16)
    return dict(c=c, runs=runs, start=starts, rec=recs, states=states, flat=flat, spins=spins, batch=batch, stream=st)


def _run_uneven(s):
    sk.reset_many(s["runs"], s["start"])
    s["batch"].advance(s["c"]["steps"])
    sk.observables_many(s["runs"], 0, 1, s["rec"])
    for r, x in zip(s["runs"], s["states"]):
        _state(r, x)
    return dict(records=s["flat"], spins=s["spins"])


def _prepare_energy(c, seed):
    g = _gen(seed)
    J = _couplings(c["N"], c["kind"], g)
    return dict(inst=sk.Instance(J), spins=_spins(c["count"], c["N"], g))


def _run_energy(s):
    return s["inst"].energy(s["spins"])


def _exact_energy(c, seed):
    g = _gen(seed)
    J = _couplings(c["N"], c["kind"], g).double()
    S = _spins(c["count"], c["N"], g).double()
    return -0.5 * ((S @ J) * S).sum(1)


def _prepare_recompute(c, seed):
    g = _gen(seed)
    inst = sk.Instance(_couplings(c["N"], c["kind"], g))
    start = _spins(c["chains"], c["N"], g)
    run = sk.Run(inst, chains=c["chains"], K=64, beta=2.0, seed=seed + 1, init=start)
    return dict(c=c, run=run, spins=torch.empty_like(start), fields=_fields(c["chains"], c["N"], c["kind"]))


def _run_recompute(s):
    s["run"].recompute(sk.SK_RECOMPUTE_RESYNC, 3, sync=False)
    return dict(spins=_state(s["run"], s["spins"], s["fields"]), fields=s["fields"])


def _exact_recompute(c, seed):
    g = _gen(seed)
    J = _couplings(c["N"], c["kind"], g).double()
    H = _spins(c["chains"], c["N"], g).double() @ J
    return dict(spins=None, fields=None if c["kind"] == PM1 else H)


def _prepare_setgen(c, seed):
    n = c["n"]
    P = np.random.Generator(np.random.PCG64(seed)).random((n, n)) / n
    return dict(P=P, out=torch.zeros(1 << n, dtype=torch.float64, device="cuda"))


def _run_setgen(s):
    return sk.set_generation(s["P"], out=s["out"])


def _exact_setgen(c, seed):
    n = c["n"]
    P = torch.from_numpy(np.random.Generator(np.random.PCG64(seed)).random((n, n)) / n)
    mask = torch.arange(1 << n, device="cuda")
    size = torch.zeros_like(mask)
    for b in range(n):
        size += (mask >> b) & 1
    out = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
    out[0] = 1.0
    for m in range(1, n):  # the masks of one cardinality, by the recursion on the first addition
        M = mask[size == m]
        tot = torch.zeros(M.numel(), dtype=torch.float64, device="cuda")
        for e in range(n):
            X = M[((M >> e) & 1) == 1]
            if not X.numel():
                continue
            a = torch.zeros(X.numel(), dtype=torch.float64, device="cuda")
            for p in range(n):
                if p != e:
                    a += float(P[e, p]) * (1 - ((X >> p) & 1)).double()
            tot[((M >> e) & 1) == 1] += a * out[X & ~(1 << e)]
        out[M] = tot / (n - m)
    return out


def _server_jobs(c):
    r = np.random.Generator(np.random.PCG64(c["mix"]))

    def lg(lo, hi):
        return int(round(math.exp(r.uniform(math.log(lo), math.log(hi)))))
    jobs = []
    for i in range(c["jobs"]):
        K = int(r.choice([1, 16, 64, 256]))
        jobs.append(dict(N=lg(64, c["n_max"]), kind=i % 2, chains=lg(1, c["chains_max"]), K=K,
                         rule=sk.SK_RULE_METROPOLIS if K == 1 else sk.SK_RULE_MCMCMC,
                         steps=lg(c["steps_max"] // 4, c["steps_max"]), beta=float(r.uniform(0.3, 3.0))))
    return jobs


def _prepare_server(c, seed):
    jobs = _server_jobs(c)
    srv = sk.Server(budget_bytes=16 << 30, quantum_steps=256)
    for i, j in enumerate(jobs):
        srv.add_couplings(i + 1, _couplings(j["N"], j["kind"], _gen(seed, i + 1)).cpu().numpy())
    return dict(srv=srv, jobs=jobs, seed=seed)


def _run_server(s):
    srv = s["srv"]
    tickets = [srv.submit(couplings_id=i + 1, seed=s["seed"] + 1, stream_id=i, **j) for i, j in enumerate(s["jobs"])]
    srv.wait_all()
    out = []
    for t, j in zip(tickets, s["jobs"]):
        E, S, flips = srv.result(t, j["chains"], j["N"])
        out.append(dict(energy=E, spins=S, flips=flips))
    return out


_FAMILIES = {
    "star": (_prepare_star, _run_star),
    "batch": (_prepare_batch, _run_batch),
    "fresh": (_prepare_fresh, _run_fresh),
    "uneven": (_prepare_uneven, _run_uneven),
    "graph": (_prepare_graph, _run_star),
    "energy": (_prepare_energy, _run_energy),
    "recompute": (_prepare_recompute, _run_recompute),
    "setgen": (_prepare_setgen, _run_setgen),
    "server": (_prepare_server, _run_server),
}


def prepare(case, seed):
    s = _FAMILIES[case["family"]][0](case, int(seed))
    s["family"] = case["family"]
    return s


def run(state):
    return _FAMILIES[state["family"]][1](state)


def exact(case, seed):
    """Energies, fields and set probabilities in 64 bits; a sampled trajectory has no
    such value (it is defined by the sampler's own arithmetic)."""
    if case["family"] == "energy":
        return _exact_energy(case, int(seed))
    if case["family"] == "recompute":
        return _exact_recompute(case, int(seed))
    if case["family"] == "setgen":
        return _exact_setgen(case, int(seed))
    return None


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _sampling(N, kind, chains, K, steps):
    """Couplings and starts read once, spins and records written once; per
    chain-step the K candidates' energies and weights (~10 operations each)
    and one multiply-add per field for one moved spin."""
    bj = 1 if kind == PM1 else 4
    return N * N * bj + chains * (2 * N + 20), float(chains) * steps * (10.0 * K + 2.0 * N)


def work(case):
    f = case["family"]
    if f in ("star", "graph"):
        K = case["K"] if f == "star" else (
            case["nodes"] or sum(case["arity"] ** d for d in range(case["depth"] + 1))) - 1
        b, o = _sampling(case["N"], case["kind"], case["chains"], K, case["steps"])
        b += 4 * case["chains"] * case["N"]  # the fields read back
        if case.get("recompute"):
            n = case["steps"] // case["recompute"]
            o += n * 2.0 * case["chains"] * case["N"] ** 2 * (1 if case["kind"] == PM1 else 3)
        return {"bytes": b, "flops": o}
    if f in ("batch", "fresh"):
        b, o = _sampling(case["N"], case["kind"], case["chains"], case["K"], case["steps"])
        return {"bytes": b * case["instances"], "flops": o * case["instances"]}
    if f == "uneven":
        w = [_sampling(x["N"], x["kind"], x["chains"], x["K"], case["steps"]) for x in _uneven(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if f == "server":
        w = [_sampling(x["N"], x["kind"], x["chains"], x["K"], x["steps"]) for x in _server_jobs(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if f == "energy":
        N, n = case["N"], case["count"]
        return {"bytes": N * N * (1 if case["kind"] == PM1 else 4) + n * (N + 8), "flops": float(n) * N * (N + 1)}
    if f == "recompute":
        N, n = case["N"], case["chains"]
        return {"bytes": N * N * (1 if case["kind"] == PM1 else 4) + n * N * 6,
                "flops": 2.0 * n * N * N * (1 if case["kind"] == PM1 else 3)}
    n = case["n"]  # set generation: the 2^n probabilities, a multiply-add per member of each subset
    return {"bytes": 8.0 * 2 ** n, "flops": float(n) * 2 ** n}
