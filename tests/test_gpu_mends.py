"""Results that single paths once got wrong: each test fails on the form it names."""
import numpy as np
import pytest

import oracle
from paper_2102_05613_gb300 import inputs, sk

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


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
