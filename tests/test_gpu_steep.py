"""Step-like transmitter release (Kp down to 1e-30 mV): T is 0 below Vp and 1
above it, in every layout, against the FP64 oracle's single step.

Tolerance: the suite's single-step bound, 1e-5.  With T exactly 0 or 1 the
gates' derivative has no error of its own; potentials keep 12 mV off Vp, which
no stage crosses (rest-like gates move V by less than 1 mV a step)."""
import numpy as np
import pytest

import oracle
from paper_1906_03958_gb300 import netgen as ng
from tests.helpers import step_error

pytestmark = pytest.mark.gpu

KPS = {"1e-30..1e-9": [1e-30, 1e-20, 1e-15, 1e-12, 1e-10, 1e-9],
       "1e-8..2e-6": [1e-8, 2e-8, 1e-7, 2e-7, 7e-7, 2e-6],
       "3e-6..1e-3": [3e-6, 5e-6, 1e-5, 3e-5, 1e-4, 1e-3]}


@pytest.mark.parametrize("layout", ["dense rows", "work items", "synapse gates", "grid"])
@pytest.mark.parametrize("kps", list(KPS))
def test_step_like_transmitter(kps, layout):
    from paper_1906_03958_gb300 import psst
    rng = np.random.default_rng(11)
    tab = ng.synapse_table(*[(ng.ACH, ng.GABA_A, ng.GABA_B)[k % 3] for k in range(6)])
    tab[:, 8] = KPS[kps]
    n, nt = 48, tab.shape[0]
    post, pre, st = np.nonzero(rng.random((n, n, nt)) < 0.2)
    spec = ng.single_network(np.zeros(n), rng.uniform(0.0, 10.0, n), post, pre, rng.uniform(0.0, 0.2, post.size), st,
                             ng.neuron_table(ng.HH), tab)
    S = spec.n_synapses
    y = np.zeros(4 * n + 2 * S, np.float32)
    y[:n] = np.where(np.arange(n) % 3 == 0, rng.uniform(14.0, 40.0, n), rng.uniform(-90.0, -50.0, n))
    for x, rest in enumerate((0.0529, 0.5961, 0.3177)):
        y[(x + 1) * n:(x + 2) * n] = rest
    pair = spec.pre.astype(np.int64) * nt + spec.syn_type
    y[4 * n:4 * n + S] = rng.uniform(0.0, 0.5, n * nt).astype(np.float32)[pair]
    second = spec.syn_params[spec.syn_type, 0] != 0
    y[4 * n + S:] = np.where(second, rng.uniform(0.0, 2.0, n * nt).astype(np.float32)[pair], 0.0)
    want, _ = oracle.integrate(spec, y.astype(np.float64), 1)
    kw = {"dense rows": {}, "work items": dict(item_chunks=2), "synapse gates": dict(gate_mode=1),
          "grid": dict(mode=psst.MODE_GRID)}[layout]
    with psst.Network(spec, init_state=y, **kw) as net:
        net.integrate(1)
        net.status()
        got = net.get_state_numpy()
    assert np.all(np.isfinite(got))
    assert step_error(got, want, n, S) <= 1e-5
