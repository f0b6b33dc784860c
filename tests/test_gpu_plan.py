"""Which kernel the planner gives a network with one gate per pair: dense rows
cost the same whatever the connectivity, work items pay per synapse, so sparse
batches keep work items.  Each choice against the FP64 oracle's single step."""
import numpy as np
import pytest

import oracle
from paper_1906_03958_gb300 import netgen as ng
from tests.helpers import step_error

pytestmark = pytest.mark.gpu


def _batch(n, p, nets, seed):
    parts = []
    for b in range(nets):
        rng = np.random.default_rng([seed, b])
        post, pre = np.nonzero(rng.random((n, n)) < p)
        if post.size == 0:
            post, pre = np.array([0]), np.array([n - 1])
        parts.append(ng.single_network(np.zeros(n), rng.uniform(0.0, 10.0, n), post, pre,
                                       rng.uniform(0.0, 2.0 / max(1.0, n * p), post.size), (pre >= 0.8 * n).astype(int),
                                       ng.neuron_table(ng.HH), ng.synapse_table(ng.ACH, ng.GABA_A)))
    return ng.concat_specs(parts)


# networks, neurons, connectivity, dense rows expected
CASES = {"many, 1%": (200, 300, 0.01, False), "many, 10%": (200, 200, 0.1, False), "many, 45%": (170, 150, 0.45, True),
         "many small": (400, 24, 0.1, True), "few, 1%": (100, 300, 0.01, False), "alone, 10%": (1, 300, 0.1, True),
         "alone, 1%": (1, 500, 0.01, True)}


@pytest.mark.parametrize("case", list(CASES))
def test_sparse_batches_keep_work_items(case):
    from paper_1906_03958_gb300 import psst
    nets, n, p, dense = CASES[case]
    spec = _batch(n, p, nets, 31)
    rng = np.random.default_rng(5)
    y = oracle.rest_state(spec).astype(np.float32)
    y[:spec.n_neurons] += rng.uniform(-7.0, 8.0, spec.n_neurons).astype(np.float32)
    y64, _ = oracle.integrate(spec, y.astype(np.float64), 1)
    out = []
    for mc in (1, 0):
        with psst.Network(spec, init_state=y, min_cluster=mc) as net:
            assert (net.info()["item_chunks"] == 0) == dense
            if mc == 0:
                net.autotune(5)
                assert (net.info()["item_chunks"] == 0) == dense
            net.integrate(1)
            net.status()
            out.append(net.get_state_numpy())
    assert step_error(out[0], y64, spec.n_neurons, spec.n_synapses) <= 1e-5
    np.testing.assert_array_equal(out[0], out[1])
