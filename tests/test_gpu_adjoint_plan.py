"""Which adjoint a handle gets at the limits of the one over dense rows (128
neurons, 4 synapse types, 160 pair slots, no duplicated synapse, all networks of
the handle), each against the FP64 oracle's adjoint (the suite's 1e-3 per
coordinate)."""
import numpy as np
import pytest

import oracle
from paper_1906_03958_gb300 import netgen as ng
from tests.helpers import grad_error

pytestmark = pytest.mark.gpu

KINDS = (ng.ACH, ng.GABA_A, ng.GABA_B, ng.ACH, ng.GABA_A)


def _network(n, types, seed, p=0.15, every_pair=False, dup=False, table=None):
    rng = np.random.default_rng(seed)
    m = rng.random((n, n, types)) < p
    if every_pair:  # each neuron's every type has a synapse
        m[(np.arange(n) + 1) % n, np.arange(n), :] = True
    post, pre, st = np.nonzero(m)
    if dup:
        post, pre, st = np.r_[post, post[:1]], np.r_[pre, pre[:1]], np.r_[st, st[:1]]
    return ng.single_network(np.zeros(n), rng.uniform(0.0, 8.0, n), post, pre, rng.uniform(0.0, 0.5 / (n * p), post.size),
                             st, ng.neuron_table(ng.HH), ng.synapse_table(*KINDS[:table or types]))


CASES = {
    "160 slots": (lambda: [_network(80, 2, 1, every_pair=True)], 1),
    "168 slots": (lambda: [_network(81, 2, 2, every_pair=True)], 2),
    "128 neurons": (lambda: [_network(128, 1, 3, every_pair=True)], 1),
    "129 neurons": (lambda: [_network(129, 1, 4, every_pair=True)], 2),
    "4 types": (lambda: [_network(36, 4, 5, every_pair=True), _network(3, 4, 6, 0.5)], 1),
    "5 types": (lambda: [_network(20, 5, 7)], 2),
    "one duplicate": (lambda: [_network(30, 2, 8), _network(25, 2, 9, dup=True)], 2),
    "one large": (lambda: [_network(30, 1, 10), _network(140, 1, 11)], 2),
}


@pytest.mark.parametrize("case", list(CASES))
def test_adjoint_at_the_planners_limits(case):
    import torch
    from paper_1906_03958_gb300 import psst
    make, kernel = CASES[case]
    spec = ng.concat_specs(make())
    steps, stride = 60, 4
    g = np.random.default_rng(2).standard_normal((steps // stride, spec.n_neurons))
    gy64, gw64, gp64 = oracle.adjoint(spec, oracle.rest_state(spec), steps, g, stride, ckpt=20)
    with psst.Network(spec, rec_stride=stride, rec_capacity=steps // stride) as net:
        assert net.info()["adjoint"] == 0
        gw, gp, gy = (x.cpu().numpy() for x in net.adjoint(steps, torch.from_numpy(g.astype(np.float32)).cuda(), 25))
        net.status()
        assert net.info()["adjoint"] == kernel
    assert grad_error(gw, gw64) <= 1e-3
    assert grad_error(gp, gp64) <= 1e-3
    assert grad_error(gy.ravel(), gy64[:4 * spec.n_neurons]) <= 1e-3
