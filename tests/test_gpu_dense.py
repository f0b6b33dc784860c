"""Networks whose synapses are held as dense rows (csrc/psst_dense.cu): sizes at
the edges of its tiles (4 rows, 32 rows, 32 columns per type), every cluster
size, against the FP64 oracle's single step and against the work-item kernel.

Tolerances: one step from the same FP32 state within the suite's 1e-5 (a row's
sum of up to 300 terms w G (V - E) carries at most ~300 * 2^-24 = 2e-5 of its
own magnitude, times dt / C = 0.01 on V); cluster sizes bit for bit.
"""
import numpy as np
import pytest

import oracle
from paper_1906_03958_gb300 import netgen as ng
from tests.helpers import step_error

pytestmark = pytest.mark.gpu

STEP_TOL = 1e-5


def _network(n, seed, p=0.4, types=3):
    """n neurons, each ordered pair (self pairs too) with a synapse of each of
    the first `types` types independently with probability p."""
    rng = np.random.default_rng(seed)
    post, pre, st = np.nonzero(rng.random((n, n, types)) < p)
    if post.size == 0:
        post, pre, st = np.array([0]), np.array([n - 1]), np.array([0])
    w = rng.uniform(0.0, 3.0 / (n * p), post.size)
    return ng.single_network(rng.integers(0, 2, n), rng.uniform(0.0, 10.0, n), post, pre, w, st,
                             ng.neuron_table(ng.PN, ng.LN), ng.synapse_table(ng.ACH, ng.GABA_A, ng.GABA_B),
                             pulse_amp=rng.uniform(0.0, 10.0, n), pulse_on=3, pulse_off=90)


def _state(spec, seed):
    """A state away from rest with equal gates within each pair."""
    rng = np.random.default_rng(seed)
    N, S, nt = spec.n_neurons, spec.n_synapses, spec.syn_params.shape[0]
    y = np.zeros(4 * N + 2 * S, np.float32)
    y[:N] = rng.uniform(-80.0, 30.0, N)
    y[N:4 * N] = rng.uniform(0.0, 1.0, 3 * N)
    net = np.repeat(np.arange(spec.n_nets), spec.net_synapses())
    pair = (spec.net_neuron_off[net].astype(np.int64) + spec.pre) * nt + spec.syn_type
    y[4 * N:4 * N + S] = rng.uniform(0.0, 1.0, N * nt).astype(np.float32)[pair]
    s = rng.uniform(0.0, 5.0, N * nt).astype(np.float32)[pair]
    y[4 * N + S:] = np.where(spec.syn_params[spec.syn_type, 0] != 0, s, 0.0)
    return y


SIZES = {
    "tiny": [(n, 0.6, 3) for n in (1, 2, 3, 4, 5, 7, 8, 9, 12)],
    "tile": [(n, 0.4, 3) for n in (15, 16, 17, 31, 32, 33, 63, 64, 65)],
    "columns": [(n, 0.9, 1) for n in (32, 33, 96, 97, 128, 129, 161)],
    "large": [(200, 0.1, 1), (239, 0.2, 2), (257, 0.3, 1), (288, 0.1, 2), (300, 0.5, 1)],
}


@pytest.mark.parametrize("sizes", list(SIZES))
def test_dense_rows_single_step_and_cluster_sizes(sizes):
    from paper_1906_03958_gb300 import psst
    spec = ng.concat_specs([_network(n, 500 + k, p, t) for k, (n, p, t) in enumerate(SIZES[sizes])])
    N, S = spec.n_neurons, spec.n_synapses
    y = _state(spec, 7)
    y64, _ = oracle.integrate(spec, y.astype(np.float64), 1, step0=2)
    first = None
    for mc in (1, 2, 4, 0):
        with psst.Network(spec, init_state=y, rec_stride=1, rec_capacity=60, min_cluster=mc) as net:
            assert net.info()["item_chunks"] == 0  # dense rows
            net.set_step(2)
            net.integrate(1)
            net.status()
            one = net.get_state_numpy()
            assert step_error(one, y64, N, S) <= STEP_TOL
            net.integrate(50)
            net.status()
            out = one, net.get_state_numpy(), net.read_record()
        if first is None:
            first = out
        for a, b in zip(out, first):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("method", ["rk4", "euler", "heun3"])
def test_dense_rows_agree_with_work_items(method):
    # the same map with the synaptic sums grouped differently, over 100 steps
    # from rest in uneven calls; a duplicated synapse and given work items
    # keep a network on the work-item kernel
    from paper_1906_03958_gb300 import psst
    spec = ng.concat_specs([_network(n, 600 + n, 0.3, 3) for n in (21, 50, 110)])
    kw = dict(method=psst.METHOD_EULER) if method == "euler" else \
        dict(tableau=([1 / 3, 2 / 3], [0.25, 0.0, 0.75])) if method == "heun3" else {}
    traj = []
    for chunks in (0, 2):
        with psst.Network(spec, rec_stride=10, rec_capacity=10, item_chunks=chunks, **kw) as net:
            assert net.info()["item_chunks"] == chunks
            for n in (1, 33, 66):
                net.integrate(n)
            net.status()
            traj.append((net.read_record(), net.get_state_numpy()))
    np.testing.assert_allclose(traj[0][0], traj[1][0], rtol=0, atol=1e-3)
    np.testing.assert_allclose(traj[0][1], traj[1][1], rtol=0, atol=1e-3)
    dup = ng.single_network(np.zeros(3), np.zeros(3), [0, 0, 1], [1, 1, 2], [0.1, 0.2, 0.1], [0, 0, 0],
                            ng.neuron_table(ng.HH), ng.synapse_table(ng.ACH))
    with psst.Network(dup) as net:
        assert net.info()["item_chunks"] > 0


# sizes at the edges of the sweep's tiles: 32 neurons, 4 and 16 pair slots
ADJ_SIZES = {
    "small": [(2, 0.9, 1), (5, 0.8, 3), (16, 0.5, 2), (31, 0.3, 3)],
    "32": [(32, 0.4, 1), (33, 0.3, 2), (63, 0.2, 1), (64, 0.2, 2)],
    "128": [(96, 0.1, 1), (97, 0.15, 1), (127, 0.1, 1), (128, 0.5, 1)],
}


@pytest.mark.parametrize("method", ["rk4", "euler", "heun3"])
@pytest.mark.parametrize("sizes", list(ADJ_SIZES))
def test_dense_adjoint_matches_oracle(sizes, method):
    # one batch of networks of uneven sizes, segments of uneven length, frames
    # that fall inside and at the ends of segments; per-coordinate bound of the
    # adjoint tests (1e-3, floor 1e-2 of the largest)
    import torch
    from paper_1906_03958_gb300 import psst
    from tests.helpers import grad_error
    spec = ng.concat_specs([_network(n, 700 + k, p, t) for k, (n, p, t) in enumerate(ADJ_SIZES[sizes])])
    N, nsteps, stride = spec.n_neurons, 90, 3
    g = np.random.default_rng(3).standard_normal((nsteps // stride, N))
    tab = ([1 / 3, 2 / 3], [0.25, 0.0, 0.75])
    kw = dict(order=1) if method == "euler" else dict(tableau=tab) if method == "heun3" else {}
    gy64, gw64, gp64 = oracle.adjoint(spec, oracle.rest_state(spec), nsteps, g, stride, ckpt=30, **kw)
    kw = dict(method=psst.METHOD_EULER) if method == "euler" else dict(tableau=tab) if method == "heun3" else {}
    with psst.Network(spec, rec_stride=stride, rec_capacity=nsteps // stride, **kw) as net:
        for ck in (40, 90, 7):
            gw, gp, gy = (x.cpu().numpy() for x in net.adjoint(nsteps, torch.from_numpy(g.astype(np.float32)).cuda(), ck))
            net.status()
            assert grad_error(gw, gw64) <= 1e-3
            assert grad_error(gp, gp64) <= 1e-3
            assert grad_error(gy.ravel(), gy64[:4 * N]) <= 1e-3
