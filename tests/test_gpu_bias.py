"""Errors that point one way.  Rounding errors of single operations average
out over a run; a mean error of a rate function, of the step's scale or of the
adjoint's Jacobian does not, it shifts every spike and scales every gradient
the same way.

Tolerances: the mean error of a rate over a 10 mV range within 2e-8 of it, a
third of FP32's unit roundoff (the sample's own noise: 1e-7 / sqrt(4,000) =
1.6e-9); a state after 200 steps within 1e-7 of its norm (3.4e-8 is the rounding
of the result itself; the rest leaves each step's rounding room to add up as a
random walk, not a drift).
"""
import numpy as np
import pytest

import oracle
from paper_1906_03958_gb300 import netgen as ng

pytestmark = pytest.mark.gpu

HEUN3 = ([1 / 3, 2 / 3], [0.25, 0.0, 0.75])


def _ratio(u):
    near = np.abs(u) < 1e-6
    u1 = np.where(near, 1.0, u)
    return np.where(near, 1.0 + 0.5 * u, u1 / -np.expm1(-u1))


def _rates64(V):
    return dict(alpha_m=_ratio((V + 40) / 10), beta_m=4 * np.exp(-(V + 65) / 18), alpha_h=0.07 * np.exp(-(V + 65) / 20),
                beta_h=1 / (1 + np.exp(-(V + 35) / 10)), alpha_n=0.1 * _ratio((V + 55) / 10),
                beta_n=0.125 * np.exp(-(V + 65) / 80))


def test_rates_have_no_mean_error():
    # one Euler step of 1,024 ms from gates 0 is 1,024 alpha, from gates 1 it is
    # 1 - 1,024 beta
    from paper_1906_03958_gb300 import psst
    lo, bins, per = -100.0, 12, 4000
    V = (lo + 10.0 * bins * (np.arange(bins * per) + 0.37) / (bins * per)).astype(np.float32)
    n = V.size
    spec = ng.independent(n)
    spec.dt = 1024.0
    got = {}
    for gate, names in ((0.0, ("alpha_m", "alpha_h", "alpha_n")), (1.0, ("beta_m", "beta_h", "beta_n"))):
        y = np.concatenate([V, np.full(3 * n, gate, np.float32)])
        with psst.Network(spec, init_state=y, method=psst.METHOD_EULER) as net:
            net.integrate(1)
            out = net.get_state_numpy().astype(np.float64)
        for x, name in enumerate(names):
            got[name] = np.abs(out[(x + 1) * n:(x + 2) * n] - gate) / 1024.0
    want = _rates64(V.astype(np.float64))
    for name in want:
        mean = (got[name] / want[name] - 1.0).reshape(bins, per).mean(axis=1)
        assert np.max(np.abs(mean)) <= 2e-8, (name, mean)


@pytest.mark.parametrize("method", ["rk4", "euler", "heun3"])
def test_trajectory_does_not_drift(method):
    from paper_1906_03958_gb300 import psst
    spec = ng.batched(24, n_min=10, n_max=80)
    spec.dt = float(np.float32(spec.dt))  # the same map on both sides
    kw = dict(method=psst.METHOD_EULER) if method == "euler" else dict(tableau=HEUN3) if method == "heun3" else {}
    ref = dict(order=1) if method == "euler" else dict(tableau=HEUN3) if method == "heun3" else {}
    y = oracle.rest_state(spec).astype(np.float32)
    y[:spec.n_neurons] += np.random.default_rng(2).uniform(-7.0, 8.0, spec.n_neurons).astype(np.float32)
    want, _ = oracle.integrate(spec, y.astype(np.float64), 200, **ref)
    with psst.Network(spec, init_state=y, **kw) as net:
        net.integrate(200)
        net.status()
        got = net.get_state_numpy().astype(np.float64)
    assert np.linalg.norm(got - want) <= 1e-7 * np.linalg.norm(want)


def _ratio_deriv(u):
    near = np.abs(u) < 1e-2
    u1 = np.where(near, 1.0, u)
    e, d = np.exp(-u1), -np.expm1(-u1)
    return np.where(near, 0.5 + u / 6 - u ** 3 / 180, (d - u1 * e) / d ** 2)


@pytest.mark.parametrize("gate", ["m", "n"])
@pytest.mark.parametrize("size", [100, 150])  # the adjoint over dense rows, over work items
def test_slopes_have_no_mean_error(size, gate):
    # two Euler steps of 1 ms of neurons that have one conductance g and start
    # with its gate closed: the first leaves V and opens the gate to y = alpha(V)
    # (h: 1 - beta_h(V)), so that dV_2/dV_0 = 1 - g d/dV [y^k h (V - E)] holds the
    # gate's slope.  Its mean error over 10 mV within 3e-8: alpha enters to the
    # second or third power, each at up to 0.5e-8, beside the slope's 2e-8.
    import torch
    from paper_1906_03958_gb300 import psst
    bins, per = 8, 3000
    n = bins * per
    V = (-100.0 + 10.0 * bins * (np.arange(n) + 0.37) / n).astype(np.float32)
    g, E = 1000.0, 50.0
    spec = ng.independent(n, n_nets=n // size, pulse=False)
    spec.dt = 1.0
    spec.i_const[:] = 0.0
    spec.neuron_params[:] = 0.0
    spec.neuron_params[:, 0] = 1.0
    spec.neuron_params[:, {"m": 1, "n": 2}[gate]] = g
    spec.neuron_params[:, {"m": 4, "n": 5}[gate]] = E
    # one synapse of weight 0 in each network (its first neuron's to itself)
    first = np.zeros(n, np.int64)
    first[spec.net_neuron_off[:-1]] = 1
    spec.row_ptr = np.concatenate([[0], np.cumsum(first)])
    spec.pre = np.zeros(spec.n_nets, np.int32)
    spec.weight = np.zeros(spec.n_nets, np.float32)
    spec.syn_type = np.zeros(spec.n_nets, np.int32)
    y = np.zeros(4 * n + 2 * spec.n_nets, np.float32)
    y[:n] = V
    y[2 * n:3 * n] = 1.0
    with psst.Network(spec, init_state=y, rec_stride=2, rec_capacity=1, method=psst.METHOD_EULER) as net:
        _, _, gy = net.adjoint(2, torch.ones((1, n), device="cuda"), 2)
        net.status()
        got = gy[0].double().cpu().numpy()
    x = V.astype(np.float64)
    if gate == "m":
        a, da = _ratio((x + 40) / 10), 0.1 * _ratio_deriv((x + 40) / 10)
        bh = 1 / (1 + np.exp(-(x + 35) / 10))
        h, dh = 1 - bh, -0.1 * bh * (1 - bh)
        want = 1 - g * (3 * a ** 2 * da * h * (x - E) + a ** 3 * dh * (x - E) + a ** 3 * h)
    else:
        a, da = 0.1 * _ratio((x + 55) / 10), 0.01 * _ratio_deriv((x + 55) / 10)
        want = 1 - g * (4 * a ** 3 * da * (x - E) + a ** 4)
    use = np.abs(want) > 2.0  # no cancellation against the 1
    err = np.where(use, got / want - 1.0, 0.0).reshape(bins, per)
    many = use.reshape(bins, per).sum(axis=1) > 2000
    assert many.sum() >= 3
    assert np.max(np.abs(err.sum(axis=1) / use.reshape(bins, per).sum(axis=1).clip(1))[many]) <= 3e-8
