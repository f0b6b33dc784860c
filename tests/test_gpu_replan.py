"""Launch plans that are made again (a state with other gates, the autotuner):
their buffers are given back, a plan that could not be made is not launched, and
work still queued keeps the plan it was launched with."""
import numpy as np
import pytest

import oracle
from paper_1906_03958_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


def _spec():
    return ng.batched(6, n_min=30, n_max=90)


def _states(spec):
    """A state with equal gates in each pair, and one without."""
    y = oracle.rest_state(spec).astype(np.float32)
    N, S = spec.n_neurons, spec.n_synapses
    z = y.copy()
    z[4 * N:4 * N + S] = np.random.default_rng(3).uniform(0.0, 0.3, S)
    return y, z


@pytest.mark.parametrize("mode", ["cta", "grid"])
def test_plans_do_not_pile_up(mode):
    from paper_1906_03958_gb300 import psst
    spec = _spec() if mode == "cta" else ng.batched(1, n_min=60, n_max=60)
    with psst.Network(spec, allocator="torch", mode=psst.MODE_GRID if mode == "grid" else psst.MODE_CTA) as net:
        used, first = [], None
        for _ in range(3):
            for y in _states(spec):
                net.set_state(y)
                net.set_step(0)
                net.integrate(3)
                used.append(sum(t.numel() for t in net._allocator.blocks.values()))
            got = net.get_state_numpy()
            first = got if first is None else first
            np.testing.assert_array_equal(got, first)
        assert used[-2:] == used[2:4]


def test_no_plan_is_not_launched():
    from paper_1906_03958_gb300 import psst
    from tests.test_gpu_adjoint_memory import _limited_allocator
    spec = _spec()
    y, z = _states(spec)
    with psst.Network(spec, init_state=z) as net:
        net.integrate(3)
        want = net.get_state_numpy()
    alloc = _limited_allocator()
    with psst.Network(spec, init_state=y, allocator=alloc) as net:
        net.integrate(1)
        net.set_state(y)  # the check's buffer is there
        alloc.limit = 0
        with pytest.raises(psst.PsstError) as e:
            net.set_state(z)
        assert e.value.code == -2  # PSST_ERR_OOM
        for call in (lambda: net.integrate(3), lambda: net.autotune(2)):
            with pytest.raises(psst.PsstError) as e:
                call()
            assert e.value.code == -6  # PSST_ERR_STATE
        alloc.limit = 1 << 40
        net.set_state(z)
        net.integrate(3)
        net.status()
        # (a batch created with this state has the same plan)
        np.testing.assert_array_equal(net.get_state_numpy(), want)


def test_queued_work_keeps_its_plan():
    import torch
    from paper_1906_03958_gb300 import psst
    spec = _spec()
    y, z = _states(spec)

    def run(wait):
        out = []
        with psst.Network(spec, init_state=y) as net, torch.cuda.stream(torch.cuda.Stream()):
            for step in ("tune", "state", "tune"):
                net.integrate(2000)
                if wait:
                    torch.cuda.synchronize()
                if step == "tune":
                    net.autotune(2)
                else:
                    out.append(net.get_state())
                    net.set_state(z)
            net.integrate(10)
            net.status()
            out.append(net.get_state())
            return [x.cpu().numpy() for x in out]

    for a, b in zip(run(False), run(True)):
        np.testing.assert_array_equal(a, b)
