"""A neuron that diverges (its input current is 1e30): the neurons that its
synapses reach follow it, the others of its network keep their bits, forward and
in the gradients."""
import numpy as np
import pytest

from paper_1906_03958_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


def _two_parts(sizes, hot):
    """Networks of two halves without a synapse between them; hot: the first
    neuron of each second half diverges."""
    parts = []
    for k, n in enumerate(sizes):
        rng = np.random.default_rng([9, k])
        m = rng.random((n, n)) < 0.5
        half = np.arange(n) < n // 2
        m &= half[:, None] == half[None, :]
        post, pre = np.nonzero(m)
        st = rng.integers(0, 3, n)[pre]
        i = rng.uniform(0.0, 8.0, n)
        if hot:
            i[n // 2] = 1e30
        parts.append(ng.single_network(np.zeros(n), i, post, pre, rng.uniform(0.0, 1.0 / n, post.size), st,
                                       ng.neuron_table(ng.HH), ng.synapse_table(ng.ACH, ng.GABA_A, ng.GABA_B)))
    return ng.concat_specs(parts)


def _first_half(spec):
    local = np.concatenate([np.arange(n) < n // 2 for n in spec.net_sizes()])
    return local, np.repeat(local, np.diff(spec.row_ptr))


@pytest.mark.parametrize("method", ["rk4", "euler"])
@pytest.mark.parametrize("cluster", [1, 2, 4])
def test_a_diverging_neuron_stays_among_its_own(cluster, method):
    from paper_1906_03958_gb300 import psst
    sizes = (10, 33, 64, 100, 150, 230)
    out = []
    for hot in (False, True):
        spec = _two_parts(sizes, hot)
        with psst.Network(spec, rec_stride=5, rec_capacity=8, min_cluster=cluster,
                          method=psst.METHOD_EULER if method == "euler" else psst.METHOD_RK4) as net:
            assert net.info()["item_chunks"] == 0  # dense rows
            for n in (7, 33):
                net.integrate(n)
            if hot:
                with pytest.raises(psst.PsstError) as e:
                    net.status()
                assert e.value.code == -4  # PSST_ERR_NONFINITE
            out.append((net.get_state_numpy(), net.read_record()))
    cool, _ = _first_half(spec)
    N = spec.n_neurons
    np.testing.assert_array_equal(out[1][1][:, cool], out[0][1][:, cool])
    for x in range(4):
        np.testing.assert_array_equal(out[1][0][x * N:(x + 1) * N][cool], out[0][0][x * N:(x + 1) * N][cool])
    assert not np.all(np.isfinite(out[1][0][:N][~cool]))


def test_its_gradients_stay_too():
    import torch
    from paper_1906_03958_gb300 import psst
    out = []
    for hot in (False, True):
        spec = _two_parts((10, 33, 64, 100), hot)
        g = np.random.default_rng(1).standard_normal((8, spec.n_neurons)).astype(np.float32)
        with psst.Network(spec, rec_stride=5, rec_capacity=8) as net:
            gw, _, gy = net.adjoint(40, torch.from_numpy(g).cuda(), 16)
            out.append((gw.cpu().numpy(), gy.cpu().numpy()))
    cool, syn = _first_half(spec)
    np.testing.assert_array_equal(out[1][0][syn], out[0][0][syn])
    np.testing.assert_array_equal(out[1][1][:, cool], out[0][1][:, cool])
    assert not np.all(np.isfinite(out[1][0][~syn]))
