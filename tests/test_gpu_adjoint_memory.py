"""psst_adjoint when device memory runs out or a network is refused: the call
reports it, and the calls after it work on complete buffers."""
import numpy as np
import pytest

from paper_1906_03958_gb300 import netgen as ng

pytestmark = pytest.mark.gpu


def _limited_allocator():
    import torch
    from paper_1906_03958_gb300 import psst

    class Limited(psst.TorchAllocator):
        """Refuses what would take the handle's memory past `limit` bytes."""

        def __init__(self, device):
            super().__init__(device)
            self.limit = 1 << 40

            def _alloc(nbytes, ctx):
                if self.used() + nbytes > self.limit:
                    return None
                t = torch.empty(int(nbytes), dtype=torch.uint8, device=f"cuda:{device}")
                self.blocks[t.data_ptr()] = t
                return t.data_ptr()

            self._alloc = psst._ALLOC_FN(_alloc)
            self.struct = psst.Allocator(self._alloc, self._free, None)

        def used(self):
            return sum(t.numel() for t in self.blocks.values())

    return Limited(0)


def _lobe(gate_mode):
    from paper_1906_03958_gb300 import psst
    _, spec = ng.differentiated(n_sets=1, seed=3, n_pn=12, n_ln=4)
    alloc = _limited_allocator()
    return psst.Network(spec, rec_stride=10, rec_capacity=400, gate_mode=gate_mode, allocator=alloc), alloc


def _adjoint(net, steps, every):
    import torch
    g = np.random.default_rng(0).standard_normal((steps // 10, net.N)).astype(np.float32)
    out = [x.cpu().numpy() for x in net.adjoint(steps, torch.from_numpy(g).cuda(), every)]
    net.status()
    return out


@pytest.mark.parametrize("gate_mode", [0, 1])  # dense rows, work items
@pytest.mark.parametrize("first", ["fails", "fits"])
def test_adjoint_after_an_allocation_that_failed(gate_mode, first):
    from paper_1906_03958_gb300 import psst
    with _lobe(gate_mode)[0] as net:
        want = _adjoint(net, 40, 40)
    net, alloc = _lobe(gate_mode)
    with net:
        # checkpoints and state copy exist, so that the adjoint's own buffers meet the limit
        net.record_checkpoints(4000, 4000)
        net.autotune(1)
        steps = 40
        if first == "fits":
            _adjoint(net, 40, 40)
            steps = 4000  # a segment buffer of its own
        alloc.limit = alloc.used() + 1024
        with pytest.raises(psst.PsstError) as e:
            _adjoint(net, steps, steps)
        assert e.value.code == -2  # PSST_ERR_OOM
        if first == "fails":
            alloc.limit = 1 << 40
        for a, b in zip(_adjoint(net, 40, 40), want):
            np.testing.assert_array_equal(a, b)


def test_adjoint_refused_twice():
    # a network of a cluster of CTAs whose adjoint does not fit one: refused, and refused again
    from paper_1906_03958_gb300 import psst
    spec = ng.batched(1, n_min=400, n_max=400)
    with psst.Network(spec, rec_stride=10, rec_capacity=4, mode=psst.MODE_CTA) as net:
        for _ in range(2):
            with pytest.raises(psst.PsstError) as e:
                _adjoint(net, 40, 40)
            assert e.value.code == -7  # PSST_ERR_UNSUPPORTED


def test_dense_adjoint_gives_way_at_a_memory_limit():
    # one synapse type, where the dense rows' records are larger: a limit that the
    # adjoint over work items just meets
    from paper_1906_03958_gb300 import psst
    rng = np.random.default_rng(8)
    n = 128
    post, pre = np.nonzero(rng.random((n, n)) < 0.1)
    spec = ng.single_network(np.zeros(n), rng.uniform(0.0, 8.0, n), post, pre, rng.uniform(0.0, 0.05, post.size),
                             np.zeros(post.size), ng.neuron_table(ng.HH), ng.synapse_table(ng.ACH))
    steps = 200

    def run(gate_mode, limit):
        alloc = _limited_allocator()
        with psst.Network(spec, rec_stride=10, rec_capacity=20, gate_mode=gate_mode, allocator=alloc) as net:
            net.record_checkpoints(steps, steps)
            net.autotune(1)
            base = alloc.used()
            if limit is not None:
                alloc.limit = base + limit
            out = _adjoint(net, steps, steps)
            again = _adjoint(net, steps, steps)
            for a, b in zip(out, again):
                np.testing.assert_array_equal(a, b)
            return out, alloc.used() - base

    general, need = run(1, None)
    dense, more = run(0, None)
    assert more > need
    got, used = run(0, need)
    assert used <= need
    for a, b, c in zip(got, general, dense):
        scale = np.abs(c).max()
        assert np.abs(a - c).max() <= 1e-4 * scale and np.abs(b - c).max() <= 1e-4 * scale
