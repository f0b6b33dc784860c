"""Performance cases of the library: the calls that programs built on it make.

Each case is one pass through the public entry points of
``paper_1906_03958_gb300`` (``psst.Network`` and ``autograd.trace``) on a
network whose size, wiring and options come from the generators, tests and
benchmark of this repository.  ``prepare`` makes what a program holds before
the call (the network on the GPU, its buffers, weights and targets), ``run``
is the call, ``work`` counts what the path cannot do without, ``exact`` is a
float64 evaluation of the same map in plain torch.

Kinds of networks:
  plain        one small excitatory network (``netgen.plain20``'s recipe)
  lobe         antennal lobes: PN/LN, cholinergic, GABA_A and slow GABA_B
  ragged       a batch of E/I networks of uneven sizes (``netgen.batched``)
  independent  uncoupled neurons (``netgen.independent``)
  sparse       one large E/I network with shot noise (``netgen.sparse_large``)
  fit          lobes with dense weight matrices, differentiated
               (``netgen.differentiated``)

The initial state is scattered around rest with open synapses, as a network
has it in the middle of a simulation.  The passes continue from each other,
as successive integrate calls do.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1906_03958_gb300 import autograd, netgen as ng, psst

# Heun's third-order method as an explicit tableau (a, b).
HEUN3 = ([1.0 / 3.0, 2.0 / 3.0], [0.25, 0.0, 0.75])


def listed():
    return [
        # Closed loop (a controller or a robot in the loop): one RK4 step per
        # call on the 20-neuron network, the state read after each.
        dict(name="closed loop, 20 neurons", kind="plain", nets=1, n=20, steps=1, method="rk4", frames=0),
        # The antennal-lobe network alone, 10 ms with its trace: the single
        # network of the benchmark, autotuned as there.
        dict(name="antennal lobe", kind="lobe", nets=1, n=120, steps=1000, method="rk4", frames=100,
             autotune=True),
        # A small study: a few dozen networks of uneven sizes, fewer than the
        # GPU has SMs.
        dict(name="ragged batch of 48", kind="ragged", nets=48, n_min=20, n_max=300, steps=200, method="rk4",
             frames=20),
        # The benchmark's batch: 4,096 networks of 20 to 300 neurons, autotuned,
        # replayed through a CUDA graph.
        dict(name="ragged batch of 4096", kind="ragged", nets=4096, n_min=20, n_max=300, steps=100, method="rk4",
             frames=10, autotune=True, graph=True),
        # Lobes whose synapses start from unequal gates (one gate per synapse),
        # as after a perturbation of single synapses.
        dict(name="unequal gates, 60 lobes", kind="lobe", nets=60, n=101, steps=100, method="rk4", frames=10,
             unequal=True),
        # Host round trip: state in from host memory, forward Euler, trace and
        # state back to host memory (a sweep driven from the CPU).
        dict(name="host round trip, Euler", kind="ragged", nets=257, n_min=20, n_max=150, steps=300,
             method="euler", frames=30, host=True),
        # Uncoupled neurons, the systems of the paper's Fig. 2b: the small end
        # of its sweep and a large odd count with shot noise.
        dict(name="1000 independent neurons", kind="independent", nets=1, n=1000, steps=500, method="rk4",
             frames=50),
        dict(name="1M independent neurons", kind="independent", nets=1, n=1000003, steps=100, method="rk4",
             frames=10, noise=True),
        # The large sparse network of the benchmark, and a mid-sized one too
        # large for a cluster of CTAs, with a third-order tableau.
        dict(name="sparse 10000", kind="sparse", nets=1, n=10000, p=0.02, steps=200, method="rk4", frames=20,
             noise=True),
        dict(name="sparse 2777, Heun", kind="sparse", nets=1, n=2777, p=0.06, steps=200, method="heun3",
             frames=20, noise=True),
        # Fitting weights and conductances: forward with recorded checkpoints,
        # loss on the trace, discrete adjoint.  The benchmark's 64 parameter
        # sets, and one small network.
        dict(name="fit of 64 lobes", kind="fit", nets=64, n=120, steps=200, method="rk4", frames=20, every=50),
        dict(name="fit of one small lobe", kind="fit", nets=1, n=37, steps=300, method="rk4", frames=300,
             every=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "lobe", "ragged", "ragged", "unequal", "host", "independent", "sparse", "fit"])
    method = rng.choice(["rk4", "rk4", "rk4", "euler", "heun3"])
    if kind == "plain":
        steps = _log_int(rng, 1, 100)
        return dict(kind="plain", nets=1, n=rng.randint(2, 64), steps=steps, method=method, frames=0)
    if kind == "lobe":
        frames = rng.randint(5, 100)
        return dict(kind="lobe", nets=_log_int(rng, 1, 128), n=rng.randint(16, 170), steps=10 * frames,
                    method=method, frames=frames, autotune=rng.random() < 0.5)
    if kind == "ragged":
        nets = _log_int(rng, 8, 2048)
        n_max = rng.randint(40, 300)
        frames = rng.randint(5, 20)
        return dict(kind="ragged", nets=nets, n_min=rng.randint(2, 40), n_max=n_max, steps=10 * frames,
                    method=method, frames=frames, graph=rng.random() < 0.5)
    if kind == "unequal":
        frames = rng.randint(2, 20)
        return dict(kind="lobe", nets=_log_int(rng, 1, 128), n=rng.randint(16, 130), steps=10 * frames,
                    method=method, frames=frames, unequal=True)
    if kind == "host":
        frames = rng.randint(2, 30)
        return dict(kind="ragged", nets=_log_int(rng, 4, 512), n_min=rng.randint(2, 20),
                    n_max=rng.randint(21, 200), steps=10 * frames, method=method, frames=frames, host=True)
    if kind == "independent":
        frames = rng.randint(5, 10)
        return dict(kind="independent", nets=rng.randint(1, 7), n=_log_int(rng, 100, 2000000), steps=10 * frames,
                    method=method, frames=frames, noise=rng.random() < 0.5)
    if kind == "sparse":
        n = _log_int(rng, 1700, 12000)
        frames = rng.randint(5, 20)
        # about 60 to 220 synapses per neuron, within what the grid mode holds
        p = rng.uniform(60.0, min(220.0, 0.1 * n)) / n
        return dict(kind="sparse", nets=1, n=n, p=p, steps=10 * frames, method=method, frames=frames, noise=True)
    steps = 10 * rng.randint(4, 20)
    stride = rng.choice([1, 10])
    return dict(kind="fit", nets=_log_int(rng, 1, 64), n=rng.randint(12, 128), steps=steps, method=method,
                frames=steps // stride, every=rng.randint(steps // 8 + 1, steps))


# ------------------------------------------------------------------ networks

def _mask_edges(rng, rows, cols, prob):
    """Edges (row, col) with probability prob of each pair of a rows x cols
    grid, in row order."""
    post, pre = [], []
    block = max(1, 20_000_000 // max(cols, 1))
    for r0 in range(0, rows, block):
        r = min(block, rows - r0)
        k = np.flatnonzero(rng.random(r * cols, dtype=np.float32) < prob)
        post.append(k // cols + r0)
        pre.append(k % cols)
    return np.concatenate(post), np.concatenate(pre)


def _ragged_edges(rng, sizes, prob):
    """Edges of a batch of networks, each ordered pair i != j of network b
    with probability prob[b]: global row, local column, network."""
    posts, pres = [], []
    first = 0
    for n, p in zip(sizes.tolist(), prob.tolist()):
        mask = rng.random((n, n), dtype=np.float32) < p
        np.fill_diagonal(mask, False)
        k = np.flatnonzero(mask)
        posts.append(k // n + first)
        pres.append(k % n)
        first += n
    net = np.repeat(np.arange(len(sizes)), [len(q) for q in posts])
    return np.concatenate(posts), np.concatenate(pres), net


def _lobe_edges(rng, n_pn, n_ln, dense):
    """Edges of one lobe, rows in order and (pre, type) within a row, and the
    largest weight of each; dense: every pair, absent ones marked False."""
    n = n_pn + n_ln
    full = np.ones((n, n), bool)
    fast = full if dense else (rng.random((n, n)) < 0.5) & ~np.eye(n, dtype=bool)
    slow = np.ones((n_pn, n_ln), bool) if dense else rng.random((n_pn, n_ln)) < 0.5
    po, pr = np.nonzero(fast)
    po2, pr2 = np.nonzero(slow)
    post = np.concatenate([po, po2])
    pre = np.concatenate([pr, pr2 + n_pn])
    st = np.concatenate([(pr >= n_pn).astype(np.int64), np.full(po2.size, 2)])
    order = np.lexsort((st, pre, post))
    post, pre, st = post[order], pre[order], st[order]
    w_max = np.array([0.3, 0.6, 0.3])[st]
    live = (post != pre) & (rng.random(post.size) < 0.5) if dense else np.ones(post.size, bool)
    return post, pre, st, w_max, live


@functools.lru_cache(maxsize=1)
def _wiring(kind, nets, n, n_min, n_max, p):
    """Who is connected to whom: the networks' sizes, CSR rows, presynaptic
    neurons, synapse types and the scale of each weight.  A case has one
    wiring; its weights, inputs and states come from the seed, as in a sweep
    over parameters and initial conditions."""
    rng = np.random.default_rng(4000)
    if kind == "plain":
        post, pre = _mask_edges(rng, n, n, 0.5)
        keep = post != pre
        post, pre = post[keep], pre[keep]
        sizes, st, scale = np.array([n]), np.zeros(pre.size), np.full(pre.size, 0.5)
    elif kind == "ragged":
        sizes = rng.integers(n_min, n_max + 1, nets)
        prob = rng.uniform(0.1, 0.5, nets).astype(np.float32)
        post, pre, net = _ragged_edges(rng, sizes, prob)
        st = pre >= np.round(0.8 * sizes)[net]
        scale = (0.5 * 10.0 / (sizes * prob))[net]
    elif kind in ("lobe", "fit"):
        n_ln = max(1, n // 4)
        parts = [_lobe_edges(rng, n - n_ln, n_ln, kind == "fit") for _ in range(nets)]
        sizes = np.full(nets, n)
        post = np.concatenate([q[0] + b * n for b, q in enumerate(parts)])
        pre, st = np.concatenate([q[1] for q in parts]), np.concatenate([q[2] for q in parts])
        scale = np.concatenate([q[3] * q[4] for q in parts])
    elif kind == "independent":
        sizes = np.diff(np.linspace(0, n, nets + 1).round().astype(np.int64))
        post, pre, st, scale = (np.zeros(0, np.int64) for _ in range(4))
    else:
        post, pre = _mask_edges(rng, n, n - 1, np.float32(p))
        pre = pre + (pre >= post)  # no self-synapse
        sizes, st, scale = np.array([n]), pre >= int(round(0.8 * n)), np.ones(pre.size)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(post, minlength=int(sizes.sum())))])
    return sizes, row_ptr.astype(np.int64), pre.astype(np.int32), st.astype(np.int32), scale.astype(np.float32)


def _spec(case, seed):
    """The case's networks with weights and inputs drawn from the seed."""
    rng = np.random.default_rng([seed, 77])
    kind, nets = case["kind"], case["nets"]
    sizes, row_ptr, pre, st, w = _wiring(kind, nets, case.get("n", 0), case.get("n_min", 0), case.get("n_max", 0),
                                         case.get("p", 0.0))
    n = int(sizes.sum())
    thresh, amp = 0, 0.0
    on, off = np.full(nets, 50, np.int64), np.full(nets, 5000, np.int64)
    ntype, ntab, stab = np.zeros(n), ng.neuron_table(ng.HH), ng.synapse_table(ng.ACH, ng.GABA_A)
    i_const, pulse = rng.uniform(0.0, 10.0, n), np.zeros(n)
    if kind == "sparse":
        w = w * rng.lognormal(-1.0, 0.5, pre.size)
    else:
        w = w * rng.random(pre.size, dtype=np.float32)
    if kind in ("plain", "independent"):
        stab = ng.synapse_table(ng.ACH)
    if kind == "ragged":
        pulse = np.where(rng.random(n) < 1.0 / 3.0, rng.uniform(0.0, 10.0, n), 0.0)
        on = rng.integers(0, 100, nets)
        off = on + rng.integers(2000, 10000, nets)
    elif kind == "independent":
        pulse = np.full(n, 10.0)
    elif kind in ("lobe", "fit"):
        n_ln = max(1, case["n"] // 4)
        types = np.r_[np.zeros(case["n"] - n_ln), np.ones(n_ln)]
        ntype, ntab, stab = np.tile(types, nets), ng.neuron_table(ng.PN, ng.LN), \
            ng.synapse_table(ng.ACH, ng.GABA_A, ng.GABA_B)
        if kind == "fit":  # each set with conductances of its own
            ntype = np.concatenate([types + 2 * b for b in range(nets)])
            ntab = np.tile(ntab, (nets, 1)).astype(np.float64)
            ntab[:, [1, 2, 3, 7]] *= 1.0 + 0.2 * rng.uniform(-1.0, 1.0, (2 * nets, 4))
        i_const = rng.uniform(0.0, 5.0, n)
        pulse = np.where(rng.random(n) < 1.0 / 3.0, 10.0 * rng.uniform(0.5, 1.0, n), 0.0)
    if case.get("noise"):
        thresh, amp = int(round(20.0 * 1e-3 * ng.DT * (1 << 24))), 20.0
    return ng.NetworkSpec(
        net_neuron_off=np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32),
        neuron_type=np.asarray(ntype, np.int32), neuron_params=np.asarray(ntab, np.float32),
        row_ptr=np.asarray(row_ptr, np.int64), pre=np.asarray(pre, np.int32), weight=np.asarray(w, np.float32),
        syn_type=np.asarray(st, np.int32), syn_params=np.asarray(stab, np.float32),
        i_const=np.asarray(i_const, np.float32), pulse_amp=np.asarray(pulse, np.float32),
        pulse_on=np.asarray(on, np.int64), pulse_off=np.asarray(off, np.int64), noise_seed=seed,
        noise_thresh=thresh, noise_amp=amp, dt=ng.DT, name="case")


def _pairs(spec):
    """Of every synapse, its (presynaptic neuron, type) pair over the batch."""
    base = np.repeat(spec.net_neuron_off[:-1].astype(np.int64), spec.net_synapses())
    return (base + spec.pre) * spec.syn_params.shape[0] + spec.syn_type


def _initial_state(case, spec, seed):
    """[V, m, h, n, r, s] around rest: potentials scattered over 15 mV, gates
    within 20% of their rest values, synapses partly open; all gates of a
    (presynaptic neuron, type) pair equal unless the case has them unequal."""
    rng = np.random.default_rng([seed, 78])
    N, S, nt = spec.n_neurons, spec.n_synapses, spec.syn_params.shape[0]
    y = np.empty(4 * N + 2 * S, np.float32)
    y[:N] = rng.uniform(-72.0, -57.0, N)
    for x, rest in enumerate((0.0529, 0.5961, 0.3177)):
        y[(x + 1) * N:(x + 2) * N] = rest * rng.uniform(0.8, 1.2, N)
    if S:
        second = spec.syn_params[spec.syn_type, 0] != 0
        if case.get("unequal"):
            r, s = rng.uniform(0.0, 0.3, S), rng.uniform(0.0, 1.0, S)
        else:
            pair = _pairs(spec)
            r = rng.uniform(0.0, 0.3, N * nt).astype(np.float32)[pair]
            s = rng.uniform(0.0, 1.0, N * nt).astype(np.float32)[pair]
        y[4 * N:4 * N + S] = r
        y[4 * N + S:] = np.where(second, s, 0.0)
    return y


def prepare(case, seed):
    spec = _spec(case, seed)
    y0 = _initial_state(case, spec, seed)
    frames = case["frames"]
    stride = case["steps"] // frames if frames else 0
    method = {"rk4": psst.METHOD_RK4, "euler": psst.METHOD_EULER}.get(case["method"], 0)
    net = psst.Network(spec, init_state=y0, rec_stride=stride, rec_capacity=max(frames, 1), method=method,
                       tableau=HEUN3 if case["method"] == "heun3" else None)
    if case.get("autotune"):
        net.autotune(50)
    if case.get("graph"):
        net.set_graph_mode(True)
    state = dict(case=case, net=net)
    if case["kind"] == "fit":
        rng = np.random.default_rng([seed, 79])
        net.record_checkpoints(case["every"], case["steps"])
        state["weight"] = torch.from_numpy(spec.weight).cuda()
        state["params"] = torch.from_numpy(spec.neuron_params).cuda()
        # the measured traces to fit: around rest, a few mV of noise
        state["target"] = torch.from_numpy(
            rng.normal(-62.0, 4.0, (frames, spec.n_neurons)).astype(np.float32)).cuda()
    elif case.get("host"):
        state["start"] = torch.from_numpy(y0).pin_memory()
        state["trace"] = torch.empty((frames, spec.n_neurons), dtype=torch.float32).pin_memory()
        state["final"] = torch.empty(net.dim, dtype=torch.float32).pin_memory()
    else:
        state["final"] = torch.empty(net.dim, dtype=torch.float32, device="cuda")
        if frames:
            state["trace"] = torch.empty((frames, spec.n_neurons), dtype=torch.float32, device="cuda")
    return state


def run(state):
    case, net = state["case"], state["net"]
    steps = case["steps"]
    if case["kind"] == "fit":
        w = state["weight"].detach().requires_grad_()
        p = state["params"].detach().requires_grad_()
        trace = autograd.trace(net, w, p, steps, case["every"])
        loss = torch.mean((trace - state["target"]) ** 2)
        loss.backward()
        return dict(trace=trace.detach(), grad_weight=w.grad, grad_params=p.grad)
    if case.get("host"):
        net.set_state(state["start"])
        net.integrate(steps)
        trace = net.read_record(out=state["trace"].numpy())
        return dict(trace=trace, final=net.get_state(out=state["final"].numpy()))
    net.integrate(steps)
    out = dict(final=net.get_state(out=state["final"]))
    if case["frames"]:
        out["trace"] = net.read_record(out=state["trace"])
    return out


# ---------------------------------------------------------------------- work

def _expected_sizes(case):
    """Neurons, synapses and used (presynaptic neuron, type) pairs."""
    kind, nets = case["kind"], case["nets"]
    if kind == "plain":
        n = case["n"]
        return n, 0.5 * n * (n - 1), n
    if kind == "ragged":
        lo, hi = case["n_min"], case["n_max"]
        k = np.arange(lo, hi + 1, dtype=np.float64)
        return nets * k.mean(), nets * 0.3 * (k * (k - 1)).mean(), nets * k.mean()
    if kind in ("lobe", "fit"):
        n, q = case["n"], max(1, case["n"] // 4)
        syn = n * n + (n - q) * q if kind == "fit" else 0.5 * (n * (n - 1) + (n - q) * q)
        return nets * n, nets * syn, nets * (n + q)
    if kind == "independent":
        return case["n"], 0, 0
    return case["n"], case["n"] * (case["n"] - 1) * case["p"], case["n"]


def work(case):
    n, syn, pairs = _expected_sizes(case)
    stages = {"rk4": 4, "euler": 1, "heun3": 3}[case["method"]] * case["steps"]
    gates = syn if case.get("unequal") else pairs
    # per stage: a neuron's rates, currents and update 80, a pair's
    # transmitter and gate 18, a synapse's multiply-add 2, of unequal gates
    # each its own update 4
    flops = stages * (80.0 * n + 18.0 * pairs + 2.0 * syn + (4.0 * gates if case.get("unequal") else 0.0))
    # state in and out (gates r, s of each synapse as the entry points have
    # it), weights, connectivity, parameters and inputs, the trace
    data = 4.0 * (2 * (4 * n + 2 * syn) + 2 * syn + 3 * n + case["frames"] * n)
    if case["kind"] == "fit":
        # backward: about twice the forward's products, and the gradients
        flops *= 3.0
        data += 4.0 * (syn + 2 * case["frames"] * n)
    return {"bytes": float(data), "flops": float(flops)}


# --------------------------------------------------------------------- exact

def _philox(step, neuron, seed):
    """Word 0 of Philox4x32-10 for counter (step lo, step hi, neuron, 0)."""
    mask = 0xFFFFFFFF
    c0 = torch.full_like(neuron, step & mask)
    c1 = torch.full_like(neuron, (step >> 32) & mask)
    c2, c3 = neuron, torch.zeros_like(neuron)
    k0, k1 = seed & mask, (seed >> 32) & mask
    for rnd in range(10):
        if rnd:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # 64-bit products, wrapped
        hi0, lo0 = (p0 >> 32) & mask, p0 & mask
        hi1, lo1 = (p1 >> 32) & mask, p1 & mask
        c0, c1, c2, c3 = hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0
    return c0


class _Model:
    """The network map in float64, one gate (r, s) per pair, or per synapse
    where the gates are unequal."""

    def __init__(self, spec, unequal):
        f8 = lambda a: torch.from_numpy(np.asarray(a, np.float64)).cuda()
        i8 = lambda a: torch.from_numpy(np.asarray(a, np.int64)).cuda()
        self.spec, self.N = spec, spec.n_neurons
        net = np.repeat(np.arange(spec.n_nets), spec.net_sizes())
        self.types = i8(spec.neuron_type)
        self.post = i8(np.repeat(np.arange(self.N), np.diff(spec.row_ptr)))
        nt = spec.syn_params.shape[0]
        pair = _pairs(spec)
        if unequal:
            self.gate, gates = i8(np.arange(pair.size)), pair
        else:
            used = np.zeros(self.N * nt, bool)
            used[pair] = True
            gates = np.flatnonzero(used)
            index = np.cumsum(used) - 1
            self.gate = i8(index[pair])
        first = np.zeros(gates.size, np.int64)
        first[self.gate.cpu().numpy()] = np.arange(pair.size)
        self.first = i8(first)  # a synapse of each gate
        self.pre = i8(gates // nt)
        tab = f8(spec.syn_params)[i8(gates % nt)].T if gates.size else torch.zeros((9, 0)).double().cuda()
        self.second = tab[0] != 0
        self.a, self.b, self.K3, self.K4, self.Kd, E, self.Vp, self.Kp = tab[1:]
        self.E = E
        self.i_const, self.pulse = f8(spec.i_const), f8(spec.pulse_amp)
        self.on, self.off = i8(spec.pulse_on[net]), i8(spec.pulse_off[net])
        self.neuron = torch.arange(self.N, device="cuda")
        self.dt = float(np.float32(spec.dt))

    def current(self, step):
        I = self.i_const + torch.where((self.on <= step) & (step < self.off), self.pulse, 0.0)
        if self.spec.noise_thresh:
            event = (_philox(step, self.neuron, int(self.spec.noise_seed)) >> 8) < self.spec.noise_thresh
            I = I + torch.where(event, float(self.spec.noise_amp), 0.0)
        return I

    def f(self, y, I, w, P):
        V, m, h, n, r, s = y

        def ratio(u):
            near = u.abs() < 1e-6
            u1 = torch.where(near, torch.ones_like(u), u)
            return torch.where(near, 1.0 + 0.5 * u, u1 / -torch.expm1(-u1))

        am, bm = ratio((V + 40.0) / 10.0), 4.0 * torch.exp(-(V + 65.0) / 18.0)
        ah, bh = 0.07 * torch.exp(-(V + 65.0) / 20.0), 1.0 / (1.0 + torch.exp(-(V + 35.0) / 10.0))
        an, bn = 0.1 * ratio((V + 55.0) / 10.0), 0.125 * torch.exp(-(V + 65.0) / 80.0)
        C, gNa, gK, gL, ENa, EK, EL, gKL, EKL = P
        ion = gNa * m ** 3 * h * (V - ENa) + gK * n ** 4 * (V - EK) + gL * (V - EL) + gKL * (V - EKL)
        dr, ds = torch.zeros_like(r), torch.zeros_like(s)
        if self.pre.numel():
            T = 1.0 / (1.0 + torch.exp(-(V[self.pre] - self.Vp) / self.Kp))
            dr = self.a * T * (1.0 - r) - self.b * r
            ds = torch.where(self.second, self.K3 * r - self.K4 * s, 0.0)
            s4 = s ** 4
            G = torch.where(self.second, s4 / torch.where(self.second, s4 + self.Kd, 1.0), r)
            zero = torch.zeros_like(V)
            A = zero.index_add(0, self.post, w * G[self.gate])
            B = zero.index_add(0, self.post, w * (G * self.E)[self.gate])
            ion = ion + V * A - B
        return [(I - ion) / C, am * (1 - m) - bm * m, ah * (1 - h) - bh * h, an * (1 - n) - bn * n, dr, ds]

    def step(self, y, k, w, P, method):
        I, dt = self.current(k), self.dt
        a, b = {"rk4": ([0.5, 0.5, 1.0], [1 / 6, 1 / 3, 1 / 3, 1 / 6]), "euler": ([], [1.0]), "heun3": HEUN3}[method]
        total, slope = None, None
        for q, weight in enumerate(b):
            z = y if q == 0 else [u + dt * a[q - 1] * d for u, d in zip(y, slope)]
            slope = self.f(z, I, w, P)
            total = [weight * d for d in slope] if q == 0 else [t + weight * d for t, d in zip(total, slope)]
        return [u + dt * t for u, t in zip(y, total)]


def exact(case, seed):
    spec = _spec(case, seed)
    y0 = _initial_state(case, spec, seed)
    model = _Model(spec, case.get("unequal", False))
    N, S = spec.n_neurons, spec.n_synapses
    full = torch.from_numpy(y0).cuda().double()
    y = [full[x * N:(x + 1) * N] for x in range(4)]
    y += [full[4 * N:4 * N + S][model.first], full[4 * N + S:][model.first]]
    fit = case["kind"] == "fit"
    w = torch.from_numpy(spec.weight).cuda().double().requires_grad_(fit)
    p = torch.from_numpy(spec.neuron_params).cuda().double().requires_grad_(fit)
    stride = case["steps"] // case["frames"] if case["frames"] else 0
    trace = []
    with torch.set_grad_enabled(fit):
        P = p[model.types].T
        for k in range(case["steps"]):
            y = model.step(y, k, w, P, case["method"])
            if stride and (k + 1) % stride == 0:
                trace.append(y[0])
        if fit:
            trace = torch.stack(trace)
            target = np.random.default_rng([seed, 79]).normal(-62.0, 4.0, trace.shape).astype(np.float32)
            torch.mean((trace - torch.from_numpy(target).cuda().double()) ** 2).backward()
            return dict(trace=trace.detach(), grad_weight=w.grad, grad_params=p.grad)
    out = dict(final=torch.cat(y[:4] + [y[4][model.gate], y[5][model.gate]]))
    if trace:
        out["trace"] = torch.stack(trace)
    if case.get("host"):
        out = {k: v.cpu().numpy() for k, v in out.items()}
    return out
