"""Selections inside the kernels, against the FP64 oracle: neurons that get rows when a
node is bounded again, and neurons with multi-neuron constraints.

Tolerance of bounds and gradients as in test_gpu_parity: 1e-4 (1 + |oracle|), gradients
relative to the largest component.
"""
import numpy as np
import pytest
import torch

import synth
from helpers import TOL, close, concat, random_node, to_params
from oracle import bab, core

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Context():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00263_gb300 import Context
    return Context


def _case(spec, eps, mnc_fn=None):
    layers = synth.make_network(spec)
    x0 = synth.make_image(spec["seed"] + 7, spec["in_shape"]).reshape(-1)
    y = synth.net_forward(layers, x0)
    C, d = synth.property_rows(int(np.argmax(y)), y.shape[0])
    lo, hi = synth.input_box(x0, eps)
    return layers, C, d, lo, hi, bab.prepare(layers, C, d, lo, hi, mnc_fn)


def test_rows_of_partly_unstable_layers(Context):
    """Nodes with 0 to 900 splits in layers of 8649 neurons (a tile of 8192 and a ragged
    one): the rows are the unstable unsplit neurons among stable and split ones, on both
    sides of neuron 8192; several nodes are collected together."""
    layers, C, d, lo, hi, prep = _case(dict(seed=98, in_shape=(1, 31, 31), layers=[
        ("conv", 9, 3, 1, 1), ("relu",), ("conv", 9, 1, 1, 0), ("relu",), ("fc", 3)]), 0.04)
    net, lo_t, hi_t, l, u, S, _, _ = prep
    rng = np.random.default_rng(21)
    nodes = [random_node(prep, rng, n_splits=k, row=k % 2) for k in (0, 7, 900)]
    for on in nodes:
        on.split_layer = 1
        for side in (slice(0, 8192), slice(8192, None)):
            open_ = (on.S[2] == 0) & (on.l[2] < 0) & (on.u[2] > 0)
            assert 0 < int(open_[side].sum()) < open_[side].numel()
    with Context(node_capacity=64) as ctx:
        prop = ctx.set_property(ctx.load_network(layers), lo, hi, C, d)
        gids = [ctx.node_root(prop, on.row) for on in nodes]
        for g, on in zip(gids, nodes):
            ctx.import_params(g, to_params(on, net.R))
        ctx.bound_batch(gids)
        for g, on in zip(gids, nodes):
            core.rebound_node(net, on, lo_t, hi_t)
            p = ctx.export_params(g)
            assert close(p.l, concat(on.l, net.R)).all() and close(p.u, concat(on.u, net.R)).all()


def _constraints(seed, counts):
    """Constraints over three neurons in which the first neurons of a layer occur counts[0],
    counts[1], ... times and every other one at least once (layers of as many neurons as
    counts or fewer: none)."""
    def fn(net, l, u, lo, hi):
        rng = np.random.default_rng(seed)
        out = {}
        for t in l:
            d, n = l[t].numel(), len(counts)
            if d <= n + 2:
                continue
            first = np.repeat(np.arange(n), counts)
            rest = n + np.concatenate([np.arange(d - n), rng.integers(0, d - n, max(0, 2 * first.size - (d - n)))])
            idx = np.stack([first, rest[:first.size], rest[-first.size:]], 1)
            P, Ph = (rng.normal(0, 0.1, idx.shape).astype(np.float32) for _ in range(2))
            out[t] = core.MNC(idx, P, Ph, rng.uniform(0.0, 0.2, first.size).astype(np.float32))
        return out
    return fn


# entries are staged 480 at a time for a row alone, 224 for the rows of a group and 448 for
# a row of a mixed group, and 1024 listed neurons make one round of a row's CTAs: neurons
# with a chunk's entries, one fewer and one more, two chunks, and 1100 listed neurons
@pytest.mark.parametrize("order", ["few", "blocks", "alternating"])
def test_gamma_terms_around_a_chunk(Context, order):
    counts = [223, 224, 225, 447, 448, 449, 479, 480, 481, 897, 961]
    spec = dict(seed=34, in_shape=(1, 4, 4), layers=[("fc", 1100), ("relu",), ("fc", 9), ("relu",), ("fc", 3)])
    cases = [_case(spec, 0.05, _constraints(5, counts)), _case(spec, 0.04, _constraints(6, counts[::-1]))]
    rng = np.random.default_rng(13)
    E = sum(counts)
    with Context(node_capacity=512, max_mnc_rows=E) as ctx:
        gnet = ctx.load_network(cases[0][0])
        gids, refs = [], []
        for layers, C, d, lo, hi, prep in cases:
            net, lo_t, hi_t, l, u, S, m, dense = prep
            assert sorted(m) == [1] and np.unique(m[1].idx).size == 1100
            prop = ctx.set_property(gnet, lo, hi, C, d)
            ctx.set_mnc(prop, 1, m[1].idx, m[1].P, m[1].Ph, m[1].p)
            on = random_node(prep, rng, n_splits=2, row=1, gamma_scale=0.02)
            on.split_layer = net.R
            refs.append(core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, dense, lo_t, hi_t))
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        SD = sum(v.numel() for v in l.values())
        which = {"few": [0, 1, 0], "blocks": [0] * 21 + [1] * 18, "alternating": [j % 2 for j in range(39)]}[order]
        lb, ga, gb, gg = ctx.bound_grad([gids[j] for j in which], SD, E)
        for i, j in enumerate(which):
            ref, _, oa, ob, og = refs[j]
            assert close(lb[i], float(ref)).all(), (i, j, lb[i], float(ref))
            o = np.concatenate([concat(oa, net.R), concat(ob, net.R), og[1].numpy()])
            g = np.concatenate([ga[i], gb[i], gg[i]])
            assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())
