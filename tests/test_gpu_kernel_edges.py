"""Kernels at the edges of their tiles and splits, against the FP64 oracle.

Tolerance of bounds and gradients as in test_gpu_parity: 1e-4 (1 + |oracle|),
gradients relative to the largest component.
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


def _rows_per_neuron(seed, counts, k):
    """Constraints over k neurons each in which the first neurons of every layer
    occur counts[0], counts[1], ... times (up to the layer's width)."""
    def fn(net, l, u, lo, hi):
        rng = np.random.default_rng(seed)
        out = {}
        for t in l:
            d = l[t].numel()
            first = np.repeat(np.arange(min(d, len(counts))), counts[:d])
            idx = np.stack([first] + [rng.integers(0, d, first.size) for _ in range(k - 1)], 1)
            P, Ph = (rng.normal(0, 0.1, idx.shape).astype(np.float32) for _ in range(2))
            p = rng.uniform(0.0, 0.2, first.size).astype(np.float32)
            out[t] = core.MNC(idx, P, Ph, p)
        return out
    return fn


# gamma terms: neurons with no entry (written as zeros by CTAs of their own) and with
# entries around one and four widths of the warp that stages them, in a network of a few
# listed neurons and in one of more than 8192 neurons; rows over 2 and 3 neurons
@pytest.mark.parametrize("spec,k", [
    (dict(seed=31, in_shape=(12,), layers=[("fc", 33), ("relu",), ("fc", 9), ("relu",), ("fc", 3)]), 3),
    (dict(seed=32, in_shape=(1, 33, 33), layers=[("conv", 8, 3, 1, 1), ("relu",), ("fc", 17), ("relu",),
                                                 ("fc", 3)]), 2),
])
def test_gamma_terms(Context, spec, k):
    counts = [0, 1, 31, 32, 33, 127, 128, 129, 300, 0, 5]
    if len(spec["in_shape"]) == 1:
        layers = synth.tiny_fc_net(spec["seed"], [12, 33, 9, 3])
        lo, hi = synth.input_box(np.random.default_rng(1).uniform(0.2, 0.8, 12), 0.1)
        C, d = synth.property_rows(0, 3)
        prep = bab.prepare(layers, C, d, lo, hi, _rows_per_neuron(5, counts, k))
    else:
        layers, C, d, lo, hi, prep = _case(spec, 0.02, _rows_per_neuron(5, counts, k))
    net, lo_t, hi_t, l, u, S, m, dense = prep
    E = sum(v.idx.shape[0] for v in m.values())
    SD = sum(l[i].numel() for i in l)
    rng = np.random.default_rng(9)
    with Context(node_capacity=64, max_mnc_rows=E + 3) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        for i in sorted(m):
            ctx.set_mnc(prop, i, m[i].idx, m[i].P, m[i].Ph, m[i].p)
        nodes = [random_node(prep, rng, n_splits=j, row=j % 2) for j in range(3)]
        gids = []
        for on in nodes:
            on.split_layer = net.R
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        lb, ga, gb, gg = ctx.bound_grad(gids, SD, E)
        best = ctx.optimize(gids, steps=1, eps_rel=1e-3)
        for j, on in enumerate(nodes):
            ref, _, oa, ob, og = core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, dense,
                                                     lo_t, hi_t)
            assert close(lb[j], float(ref)).all()
            o = np.concatenate([concat(oa, net.R), concat(ob, net.R),
                                *(og[i].numpy() for i in sorted(og))])
            g = np.concatenate([ga[j], gb[j], gg[j]])
            assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())
            top, *_ = core.optimize(net, on, dense, lo_t, hi_t, core.AdamHP(steps=1, eps_rel=1e-3))
            assert close(best[j], top).all()


# windowed rows: stride classes of one to more than three taps,
# kernels smaller than the stride, 1, 2, 3, 4, 5 and 8 input
# channels, windows cut by the padding, a row count that is not a multiple of
# the rows per CTA, splits in the layers that the rows pass
@pytest.mark.parametrize("layers,shape", [
    ([("conv", 3, 3, 1, 1), ("relu",), ("conv", 5, 2, 2, 0), ("relu",), ("conv", 3, 3, 1, 1), ("relu",),
      ("fc", 3)], (2, 7, 9)),
    ([("conv", 4, 4, 3, 2), ("relu",), ("conv", 8, 5, 1, 2), ("relu",), ("conv", 7, 3, 2, 1), ("relu",),
      ("fc", 3)], (1, 13, 11)),
    ([("conv", 8, 1, 1, 0), ("relu",), ("conv", 12, 4, 1, 1), ("relu",), ("conv", 5, 1, 2, 0), ("relu",),
      ("fc", 3)], (3, 6, 5)),
    ([("conv", 2, 3, 4, 1), ("relu",), ("conv", 6, 3, 1, 2), ("relu",), ("fc", 3)], (5, 17, 14)),
    # one row per CTA: the window at the input holds 54 x 54 values of 4 channels
    ([("conv", 4, 4, 2, 1), ("relu",), ("conv", 4, 12, 2, 1), ("relu",), ("conv", 2, 8, 2, 0), ("relu",),
      ("fc", 3)], (4, 72, 72)),
])
def test_window_rows(Context, layers, shape):
    layers, C, d, lo, hi, prep = _case(dict(seed=41, in_shape=shape, layers=layers), 0.05)
    net, lo_t, hi_t, l, u, S, _, _ = prep
    rng = np.random.default_rng(2)
    with Context(node_capacity=64) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        for i in l:
            gl, gu = ctx.root_bounds(prop, i)
            assert close(gl, l[i].numpy()).all() and close(gu, u[i].numpy()).all(), i
        for j in range(3):
            on = random_node(prep, rng, n_splits=j + 1, row=j % 2)
            on.split_layer = 1
            gid = ctx.node_root(prop, on.row)
            ctx.import_params(gid, to_params(on, net.R))
            ctx.bound_batch([gid])
            core.rebound_node(net, on, lo_t, hi_t)
            p = ctx.export_params(gid)
            assert close(p.l, concat(on.l, net.R)).all() and close(p.u, concat(on.u, net.R)).all()


def test_row_roots_are_created_by_the_first_step(Context):
    """Started properties hold the slots of their row root nodes without
    creating them: other nodes cannot take those slots, the queue counts them, and
    the first step finds them."""
    from paper_2205_00263_gb300.api import MnbabError
    layers, C, d, lo, hi, _ = _case(dict(seed=43, in_shape=(1, 6, 6), layers=[
        ("conv", 3, 3, 1, 1), ("relu",), ("fc", 4)]), 0.05)
    rows = C.shape[0]
    cap = 64  # the pad slot, two properties (root and rows), other nodes
    with Context(node_capacity=cap) as ctx, Context(node_capacity=256) as big:
        net = ctx.load_network(layers)
        a, b = (ctx.set_property(net, lo, hi, C, d) for _ in range(2))
        ctx.root_bounds(a, 1)
        assert ctx.queue_size(a) == rows and ctx.queue_size(b) == rows
        extra = [ctx.node_root(a, 0) for _ in range(cap - 1 - 2 * (rows + 1))]
        with pytest.raises(MnbabError):
            ctx.node_root(a, 0)
        for n in extra:
            ctx.node_free(n)
        net2 = big.load_network(layers)
        ref = big.set_property(net2, lo, hi, C, d)
        assert big.bab_step([ref], max_nodes=rows, steps=2)["nodes_bounded"] == rows
        assert ctx.bab_step([a, b], max_nodes=2 * rows, steps=2)["nodes_bounded"] == 2 * rows
        for p in (a, b):
            assert [(r["row"], r["seq"], r["lb"]) for r in ctx.trace(p)] == \
                   [(r["row"], r["seq"], r["lb"]) for r in big.trace(ref)]


# tensor-core convolutions in both directions (forced by gemm_path 2): strides
# 1 to 4, kernels below and above the stride, padding beyond the kernel's reach, planes
# smaller than a tile and rows across tiles, channel counts that are not multiples of 8 or 16,
# one to four chunks of 16 channels and 1 to 16 stride classes; one row and 700, four to a CTA
@pytest.mark.parametrize("layers,shape", [
    ([("conv", 9, 5, 3, 2), ("relu",), ("conv", 17, 2, 4, 1), ("relu",), ("fc", 3)], (8, 22, 15)),
    ([("conv", 24, 3, 1, 2), ("relu",), ("conv", 48, 5, 2, 2), ("relu",), ("fc", 3)], (10, 6, 9)),
    ([("conv", 40, 1, 2, 0), ("relu",), ("conv", 64, 3, 1, 0), ("relu",), ("conv", 8, 1, 1, 0), ("relu",),
      ("fc", 3)], (9, 9, 7)),
    ([("conv", 16, 4, 2, 1), ("relu",), ("conv", 33, 4, 2, 1), ("relu",), ("fc", 3)], (12, 32, 20)),
])
def test_tensor_core_convolutions(Context, layers, shape):
    layers, C, d, lo, hi, prep = _case(dict(seed=51, in_shape=shape, layers=layers), 0.01)
    net, lo_t, hi_t, l, u, S, _, _ = prep
    SD = sum(l[i].numel() for i in l)
    rng = np.random.default_rng(4)
    nodes = [random_node(prep, rng, n_splits=j, row=j % 2) for j in range(3)]
    refs = []
    for on in nodes:
        on.split_layer = net.R
        refs.append(core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, None, lo_t, hi_t))
    with Context(node_capacity=2048, gemm_path=2) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        gids = []
        for on in nodes:
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        for batch in ([0], [j % 3 for j in range(700)]):
            lb, ga, gb, _ = ctx.bound_grad([gids[j] for j in batch], SD, 0)
            for i in list(range(min(3, len(batch)))) + [len(batch) - 1]:
                ref, _, oa, ob, _ = refs[batch[i]]
                assert close(lb[i], float(ref)).all(), (batch[i], lb[i], float(ref))
                o = np.concatenate([concat(oa, net.R), concat(ob, net.R)])
                g = np.concatenate([ga[i], gb[i]])
                assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())
            assert all((lb[j::3] == lb[j]).all() or np.abs(lb[j::3] - lb[j]).max() <= 1e-6 * (1 + abs(lb[j]))
                       for j in range(min(3, len(batch))))


# row-resident convolutions in both directions and starting rows (gemm_path 1, layers
# too small for the implicit GEMM): kernels of 3 and 4 with and without padding, and
# others; strides 1 to 3; channel counts that are no multiple of a block; one input
# channel (several items per thread) with a last round that is not full; planes split
# into chunks whose first and last input rows are cut off; one row and several
@pytest.mark.parametrize("layers,shape", [
    ([("conv", 5, 3, 1, 1), ("relu",), ("conv", 6, 2, 2, 0), ("relu",), ("fc", 7), ("relu",), ("fc", 3)], (3, 9, 7)),
    ([("conv", 8, 4, 2, 1), ("relu",), ("conv", 9, 5, 3, 2), ("relu",), ("fc", 3)], (1, 29, 31)),
    ([("conv", 6, 4, 2, 0), ("relu",), ("conv", 12, 3, 1, 0), ("relu",), ("fc", 3)], (1, 28, 20)),
    ([("conv", 8, 3, 1, 1), ("relu",), ("conv", 16, 1, 2, 0), ("relu",), ("conv", 11, 3, 1, 2), ("relu",),
      ("fc", 3)], (3, 21, 20)),
    ([("conv", 4, 7, 1, 3), ("relu",), ("conv", 3, 3, 2, 1), ("relu",), ("fc", 3)], (2, 6, 40)),
])
def test_row_convolutions(Context, layers, shape):
    layers, C, d, lo, hi, prep = _case(dict(seed=61, in_shape=shape, layers=layers), 0.01)
    net, lo_t, hi_t, l, u, S, _, _ = prep
    SD = sum(l[i].numel() for i in l)
    rng = np.random.default_rng(6)
    nodes = [random_node(prep, rng, n_splits=2 * j, row=j % 2) for j in range(3)]
    refs = []
    for on in nodes:
        on.split_layer = net.R
        refs.append(core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, None, lo_t, hi_t))
    with Context(node_capacity=1024, gemm_path=1) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        for i in l:
            gl, gu = ctx.root_bounds(prop, i)
            assert close(gl, l[i].numpy()).all() and close(gu, u[i].numpy()).all(), i
        gids = []
        for on in nodes:
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        for batch in ([0], [1, 2], [j % 3 for j in range(160)]):
            lb, ga, gb, _ = ctx.bound_grad([gids[j] for j in batch], SD, 0)
            for i in list(range(min(3, len(batch)))) + [len(batch) - 1]:
                ref, _, oa, ob, _ = refs[batch[i]]
                assert close(lb[i], float(ref)).all(), (batch[i], lb[i], float(ref))
                o = np.concatenate([concat(oa, net.R), concat(ob, net.R)])
                g = np.concatenate([ga[i], gb[i]])
                assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())


# stride-1 convolutions back to at most three input channels (128-position chunks per
# warp, many rows): 3x3 and 5x5 kernels, padding from none to the kernel's reach,
# planes that are no multiple of a chunk or of a CTA's chunks, chunks that start inside
# a row, source channels that are no multiple of a stage; a plane width that is no
# multiple of four takes the other kernel
@pytest.mark.parametrize("layers,shape", [
    ([("conv", 21, 3, 1, 1), ("relu",), ("conv", 4, 2, 2, 0), ("relu",), ("fc", 3)], (3, 30, 36)),
    ([("conv", 16, 5, 1, 2), ("relu",), ("conv", 4, 3, 3, 0), ("relu",), ("fc", 3)], (2, 27, 28)),
    ([("conv", 30, 5, 1, 4), ("relu",), ("conv", 4, 4, 4, 0), ("relu",), ("fc", 3)], (1, 28, 28)),
    ([("conv", 23, 3, 1, 0), ("relu",), ("conv", 4, 2, 2, 0), ("relu",), ("fc", 3)], (3, 32, 32)),
    ([("conv", 20, 3, 1, 1), ("relu",), ("conv", 4, 2, 2, 0), ("relu",), ("fc", 3)], (3, 31, 34)),
])
def test_convolution_to_few_channels(Context, layers, shape):
    layers, C, d, lo, hi, prep = _case(dict(seed=71, in_shape=shape, layers=layers), 0.01)
    net, lo_t, hi_t, l, u, S, _, _ = prep
    SD = sum(l[i].numel() for i in l)
    rng = np.random.default_rng(8)
    nodes = [random_node(prep, rng, n_splits=3 * j, row=j % 2) for j in range(2)]
    refs = []
    for on in nodes:
        on.split_layer = net.R
        refs.append(core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, None, lo_t, hi_t))
    with Context(node_capacity=1024, gemm_path=1) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        gids = []
        for on in nodes:
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        for batch in ([0, 1], [j % 2 for j in range(90)], [j % 2 for j in range(400)]):
            lb, ga, gb, _ = ctx.bound_grad([gids[j] for j in batch], SD, 0)
            for i in (0, 1, len(batch) - 1):
                ref, _, oa, ob, _ = refs[batch[i]]
                assert close(lb[i], float(ref)).all(), (batch[i], lb[i], float(ref))
                o = np.concatenate([concat(oa, net.R), concat(ob, net.R)])
                g = np.concatenate([ga[i], gb[i]])
                assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())


# dense products of a few rows (gemm_path 1): widths that are no multiple of four (no
# 16-byte copies), of a tile or of a step of the reduction, reductions shorter than a
# step and than the ring of steps, split reductions with a short last part; one row,
# rows that end inside a tile, and enough for 64 x 64 tiles
@pytest.mark.parametrize("dims", [(13, 9, 5, 3), (50, 129, 70, 4), (64, 304, 68, 3), (31, 515, 257, 6),
                                  (520, 1300, 33, 3)])
def test_dense_products(Context, dims):
    layers = []
    for n in dims[1:]:
        layers += [("fc", n), ("relu",)]
    layers, C, d, lo, hi, prep = _case(dict(seed=81, in_shape=(1, 1, dims[0]), layers=layers[:-1]), 0.02)
    net, lo_t, hi_t, l, u, S, _, _ = prep
    SD = sum(l[i].numel() for i in l)
    rng = np.random.default_rng(9)
    nodes = [random_node(prep, rng, n_splits=2 * j, row=j % 2) for j in range(2)]
    refs = []
    for on in nodes:
        on.split_layer = net.R
        refs.append(core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, None, lo_t, hi_t))
    with Context(node_capacity=4096, gemm_path=1) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        for i in l:
            gl, gu = ctx.root_bounds(prop, i)
            assert close(gl, l[i].numpy()).all() and close(gu, u[i].numpy()).all(), i
        gids = []
        for on in nodes:
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        for batch in ([1], [j % 2 for j in range(45)], [j % 2 for j in range(1000)]):
            lb, ga, gb, _ = ctx.bound_grad([gids[j] for j in batch], SD, 0)
            for i in {0, min(1, len(batch) - 1), len(batch) - 1}:
                ref, _, oa, ob, _ = refs[batch[i]]
                assert close(lb[i], float(ref)).all(), (batch[i], lb[i], float(ref))
                o = np.concatenate([concat(oa, net.R), concat(ob, net.R)])
                g = np.concatenate([ga[i], gb[i]])
                assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())


# gamma terms of rows in groups (from 32 rows on): groups of one property and of
# several, a last group that is not full, a property without constraints among them
@pytest.mark.parametrize("order", ["blocks", "alternating"])
def test_gamma_terms_of_row_groups(Context, order):
    spec = dict(seed=33, in_shape=(1, 5, 5), layers=[("fc", 21), ("relu",), ("fc", 9), ("relu",), ("fc", 3)])
    cases = [_case(spec, 0.05, _rows_per_neuron(5, (300, 1, 40, 0, 229), 3)),
             _case(spec, 0.04, _rows_per_neuron(6, (7, 230), 2)), _case(spec, 0.06)]
    rng = np.random.default_rng(12)
    E = [sum(v.idx.shape[0] for v in (c[5][6] or {}).values()) for c in cases]
    with Context(node_capacity=512, max_mnc_rows=max(E)) as ctx:
        gnet = ctx.load_network(cases[0][0])
        gids, refs = [], []
        for layers, C, d, lo, hi, prep in cases:
            net, lo_t, hi_t, l, u, S, m, dense = prep
            prop = ctx.set_property(gnet, lo, hi, C, d)
            for t in sorted(m or {}):
                ctx.set_mnc(prop, t, m[t].idx, m[t].P, m[t].Ph, m[t].p)
            on = random_node(prep, rng, n_splits=2, row=1)
            on.split_layer = net.R
            refs.append(core.bound_and_grad(net, on, on.alpha, on.beta, on.gamma, dense, lo_t, hi_t))
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        SD = sum(v.numel() for v in l.values())
        which = [0] * 14 + [1] * 15 + [2] * 9 if order == "blocks" else [j % 3 for j in range(39)]
        lb, ga, gb, gg = ctx.bound_grad([gids[j] for j in which], SD, max(E))
        flat, at = np.concatenate([ga, gb, gg], 1).reshape(-1), 0  # a node: alpha, beta, its gammas
        for i, j in enumerate(which):
            ref, _, oa, ob, og = refs[j]
            assert close(lb[i], float(ref)).all(), (i, j, lb[i], float(ref))
            o = np.concatenate([concat(oa, net.R), concat(ob, net.R),
                                *(og[t].numpy() for t in sorted(og or {}))])
            g = flat[at:at + 2 * SD + E[j]]
            at += g.size
            assert np.abs(g - o).max() <= TOL * (1 + np.abs(o).max())


# rows of unstable neurons: a second layer of 8649 neurons (a tile of 8192 and a ragged
# one), of 7 and of 33
@pytest.mark.parametrize("layers,shape", [
    ([("conv", 9, 3, 1, 1), ("relu",), ("conv", 9, 1, 1, 0), ("relu",), ("fc", 3)], (1, 31, 31)),
    ([("fc", 40), ("relu",), ("fc", 7), ("relu",), ("fc", 33), ("relu",), ("fc", 3)], (1, 5, 5)),
])
def test_rows_of_unstable_neurons(Context, layers, shape):
    layers, C, d, lo, hi, prep = _case(dict(seed=91, in_shape=shape, layers=layers), 0.05)
    l, u = prep[3], prep[4]
    with Context(node_capacity=64) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        for i in l:
            gl, gu = ctx.root_bounds(prop, i)
            assert close(gl, l[i].numpy()).all() and close(gu, u[i].numpy()).all(), i


# the fused optimisation loop: FC outputs that give a warp one, two, four and seven
# at a time and more than one round of them, FC inputs that are no multiple of four,
# stride classes of one, two and three taps, planes whose last pair of positions is
# half empty; on both the SIMT (1) and the tensor-core (0) form
@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("layers,shape", [
    ([("fc", 130), ("relu",), ("fc", 65), ("relu",), ("fc", 33), ("relu",), ("fc", 17), ("relu",), ("fc", 3)],
     (1, 5, 6)),
    ([("conv", 6, 5, 2, 2), ("relu",), ("conv", 8, 3, 3, 1), ("relu",), ("fc", 113), ("relu",), ("fc", 4)],
     (1, 13, 11)),
    ([("conv", 8, 3, 1, 1), ("relu",), ("conv", 4, 2, 3, 0), ("relu",), ("fc", 31), ("relu",), ("fc", 3)],
     (2, 9, 7)),
])
def test_fused_optimisation_layers(Context, layers, shape, path):
    layers, C, d, lo, hi, prep = _case(dict(seed=95, in_shape=shape, layers=layers), 0.03)
    net, lo_t, hi_t = prep[:3]
    dense = prep[7]
    rng = np.random.default_rng(13)
    with Context(node_capacity=64, gemm_path=path) as ctx:
        gnet = ctx.load_network(layers)
        prop = ctx.set_property(gnet, lo, hi, C, d)
        nodes = [random_node(prep, rng, n_splits=j, row=j % 2, gamma_scale=0.0) for j in range(4)]
        gids = []
        for on in nodes:
            on.split_layer = net.R
            gids.append(ctx.node_root(prop, on.row))
            ctx.import_params(gids[-1], to_params(on, net.R))
        best = ctx.optimize(gids, steps=5)
        for j, on in enumerate(nodes):
            top, *_ = core.optimize(net, on, dense, lo_t, hi_t, core.AdamHP(steps=5))
            assert close(best[j], top).all(), (j, best[j], top)


def test_autotune_first_thing(Context):
    """Every variant of every layer runs in a context that has launched nothing
    else: layers whose staging takes exactly 48 KB of dynamic shared memory beside
    their kernel's static variables (stride-2 transposed convolutions from 64 x 8 x 8
    and 32 x 16 x 16)."""
    layers = synth.make_network(dict(seed=97, in_shape=(32, 32, 32), layers=[
        ("conv", 32, 4, 2, 1), ("relu",), ("conv", 64, 3, 1, 1), ("relu",), ("conv", 64, 4, 2, 1),
        ("relu",), ("fc", 3)]))
    with Context(node_capacity=512) as ctx:
        net = ctx.load_network(layers)
        recs = ctx.autotune(net, max_rows=64)
        assert recs and all(r["variant"] != "auto" for r in recs)
