"""Limits of a launch's shared memory: sizes just below 48 KB, which exceed what a launch
may take without leave together with the kernel's static shared memory, and launches that
are refused."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from helpers import close, fc_case
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


# the sweep of dense rows (32 bytes for each neuron of the widest layer: 49,152), the
# optimisation loop (15 bytes a neuron and 4 an input: 49,120) and the pre-attack
# (12 and 4: 49,120), each in a network that no other test loads
@pytest.mark.parametrize("call,dims", [("roots", (20, 1536, 3, 3)), ("optimize", (280, 3200, 3)),
                                       ("attack", (280, 4000, 3))])
def test_just_below_48_kb(Context, call, dims):
    layers, C, d, lo, hi, prep = fc_case(7, dims, 0.02)
    net, lo_t, hi_t, l, u, S, _, dense = prep
    with Context(node_capacity=16) as ctx:
        prop = ctx.set_property(ctx.load_network(layers), lo, hi, C, d)
        if call == "roots":
            for t in l:
                gl, gu = ctx.root_bounds(prop, t)
                assert close(gl, l[t].numpy()).all() and close(gu, u[t].numpy()).all()
        elif call == "optimize":
            best = ctx.optimize([ctx.node_root(prop, 0)], steps=2)
            node = bab.root_node(net, 0, l, u, S, None)
            top, *_ = core.optimize(net, node, dense, lo_t, hi_t, core.AdamHP(steps=2))
            assert close(best[0], top).all()
        else:
            x = ((lo + hi) / 2).astype(np.float32)
            best, _ = ctx.attack(prop, x[None], 1)
            mid = net.forward(torch.as_tensor(x, dtype=lo_t.dtype)[None])[0].numpy()
            assert (best <= mid + 1e-4 * (1 + np.abs(mid))).all() and np.isfinite(best).all()


# a convolution and a dense product on the tensor cores, the fused optimisation loop
@pytest.mark.parametrize("call,path,shape,layers", [
    ("bound", 2, (16, 8, 8), [("conv", 16, 3, 1, 1), ("relu",), ("fc", 3)]),
    ("bound", 2, (40,), [("fc", 72), ("relu",), ("fc", 64), ("relu",), ("fc", 3)]),
    ("optimize", 1, (40,), [("fc", 3000), ("relu",), ("fc", 3)]),
])
def test_refused_launch_is_reported(Context, call, path, shape, layers):
    """An error that is pending on the thread, as a refused launch leaves it, is reported by
    the call whose later launches raise a kernel's shared-memory limit; the next call gives
    the values of a call without it."""
    from paper_2205_00263_gb300 import MnbabError
    layers = synth.make_network(dict(seed=11, in_shape=shape, layers=layers))
    x = np.random.default_rng(3).uniform(0.2, 0.8, int(np.prod(shape))).astype(np.float32)
    C, d = synth.property_rows(0, 3)
    lo, hi = synth.input_box(x, 0.02)
    cudart = ctypes.CDLL("libcudart.so.13")  # the one that the library loaded
    with Context(node_capacity=16, gemm_path=path) as ctx:
        prop = ctx.set_property(ctx.load_network(layers), lo, hi, C, d)
        nodes = [ctx.node_root(prop, r) for r in range(2)]
        start = [ctx.export_params(n) for n in nodes]

        def run():
            for n, p in zip(nodes, start):
                ctx.import_params(n, p)
            pending()
            return ctx.optimize(nodes, steps=2) if call == "optimize" else ctx.bound_batch(nodes)[0]

        pending = lambda: None  # noqa: E731
        want = run()
        pending = lambda: cudart.cudaGetDevice(None)  # noqa: E731
        with pytest.raises(MnbabError):
            run()
        pending = lambda: None  # noqa: E731
        assert (run() == want).all()
