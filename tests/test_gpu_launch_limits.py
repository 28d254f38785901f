"""Launches whose dynamic shared memory is just below 48 KB: with the kernel's static
shared memory they exceed what a launch may take without leave."""
import numpy as np
import pytest
import torch

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
