"""Node pools that are too small: a call that finds too few slots is refused with
MNBAB_E_BUDGET and leaves every property's open nodes open, so that later calls end as
in a large pool."""
import numpy as np
import pytest
import torch

from helpers import fc_case

pytestmark = pytest.mark.gpu

STEPS = 3
ROWS = 3


@pytest.fixture(scope="module")
def Context():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00263_gb300 import Context
    return Context


def _property(ctx, net, case):
    _, C, d, lo, hi, _ = case
    return ctx.set_property(net, lo, hi, C, d)


def _refused(call):
    from paper_2205_00263_gb300 import _lib as L
    from paper_2205_00263_gb300.api import MnbabError
    with pytest.raises(MnbabError) as e:
        call()
    assert e.value.code == L.E_BUDGET


def _key(ctx, prop):
    return [(r["seq"], r["row"], r["verdict"], r["split_layer"], r["split_neuron"], r["lb"])
            for r in ctx.trace(prop)]


def _case():
    """Falsified by the oracle at its 16th node; every row's root node branches."""
    return fc_case(38, (10, 16, 12, ROWS + 1), 0.15)


@pytest.mark.parametrize("refused_by", ["step", "bounds"])
def test_refused_start_leaves_the_started_ones(Context, refused_by):
    """The third property's start finds a slot for its root but not for its row root
    nodes, and takes none; the two started before it keep theirs."""
    case = _case()
    with Context(node_capacity=1 + 2 * (ROWS + 1) + ROWS) as ctx, Context(node_capacity=256) as big:
        net, ref_net = ctx.load_network(case[0]), big.load_network(case[0])
        a, b, c = (_property(ctx, net, case) for _ in range(3))
        ref = _property(big, ref_net, case)
        if refused_by == "step":
            _refused(lambda: ctx.bab_step([a, b, c], max_nodes=1, steps=STEPS))
        else:
            _refused(lambda: ctx.root_bounds(a, 1))
        assert ctx.queue_size(c) == 0
        big.bab_step([ref], max_nodes=1, steps=STEPS)
        for p in (a, b):
            ctx.bab_step([p], max_nodes=1, steps=STEPS)
            assert _key(ctx, p) == _key(big, ref) and len(_key(ctx, p)) == 1
            assert ctx.queue_size(p) == big.queue_size(ref) == ROWS + 1
        _refused(lambda: ctx.bab_step([c], max_nodes=1, steps=STEPS))
        assert ctx.queue_size(c) == 0 and _key(ctx, c) == []


def test_refused_children_leave_their_nodes_open(Context):
    """A step whose nodes branch finds room for one child: its nodes are open again and
    nothing is decided.  With room the property ends as in a large pool (falsified, where
    a queue that had lost its nodes read as verified)."""
    case = _case()
    cap = 64
    with Context(node_capacity=cap) as ctx, Context(node_capacity=256) as big:
        net, ref_net = ctx.load_network(case[0]), big.load_network(case[0])
        a, ref = _property(ctx, net, case), _property(big, ref_net, case)
        extra = [ctx.node_root(a, 0) for _ in range(cap - 1 - (ROWS + 1) - 1)]
        _refused(lambda: ctx.bab_step([a], max_nodes=ROWS, steps=STEPS))
        assert ctx.queue_size(a) == ROWS and _key(ctx, a) == []
        assert ctx.status(a)[0] == 0
        assert [ctx.verdict(a, r)[0] for r in range(-1, ROWS)] == [0] * (ROWS + 1)
        for n in extra:
            ctx.node_free(n)
        for c, p in ((ctx, a), (big, ref)):
            while c.bab_step([p], max_nodes=ROWS, steps=STEPS)["nodes_bounded"]:
                pass
        assert ctx.verdict(a)[0] == big.verdict(ref)[0] == -1
        seqs = [k[0] for k in _key(ctx, a)]
        assert seqs == sorted(seqs) and seqs[:ROWS] == list(range(ROWS))
