"""One context per host thread: two threads whose networks take the same kernels with
different amounts of shared memory, each as if it were alone.  The shared-memory limit of
a kernel belongs to the device, not to a context."""
import threading

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

CALLS = 10000


@pytest.fixture(scope="module")
def Context():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00263_gb300 import Context
    return Context


def _calls(Context, spec, gemm_path, fused, calls, go=lambda i: True):
    """The values of `calls` calls that re-bound a root node and bound it (and optimise and
    attack it), which are all the same; go(i): whether to make call i."""
    layers = synth.make_network(spec)
    x = synth.make_image(spec["seed"], spec["in_shape"]).reshape(-1)
    lo, hi = synth.input_box(x, 0.02)
    C, d = synth.property_rows(0, 3)
    first = None
    with Context(node_capacity=16, gemm_path=gemm_path) as ctx:
        net = ctx.load_network(layers)
        prop = ctx.set_property(net, lo, hi, C, d)
        node = ctx.node_root(prop, 0)
        start = ctx.export_params(node)
        start.split_layer = 1  # the layers above are bounded again
        for i in range(calls):
            if not go(i):
                break
            ctx.import_params(node, start)
            got = list(ctx.bound_batch([node]))
            if fused:
                got += [ctx.optimize([node], steps=1), ctx.attack(prop, np.stack([lo, hi]), 1)[0]]
            got = np.concatenate([np.ravel(g) for g in got])
            first = got if first is None else first
            assert (got == first).all(), (i, got, first)
    return first


# a pair of networks: the first one's launches take more than the second one's limit
@pytest.mark.parametrize("gemm_path,fused,large,small", [
    # tensor-core convolutions: 73 KB (64 channels, a reduction of 1024) and 17 KB
    pytest.param(2, False, dict(seed=3, in_shape=(64, 6, 6), layers=[("conv", 64, 4, 2, 1), ("relu",), ("fc", 3)]),
                 dict(seed=4, in_shape=(8, 6, 6), layers=[("conv", 9, 3, 1, 1), ("relu",), ("fc", 3)]),
                 id="tensor_core_convolutions"),
])
def test_two_threads(Context, gemm_path, fused, large, small):
    alone = [_calls(Context, s, gemm_path, fused, 1) for s in (large, small)]
    failed, ready = [], threading.Barrier(2)

    def run(spec, want):
        try:
            got = _calls(Context, spec, gemm_path, fused, CALLS,
                         lambda i: not failed and (i > 0 or ready.wait(60) >= 0))
            assert failed or (got == want).all(), (got, want)
        except BaseException as e:  # noqa: BLE001 - handed to the test's thread
            failed.append(e)
            ready.abort()

    threads = [threading.Thread(target=run, args=v) for v in zip((large, small), alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]
