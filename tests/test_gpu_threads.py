"""One context per host thread: two threads whose networks take the same kernels with
different amounts of shared memory, each as if it were alone.  The shared-memory limit of
a kernel belongs to the device, not to a context."""
import threading

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

@pytest.fixture(scope="module")
def Context():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00263_gb300 import Context
    return Context


def _calls(Context, spec, gemm_path, nodes, fused, calls, go=lambda i: True):
    """The values of `calls` calls that re-bound root nodes, two rows a launch, and bound
    them (and optimise and attack), which are all the same; go(i): whether to make call i."""
    layers = synth.make_network(spec)
    x = np.random.default_rng(spec["seed"]).uniform(0.2, 0.8, spec["in_shape"]).reshape(-1)
    lo, hi = synth.input_box(x, 0.05)
    C, d = synth.property_rows(0, 3)
    first = None
    with Context(node_capacity=32, gemm_path=gemm_path, row_chunk=2) as ctx:
        net = ctx.load_network(layers)
        prop = ctx.set_property(net, lo, hi, C, d)
        ids = [ctx.node_root(prop, 0) for _ in range(nodes)]
        start = ctx.export_params(ids[0])
        start.split_layer = 1  # the layers above are bounded again
        for i in range(calls):
            if not go(i):
                break
            for n in ids:
                ctx.import_params(n, start)
            got = list(ctx.bound_batch(ids))
            if fused:
                got += [ctx.optimize(ids, steps=1), ctx.attack(prop, np.stack([lo, hi]), 1)[0]]
            got = np.concatenate([np.ravel(g) for g in got])
            first = got if first is None else first
            assert (got == first).all(), (i, got, first)
    return first


# a pair of networks: the first one's launches take more than the second one's limit
@pytest.mark.parametrize("gemm_path,nodes,fused,calls,large,small", [
    # tensor-core convolutions: 73 KB (64 channels, a reduction of 1024) and 17 KB
    pytest.param(2, 1, False, 10000, dict(seed=3, in_shape=(64, 6, 6), layers=[("conv", 64, 4, 2, 1), ("relu",), ("fc", 3)]),
                 dict(seed=4, in_shape=(8, 6, 6), layers=[("conv", 9, 3, 1, 1), ("relu",), ("fc", 3)]),
                 id="tensor_core_convolutions"),
    # windowed rows: 209 KB (four rows of 54 x 54 values of 4 channels and 12 x 12 of 12)
    # and 81 KB
    pytest.param(1, 8, False, 200, dict(seed=5, in_shape=(4, 54, 54), layers=[("conv", 12, 10, 4, 0), ("relu",),
                                                                      ("conv", 16, 12, 1, 0), ("relu",), ("fc", 3)]),
                 dict(seed=6, in_shape=(4, 34, 34), layers=[("conv", 12, 10, 4, 0), ("relu",), ("conv", 16, 7, 1, 0),
                                                            ("relu",), ("fc", 3)]),
                 id="windowed_rows"),
    # fused kernels: dense-row sweeps (198 and 134 KB), the optimisation loop (93 and 63 KB)
    # and the pre-attack (74 and 50 KB)
    pytest.param(0, 2, True, 60, dict(seed=7, in_shape=(30,), layers=[("fc", 6200), ("relu",), ("fc", 64), ("relu",),
                                                                        ("fc", 3)]),
                 dict(seed=8, in_shape=(30,), layers=[("fc", 4200), ("relu",), ("fc", 64), ("relu",), ("fc", 3)]),
                 id="fused_kernels"),
])
def test_two_threads(Context, gemm_path, nodes, fused, calls, large, small):
    alone = [_calls(Context, s, gemm_path, nodes, fused, 1) for s in (large, small)]
    failed, ready = [], threading.Barrier(2)

    def run(spec, want):
        try:
            got = _calls(Context, spec, gemm_path, nodes, fused, calls,
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
