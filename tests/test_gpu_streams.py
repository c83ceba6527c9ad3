"""Contexts on their own CUDA streams, advanced concurrently (the oblique
rotator's inclination sweep runs one context per inclination this way):
every context owns its device memory, step graph and scratch, so interleaved
launches on several streams give bit-for-bit the states of each context
advanced alone."""
import math

import numpy as np
import pytest

import ffe_workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ffe():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2404_01531_gb300 import ffe
    ffe.load()
    return ffe


def test_concurrent_contexts_on_their_own_streams_equal_sequential_runs(ffe):
    cfgs = [W.pulsar(r_lc=5.0, chi=math.radians(c), n_ang=2, n_rad=4, P=5, r_out=20.0) for c in (0.0, 60.0, 90.0)]
    alone = []
    for cfg in cfgs:
        ctx = ffe.Context(cfg)
        ctx.set_initial()
        ctx.step(12)
        alone.append(ctx.download())
        assert ctx.status() == 0
        ctx.close()
    streams = [torch.cuda.Stream() for _ in cfgs]
    ctxs = [ffe.Context(cfg, stream=s) for cfg, s in zip(cfgs, streams)]
    for c in ctxs:
        c.set_initial()
    for _ in range(4):
        for c in ctxs:
            c.step(3)
    torch.cuda.synchronize()
    for c, (U, m) in zip(ctxs, alone):
        Uc, mc = c.download()
        assert c.status() == 0
        assert np.array_equal(mc, m)
        assert np.array_equal(Uc, U)
        c.close()


def test_step_captured_by_the_caller(ffe):
    """A caller that captures the context's stream gets the step's launches themselves, also from a
    context that has its own step graph: replays advance the state as steps do."""
    cfg = W.pulsar(r_lc=5.0, chi=math.radians(60.0), n_ang=2, n_rad=4, P=5, r_out=20.0)
    s = torch.cuda.Stream()
    own, ref = ffe.Context(cfg, stream=s), ffe.Context(cfg, stream=s)
    for c in (own, ref):
        c.set_initial()
        c.step(4)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
        own.step(1)
    with torch.cuda.stream(s):
        for _ in range(3):
            g.replay()
    ref.step(3)
    torch.cuda.synchronize()
    (Ua, ma), (Ub, mb) = own.download(), ref.download()
    assert np.array_equal(ma, mb) and np.array_equal(Ua, Ub)
    assert own.status() == 0
    for c in (own, ref):
        c.close()
