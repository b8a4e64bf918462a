"""Which form a ciphertext-diagonal product takes: the integer form for few diagonals, and where the
tensor cores' scratch cannot grow (a stream under capture); the same residues either way."""
import gc

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _setup(n, cols, count):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(13, [60, 40, 40], [60], 3, seed=2)
    rng = np.random.default_rng(n + count)
    W = torch.from_numpy(rng.normal(size=(n, cols))).cuda()
    host = np.stack([rng.integers(0, q, size=(count, 2, ctx.n)) for q in ctx.primes[:3]], axis=2)
    data = torch.from_numpy(np.ascontiguousarray(host)).cuda()
    return he, ctx, W, [he.Ciphertext(data[i], 2, 2.0**40) for i in range(count)]


def _narrow(he, ctx, W, cts):
    outs = []
    for k in range(0, W.shape[1], 4):
        outs += ctx.cdiag_matmult(he.WeightMatrix(ctx, W[:, k : k + 4].contiguous(), 2), cts)
    return outs


@pytest.mark.parametrize("n,count,tensor", [(64, 1, False), (64, 19, False), (64, 20, True), (32, 32, True), (4096, 24, False), (4096, 25, True), (16, 16, False)])
def test_by_diagonals(n, count, tensor):
    import torch

    he, ctx, W, cts = _setup(n, 8, count)
    wm = he.WeightMatrix(ctx, W, 2)
    ctx.synchronize()
    ctx.set_wait_limit(0)  # only the tensor-core form has waits that can give up
    ctx.cdiag_matmult(wm, cts)
    if tensor:
        with pytest.raises(he.HEError) as e:
            ctx.synchronize()
        assert e.value.status == he.HE_ETIMEOUT
    ctx.synchronize()
    ctx.set_wait_limit()
    for g, w in zip(ctx.cdiag_matmult(wm, cts), _narrow(he, ctx, W, cts)):
        assert torch.equal(g.data, w.data)


def test_under_capture_without_the_scratch():
    import torch

    with torch.cuda.stream(torch.cuda.Stream()):
        he, ctx, W, cts = _setup(64, 8, 64)
        wm = he.WeightMatrix(ctx, W, 2)
        want = [c.data.clone() for c in ctx.cdiag_matmult(wm, cts)]
        torch.cuda.synchronize()
        few = ctx.fork()
        outs = [few.new_ct(1) for _ in want]
        few.cdiag_matmult(wm, cts[:19], outs)
        few.synchronize()
        gc.collect()  # contexts of earlier tests, whose release would end the capture
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=few.stream):
            few.cdiag_matmult(wm, cts, outs)
        graph.replay()
        torch.cuda.synchronize()
        for g, w in zip(outs, want):
            assert torch.equal(g.data, w)
