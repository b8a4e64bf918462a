"""he_rotate_many where the scratch for 128 rotations cannot be had: the same ciphertexts in smaller
chunks, on a stream under capture whose scratch was warmed by 64 rotations, and with little device
memory left."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _setup(log_n, qb, pb, dnum, count, seed):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(log_n, qb, pb, dnum, seed=seed)
    steps = [1 + i % 3 for i in range(count)]
    ctx.keygen([1, 2, 3])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    low = min(ctx.primes[: len(qb)])
    cts = [he.Ciphertext(torch.randint(0, low, (2, len(qb), ctx.n), generator=g, device="cuda"), len(qb) - 1, 2.0**40) for _ in range(count)]
    return he, ctx, steps, cts


@pytest.mark.parametrize("warm", [64, 40])
def test_under_capture(warm):
    import torch

    with torch.cuda.stream(torch.cuda.Stream()):
        he, ctx, steps, cts = _setup(13, [60, 40, 40], [60], 3, 131, 7)
        ctx.rotate_many(cts[:warm], steps[:warm])
        outs = [ctx.new_ct(2) for _ in cts]
        ctx.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=ctx.stream):
            ctx.rotate_many(cts, steps, outs)
        graph.replay()
        torch.cuda.current_stream().synchronize()
        for g, c, s in zip(outs, cts, steps):
            assert torch.equal(g.data, ctx.rotate(c, s).data)


def test_with_little_memory():
    import torch

    he, ctx, steps, cts = _setup(14, [60] + [40] * 15, [60] * 4, 4, 100, 9)
    outs = [ctx.new_ct(15) for _ in cts]
    one = ctx.rotate(cts[0], 1)  # loads the code of the single rotation too
    n = ctx.n
    each = 8 * n * (16 + 4 * 20 + 2 * 4 + 2 * 16)  # scratch words of one rotation: c1, ModUp digits, ModDown
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    ballast = torch.empty(free - 80 * each, dtype=torch.uint8, device="cuda")  # holds 64 rotations, not 100
    ctx.rotate_many(cts, steps, outs)
    ctx.synchronize()
    del ballast
    torch.cuda.empty_cache()
    assert torch.equal(outs[0].data, one.data)
    for g, c, s in zip(outs, cts, steps):
        assert torch.equal(g.data, ctx.rotate(c, s).data)
