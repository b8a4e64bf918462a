"""The tensor-core ciphertext-diagonal product over primes of every size it accepts (two and three
20-bit digits, 6 to 15 moduli), at the line between the forms in columns, and on a forked context: the
residues of the general form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _setup(qb, pb, dnum, n, cols, count, log_n=12):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(log_n, qb, pb, dnum, seed=6)
    level = len(qb) - 1
    rng = np.random.default_rng(sum(qb) + n + cols + count)
    W = torch.from_numpy(rng.normal(size=(n, cols)) * 2.0 ** rng.integers(-6, 10)).cuda()
    host = np.stack([rng.integers(0, q, size=(count, 2, ctx.n)) for q in ctx.primes[: level + 1]], axis=2)
    host[:, :, :, :32] = np.array(ctx.primes[: level + 1], dtype=np.int64)[None, None, :, None] - 1
    data = torch.from_numpy(np.ascontiguousarray(host)).cuda()
    return he, ctx, W, level, [he.Ciphertext(data[i], level, 2.0**20) for i in range(count)]


def _general(he, ctx, W, level, cts):
    outs = []
    for k in range(0, W.shape[1], 6):
        outs += ctx.cdiag_matmult(he.WeightMatrix(ctx, W[:, k : k + 6].contiguous(), level), cts)
    return outs


@pytest.mark.parametrize("qb", [[30, 25], [39, 35], [41, 42], [45, 30], [47, 49], [50, 45], [53, 51], [55, 57], [59, 58], [60, 59]])
@pytest.mark.parametrize("n,count", [(256, 256), (64, 37)])
def test_prime_sizes(qb, n, count):
    import torch

    he, ctx, W, level, cts = _setup(qb, [60], 2, n, 8, count)
    for g, w in zip(ctx.cdiag_matmult(he.WeightMatrix(ctx, W, level), cts), _general(he, ctx, W, level, cts)):
        assert torch.equal(g.data, w.data)


def test_columns_at_the_line():
    import torch

    he, ctx, W, level, cts = _setup([60, 40, 40], [60], 3, 128, 8, 100, log_n=13)
    want = _general(he, ctx, W, level, cts)
    for cols in (7, 8):
        got = ctx.cdiag_matmult(he.WeightMatrix(ctx, W[:, :cols].contiguous(), level), cts)
        for g, w in zip(got[:6], want):  # the encoder pairs columns: the seventh alone rounds by itself
            assert torch.equal(g.data, w.data)


def test_on_a_fork():
    import torch

    he, ctx, W, level, cts = _setup([50, 40], [60], 2, 64, 9, 64)
    want = _general(he, ctx, W, level, cts)
    wm = he.WeightMatrix(ctx, W, level)
    torch.cuda.synchronize()
    fork = ctx.fork()
    with torch.cuda.stream(fork.stream):
        own = he.WeightMatrix(fork, W, level)
        both = [fork.cdiag_matmult(wm, cts), fork.cdiag_matmult(own, cts)]
    fork.synchronize()
    both.append(ctx.cdiag_matmult(own, cts))
    for got in both:
        for g, w in zip(got, want):
            assert torch.equal(g.data, w.data)
