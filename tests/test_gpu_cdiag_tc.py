"""The tensor-core form of the ciphertext-diagonal product (weights of at least 8 columns) against
the general form (fewer columns): the same residues, bit for bit, over rings, levels, weight periods
around the tile's block sizes, diagonal counts around the launch's 256, and column counts around the
instruction's 128; residues and weights that fill the primes' whole range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RINGS = {12: ([40, 20], [40], 2), 13: ([60, 40, 40], [60], 3), 14: ([60] + [40] * 6, [60, 60, 60], 3)}


@pytest.fixture(scope="module")
def he():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he as h

    return h


_CTX = {}


def _ctx(he, log_n):
    if log_n not in _CTX:
        qb, pb, dnum = RINGS[log_n]
        _CTX[log_n] = he.Context(log_n, qb, pb, dnum, seed=3)
    return _CTX[log_n]


def _cts(he, ctx, count, level, rng, top=False):
    import torch

    out = []
    for _ in range(count):
        d = np.empty((2, level + 1, ctx.n), dtype=np.int64)
        for l in range(level + 1):
            q = ctx.primes[l]
            d[:, l] = q - 1 if top else rng.integers(0, q, size=(2, ctx.n))
        out.append(he.Ciphertext(torch.from_numpy(d).cuda(), level, 2.0**40))
    return out


def _general(he, ctx, W, cts, level):
    outs = []
    for k in range(0, W.shape[1], 6):  # an even count: the encoder pairs neighbouring columns
        outs += ctx.cdiag_matmult(he.WeightMatrix(ctx, W[:, k:k + 6].contiguous(), level), cts)
    return outs


# (log N, level, weight rows n, diagonals, columns)
CASES = [(12, 1, 8, 8, 8), (12, 1, 64, 3, 9), (12, 1, 2048, 65, 8), (13, 2, 128, 128, 17), (13, 1, 256, 255, 127), (13, 2, 4096, 257, 129),
         (14, 6, 8, 1, 8), (14, 6, 256, 256, 130), (14, 3, 512, 300, 12), (14, 2, 4096, 256, 40), (14, 1, 8192, 1024, 8), (14, 6, 16, 16, 8)]


@pytest.mark.parametrize("log_n,level,n,count,cols", CASES)
def test_same_residues_as_general_form(he, log_n, level, n, count, cols):
    import torch

    ctx = _ctx(he, log_n)
    rng = np.random.default_rng(log_n * 1000 + n + count + cols)
    cts = _cts(he, ctx, count, level, rng)
    W = torch.from_numpy(rng.normal(size=(n, cols)) * 2.0 ** rng.integers(-8, 16)).cuda()
    got = ctx.cdiag_matmult(he.WeightMatrix(ctx, W, level), cts)
    for g, w in zip(got, _general(he, ctx, W, cts, level)):
        assert g.level == w.level and g.scale == w.scale
        assert torch.equal(g.data, w.data)


@pytest.mark.parametrize("log_n,n,count", [(13, 256, 256), (14, 1024, 256)])
def test_largest_residues(he, log_n, n, count):
    """Every ciphertext residue q - 1, constant weights of either sign: the largest sums."""
    import torch

    ctx = _ctx(he, log_n)
    rng = np.random.default_rng(5)
    level = len(RINGS[log_n][0]) - 1
    cts = _cts(he, ctx, count, level, rng, top=True)
    W = torch.full((n, 9), 0.5, dtype=torch.float64)
    W[:, 1] = -0.5
    W[:, 2] = 0.25
    W[:, 3] = -0.499999
    W[:, 4] = 2.0**19
    W[::2, 5] = -0.5
    W = W.cuda()
    got = ctx.cdiag_matmult(he.WeightMatrix(ctx, W, level), cts)
    for g, w in zip(got, _general(he, ctx, W, cts, level)):
        assert torch.equal(g.data, w.data)
