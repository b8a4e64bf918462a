"""The tensor-core ciphertext-diagonal product in several passes over the diagonals, on chains of 40-bit
primes, whose short last pass takes more operand scratch than a full one: the residues of the general
form (fewer columns), from a context whose scratch no earlier call has grown."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,qb,pb,dnum,n,count", [(12, [40, 20], [40], 2, 512, 449), (14, [40] * 7, [40, 40, 40], 3, 512, 300),
                                                      (13, [50, 40, 40], [60], 3, 1024, 545)])
def test_same_residues_as_general_form(log_n, qb, pb, dnum, n, count):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    level = len(qb) - 1
    ctx, ref = he.Context(log_n, qb, pb, dnum, seed=3), he.Context(log_n, qb, pb, dnum, seed=3)
    rng = np.random.default_rng(count)
    W = torch.from_numpy(rng.normal(size=(n, 8))).cuda()
    wm = he.WeightMatrix(ctx, W, level)
    host = np.stack([rng.integers(0, q, size=(count, 2, ctx.n)) for q in ctx.primes[: level + 1]], axis=2)
    data = torch.from_numpy(np.ascontiguousarray(host)).cuda()
    cts = [he.Ciphertext(data[i], level, 2.0**20) for i in range(count)]
    got = ctx.cdiag_matmult(wm, cts)
    for k in (0, 4):
        want = ref.cdiag_matmult(he.WeightMatrix(ref, W[:, k : k + 4].contiguous(), level), cts)
        for g, w in zip(got[k : k + 4], want):
            assert torch.equal(g.data, w.data)
