"""MatMults of one diagonal (m n <= N/2, or one column): the product and its rescale run in one launch
and their matrix is encoded straight from X; the same ciphertexts as the separate launches of
he_matmult_plain_cipher_noalloc, for every level and row-block count, and X y after decryption."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RINGS = {10: ([60, 40, 40], [60], 3), 12: ([40, 20], [40], 2), 13: ([60, 40, 40], [60], 3), 14: ([60] + [40] * 6, [60, 60, 60], 3)}


@pytest.mark.parametrize("log_n", sorted(RINGS))
@pytest.mark.parametrize("shape", ["16x13", "1xS", "2Sx1", "one"])
def test_one_diagonal(log_n, shape):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    qb, pb, dnum = RINGS[log_n]
    ctx = he.Context(log_n, qb, pb, dnum, seed=4)
    m, n = {"16x13": (16, 13), "1xS": (1, ctx.slots), "2Sx1": (2 * ctx.slots, 1), "one": (1, 1)}[shape]
    plan = he.Plan(m, n, ctx.slots)
    assert plan.m_prime == 1 and plan.col_blocks == 1
    rng = np.random.default_rng(m + n)
    X, y = rng.normal(size=(m, n)), rng.uniform(-1, 1, n)
    scale = 2.0**20 if log_n == 12 else 2.0**40
    for level in range(1, len(qb)):
        pm = ctx.encode_matrix(plan, torch.from_numpy(X).cuda(), level)
        cts = ctx.encrypt_vector(plan, torch.from_numpy(y).cuda(), scale, level, 5)
        outs = ctx.matmult(plan, pm, cts)
        want = ctx.matmult_noalloc(plan, pm, cts, [ctx.new_ct(level - 1) for _ in range(plan.row_blocks)])
        for g, w in zip(outs, want):
            assert g.level == w.level and g.scale == w.scale and torch.equal(g.data, w.data)
        if level == len(qb) - 1:
            # scale 2^20: noise near 1e-3 per slot, summed over the n slots of an output (at most 2048)
            tol = 5e-2 * max(1.0, np.sqrt(n / 64)) if log_n == 12 else 1e-4
            assert np.abs(ctx.matmult_decrypt(plan, outs).cpu().numpy() - X @ y).max() < tol
