"""MatMults of two and more row blocks take them in pairs that share a step's key product: the same
ciphertexts as the row blocks one by one (a pinned loop-kernel variant), for one to four digits, two and
four row blocks, one and two column blocks and both ends of the diagonal counts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# ring, Q and P bits, digits
RINGS = {
    "n1024-3": (10, [60, 40, 40], [60], 3),
    "n4096-2": (12, [40, 20], [40], 2),
    "n8192-3": (13, [60, 40, 40], [60], 3),
    "n8192-2": (13, [60, 40, 40], [60, 60], 2),
    "n16384-4": (14, [60, 40, 40, 40], [60], 4),
}


@pytest.mark.parametrize("ring", sorted(RINGS))
@pytest.mark.parametrize("shape", ["2Sx2", "2S+1x5", "3Sx37", "4Sx130", "2SxS+3"])
def test_row_pairs(ring, shape):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    log_n, qb, pb, dnum = RINGS[ring]
    ctx = he.Context(log_n, qb, pb, dnum, seed=4)
    S = ctx.slots
    m, n = {"2Sx2": (2 * S, 2), "2S+1x5": (2 * S + 1, 5), "3Sx37": (3 * S, 37), "4Sx130": (4 * S, 130), "2SxS+3": (2 * S, S + 3)}[shape]
    if shape == "2SxS+3" and log_n != 10:
        pytest.skip("two column blocks on the smallest ring")
    plan = he.Plan(m, n, S)
    assert plan.row_blocks >= 2
    ctx.keygen(list(range(1, plan.m_prime)))
    rng = np.random.default_rng(m + n)
    X, y = rng.normal(size=(m, n)), rng.uniform(-1, 1, n)
    scale = 2.0**20 if log_n == 12 else 2.0**40
    for level in range(1, len(qb)):
        pm = ctx.encode_matrix(plan, torch.from_numpy(X).cuda(), level)
        cts = ctx.encrypt_vector(plan, torch.from_numpy(y).cuda(), scale, level, 5)
        first = ctx.matmult(plan, pm, cts)  # unfused: row blocks in pairs, up to three digits
        again = ctx.matmult(plan, pm, cts)  # the same, or the fused key tables where they are faster
        counts = []
        pm.set_key_fusion(False)
        for pin in (False, True):
            if pin:
                pm.set_variant(0)
            n0 = ctx.launch_count()
            ones = ctx.matmult(plan, pm, cts)
            counts.append(ctx.launch_count() - n0)
        digits = -(-(level + 1) // -(-len(qb) // dnum))
        saved = plan.row_blocks // 2 * plan.col_blocks if digits <= 3 else 0
        assert counts[1] - counts[0] == saved
        for a, b, w in zip(first, again, ones):
            assert a.level == b.level == w.level and a.scale == b.scale == w.scale
            assert torch.equal(a.data, w.data) and torch.equal(b.data, w.data)
