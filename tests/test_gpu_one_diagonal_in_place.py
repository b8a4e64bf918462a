"""MatMult of one diagonal with an output in its input's buffer: the same ciphertexts as into separate
buffers, for every level, with the output at the buffer's start and at its end, and with two row blocks
(the second output in place)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RINGS = {10: ([60, 40, 40], [60], 3), 12: ([40, 20], [40], 2), 13: ([60, 40, 40], [60], 3), 14: ([60] + [40] * 6, [60, 60, 60], 3)}


@pytest.mark.parametrize("log_n", sorted(RINGS))
@pytest.mark.parametrize("rows", [1, 2])
def test_output_in_the_inputs_buffer(log_n, rows):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    qb, pb, dnum = RINGS[log_n]
    ctx = he.Context(log_n, qb, pb, dnum, seed=4)
    m, n = (16, 13) if rows == 1 else (2 * ctx.slots, 1)
    plan = he.Plan(m, n, ctx.slots)
    assert plan.m_prime == 1 and plan.col_blocks == 1 and plan.row_blocks == rows
    rng = np.random.default_rng(log_n)
    X, y = torch.from_numpy(rng.normal(size=(m, n))).cuda(), torch.from_numpy(rng.uniform(-1, 1, n)).cuda()
    for level in range(1, len(qb)):
        pm = ctx.encode_matrix(plan, X, level)
        (ct,) = ctx.encrypt_vector(plan, y, 2.0**20, level, 5)
        want = [w.data.clone() for w in ctx.matmult(plan, pm, [ct])]
        words = 2 * level * ctx.n
        for at in (0, ct.data.numel() - words):
            buf = ct.data.reshape(-1).clone()
            outs = [he.Ciphertext(torch.empty_like(want[0]), level - 1, 0.0) for _ in range(rows - 1)]
            outs.append(he.Ciphertext(buf[at : at + words].view(2, level, ctx.n), level - 1, 0.0))
            ctx.matmult(plan, pm, [he.Ciphertext(buf.view_as(ct.data), level, ct.scale)], outs)
            for g, w in zip(outs, want):
                assert torch.equal(g.data, w)
