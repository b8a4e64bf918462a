"""Decryption and decode in one launch: the doubles of the separate launches, which a product of more
row blocks than the fused launch takes (17 and more) still runs; both epilogues (slots, and the lazy
rotate-and-sum of he_matmult_decrypt with and without a mask), every ring with clusters, mixed levels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n", [10, 11, 12, 13, 14])
@pytest.mark.parametrize("n", [1, 6, 300])
def test_decrypt_fused(log_n, n):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(log_n, [60, 40, 40], [60], 3, seed=4)
    S = ctx.slots
    rng = np.random.default_rng(log_n)
    z = torch.from_numpy(rng.normal(size=(32, S))).cuda()
    cts = [ctx.encrypt(ctx.encode(z[r], 2.0**40, r % 3), r) for r in range(32)]
    slots = torch.empty((32, S), dtype=torch.float64, device="cuda")
    for r, c in enumerate(cts):
        ctx.decrypt(c, slots[r])
    assert (slots - z).abs().max().item() < 1e-4
    for blocks in (1, 2, 16, 32):
        plan = he.Plan(blocks * S, n, S)
        assert plan.row_blocks == blocks
        for mask in (None, z[:blocks].flip(1).contiguous()):
            separate = ctx.matmult_decode(plan, slots[:blocks], mask=mask)
            assert torch.equal(ctx.matmult_decrypt(plan, cts[:blocks], mask=mask), separate)
