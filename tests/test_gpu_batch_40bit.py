"""The batch's accumulators for 40-bit primes: the ciphertexts of single products (whose loop keeps the
general ones), for one to three digits, primes near and far from 2^40 in one ring, every staged loop
variant, the longest plan of the ring and operands at the top of their range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RINGS = {"n1024-3": (10, [60, 40, 40], [60], 3), "n1024-2": (10, [40, 40, 40, 40], [40, 40], 2),
         "n1024-1": (10, [40, 40], [40, 40], 1), "n16384-3": (14, [60] + [40] * 6, [60, 60, 60], 3)}


@pytest.mark.parametrize("ring", sorted(RINGS))
@pytest.mark.parametrize("top", [False, True])
def test_batch_40bit(ring, top):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    log_n, qb, pb, dnum = RINGS[ring]
    ctx = he.Context(log_n, qb, pb, dnum, seed=4)
    S, level = ctx.slots, ctx.L - 1
    shapes = [(S, S), (2, S), (37, 9)] if log_n == 10 else [(64, 100), (5, 3)]
    rng = np.random.default_rng(7)
    plans, pms, cts = [], [], []
    for i, (m, n) in enumerate(shapes):
        plan = he.Plan(m, n, S)
        ctx.keygen(list(range(1, plan.m_prime)))
        plans.append(plan)
        pms.append(ctx.encode_matrix(plan, torch.from_numpy(rng.normal(size=(m, n))).cuda(), level))
        ct = ctx.encrypt_vector(plan, torch.from_numpy(rng.uniform(-1, 1, n)).cuda(), 2.0**30, level, 5 + i)[0]
        if top:  # every residue of both components q - 1
            q = torch.tensor(ctx.primes[: level + 1], dtype=torch.int64, device="cuda")
            ct.data.copy_((q - 1).view(1, -1, 1).expand(2, -1, ctx.n).reshape(ct.data.shape))
        cts.append(ct)
    want = [ctx.matmult(p, pm, [c])[0] for p, pm, c in zip(plans, pms, cts)]
    batch = he.Batch(ctx, plans, pms)
    for v in (4, 5, 6, 7):
        batch.set_variant(v)
        for o, w in zip(batch.run(cts), want):
            assert o.level == w.level and torch.equal(o.data, w.data)
