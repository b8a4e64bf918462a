"""The two-phase transform's unreduced inputs (signed coefficients lifted by a multiple of the prime,
reduced only past 2^60) and its folds at the end: the encoded matrix equals the one-CTA form's, which
reduces its inputs, at every magnitude of the coefficients and for primes of every class."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,qb,pb,dnum", [(12, [40, 20], [40], 2), (13, [60, 40, 40], [60], 3), (13, [59, 58, 41, 30], [57], 4), (14, [60] + [40] * 6, [60, 60, 60], 3)])
@pytest.mark.parametrize("mag", [0, 10, 18, 21, 30])
def test_encoded_matrix_same_in_both_forms(log_n, qb, pb, dnum, mag):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(log_n, qb, pb, dnum, seed=2)
    rng = np.random.default_rng(mag)
    plan = he.Plan(32, ctx.slots, ctx.slots)
    X = rng.normal(size=(32, ctx.slots))
    X[::3] = np.abs(X[::3])  # a large mean: one large coefficient
    X[1::3] = -np.abs(X[1::3])
    X = torch.from_numpy(X * 2.0**mag).cuda()
    got = []
    for form in (0, 2):
        ctx.set_ntt_form(form)
        got.append(ctx.encode_matrix(plan, X, len(qb) - 1).export())
    assert torch.equal(got[0], got[1])
