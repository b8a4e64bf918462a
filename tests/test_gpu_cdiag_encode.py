"""The diagonal plaintexts of he_cdiag_encode_matrix, whose transforms run as one pair of launches over
a table of outputs: every limb is the transform of the same integer coefficients (the inverse and
forward transforms of he_pt_export / he_pt_import are other kernels), for diagonal counts around a
table's 256 outputs and around the cluster form's limit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RINGS = {11: ([60, 40], [60], 2), 12: ([40, 20], [40], 2), 13: ([60, 40, 40], [60], 3), 14: ([60] + [40] * 6, [60, 60, 60], 3)}


@pytest.mark.parametrize("log_n,m,n", [(11, 32, 64), (12, 16, 32), (12, 512, 512), (12, 64, 2048), (13, 256, 512), (14, 4, 4), (14, 8192, 16), (14, 16, 8192)])
def test_limbs_transform_the_same_coefficients(log_n, m, n):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    qb, pb, dnum = RINGS[log_n]
    ctx = he.Context(log_n, qb, pb, dnum, seed=1)
    rng = np.random.default_rng(m + n)
    level, scale = len(qb) - 1, 2.0**20 if log_n == 12 else 2.0**35
    pts = ctx.cdiag_encode_matrix(torch.from_numpy(rng.uniform(-1, 1, (m, n))).cuda(), scale, level)
    assert len(pts) == min(m, n)
    for p in pts:
        coef = ctx.pt_export(p)
        assert torch.equal(ctx.pt_import(coef, level, scale).data, p.data)
        c = he.as_u64(coef)
        q = [int(v) for v in ctx.primes[: level + 1]]
        signed = np.where(c[0] > q[0] // 2, c[0].astype(np.int64) - np.int64(q[0]), c[0].astype(np.int64))
        assert np.abs(signed).max() > 0
        for l in range(1, level + 1):
            assert np.array_equal(np.mod(signed, np.int64(q[l])).astype(np.uint64), c[l])
