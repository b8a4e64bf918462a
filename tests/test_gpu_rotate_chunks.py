"""he_rotate_many over its chunks (128 rotations) and transforms: every NTT form and key-switch variant
gives the residues of single rotations, at the largest conversion (four primes per digit, four special
primes, all near 2^60) and with the primes of the parameter sets."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,qb,pb,dnum,count", [(12, [60] * 8, [60] * 4, 2, 33), (12, [59] * 4 + [58] * 4, [59] * 4, 2, 17), (13, [60, 40, 40], [60], 3, 131),
                                                    (14, [60] + [40] * 6, [60, 60, 60], 3, 12)])
def test_forms_match_single_rotations(log_n, qb, pb, dnum, count):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(log_n, qb, pb, dnum, seed=7)
    rng = np.random.default_rng(count)
    level = len(qb) - 1
    cts = []
    for _ in range(count):
        d = np.stack([rng.integers(0, ctx.primes[l], size=(2, ctx.n)) for l in range(level + 1)], axis=1)
        d[:, :, :64] = np.array(ctx.primes[: level + 1], dtype=np.int64)[None, :, None] - 1
        cts.append(he.Ciphertext(torch.from_numpy(np.ascontiguousarray(d)).cuda(), level, 2.0**40))
    steps = [int(s) for s in rng.integers(1, ctx.slots, size=count)]
    ctx.keygen(sorted(set(steps)))
    want = [ctx.rotate(c, s) for c, s in zip(cts, steps)]
    for form, variant in [(0, 0), (2, 2), (2, 1), (-1, -1)]:
        ctx.set_ntt_form(form)
        ctx.set_keyswitch_variant(variant)
        for g, w in zip(ctx.rotate_many(cts, steps), want):
            assert torch.equal(g.data, w.data)
        for g, s in zip(ctx.rotate_hoisted(cts[0], steps), steps):
            assert torch.equal(g.data, ctx.rotate(cts[0], s).data)
