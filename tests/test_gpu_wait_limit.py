"""A bounded wait of the tensor-core product that gives up (a limit of no polls at all): the calls that
hand out its results say so until he_synchronize has reported it, once on each context of the family,
and everything works again afterwards."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_a_wait_that_gives_up_is_reported_and_cleared():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_00482_gb300 import he

    ctx = he.Context(12, [40, 20], [40], 2, seed=3)
    other = ctx.fork(torch.cuda.Stream())
    n = 128
    rng = np.random.default_rng(1)
    W = torch.from_numpy(rng.normal(size=(n, 8))).cuda()
    wide, narrow = he.WeightMatrix(ctx, W, 1), he.WeightMatrix(ctx, W[:, :4].contiguous(), 1)
    host = np.stack([rng.integers(0, q, size=(n, 2, ctx.n)) for q in ctx.primes[:2]], axis=2)
    data = torch.from_numpy(np.ascontiguousarray(host)).cuda()
    cts = [he.Ciphertext(data[i], 1, 2.0**20) for i in range(n)]
    want = ctx.cdiag_matmult(wide, cts)
    slots = torch.zeros((8, ctx.slots), dtype=torch.float64, device="cuda")
    plan = he.Plan(8, 8, ctx.slots)

    def gives_up(call, *args):
        with pytest.raises(he.HEError) as e:
            call(*args)
        assert e.value.status == he.HE_ETIMEOUT

    ctx.synchronize()
    ctx.set_wait_limit(0)
    outs = ctx.cdiag_matmult(wide, cts)
    gives_up(ctx.ct_export_host, outs[0])  # waits for the stream
    for c in (ctx, other):
        gives_up(c.decrypt, want[0])
        gives_up(c.matmult_decrypt, plan, want[:1])
        gives_up(c.cdiag_decode, n, n, slots)
        gives_up(c.cdiag_matmult, wide, cts)
    for g, w in zip(ctx.cdiag_matmult(narrow, cts), want):  # no bounded wait in the general form
        assert torch.equal(g.data, w.data)
    ctx.set_wait_limit()
    for c in (ctx, other):
        gives_up(c.synchronize)
        c.synchronize()
        c.decrypt(want[0])
    for g, w in zip(ctx.cdiag_matmult(wide, cts), want):
        assert torch.equal(g.data, w.data)
    ctx.synchronize()
    with pytest.raises(he.HEError):
        ctx.set_wait_limit((1 << 21) + 1)
    with pytest.raises(he.HEError):
        ctx.set_wait_limit(-1)
