"""The work that programs have this library do, as cases that can be timed and compared.

A case is one public call, or one party's step made of such calls, at one size:

  linr_step      a VFL-LinR iteration's product from fp64 inputs to fp64 results: the matrix is
                 encoded again (a new batch), the vector encrypted, multiplied, the product
                 decrypted and its slots summed
  matmult        the encrypted product alone, on a matrix that was encoded once (fixed features)
  batch          many uneven products in one call
  rotate_hoisted many rotations of one ciphertext
  rotate_many    one rotation each of many ciphertexts
  cdiag_encode   a VFL-NN activation matrix into its diagonal plaintexts
  cdiag_forward  the VFL-NN layer product on encrypted diagonals
  cdiag_transpose the diagonals of the transposed matrix, for the backward pass
  cdiag_decrypt  the layer product's ciphertexts into the cleartext matrix

Rings are the parameter sets of paper_2405_00482_gb300.inputs, named by their ring degree.  The
results of a call on many ciphertexts lie one after another in one buffer, as a program that sends
them on keeps them; the two calls whose Python form allocates each result go through the C ABI.
"""
import math

import torch

from paper_2405_00482_gb300 import he, inputs

RINGS = {4096: inputs.PARAMS_SMALL, 8192: inputs.PARAMS_N8192, 16384: inputs.PARAMS_N16384}


def listed():
    return [
        # the benchmark's smallest product, X^T [[r]] with X 64 x 16: every launch counts
        {"name": "linr_step_16x64", "kind": "linr_step", "ring": 4096, "m": 16, "n": 64},
        {"name": "matmult_16x64", "kind": "matmult", "ring": 4096, "m": 16, "n": 64},
        # the benchmark's gradient and forward products of a 1024 x 256 batch
        {"name": "linr_step_256x1024", "kind": "linr_step", "ring": 8192, "m": 256, "n": 1024},
        {"name": "matmult_1024x256", "kind": "matmult", "ring": 8192, "m": 1024, "n": 256},
        # a ragged product cut into two row blocks (m above the slot count)
        {"name": "matmult_5000x300", "kind": "matmult", "ring": 8192, "m": 5000, "n": 300},
        # the benchmark's uneven jobs, batch 128..4096 and features 16..512 each
        {"name": "batch_64", "kind": "batch", "ring": 8192, "jobs": 64},
        # the rotation counts of the benchmark: the m' - 1 = 63 of the gradient product
        {"name": "rotate_hoisted_63", "kind": "rotate_hoisted", "ring": 8192, "count": 63, "level": 2},
        {"name": "rotate_many_63", "kind": "rotate_many", "ring": 8192, "count": 63, "level": 2},
        # the benchmark's VFL neural layer: activations 4096 x 256, weights 256 x 128
        {"name": "cdiag_encode_4096x256", "kind": "cdiag_encode", "ring": 16384, "m": 4096, "n": 256},
        {"name": "cdiag_forward_4096x256x128", "kind": "cdiag_forward", "ring": 16384, "m": 4096, "n": 256, "cols": 128},
        {"name": "cdiag_transpose_4096x256", "kind": "cdiag_transpose", "ring": 16384, "m": 4096, "n": 256},
        # a narrower layer's result, decrypted column by column
        {"name": "cdiag_decrypt_256x4096x37", "kind": "cdiag_decrypt", "ring": 16384, "m": 256, "n": 4096, "cols": 37},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["linr_step", "matmult", "batch", "rotate_hoisted", "rotate_many", "cdiag_encode", "cdiag_forward", "cdiag_transpose",
                       "cdiag_decrypt"])
    if kind in ("linr_step", "matmult"):
        # batches of 16..8192 rows and 8..512 features; the gradient multiplies by the transpose
        ring = rng.choice([4096, 8192, 8192])
        b, f = _log_int(rng, 16, 8192 if ring == 8192 else 1024), _log_int(rng, 8, 512 if ring == 8192 else 128)
        m, n = (f, b) if rng.random() < 0.5 else (b, f)
        return {"kind": kind, "ring": ring, "m": m, "n": n}
    if kind == "batch":
        return {"kind": kind, "ring": 8192, "jobs": _log_int(rng, 2, 48)}
    if kind in ("rotate_hoisted", "rotate_many"):
        ring = rng.choice([4096, 8192, 16384])
        top = RINGS[ring].top
        return {"kind": kind, "ring": ring, "count": _log_int(rng, 1, 160), "level": rng.choice([top, top, rng.randint(1, top)])}
    m, n = 1 << rng.randint(4, 13), 1 << rng.randint(4, 8)
    if rng.random() < 0.4:
        m, n = n, m
    case = {"kind": kind, "ring": 16384, "m": m, "n": n}
    if kind in ("cdiag_forward", "cdiag_decrypt"):
        case["cols"] = _log_int(rng, 1, 128 if kind == "cdiag_forward" else 64)
    return case


# ---- inputs: plain torch, from the seed alone ----
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _normal(g, *shape, scale=1.0):
    return scale * torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")


def _uniform(g, *shape):
    return 2.0 * torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") - 1.0


def _matrix_and_vector(case, seed):
    """Features ~ N(0, 1), residuals or weights ~ U[-1, 1]."""
    g = _gen(seed)
    return _normal(g, case["m"], case["n"]), _uniform(g, case["n"])


def _layer(case, seed):
    """Activations ~ U[-1, 1], weights ~ N(0, 1 / rows)."""
    g = _gen(seed)
    a = _uniform(g, case["m"], case["n"])
    w = _normal(g, case["n"], case["cols"], scale=case["n"] ** -0.5) if "cols" in case else None
    return a, w


def _job_shapes(case, seed):
    """(features, batch) of each job: 16..512 and 128..4096.  The shapes belong to the case; only
    the values follow the seed."""
    g = torch.Generator()
    g.manual_seed(case["jobs"])
    b = torch.randint(128, 4097, (case["jobs"],), generator=g).tolist()
    f = torch.randint(16, 513, (case["jobs"],), generator=g).tolist()
    return list(zip(f, b))


def _results(ctx, count, level):
    """One buffer of `count` ciphertexts, and the ciphertexts in it."""
    buf = torch.empty((count, 2, level + 1, ctx.n), dtype=torch.int64, device=ctx.device)
    return buf, [he.Ciphertext(buf[i], level, 0.0) for i in range(count)]


def _context(case, seed):
    p = RINGS[case["ring"]]
    return p, he.Context(p.log_n, list(p.q_bits), list(p.p_bits), p.dnum, seed=seed)


def prepare(case, seed):
    p, ctx = _context(case, seed)
    kind, st = case["kind"], {"case": case, "p": p, "ctx": ctx, "nonce": 1000 * (seed % 1000003)}
    if kind in ("linr_step", "matmult"):
        X, v = _matrix_and_vector(case, seed)
        plan = he.Plan(case["m"], case["n"], ctx.slots)
        ctx.keygen(plan.rotation_steps)
        st["buf"], st["outs"] = _results(ctx, plan.row_blocks, p.top - 1)
        st.update(plan=plan, X=X, v=v, pm=ctx.encode_matrix(plan, X, p.top))
        st["cts"] = ctx.encrypt_vector(plan, v, p.scale, p.top, st["nonce"])
        st["y"] = torch.empty(plan.m, dtype=torch.float64, device=ctx.device)
    elif kind == "batch":
        g = _gen(seed)
        plans = [he.Plan(m, n, ctx.slots) for m, n in _job_shapes(case, seed)]
        ctx.keygen(list(range(1, max(q.m_prime for q in plans))))
        pms = [ctx.encode_matrix(q, _normal(g, q.m, q.n), p.top) for q in plans]
        st["cts"] = [ctx.encrypt_vector(q, _uniform(g, q.n), p.scale, p.top, st["nonce"] + i)[0] for i, q in enumerate(plans)]
        st["batch"] = he.Batch(ctx, plans, pms)
        st["buf"], st["outs"] = _results(ctx, len(plans), p.top - 1)
    elif kind in ("rotate_hoisted", "rotate_many"):
        g, count = _gen(seed), case["count"]
        steps = [i % (ctx.slots - 1) + 1 for i in range(count)]
        ctx.keygen(sorted(set(steps)))
        st["cts"] = [ctx.encrypt(ctx.encode(_uniform(g, ctx.slots), p.scale, case["level"]), st["nonce"] + i)
                     for i in range(1 if kind == "rotate_hoisted" else count)]
        st["steps"] = steps
        st["buf"], st["outs"] = _results(ctx, count, case["level"])
    else:
        a, w = _layer(case, seed)
        st["A"] = a
        diag = min(case["m"], case["n"])
        if kind == "cdiag_encode":
            st["buf"] = torch.empty((diag, p.top + 1, ctx.n), dtype=torch.int64, device=ctx.device)
            st["c_outs"] = (he.HePt * diag)(*[he.HePt(st["buf"][i].data_ptr(), p.top, 0.0) for i in range(diag)])
        else:
            pts = ctx.cdiag_encode_matrix(a, p.scale, p.top)
            st["cts"] = [ctx.encrypt(q, st["nonce"] + i) for i, q in enumerate(pts)]
        if kind == "cdiag_transpose":
            ctx.keygen(he.Context.cdiag_transpose_steps(case["m"], case["n"]))
            st["buf"], outs = _results(ctx, diag, p.top)
            st["c_ins"] = (he.HeCt * diag)(*[c.c() for c in st["cts"]])
            st["c_outs"] = (he.HeCt * diag)(*[c.c() for c in outs])
        if w is not None:
            st["W"] = he.WeightMatrix(ctx, w, p.top)
            st["buf"], st["outs"] = _results(ctx, case["cols"], p.top - 1)
        if kind == "cdiag_decrypt":
            ctx.cdiag_matmult(st["W"], st["cts"], st["outs"])
            del st["cts"]
            st["slots"] = torch.empty((case["cols"], ctx.slots), dtype=torch.float64, device=ctx.device)
    return st


def _ok(status, what):
    if status != he.HE_OK:
        raise he.HEError(status, what)


def run(st):
    case, ctx, p = st["case"], st["ctx"], st["p"]
    kind = case["kind"]
    if kind == "linr_step":
        plan = st["plan"]
        ctx.encode_matrix(plan, st["X"], p.top, out=st["pm"])
        cts = ctx.encrypt_vector(plan, st["v"], p.scale, p.top, st["nonce"], outs=st["cts"])
        outs = ctx.matmult(plan, st["pm"], cts, st["outs"])
        return {"product": st["buf"], "y": ctx.matmult_decrypt(plan, outs, out=st["y"])}
    if kind == "matmult":
        ctx.matmult(st["plan"], st["pm"], st["cts"], st["outs"])
    elif kind == "batch":
        st["batch"].run(st["cts"], st["outs"])
    elif kind == "rotate_hoisted":
        ctx.rotate_hoisted(st["cts"][0], st["steps"], st["outs"])
    elif kind == "rotate_many":
        ctx.rotate_many(st["cts"], st["steps"], st["outs"])
    elif kind == "cdiag_encode":
        _ok(he.lib().he_cdiag_encode_matrix(ctx.handle, st["A"].data_ptr(), case["m"], case["n"], p.scale, p.top, st["c_outs"]),
            "he_cdiag_encode_matrix")
    elif kind == "cdiag_forward":
        ctx.cdiag_matmult(st["W"], st["cts"], st["outs"])
    elif kind == "cdiag_transpose":
        _ok(he.lib().he_cdiag_transpose(ctx.handle, st["c_ins"], case["m"], case["n"], st["c_outs"]), "he_cdiag_transpose")
    else:
        for k, c in enumerate(st["outs"]):
            ctx.decrypt(c, st["slots"][k])
        return ctx.cdiag_decode(case["m"], case["n"], st["slots"])
    return st["buf"]


def exact(case, seed):
    """The cleartext products; ciphertexts and plaintext polynomials have no such value."""
    if case["kind"] == "linr_step":
        X, v = _matrix_and_vector(case, seed)
        return {"product": None, "y": X @ v}
    if case["kind"] == "cdiag_decrypt":
        a, w = _layer(case, seed)
        return a @ w
    return None


# ---- the work of one pass: residues are 8 bytes; a modular multiply-add counts as two operations ----
def _pow2(v):
    return 1 << max(0, (v - 1).bit_length())


def _product_work(p, m, n, encode):
    slots, N, nq, K = p.slots, p.n, p.top + 1, len(p.p_bits)
    ext, alpha = nq + K, -(-len(p.q_bits) // p.dnum)
    ndig = -(-nq // alpha)
    mp, np_ = _pow2(m), _pow2(n)
    mb, nb = min(mp, slots), min(np_, slots)
    R, C = mp // mb, np_ // nb
    diag = max(1, mb * nb // slots)
    keys = 8 * N * (diag - 1) * 2 * ndig * ext
    loop = 2 * N * R * C * ((diag - 1) * (2 * ndig * ext + 2 * ext + nq) + 2 * nq)
    log_n = p.log_n
    ntt = N // 2 * log_n
    if encode:  # fp64 matrix and vector in, fp64 results and the product's ciphertexts out
        words = m * n + n + m + R * 2 * p.top * N
        return {"bytes": 8 * words + keys, "flops": loop + 2 * ntt * (R * C * diag * ext + 2 * C * nq) + 10 * ntt * (R * C * diag + C + R) // 2}
    words = R * C * diag * ext * N + C * 2 * nq * N + R * 2 * p.top * N
    return {"bytes": 8 * words + keys, "flops": loop + 2 * ntt * (C * ndig * ext + 2 * R * (nq + K))}


def work(case):
    p = RINGS[case["ring"]]
    N, kind, K = p.n, case["kind"], len(p.p_bits)
    ntt = N // 2 * p.log_n
    if kind in ("linr_step", "matmult"):
        return _product_work(p, case["m"], case["n"], kind == "linr_step")
    if kind == "batch":
        each = [_product_work(p, m, n, False) for m, n in _job_shapes(case, 0)]
        top = max(max(1, _pow2(m) * _pow2(n) // p.slots) for m, n in _job_shapes(case, 0))
        key = 8 * N * 2 * p.dnum * (p.top + 1 + K)
        own = sum(max(1, _pow2(m) * _pow2(n) // p.slots) - 1 for m, n in _job_shapes(case, 0))
        # the jobs share the rotation keys of the longest one
        return {"bytes": sum(w["bytes"] for w in each) - key * own + key * (top - 1), "flops": sum(w["flops"] for w in each)}
    if kind in ("rotate_hoisted", "rotate_many", "cdiag_transpose"):
        nq = p.top + 1 if kind == "cdiag_transpose" else case["level"] + 1
        count = min(case["m"], case["n"]) if kind == "cdiag_transpose" else case["count"]
        ext, alpha = nq + K, -(-len(p.q_bits) // p.dnum)
        ndig = -(-nq // alpha)
        ins = 1 if kind == "rotate_hoisted" else count
        modup = nq + ndig * ext - nq
        return {"bytes": 8 * N * (2 * nq * (ins + count) + count * 2 * ndig * ext),
                "flops": 2 * N * count * 2 * ndig * ext + 2 * ntt * (ins * modup + count * 2 * (K + nq))}
    m, n, nq = case["m"], case["n"], p.top + 1
    diag = min(m, n)
    if kind == "cdiag_encode":
        return {"bytes": 8 * (m * n + diag * nq * N), "flops": diag * (2 * ntt * nq + 5 * ntt)}
    cols = case["cols"]
    if kind == "cdiag_forward":
        return {"bytes": 8 * (diag * 2 * nq * N + n * cols + cols * 2 * p.top * N),
                "flops": 2 * diag * cols * 2 * nq * N + 2 * ntt * cols * 2 * nq}
    return {"bytes": 8 * (cols * 2 * p.top * N + m * cols), "flops": cols * (2 * N + 2 * ntt + 5 * ntt)}
