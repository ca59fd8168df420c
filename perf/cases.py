"""The performance cases of the exact RNS product and the Smith-form calls.

Each case is one call (or the three calls of the separate steps) that a program
using the library makes, through the public binding `smf`: exact products from
the smallest to the bench size, a batch of uneven products, the separate
reduce / residue product / CRT steps, conversion between bases, p-adic lifting,
A^-1 mod p, determinants and local Smith forms modulo primes, and the whole
Smith form.  Sizes come from the repository's configurations, tests and bench.
"""
import math

import numpy as np
import torch

from paper_2605_19254_gb300 import inputs, smf

DEV = "cuda:0"
P24 = (1 << 24) - 3  # 16777213, the largest prime below 2^24
Q31 = (2147483647, 2147483629, 2147483587, 2147483579)  # the largest primes below 2^31


def listed():
    return [
        # the smallest products: the constructed n = 64 Smith workload's matrix size times a narrow block
        dict(name="matmul_64", kind="matmul", m=64, k=64, n=16, a_bits=7, a_words=1, b_words=8, host=False,
             form="limb"),
        # the bench product: small-entry matrix times a wide block of 512-bit integers
        dict(name="matmul_4096", kind="matmul", m=4096, k=4096, n=256, a_bits=20, a_words=1, b_words=8, host=False,
             form="limb"),
        # both operands big (products of massaged matrices); odd sizes
        dict(name="matmul_wide_1009", kind="matmul", m=1009, k=1009, n=100, a_bits=0, a_words=4, b_words=8,
             host=False, form="limb"),
        # operands and result in pinned host memory: the copy pipeline, end to end
        dict(name="matmul_host_2003", kind="matmul", m=2003, k=2003, n=128, a_bits=20, a_words=1, b_words=8,
             host=True, form="limb"),
        # the batched workload: 512 products of uneven n, entries of 7 and 20 bits in turn
        dict(name="grouped_512", kind="grouped", count=512, cols=128, lo=32, hi=1024, b_words=8, shapes=0),
        # the three steps called one by one on residues the program keeps (ragged sizes)
        dict(name="steps_1500", kind="steps", m=1500, k=1500, n=250, a_bits=20, b_words=8),
        # residues of a 4096 x 256 matrix of products taken to the next basis
        dict(name="convert_1m", kind="convert", count=4096 * 256, bound=543, bound_to=543),
        # Phase 1's lifting loop: a few tens of digits of A^-1 B
        dict(name="lift_1024", kind="lift", n=1024, cols=64, a_bits=20, b_bits=40, steps=32),
        # the lifting's initialization, odd n
        dict(name="inverse_1500", kind="inverse", n=1500, a_bits=20),
        # Phase 3's check: det A modulo four 31-bit primes, on a paper-sized matrix
        dict(name="det_2003", kind="det", n=2003, a_bits=11, primes=4),
        # Phase 2's last iteration: local Smith forms at three primes
        dict(name="local_1009", kind="local", n=1009, form="2:9,3:6,5:4"),
        # the whole Smith form of a planted matrix (half the batched Smith workload is built so)
        dict(name="smith_1009", kind="smith", n=1009, planted=True, a_bits=0),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["matmul", "matmul", "matmul", "grouped", "steps", "convert", "lift", "inverse", "det", "local",
                       "smith"])
    if kind == "matmul":
        wide = rng.random() < 0.3
        host = not wide and rng.random() < 0.25
        form = "fp64" if not host and rng.random() < 0.15 else "limb"
        top = 512 if form == "fp64" else 1500 if wide else 4096
        return dict(kind=kind, m=_log(rng, 16, top), k=_log(rng, 16, top), n=_log(rng, 8, 256),
                    a_bits=0 if wide else rng.choice([7, 10, 20, 40]), a_words=rng.choice([2, 3, 4, 8]) if wide else 1,
                    b_words=rng.choice([1, 3, 4, 8, 8]), host=host, form=form)
    if kind == "grouped":
        return dict(kind=kind, count=_log(rng, 2, 512), cols=rng.choice([16, 33, 64, 100, 128]), lo=32,
                    hi=rng.choice([128, 512, 1024]), b_words=rng.choice([2, 4, 8]), shapes=rng.randrange(1000))
    if kind == "steps":
        return dict(kind=kind, m=_log(rng, 32, 4096), k=_log(rng, 32, 4096), n=_log(rng, 8, 256),
                    a_bits=rng.choice([7, 20]), b_words=rng.choice([1, 2, 4, 8]))
    if kind == "convert":
        return dict(kind=kind, count=_log(rng, 1000, 1 << 21), bound=rng.randint(60, 700),
                    bound_to=rng.randint(60, 700))
    if kind == "lift":
        return dict(kind=kind, n=_log(rng, 64, 2003), cols=rng.choice([16, 32, 64, 65]),
                    a_bits=rng.choice([7, 10, 20]), b_bits=rng.choice([10, 40]), steps=rng.randint(8, 64))
    if kind == "inverse":
        return dict(kind=kind, n=_log(rng, 32, 2600), a_bits=rng.choice([7, 20, 40]))
    if kind == "det":
        return dict(kind=kind, n=_log(rng, 32, 2600), a_bits=rng.choice([7, 11, 20]), primes=rng.choice([1, 2, 4]))
    if kind == "local":
        return dict(kind=kind, n=_log(rng, 32, 1009),
                    form=rng.choice(["2:9,3:6,5:4", "2:4", "3:5,7:3", "2:12,3:8,5:5,7:4,11:3"]))
    return dict(kind=kind, n=_log(rng, 32, 701), planted=rng.random() < 0.5, a_bits=rng.choice([7, 20]))


# ---------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape, bits):
    """int64 uniform on [-2^bits, 2^bits], on the GPU."""
    return torch.randint(-(1 << bits), (1 << bits) + 1, shape, dtype=torch.int64, device=DEV, generator=g)


def _words(g, shape, words):
    """Random signed (64 words)-bit integers."""
    return torch.randint(-(1 << 63), (1 << 63) - 1, tuple(shape) + (words,), dtype=torch.int64, device=DEV,
                         generator=g)


def _a_bits(case):
    return case["a_bits"] or 64 * case["a_words"] - 1


def _out_words(k, a_bits, b_bits):
    return (k.bit_length() + a_bits + b_bits + 2 + 63) // 64


def _planted(seed, n):
    """U diag(s) V with s ending in a chain of small factors, as the batched Smith workload builds it."""
    tail = inputs.divisibility_chain(seed, "s", int(inputs.uniform_int(seed, "t", (1,), 4, 8)[0]))
    A = inputs.smith_known_matrix_np(seed, [1] * (n - len(tail)) + tail, 2 * n)
    return A, max(1, int(np.abs(A).max()).bit_length())


def _planted_local(seed, n, primes):
    """U diag(s) V whose last factors are random products of the given primes: deep local forms."""
    length = min(n - 1, 12)
    f = inputs.uniform_int(seed, "f", (length,), 0, len(primes) - 1)
    s, cur = [], 1
    for j in range(length):
        cur *= primes[int(f[j])]
        s.append(cur)
    A = inputs.smith_known_matrix_np(seed, [1] * (n - length) + s, n)
    return A, max(1, int(np.abs(A).max()).bit_length())


def prepare(case, seed):
    kind = case["kind"]
    form = smf.SMF_FORM_FP64 if kind == "matmul" and case["form"] == "fp64" else smf.SMF_FORM_INT8LIMB
    ctx = smf.Context(0, form)
    g = _gen(seed)
    st = dict(kind=kind, ctx=ctx)
    if kind == "matmul":
        m, k, n = case["m"], case["k"], case["n"]
        ab = _a_bits(case)
        A = _words(g, (m, k), case["a_words"]) if case["a_bits"] == 0 else _uniform(g, (m, k, 1), ab)
        B = _words(g, (k, n), case["b_words"])
        W = _out_words(k, ab, 64 * case["b_words"] - 1)
        if case["host"]:
            A, B = A.cpu().pin_memory(), B.cpu().pin_memory()
            C = torch.zeros((m, n, W), dtype=torch.int64).pin_memory()
        else:
            C = torch.zeros((m, n, W), dtype=torch.int64, device=DEV)
        need = ctx.rns_matmul_workspace(A, B, C, a_bits=case["a_bits"])
        st.update(A=A, B=B, C=C, a_bits=case["a_bits"], ws=torch.empty(need, dtype=torch.uint8, device=DEV))
    elif kind == "grouped":
        shapes = inputs.batched_shapes(case["shapes"], case["count"], case["lo"], case["hi"])
        bits = [b for _, b in shapes]
        As = [_uniform(g, (n, n, 1), b) for n, b in shapes]
        Bs = [_words(g, (n, case["cols"]), case["b_words"]) for n, _ in shapes]
        # the results lie in one buffer, one block per product
        Ws = [_out_words(n, b, 64 * case["b_words"] - 1) for n, b in shapes]
        sizes = [n * case["cols"] * w for (n, _), w in zip(shapes, Ws)]
        starts = np.concatenate([[0], np.cumsum([(s + 1) // 2 * 2 for s in sizes])])
        C = torch.zeros(int(starts[-1]), dtype=torch.int64, device=DEV)
        Cs = [C[int(o):int(o) + s].view(n, case["cols"], w) for o, s, (n, _), w in zip(starts, sizes, shapes, Ws)]
        need = ctx.rns_matmul_grouped_workspace(As, Bs, Cs, a_bits=bits)
        st.update(As=As, Bs=Bs, Cs=Cs, C=C, bits=bits, ws=torch.empty(need, dtype=torch.uint8, device=DEV))
    elif kind == "steps":
        m, k, n = case["m"], case["k"], case["n"]
        bb = 64 * case["b_words"] - 1
        basis = ctx.basis_create(k.bit_length() + case["a_bits"] + bb)
        L = len(basis.primes)
        A = _uniform(g, (m, k), case["a_bits"]).to(torch.int32)  # its own residues modulo every prime
        B = _words(g, (k, n), case["b_words"])
        W = _out_words(k, case["a_bits"], bb)
        W = max(W, (math.prod(basis.primes).bit_length() + 63) // 64)
        need = ctx.residue_gemm_workspace(basis, m, n, k, True)
        st.update(basis=basis, A=A, B=B, m=m, k=k, n=n, ws=torch.empty(need, dtype=torch.uint8, device=DEV),
                  rB=torch.zeros((L, k, n), dtype=torch.int32, device=DEV),
                  rC=torch.zeros((L, m, n), dtype=torch.int32, device=DEV),
                  C=torch.zeros((m, n, W), dtype=torch.int64, device=DEV))
    elif kind == "convert":
        src = ctx.basis_create(case["bound"])
        dst = ctx.basis_create(case["bound_to"], min(src.primes))
        p = torch.tensor(src.primes, dtype=torch.int64, device=DEV)
        r = (torch.randint(0, 1 << 62, (len(src.primes), case["count"]), dtype=torch.int64, device=DEV, generator=g)
             % p[:, None]).to(torch.int32)
        st.update(src=src, dst=dst, r=r,
                  out=torch.zeros((len(dst.primes), case["count"]), dtype=torch.int32, device=DEV))
    elif kind in ("lift", "inverse"):
        n = case["n"]
        basis = ctx.basis_create(20, P24 + 1)  # the one prime 2^24 - 3
        A = _uniform(g, (n, n, 1), case["a_bits"])
        inv = torch.zeros((n, n), dtype=torch.int32, device=DEV)
        ws = torch.empty(ctx.inverse_mod_p_workspace(n), dtype=torch.uint8, device=DEV)
        st.update(basis=basis, A=A, inv=inv, a_bits=case["a_bits"], ws=ws)
        if kind == "lift":
            ctx.inverse_mod_p(basis, A, inv, a_bits=case["a_bits"], workspace=ws)
            ctx.status_sync()
            B = _uniform(g, (n, case["cols"], 1), case["b_bits"])
            need = ctx.padic_lift_workspace(basis, A, B, a_bits=case["a_bits"], b_bits=case["b_bits"])
            st.update(B=B, b_bits=case["b_bits"], steps=case["steps"],
                      X=torch.zeros((case["steps"], n, case["cols"]), dtype=torch.int32, device=DEV),
                      R=torch.zeros((n, case["cols"], 1), dtype=torch.int64, device=DEV),
                      ws=torch.empty(need, dtype=torch.uint8, device=DEV))
    elif kind == "det":
        st.update(A=_uniform(g, (case["n"], case["n"], 1), case["a_bits"]), a_bits=case["a_bits"],
                  q=list(Q31[:case["primes"]]))
    elif kind == "local":
        qe = [tuple(int(v) for v in t.split(":")) for t in case["form"].split(",")]
        A, bits = _planted_local(seed, case["n"], [q for q, _ in qe])
        st.update(A=torch.from_numpy(A[..., None]).to(DEV), a_bits=bits, q=[q for q, _ in qe], e=[e for _, e in qe])
    else:
        if case["planted"]:
            A, bits = _planted(seed, case["n"])
        else:
            A, bits = inputs.uniform_int(seed, "A", (case["n"], case["n"]), -(1 << case["a_bits"]),
                                         1 << case["a_bits"]), case["a_bits"]
        st.update(A=torch.from_numpy(np.ascontiguousarray(A[..., None])), a_bits=bits)
    return st


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "matmul":
        ctx.rns_matmul(st["A"], st["B"], st["C"], a_bits=st["a_bits"], workspace=st["ws"])
        return st["C"]
    if kind == "grouped":
        ctx.rns_matmul_grouped(st["As"], st["Bs"], st["Cs"], a_bits=st["bits"], workspace=st["ws"])
        return st["C"]
    if kind == "steps":
        ctx.rns_reduce(st["basis"], st["B"], st["rB"])
        ctx.residue_gemm(st["basis"], st["A"], 0, st["rB"], st["rC"], st["m"], st["n"], st["k"], workspace=st["ws"])
        ctx.crt_reconstruct(st["basis"], st["rC"], st["C"])
        return {"residues": st["rC"], "product": st["C"]}
    if kind == "convert":
        ctx.base_convert(st["src"], st["dst"], st["r"], st["out"])
        return st["out"]
    if kind == "lift":
        ctx.padic_lift(st["basis"], st["A"], st["inv"], st["B"], st["steps"], st["X"], st["R"], a_bits=st["a_bits"],
                       b_bits=st["b_bits"], workspace=st["ws"])
        return {"digits": st["X"], "residual": st["R"]}
    if kind == "inverse":
        ctx.inverse_mod_p(st["basis"], st["A"], st["inv"], a_bits=st["a_bits"], workspace=st["ws"])
        return st["inv"]
    if kind == "det":
        return np.array(ctx.det_mod(st["A"], st["q"], a_bits=st["a_bits"]), dtype=np.int64)
    if kind == "local":
        counts = ctx.smith_local(st["A"], st["q"], st["e"], a_bits=st["a_bits"])
        return np.array([c for cs in counts for c in cs], dtype=np.int64)
    s, _, attempts = ctx.smith_form(st["A"], seed=1, a_bits=st["a_bits"])
    data = [v.to_bytes((v.bit_length() + 31) // 32 * 4, "little") for v in s]
    return {"limbs": np.frombuffer(b"".join(data), dtype=np.uint32).astype(np.int64),
            "lengths": np.array([len(d) // 4 for d in data], dtype=np.int64), "attempts": attempts}


# ---------------------------------------------------------------------------


def _product_ops(m, k, n, a_bits, b_bits):
    """Multiply-adds of 8-bit digits that the schoolbook product of these entries takes."""
    return 2 * m * k * n * -(-(a_bits + 1) // 8) * -(-(b_bits + 1) // 8)


def _primes(bound):
    return -(-(bound + 1) // 24)


def work(case):
    """Each input read once and each output written once; operations counted in 8-bit digit products
    (exact products and conversions), in word multiply-adds (eliminations) or in digit products per step."""
    kind = case["kind"]
    if kind == "matmul":
        m, k, n = case["m"], case["k"], case["n"]
        ab, bb = _a_bits(case), 64 * case["b_words"] - 1
        W = _out_words(k, ab, bb)
        return {"bytes": 8 * (m * k * case["a_words"] + k * n * case["b_words"] + m * n * W),
                "flops": _product_ops(m, k, n, ab, bb)}
    if kind == "grouped":
        total, ops = 0, 0
        bb = 64 * case["b_words"] - 1
        for n, b in inputs.batched_shapes(case["shapes"], case["count"], case["lo"], case["hi"]):
            total += 8 * (n * n + n * case["cols"] * (case["b_words"] + _out_words(n, b, bb)))
            ops += _product_ops(n, n, case["cols"], b, bb)
        return {"bytes": total, "flops": ops}
    if kind == "steps":
        m, k, n = case["m"], case["k"], case["n"]
        bb = 64 * case["b_words"] - 1
        L = _primes(k.bit_length() + case["a_bits"] + bb)
        W = _out_words(k, case["a_bits"], bb)
        # the residues of B and of C are results of a call and inputs of the next
        return {"bytes": 4 * m * k + 8 * k * n * case["b_words"] + 8 * L * k * n + 8 * L * m * n + 8 * m * n * W,
                "flops": _product_ops(m, k, n, case["a_bits"], bb)}
    if kind == "convert":
        a, b = _primes(case["bound"]), _primes(case["bound_to"])
        return {"bytes": 4 * case["count"] * (a + b), "flops": 2 * 9 * case["count"] * a * b}
    if kind == "lift":
        n, m = case["n"], case["cols"]
        da = -(-(case["a_bits"] + 1) // 8)
        return {"bytes": 8 * n * n + 4 * n * n + 16 * n * m + 4 * case["steps"] * n * m,
                "flops": case["steps"] * 2 * n * n * m * (9 + 3 * da)}
    if kind == "inverse":
        n = case["n"]
        return {"bytes": 8 * n * n + 4 * n * n, "flops": 2 * 9 * n ** 3}
    if kind == "det":
        n = case["n"]
        return {"bytes": 8 * n * n, "flops": case["primes"] * 2 * n ** 3 // 3}
    if kind == "local":
        n = case["n"]
        return {"bytes": 8 * n * n, "flops": len(case["form"].split(",")) * 2 * n ** 3 // 3}
    n = case["n"]
    # A^-1 mod p, about 2 log2 det A / 24 lifting digits of 32 columns, four determinants
    bits = case["a_bits"] or 20
    return {"bytes": 8 * n * n, "flops": 18 * n ** 3 + n * bits // 12 * 2 * n * n * 32 * 18 + 8 * n ** 3 // 3}


def exact(case, seed):
    """Every output is a whole number (multi-word integers, residues, counts), compared for equality:
    64-bit floating point holds none of the multi-word results, so there is nothing to give here."""
    return None
