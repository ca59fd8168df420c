"""Eliminations of matrices whose panels do not fit the cluster at full width:
A^-1 mod p with panels reduced by narrower ones, singular matrices over several
panels, and determinants and local forms whose moduli go in smaller groups."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def smf():
    from paper_2605_19254_gb300 import build, smf as _smf
    build.build()
    return _smf


@pytest.fixture(scope="module")
def ctx(smf):
    c = smf.Context(0, smf.SMF_FORM_INT8LIMB)
    yield c
    c.destroy()


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _mul(A, v, p):
    """A v mod p for A below 2^24 and v below 2^24, exact: 24 x 12-bit products of up to 2^14 terms below 2^50."""
    a = A.to(torch.float64)
    lo, hi = (v & 0xFFF).to(torch.float64), (v >> 12).to(torch.float64)
    return (((a @ hi).to(torch.int64) % p) * 4096 + (a @ lo).to(torch.int64)) % p


# panels of 128 columns reduced by panels of 64 (the last panel of 22 columns: one) and of 32 (the last
# of 103 columns: 32, 32, 32 and 7)
@pytest.mark.parametrize("n", [5910, 12007])
def test_inverse_by_narrow_panels(ctx, n):
    pb = ctx.basis_create(20)
    p = int(pb.primes[0])
    g = _gen(n)
    A = torch.randint(0, p, (n, n), dtype=torch.int64, device="cuda", generator=g)
    C = torch.full((n, n), -1, dtype=torch.int32, device="cuda")
    ctx.inverse_mod_p(pb, A[..., None], C, a_bits=24)
    ctx.status_sync()
    assert int(C.min()) >= 0 and int(C.max()) < p
    # C A v = v and A C v = v for random v (a wrong C passes with probability below p^-8)
    v = torch.randint(0, p, (n, 8), dtype=torch.int64, device="cuda", generator=g)
    assert torch.equal(_mul(C, _mul(A, v, p), p), v)
    assert torch.equal(_mul(A, _mul(C, v, p), p), v)
    pb.destroy()


# one column short of full rank, found in the last of five panels, and in a narrow panel; the context is usable after
@pytest.mark.parametrize("n", [513, 640, 5910])
def test_singular_over_several_panels(ctx, smf, n):
    pb = ctx.basis_create(20)
    p = int(pb.primes[0])
    A = torch.randint(0, p, (n, n), dtype=torch.int64, device="cuda", generator=_gen(n))
    for row, other in ((17, 4), (n - 1, n - 2)):
        B = A.clone()
        B[row] = B[other]
        C = torch.zeros((n, n), dtype=torch.int32, device="cuda")
        ctx.inverse_mod_p(pb, B[..., None].contiguous(), C, a_bits=24)
        with pytest.raises(smf.SmfError) as e:
            ctx.status_sync()
        assert e.value.code == smf.SMF_E_SINGULAR
    A[:, 3] = 0  # no pivot in the first panel
    ctx.inverse_mod_p(pb, A[..., None].contiguous(), C, a_bits=24)
    with pytest.raises(smf.SmfError) as e:
        ctx.status_sync()
    assert e.value.code == smf.SMF_E_SINGULAR
    ctx.inverse_mod_p(pb, torch.eye(n, dtype=torch.int64, device="cuda")[..., None].contiguous(), C, a_bits=1)
    ctx.status_sync()
    assert torch.equal(C, torch.eye(n, dtype=torch.int32, device="cuda"))
    pb.destroy()


def _planted(n, diag, seed):
    """Unit lower x diag x unit upper, a few entries a row: exact in float32 sums (below 2^24)."""
    g = _gen(seed)

    def tri(up):
        T = torch.randint(-1, 2, (n, n), device="cuda", generator=g).float() * (torch.rand((n, n), device="cuda", generator=g) < 0.01)
        return (T.triu(1) if up else T.tril(-1)) + torch.eye(n, device="cuda")

    A = tri(False) @ (diag[:, None] * tri(True))
    assert float(A.abs().max()) < 2 ** 23
    return A.to(torch.int64)[..., None].contiguous()


# four moduli in two groups of two, and one at a time
@pytest.mark.parametrize("n", [10750, 11600])
def test_moduli_in_smaller_groups(ctx, n):
    tail = [2, 6, 6, 12, 60, 360]
    diag = torch.ones(n, device="cuda")
    diag[-len(tail):] = torch.tensor(tail, dtype=torch.float32)
    A = _planted(n, diag, n)
    bits = int(A.abs().max()).bit_length()
    q = [2147483647, 2147483629, 7, 2147483587, 11]
    det = 2 * 6 * 6 * 12 * 60 * 360
    assert ctx.det_mod(A, q, a_bits=bits) == [det % v for v in q]
    qe = [(2, 5), (3, 3), (5, 2), (7, 1)]
    got = ctx.smith_local(A, [v for v, _ in qe], [e for _, e in qe], a_bits=bits)
    assert got == [[n] + [sum(s % v ** t == 0 for s in tail) for t in range(1, e + 1)] for v, e in qe]


# The column loops of 32-bit moduli, which a threshold above n leaves: determinants and local forms, one
# lane (a pivot step and an update a column) and four in lockstep, against the planted factors.
@pytest.mark.parametrize("n", [1, 65, 300])
def test_column_loops(ctx, n):
    tail = [2, 6, 6, 60, 360, 2520][-min(n, 6):]
    diag = torch.ones(n, device="cuda")
    diag[-len(tail):] = torch.tensor(tail, dtype=torch.float32)
    A = _planted(n, diag, n)
    bits = max(1, int(A.abs().max()).bit_length())
    det = 1
    for v in tail:
        det *= v
    ctx.set_elim_panels(1 << 30)
    try:
        for q in ([2147483647], [2147483647, 11, 2147483629, 13], [65537, 11, 13, 17, 19]):
            assert ctx.det_mod(A, q, a_bits=bits) == [det % v for v in q]
        for qe in ([(2, 5)], [(3, 3)], [(2, 30)], [(2, 5), (3, 3)], [(2, 5), (3, 3), (5, 2), (7, 1)],
                   [(2, 1), (3, 1), (5, 1), (7, 1), (11, 1)]):
            got = ctx.smith_local(A, [v for v, _ in qe], [e for _, e in qe], a_bits=bits)
            want = [[n] + [sum(s % v ** t == 0 for s in tail) for t in range(1, e + 1)] for v, e in qe]
            assert got == want
    finally:
        ctx.set_elim_panels(0)
