"""A^-1 mod p one column at a time (two launches a column), where panels are not
taken: a single entry, and above 512 columns the FP64 form and primes whose
residues take four digits; singular matrices among them."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def smf():
    from paper_2605_19254_gb300 import build, smf as _smf
    build.build()
    return _smf


def _mul(A, B, p):
    """A B mod p for entries below 2^26, exact: 26 x 13-bit products of up to 2^11 terms below 2^50."""
    a = A.to(torch.float64)
    lo, hi = (B & 0x1FFF).to(torch.float64), (B >> 13).to(torch.float64)
    return (((a @ hi).to(torch.int64) % p) * 8192 + (a @ lo).to(torch.int64)) % p


@pytest.mark.parametrize("form,p_max", [("fp64", 0), ("fp64", 1022), ("limb", 1 << 26)])
@pytest.mark.parametrize("n", [1, 513, 700])
def test_columns(smf, form, p_max, n):
    ctx = smf.Context(0, smf.SMF_FORM_FP64 if form == "fp64" else smf.SMF_FORM_INT8LIMB)
    pb = ctx.basis_create(7, p_max)
    p = int(pb.primes[0])
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    # a product of triangular matrices with unit diagonals, its rows permuted: columns whose pivot is below
    eye = torch.eye(n, dtype=torch.int64, device="cuda")
    L = torch.randint(0, p, (n, n), dtype=torch.int64, device="cuda", generator=g).tril(-1) + eye
    U = torch.randint(0, p, (n, n), dtype=torch.int64, device="cuda", generator=g).triu(1) + eye
    perm = torch.randperm(n, device="cuda", generator=g)
    A = _mul(L, U, p)[perm].contiguous()
    C = torch.full((n, n), -1, dtype=torch.int32, device="cuda")
    ctx.inverse_mod_p(pb, A[..., None].contiguous(), C, a_bits=26)
    ctx.status_sync()
    assert int(C.min()) >= 0 and int(C.max()) < p
    assert torch.equal(_mul(C, A, p), eye)
    S = A.clone()
    if n > 1:
        S[n - 1] = (S[0] + S[n // 2]) % p
    else:
        S.zero_()
    ctx.inverse_mod_p(pb, S[..., None].contiguous(), C, a_bits=26)
    with pytest.raises(smf.SmfError) as e:
        ctx.status_sync()
    assert e.value.code == smf.SMF_E_SINGULAR
    ctx.inverse_mod_p(pb, A[..., None].contiguous(), C, a_bits=26)  # the context is usable after
    ctx.status_sync()
    assert torch.equal(_mul(C, A, p), eye)
    pb.destroy()
    ctx.destroy()


def test_no_basis_of_even_primes(smf):
    """The smallest prime of a basis is 3 (the divisions by p of the lifting's steps are products with its
    inverse modulo 2^64), and the inverse and the lifting hold for it."""
    ctx = smf.Context(0, smf.SMF_FORM_INT8LIMB)
    with pytest.raises(smf.SmfError):
        ctx.basis_create(0, 3)
    pb = ctx.basis_create(0, 4)
    assert [int(q) for q in pb.primes] == [3]
    n, m, steps = 40, 9, 6
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    eye = torch.eye(n, dtype=torch.int64, device="cuda")
    A = (torch.randint(-1, 2, (n, n), dtype=torch.int64, device="cuda", generator=g).tril(-1) + eye)[..., None].contiguous()
    C = torch.zeros((n, n), dtype=torch.int32, device="cuda")
    ctx.inverse_mod_p(pb, A, C, a_bits=1)
    B = torch.randint(-200, 201, (n, m, 1), dtype=torch.int64, device="cuda", generator=g)
    X = torch.full((steps, n, m), -1, dtype=torch.int32, device="cuda")
    R = torch.zeros((n, m, 1), dtype=torch.int64, device="cuda")
    ctx.padic_lift(pb, A, C, B, steps, X, R, a_bits=1, b_bits=8)
    ctx.status_sync()
    assert int(X.min()) >= 0 and int(X.max()) <= 2
    total = sum(X[i].to(torch.float64) * 3 ** i for i in range(steps))
    left = (A[..., 0].to(torch.float64) @ total).to(torch.int64) + R[..., 0] * 3 ** steps
    assert torch.equal(left, B[..., 0])
    pb.destroy()
    ctx.destroy()
