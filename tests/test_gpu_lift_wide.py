"""Lifting with very many right-hand sides: more tiles of columns than the second
and third dimensions of a grid take."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(3, 524_281), (33, 600_001)])
def test_lift_of_many_columns(n, m):
    from paper_2605_19254_gb300 import build, smf
    build.build()
    ctx = smf.Context(0, smf.SMF_FORM_INT8LIMB)
    basis = ctx.basis_create(20)
    p = int(basis.primes[0])
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    steps, eye = 2, torch.eye(n, dtype=torch.int64, device="cuda")
    A = eye + torch.triu(torch.randint(-3, 4, (n, n), device="cuda", generator=g), 1)
    C = torch.zeros((n, n), dtype=torch.int32, device="cuda")
    ctx.inverse_mod_p(basis, A[..., None].contiguous(), C, a_bits=2)
    B = torch.randint(-(1 << 30), 1 << 30, (n, m, 1), dtype=torch.int64, device="cuda", generator=g)
    X = torch.full((steps, n, m), -1, dtype=torch.int32, device="cuda")
    R = torch.zeros((n, m, 1), dtype=torch.int64, device="cuda")
    ctx.padic_lift(basis, A[..., None].contiguous(), C, B, steps, X, R, a_bits=2, b_bits=30)
    ctx.status_sync()
    # A (X_0 + p X_1) + p^2 R = B; |A X| < 2^31 and |R| < 2^10: every term below 2^60, sums in float64 exact per digit
    Af = A.to(torch.float64)
    ax = [(Af @ X[i].to(torch.float64)).to(torch.int64) for i in range(steps)]
    assert int(X.min()) >= 0 and int(X.max()) < p
    assert torch.equal(ax[0] + p * ax[1] + p * p * R[..., 0], B[..., 0])
    basis.destroy()
    ctx.destroy()
