"""The lifting's step kernels at the edges of their 32 x 8 tiles and of their
arithmetic: digits in [0, p) with A sum X_i p^i + p^k R = B in Python's integers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_19254_gb300 import build, smf
    build.build()
    c = smf.Context(0, smf.SMF_FORM_INT8LIMB)
    yield c
    c.destroy()


@pytest.mark.parametrize("n,m,pad", [(1, 1, 0), (31, 8, 0), (32, 9, 1), (33, 7, 0), (70, 17, 3)])
@pytest.mark.parametrize("a_bits,b_bits,p_bits", [(1, 1, 24), (7, 61, 24), (24, 40, 24), (20, 50, 12), (20, 20, 4)])
def test_lift_edges(ctx, n, m, pad, a_bits, b_bits, p_bits):
    steps = 5
    basis = ctx.basis_create(p_bits - 3, 1 << p_bits)
    p = int(basis.primes[0])
    assert len(basis.primes) == 1 and p < 1 << p_bits
    rng = np.random.default_rng(n * 1000 + a_bits)
    # unit lower triangular times unit upper triangular modulo p, entries within the bound
    A = np.tril(rng.integers(-1, 2, (n, n)), -1) + np.eye(n, dtype=np.int64)
    A = A + np.diag(rng.integers(0, max(1, (1 << a_bits) // (2 * p)) + 1, n)) * p if (1 << a_bits) > 2 * p else A
    B = rng.integers(-(1 << b_bits), (1 << b_bits) + 1, (n, m))
    B.flat[0] = 1 << b_bits
    B.flat[-1] = -(1 << b_bits)
    dA = torch.from_numpy(np.ascontiguousarray(A[..., None])).cuda()
    inv = torch.zeros((n, n), dtype=torch.int32, device="cuda")
    ctx.inverse_mod_p(basis, dA, inv, a_bits=a_bits)
    dB = torch.from_numpy(np.ascontiguousarray(B[..., None])).cuda()
    X = torch.full((steps, n, m), -1, dtype=torch.int32, device="cuda")
    R = torch.full((n, m + pad, 1), 99, dtype=torch.int64, device="cuda")
    ctx.padic_lift(basis, dA, inv, dB, steps, X, R[:, :m], a_bits=a_bits, b_bits=b_bits)
    ctx.status_sync()
    x, r = X.cpu().numpy(), R.cpu().numpy()[..., 0]
    assert x.min() >= 0 and x.max() < p and (r[:, m:] == 99).all()
    total = sum(x[i].astype(object) * p ** i for i in range(steps))
    assert (A.astype(object) @ total + r[:, :m].astype(object) * p ** steps == B).all()
    basis.destroy()


def test_wrong_inverse_is_reported(ctx):
    from paper_2605_19254_gb300 import smf
    basis = ctx.basis_create(20, (1 << 24) - 2)
    n, m = 40, 9
    A = torch.eye(n, dtype=torch.int64, device="cuda")[..., None].contiguous() * 3
    C = torch.eye(n, dtype=torch.int32, device="cuda")  # not 1/3
    B = torch.ones((n, m, 1), dtype=torch.int64, device="cuda")
    X = torch.zeros((2, n, m), dtype=torch.int32, device="cuda")
    R = torch.zeros((n, m, 1), dtype=torch.int64, device="cuda")
    ctx.padic_lift(basis, A, C, B, 2, X, R, a_bits=2, b_bits=1)
    with pytest.raises(smf.SmfError):
        ctx.status_sync()
    basis.destroy()
