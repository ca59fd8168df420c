"""The panel kernels of the eliminations (one cluster per panel): sizes at the
edges of panels, blocks and rows per block, against the defining identity or
the oracle.  Everything is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2605_19254_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_19254_gb300 import build, smf
    build.build()
    c = smf.Context(0, smf.SMF_FORM_INT8LIMB)
    yield c
    c.destroy()


# one panel up to n = 512 (fewer than 16 blocks below n = 128), panels of 128
# above: a last panel of 1, 127 and 128 columns; dense rows, and a permuted
# triangular matrix whose columns have one pivot row left (in any block)
@pytest.mark.parametrize("p_max", [0, 1022])
@pytest.mark.parametrize("n", [2, 15, 16, 17, 127, 128, 129, 511, 512, 513, 639, 640])
def test_inverse_by_panels(ctx, n, p_max):
    pb = ctx.basis_create(7, p_max)
    p = int(pb.primes[0])
    rng = np.random.default_rng(n)
    tri = np.triu(inputs.uniform_int(n, "T", (n, n), 0, p - 1), 1) + np.diag(inputs.uniform_int(n, "D", (n,), 1, p - 1))
    cases = [tri[rng.permutation(n)][:, rng.permutation(n)]]
    if p_max == 0:  # a random matrix is nonsingular modulo a 24-bit prime but for a chance of 2^-24
        cases.append(inputs.uniform_int(n, "A", (n, n), 0, p - 1))
    for A in cases:
        C = torch.full((n, n), -1, dtype=torch.int32, device="cuda")
        ctx.inverse_mod_p(pb, torch.from_numpy(A[..., None].copy()).cuda(), C, a_bits=24)
        ctx.status_sync()
        C = C.cpu().numpy().astype(np.int64)
        assert C.min() >= 0 and C.max() < p
        lo, hi = A & 0xFFF, A >> 12  # 24-bit by 12-bit products of n <= 640 terms: exact in float64
        f = C.astype(np.float64)
        prod = ((f @ hi.astype(np.float64)).astype(np.int64) % p * 4096 + (f @ lo.astype(np.float64)).astype(np.int64)) % p
        assert np.array_equal(prod, np.eye(n, dtype=np.int64))
    pb.destroy()


# determinants and local forms by panels of 32 columns at every size: one to
# four lanes, all moduli odd and small, odd up to 31 bits, and with a power of two
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 130, 513])
@pytest.mark.parametrize("q", [(2,), (101, 2), (65537, 3, 268435399), (2147483647, 2, 2147483629, 5)])
def test_det_by_panels(ctx, orc, n, q):
    A = inputs.uniform_int(n, "A", (n, n), -(1 << 20), 1 << 20)
    ctx.set_elim_panels(1)
    try:
        got = ctx.det_mod(torch.from_numpy(A[..., None].copy()).cuda(), list(q), a_bits=20)
    finally:
        ctx.set_elim_panels(0)
    assert got == [orc.det_mod(A, v) for v in q]


@pytest.mark.parametrize("n", [12, 31, 33, 64, 65, 200, 520])
@pytest.mark.parametrize("qe", [((2, 9), (3, 6), (5, 4)), ((2, 30),), ((3, 19), (46337, 2)), ((3, 3), (5, 2)),
                                ((7, 2), (2, 1), (3, 2), (11, 1), (13, 3))])
def test_local_by_panels(ctx, n, qe):
    # s: a chain of products of the primes, below 2^34 so that the entries fit 64 bits
    primes = [q for q, _ in qe]
    s, cur = [], 1
    for k in range(min(n, 9)):
        q = primes[k % len(primes)]
        cur *= q if cur * q < 1 << 34 else 1
        s.append(cur)
    s = [1] * (n - len(s)) + s
    A = inputs.smith_known_matrix_np(n, s, n)
    ctx.set_elim_panels(1)
    try:
        got = ctx.smith_local(torch.from_numpy(A[..., None].copy()).cuda(), primes, [e for _, e in qe], a_bits=62)
    finally:
        ctx.set_elim_panels(0)
    assert got == [[sum(v % q ** t == 0 for v in s) for t in range(e + 1)] for q, e in qe]
