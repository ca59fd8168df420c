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
