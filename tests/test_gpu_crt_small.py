"""CRT and base conversion against Python's integers: values x + (M - 1)/2 = y with
y / M at every distance from 0 and 1, where the quotient is settled by the fp32
sum, in fixed point, or limb by limb (mixed radix)."""
import math

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


def _values(M):
    """x = y - (M - 1)/2 for y near 0 and M at every scale, and in between."""
    ys = {0, 1, M - 1, M - 2, M // 2}
    for k in range(1, 80):
        for d in (-1, 0, 1, 12345):
            for y in ((M >> k) + d, M - 1 - (M >> k) + d, M * 3 // 7 + (M >> k) + d):
                ys.add(y % M)
    return [y - (M - 1) // 2 for y in sorted(ys)]


def _basis(ctx, L, p_max):
    return ctx.basis_create(max(1, int(L * (math.log2(p_max) - 0.01 if p_max > 60 else 5.2)) - 3), p_max)


@pytest.mark.parametrize("L,p_max", [(L, p) for p in (1 << 24, 1 << 26, 1 << 11, 60) for L in (1, 2, 3, 5, 8, 9)] +
                         [(L, 1 << 24) for L in (12, 13, 16, 17, 24, 31, 48)])
def test_quotients(ctx, L, p_max):
    b = _basis(ctx, L, p_max)
    primes = [int(p) for p in b.primes]
    M = math.prod(primes)
    vals = _values(M)
    W = M.bit_length() // 64 + 1
    r = np.array([[x % p for x in vals] for p in primes], dtype=np.int32)
    X = torch.full((1, len(vals), W), 77, dtype=torch.int64, device="cuda")
    ctx.crt_reconstruct(b, torch.from_numpy(r[:, None, :].copy()).cuda(), X)
    ctx.status_sync()
    want = np.frombuffer(b"".join(x.to_bytes(8 * W, "little", signed=True) for x in vals), dtype=np.int64)
    assert np.array_equal(X.cpu().numpy().ravel(), want)
    b.destroy()


# targets in pairs with the source: few and many primes, below and above eight together
@pytest.mark.parametrize("L,LQ", [(1, 1), (1, 6), (1, 7), (2, 5), (3, 4), (4, 4), (6, 1), (7, 1), (1, 17), (9, 2), (24, 8), (48, 3)])
def test_conversion_quotients(ctx, L, LQ):
    src = _basis(ctx, L, 1 << 24)
    dst = _basis(ctx, LQ, min(int(p) for p in src.primes))
    assert (len(src.primes), len(dst.primes)) == (L, LQ)
    vals = _values(math.prod(int(p) for p in src.primes))
    r = torch.from_numpy(np.array([[x % int(p) for x in vals] for p in src.primes], dtype=np.int32)).cuda()
    out = torch.full((LQ, len(vals)), -1, dtype=torch.int32, device="cuda")
    ctx.base_convert(src, dst, r, out)
    ctx.status_sync()
    assert np.array_equal(out.cpu().numpy(), np.array([[x % int(p) for x in vals] for p in dst.primes], dtype=np.int32))
    src.destroy()
    dst.destroy()
