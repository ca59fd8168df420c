"""CRT of up to nine primes against Python's integers: values x + (M - 1)/2 = y
with y / M at every distance from 0 and 1, where the quotient is settled by the
fp32 sum, in fixed point, or by mixed radix."""
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


@pytest.mark.parametrize("p_max", [1 << 24, 1 << 26, 1 << 11, 60])
@pytest.mark.parametrize("L", [1, 2, 3, 5, 8, 9])
def test_quotients(ctx, L, p_max):
    b = ctx.basis_create(max(1, int(L * (math.log2(p_max) - 0.01 if p_max > 60 else 5.2)) - 3), p_max)
    primes = [int(p) for p in b.primes]
    M = math.prod(primes)
    H = (M - 1) // 2
    ys = {0, 1, M - 1, M - 2, M // 2}
    for k in range(1, 80):
        for d in (-1, 0, 1, 12345):
            for y in ((M >> k) + d, M - 1 - (M >> k) + d, M * 3 // 7 + (M >> k) + d):
                ys.add(y % M)
    vals = [y - H for y in sorted(ys)]
    W = M.bit_length() // 64 + 1
    r = np.array([[x % p for x in vals] for p in primes], dtype=np.int32)
    X = torch.full((1, len(vals), W), 77, dtype=torch.int64, device="cuda")
    ctx.crt_reconstruct(b, torch.from_numpy(r[:, None, :].copy()).cuda(), X)
    ctx.status_sync()
    want = np.frombuffer(b"".join(x.to_bytes(8 * W, "little", signed=True) for x in vals), dtype=np.int64)
    assert np.array_equal(X.cpu().numpy().ravel(), want)
    b.destroy()
