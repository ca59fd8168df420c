"""Eliminations whose passes go beside the next panel (from about n = 770 with four
moduli, 1500 with one) against the same elimination one column at a time, and local
forms with deferred columns against their planted factors."""
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


Q31 = [2147483647, 2147483629, 2147483587, 2147483579]


@pytest.mark.parametrize("n,primes", [(761, 4), (775, 4), (1057, 2), (1100, 2), (1089, 3), (1500, 1)])
def test_dets(ctx, n, primes):
    A = torch.from_numpy(inputs.uniform_int(n, "A", (n, n), -100, 100)[..., None].copy()).cuda()
    q = Q31[:primes]
    got = [ctx.det_mod(A, q, a_bits=7) for _ in range(3)]
    ctx.set_elim_panels(1 << 30)
    want = ctx.det_mod(A, q, a_bits=7)
    ctx.set_elim_panels(0)
    assert got == [want] * 3


@pytest.mark.parametrize("n", [800, 1100])
def test_local_forms(ctx, n):
    """U diag(s) V with blocks of 2, 3 and 5: columns without a joint unit all along."""
    s = [1] * (n - 60) + [2] * 20 + [6] * 20 + [60] * 20
    A = inputs.smith_known_matrix_np(n, s, n)
    dA = torch.from_numpy(A[..., None].copy()).cuda()
    q, e = [2, 3, 5], [4, 3, 2]
    bits = max(1, int(np.abs(A).max()).bit_length())
    for _ in range(3):
        got = ctx.smith_local(dA, q, e, a_bits=bits)
        for p, k, c in zip(q, e, got):
            assert list(c) == [sum(v % p ** t == 0 for v in s) for t in range(k + 1)]
