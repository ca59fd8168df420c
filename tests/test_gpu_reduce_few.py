"""Reductions of large matrices of short entries modulo few primes, which go by limb
sums: the same results as their parts, which are small enough for digit products."""
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


def _words(rows, cols, pad, W, seed, bits=None):
    """Random entries (sign-extended from `bits`), both ends among them, rows cols + pad entries apart."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    X = torch.randint(-(1 << 63), (1 << 63) - 1, (rows, cols + pad, W), dtype=torch.int64, device="cuda", generator=g)
    if bits is not None:
        X[..., 0] >>= 63 - bits
        X[..., 1:] = X[..., :1] >> 63
    X[0, 0], X[-1, cols - 1], X[rows // 2, 0] = 0, -1, 0
    X[rows // 2, 0, 0] = 1
    if bits is None:
        X[1, 0, -1], X[2, 0, -1] = -(1 << 63), (1 << 63) - 1
        X[1, 0, :-1], X[2, 0, :-1] = 0, -1
    else:
        X[1, 0], X[2, 0] = 0, -1
        X[1, 0, 0], X[2, 0, 0] = 1 << bits, -(1 << bits)
    return X[:, :cols]


@pytest.mark.parametrize("bound,W", [(20, 1), (20, 2), (20, 4), (40, 1), (40, 2), (60, 1)])
@pytest.mark.parametrize("rows,cols,pad", [(512, 512, 0), (1031, 257, 1), (3, 90_001, 2), (300_000, 1, 0)])
def test_canonical(ctx, bound, W, rows, cols, pad):
    b = ctx.basis_create(bound)
    L = len(b.primes)
    X = _words(rows, cols, pad if W % 2 else 2 * pad, W, rows + W)
    out = torch.full((L, rows, cols), -1, dtype=torch.int32, device="cuda")
    ctx.rns_reduce(b, X, out)
    step = max(1, (1 << 17) // cols)
    for r in range(0, rows, step):
        part = X[r:r + step].clone()  # (an aligned copy)
        for c in range(0, cols, 1 << 17):
            p = part[:, c:c + (1 << 17)].clone()  # (an aligned copy)
            want = torch.empty((L,) + tuple(p.shape[:2]), dtype=torch.int32, device="cuda")
            ctx.rns_reduce(b, p, want)
            assert torch.equal(out[:, r:r + step, c:c + (1 << 17)], want)
    ctx.status_sync()
    b.destroy()


# a_bits + 64 Wb - 1 + log2 k gives 4 to 13 primes, on both sides of the rule
@pytest.mark.parametrize("Wb,a_bits", [(1, 1), (1, 20), (1, 40), (1, 63), (2, 1), (2, 20), (2, 63)])
@pytest.mark.parametrize("k,n,pad", [(128, 2100, 0), (300, 1003, 1), (4097, 129, 0)])
def test_transposed(ctx, Wb, a_bits, k, n, pad):
    m = 5
    A = _words(m, k, 0, 1, k, min(a_bits, 62)) if a_bits < 63 else _words(m, k, 0, 1, k)
    B = _words(k, n, pad, Wb, n + Wb)
    W = (64 * Wb + a_bits + k.bit_length() + 66) // 64
    C = torch.zeros((m, n, W), dtype=torch.int64, device="cuda")
    ctx.rns_matmul(A, B, C, a_bits=a_bits)
    step = (1 << 18) // k // 2
    for c in range(0, n, step):
        p = B[:, c:c + step].clone()  # (an aligned copy)
        want = torch.zeros((m, p.shape[1], W), dtype=torch.int64, device="cuda")
        ctx.rns_matmul(A, p, want, a_bits=a_bits)
        assert torch.equal(C[:, c:c + step], want)
    ctx.status_sync()


@pytest.mark.parametrize("W,bits", [(1, 30), (1, 62), (2, 40)])
def test_declared_bound(ctx, smf, W, bits):
    k, n = 256, 1100
    A = torch.ones((3, k, 1), dtype=torch.int64, device="cuda")
    B = _words(k, n, 0, W, bits, bits)
    C = torch.zeros((3, n, W + 1), dtype=torch.int64, device="cuda")
    ctx.rns_matmul(A, B, C, a_bits=1, b_bits=bits)  # both ends of the bound are allowed
    ctx.status_sync()
    for x in ((1 << bits) + 1, -(1 << bits) - 1):
        D = B.clone()
        D[k - 1, n - 3, 0] = x
        D[k - 1, n - 3, 1:] = x >> 63
        ctx.rns_matmul(A, D, C, a_bits=1, b_bits=bits)
        with pytest.raises(smf.SmfError) as e:
            ctx.status_sync()
        assert e.value.code == smf.SMF_E_BOUND
