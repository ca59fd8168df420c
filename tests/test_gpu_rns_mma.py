"""CRT and base conversion on the tensor cores, against Python's integers: every
size of the kernels' tables at its edges, ragged and unaligned residue planes,
values whose carries pass many limbs and whose quotient is settled exactly."""
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


def _values(M, count, seed):
    H = (M - 1) // 2
    v = [0, -1, 1, H, -H, H - 1, 1 - H, M // 3, -(M // 3), H // 2]
    v += [s * (1 << b) for b in range(0, M.bit_length() - 2, 13) for s in (1, -1)]
    rng = np.random.default_rng(seed)
    while len(v) < count:
        v.append(int.from_bytes(rng.bytes(M.bit_length() // 8 + 8), "little") % M - H)
    at = rng.permutation(len(v))[:count]
    return [v[i] for i in at]


def _planes(vals, primes, shift):
    """[L][count] residues on the GPU, the first plane `shift` words past a 16-byte boundary."""
    r = np.array([[x % p for x in vals] for p in primes], dtype=np.int32)
    buf = torch.zeros(r.size + 8, dtype=torch.int32, device="cuda")
    out = buf[shift:shift + r.size].view(r.shape)
    out.copy_(torch.from_numpy(r))
    return out


# (bits, largest prime): 1, 2, 8, 9, 16, 17, 24, 25, 32, 33, 47 and 48 primes, and small ones
BASES = [(20, 0), (40, 0), (191, 0), (200, 0), (383, 0), (390, 0), (575, 0), (580, 0), (767, 0), (780, 0), (1120, 0),
         (1150, 0), (100, 1 << 11), (9, 50)]


@pytest.mark.parametrize("bits,pmax", BASES)
@pytest.mark.parametrize("rows,cols,pad,shift", [(1, 1, 0, 0), (4, 33, 0, 0), (7, 19, 3, 0), (25, 16, 0, 1)])
def test_crt(ctx, bits, pmax, rows, cols, pad, shift):
    basis = ctx.basis_create(bits, pmax)
    M = math.prod(int(p) for p in basis.primes)
    vals = _values(M, rows * cols, bits)
    W = M.bit_length() // 64 + 1 + (bits % 3)
    buf = torch.full((rows, cols + pad, W), 77, dtype=torch.int64, device="cuda")
    ctx.crt_reconstruct(basis, _planes(vals, basis.primes, shift), buf[:, :cols])
    ctx.status_sync()
    got = buf.cpu().numpy()
    want = np.frombuffer(b"".join(x.to_bytes(8 * W, "little", signed=True) for x in vals), dtype=np.int64)
    assert np.array_equal(got[:, :cols], want.reshape(rows, cols, W))
    assert (got[:, cols:] == 77).all()
    basis.destroy()


@pytest.mark.parametrize("bits,pmax", BASES)
@pytest.mark.parametrize("to_bits,to_pmax,count,shift", [(20, 0, 1, 0), (200, 0, 33, 0), (575, 0, 132, 0),
                                                         (1150, 0, 260, 1), (90, 1 << 12, 400, 0), (8, 40, 31, 0)])
def test_convert(ctx, bits, pmax, to_bits, to_pmax, count, shift):
    src, dst = ctx.basis_create(bits, pmax), ctx.basis_create(to_bits, to_pmax)
    vals = _values(math.prod(int(p) for p in src.primes), count, bits + to_bits)
    out = torch.full((len(dst.primes) * count + 8,), -1, dtype=torch.int32, device="cuda")
    view = out[shift:shift + len(dst.primes) * count].view(len(dst.primes), count)
    ctx.base_convert(src, dst, _planes(vals, src.primes, shift), view)
    ctx.status_sync()
    want = np.array([[x % int(q) for x in vals] for q in dst.primes], dtype=np.int32)
    assert np.array_equal(view.cpu().numpy(), want)
    assert (out[:shift] == -1).all() and (out[shift + view.numel():] == -1).all()
    src.destroy()
    dst.destroy()


def _ints(t):
    w = t.cpu().numpy()
    return [int.from_bytes(x.tobytes(), "little", signed=True) for x in w.reshape(-1, w.shape[-1])]


def _entries(rows, cols, pad, W, seed, bits=None):
    """[rows, cols, W] words on the GPU with extreme values first, rows cols + pad entries apart."""
    b = 64 * W - 1 if bits is None else bits
    top = (1 << b) - (bits is None)
    v = [0, -1, 1, top, -(1 << b), 1 << (b // 2), -(1 << (b // 2)), 255, -256]
    v = [x for x in v if -(1 << b) <= x <= top]
    rng = np.random.default_rng(seed)
    while len(v) < rows * cols:
        v.append(int.from_bytes(rng.bytes(8 * W + 8), "little") % ((1 << (b + 1)) - 1) - (1 << b) + 1)
    v = v[:rows * cols]
    data = b"".join(x.to_bytes(8 * W, "little", signed=True) for x in v)
    buf = torch.zeros((rows, cols + pad, W), dtype=torch.int64, device="cuda")
    buf[:, :cols] = torch.from_numpy(np.frombuffer(data, dtype=np.int64).reshape(rows, cols, W).copy()).cuda()
    return buf[:, :cols], v


@pytest.mark.parametrize("bits,pmax", [(20, 0), (200, 0), (575, 0), (1150, 0), (1530, 0), (100, 1 << 11), (9, 50)])
@pytest.mark.parametrize("W", [1, 2, 3, 4, 8])
@pytest.mark.parametrize("rows,cols,pad", [(1, 1, 0), (5, 32, 0), (3, 67, 2), (9, 36, 1)])
def test_reduce(ctx, bits, pmax, W, rows, cols, pad):
    basis = ctx.basis_create(bits, pmax)
    X, v = _entries(rows, cols, pad, W, bits + W)
    L = len(basis.primes)
    out = torch.full((L, rows, cols), -1, dtype=torch.int32, device="cuda")
    ctx.rns_reduce(basis, X, out)
    ctx.status_sync()
    want = np.array([[x % int(p) for x in v] for p in basis.primes], dtype=np.int32)
    assert np.array_equal(out.cpu().numpy().reshape(L, -1), want)
    basis.destroy()


@pytest.mark.parametrize("grouped", [False, True])
@pytest.mark.parametrize("Wa,Wb", [(1, 8), (2, 1), (4, 8), (8, 2), (3, 4)])
@pytest.mark.parametrize("m,k,n,pad", [(3, 5, 2, 0), (33, 36, 17, 0), (20, 65, 9, 1)])
def test_digits(ctx, Wa, Wb, m, k, n, pad, grouped):
    A, va = _entries(m, k, pad, Wa, 1)
    B, vb = _entries(k, n, pad, Wb, 2)
    W = (64 * (Wa + Wb) + k.bit_length() + 64) // 64
    C = torch.zeros((m, n, W), dtype=torch.int64, device="cuda")
    if grouped:
        ctx.rns_matmul_grouped([A], [B], [C])
    else:
        ctx.rns_matmul(A, B, C)
    ctx.status_sync()
    want = [sum(va[i * k + t] * vb[t * n + j] for t in range(k)) for i in range(m) for j in range(n)]
    assert _ints(C) == want


@pytest.mark.parametrize("W,bits", [(1, 30), (1, 62), (2, 64), (4, 31), (4, 95), (8, 100), (8, 510), (8, 32)])
def test_declared_bound(ctx, W, bits):
    from paper_2605_19254_gb300 import smf
    k, n = 40, 35
    A = torch.ones((4, k, 1), dtype=torch.int64, device="cuda")
    C = torch.zeros((4, n, W + 2), dtype=torch.int64, device="cuda")
    B, v = _entries(k, n, 0, W, bits, bits)  # both ends of the bound are allowed
    ctx.rns_matmul(A, B, C, a_bits=1, b_bits=bits)
    ctx.status_sync()
    assert _ints(C)[:n] == [sum(v[t * n + j] for t in range(k)) for j in range(n)]
    for x in ((1 << bits) + 1, -(1 << bits) - 1, 1 << (bits + 1) if bits < 64 * W - 2 else (1 << bits) + (1 << (bits - 1))):
        B2 = B.clone()
        B2[k - 1, n - 2] = torch.from_numpy(np.frombuffer(x.to_bytes(8 * W, "little", signed=True), dtype=np.int64).copy()).cuda()
        ctx.rns_matmul(A, B2, C, a_bits=1, b_bits=bits)
        with pytest.raises(smf.SmfError) as e:
            ctx.status_sync()
        assert e.value.code == smf.SMF_E_BOUND


@pytest.mark.parametrize("a_bits", [1, 7, 15, 20])  # one, two and three digits
@pytest.mark.parametrize("k,pad", [(1, 0), (7, 0), (8, 0), (8, 1), (9, 1), (40, 8), (65, 0)])  # (odd row lengths: 8-byte aligned rows)
def test_grouped_split(ctx, a_bits, k, pad):
    m, n = 35, 6
    _, va = _entries(m, k, 0, 1, a_bits + k, a_bits)
    A = torch.zeros((m, k + pad, 1), dtype=torch.int64, device="cuda")[:, :k]
    A.copy_(torch.tensor(va, dtype=torch.int64).view(m, k, 1))
    B, vb = _entries(k, n, 0, 2, 3)
    C = torch.zeros((m, n, 3), dtype=torch.int64, device="cuda")
    ctx.rns_matmul_grouped([A], [B], [C], a_bits=a_bits)
    ctx.status_sync()
    assert _ints(C) == [sum(va[i * k + t] * vb[t * n + j] for t in range(k)) for i in range(m) for j in range(n)]
    from paper_2605_19254_gb300 import smf
    A[m - 1, k - 1, 0] = (1 << a_bits) + 1
    ctx.rns_matmul_grouped([A], [B], [C], a_bits=a_bits)
    with pytest.raises(smf.SmfError) as e:
        ctx.status_sync()
    assert e.value.code == smf.SMF_E_BOUND
