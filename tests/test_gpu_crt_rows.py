"""CRT into matrices whose rows lie further apart than they are long: the same
words as into a matrix without gaps, and nothing written between the rows."""
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


# rows shorter than a warp's 32 entries (several ends of a row between two words of a lane) and longer
@pytest.mark.parametrize("rows,cols,pad", [(700, 1, 1), (301, 2, 5), (97, 5, 1), (33, 31, 2), (5, 1000, 64)])
@pytest.mark.parametrize("bound,W", [(20, 1), (170, 3), (543, 9), (543, 33), (1100, 18)])
def test_gaps(ctx, rows, cols, pad, bound, W):
    b = ctx.basis_create(bound)
    g = torch.Generator(device="cuda")
    g.manual_seed(rows * W)
    r = torch.stack([torch.randint(0, int(p), (rows, cols), dtype=torch.int32, device="cuda", generator=g)
                     for p in b.primes])
    want = torch.zeros((rows, cols, W), dtype=torch.int64, device="cuda")
    ctx.crt_reconstruct(b, r, want)
    buf = torch.full((rows, cols + pad, W), 77, dtype=torch.int64, device="cuda")
    ctx.crt_reconstruct(b, r, buf[:, :cols])
    ctx.status_sync()
    assert torch.equal(buf[:, :cols], want)
    assert bool((buf[:, cols:] == 77).all())
    b.destroy()
