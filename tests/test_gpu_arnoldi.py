"""GPU check of the correction solve's Arnoldi pass against FP64: solves cannot show its errors, as
the outer iteration absorbs them.

C -= A y: a and y are rounded to FP32 (2^-24 each) and p terms summed by FP32 FMAs, so each entry is
within (p + 2) 2^-24 sum_i |a_i y_i| (first order; one more 2^-24 covers the rest), values below the
FP32 normal range within 2^-126 (1 + sum |y|).  G = A^T C adds FP32 products of at most 21 rows per
thread here, five steps in the warp and eight warps, of operands rounded once: 36 roundings, 40
2^-24 sum |a c|; the norm is in FP64.
"""
import pytest

from gpu_common import torch, require_gpu

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _case(p, rows, batch, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)

    def r(*n):
        return torch.randn(*n, generator=g, dtype=torch.float64, device="cuda")

    lda, bsa = rows + 3, (p + 1) * (rows + 3)
    A, Y, C = r(batch, p + 1, lda), r(batch, 17), r(batch, rows + 5)
    return A, lda, bsa, Y, C


def _run(ctx, A, lda, bsa, p, Y, C, rows, gram, batch):
    from paper_2111_02534_gb300 import tps
    G = torch.full((batch, 17), float("nan"), dtype=torch.float64, device="cuda")
    st = tps._lib.tps_selftest_arnoldi_pass(
        ctx._h, A.data_ptr(), lda, bsa, p, Y.data_ptr(), 17, C.data_ptr(), C.stride(0), rows,
        int(gram), G.data_ptr(), 17, batch, torch.cuda.current_stream().cuda_stream)
    assert st == tps.OK
    torch.cuda.synchronize()
    return G


# every width of the kernel and one below it; single rows, remainders of a block and of a pair of
# rows, several chunks; integer conversions from 2^20 rows on
@pytest.mark.parametrize("p,rows,batch", [(1, 1, 1), (2, 255, 3), (3, 256, 1), (4, 513, 2),
                                          (5, 1025, 3), (8, 4099, 1), (9, 70001, 2),
                                          (16, 131584, 3), (1, (1 << 20) + 7, 1), (3, 1 << 20, 2),
                                          (8, (1 << 20) + 255, 1), (16, (1 << 20) + 1025, 3)])
@pytest.mark.parametrize("gram", [True, False])
def test_update_and_product(p, rows, batch, gram):
    require_gpu()
    from paper_2111_02534_gb300 import tps
    ctx = tps.Context(1, 0)
    A, lda, bsa, Y, C0 = _case(p, rows, batch, 5 + p)
    A[:, :p, :rows:7] *= 1e-42        # FP32 subnormals
    A[:, :p, 3:rows:11] *= 1e-300     # below FP32 altogether
    C = C0.clone()
    G = _run(ctx, A, lda, bsa, p, Y, C, rows, gram, batch)
    a, y = A[:, :p, :rows], Y[:, :p]
    want = C0[:, :rows] - torch.einsum("bpr,bp->br", a, y)
    size = torch.einsum("bpr,bp->br", a.abs(), y.abs())
    tiny = 2.0 ** -126 * (1 + y.abs().sum(1, keepdim=True))
    bound = (p + 3) * U * size + tiny + 2.0 ** -52 * (C0[:, :rows].abs() + size)
    assert bool(((C[:, :rows] - want).abs() <= bound).all())
    assert torch.equal(C[:, rows:], C0[:, rows:])
    c = C[:, :rows]  # the products are of the column as the pass left it
    if gram:
        want = torch.einsum("bpr,br->bp", a, c)
        size = torch.einsum("bpr,br->bp", a.abs(), c.abs())
        tiny = 2.0 ** -126 * (1 + c.abs().sum(1, keepdim=True))
        assert bool(((G[:, :p] - want).abs() <= 40 * U * size + tiny).all())
        assert bool(G[:, p:].isnan().all())
    else:
        want = (c * c).sum(1)
        assert bool(((G[:, 0] - want).abs() <= 1e-13 * want).all())
        assert bool(G[:, 1:].isnan().all())
    ctx.close()


def test_integer_conversion_rounds_to_nearest():
    # columns 0 and a (odd columns are converted by integer instructions), y = (0, 1), C = 0: C
    # becomes minus the FP32 value of each entry.  Halfway cases, the ends of the normal range, and
    # what lies beyond it
    require_gpu()
    from paper_2111_02534_gb300 import tps
    ctx = tps.Context(1, 0)
    rows = 1 << 20
    g = torch.Generator(device="cuda").manual_seed(1)
    bits = torch.randint(-(1 << 62), 1 << 62, (rows,), generator=g, device="cuda")
    a = bits.view(torch.float64).clone()          # every exponent, NaN and infinity among them
    x = torch.randn(rows // 2, generator=g, dtype=torch.float64, device="cuda")
    f = x.float().double()
    a[:rows // 2] = f
    half = torch.ldexp(f.sign(), torch.frexp(f)[1] - 25)
    a[:rows // 4] += half[:rows // 4]             # the middle between two FP32 numbers
    a[:8] = torch.tensor([0.0, -0.0, 1 + 2.0 ** -24, -(1 + 2.0 ** -24), 2.0 ** -126,
                          2.0 ** -127, 3.4028234663852886e38, 3.4028235677973366e38],
                         dtype=torch.float64, device="cuda")
    A = torch.stack([torch.zeros_like(a), a])
    C = torch.zeros(1, rows, dtype=torch.float64, device="cuda")
    Y = torch.zeros(1, 17, dtype=torch.float64, device="cuda")
    Y[0, 1] = 1.0
    _run(ctx, A, rows, 2 * rows, 2, Y, C, rows, False, 1)
    got, want = -C[0], a.float().double()
    small = a.abs() < 2.0 ** -126                  # flushed, or kept
    assert bool((got[small].abs() <= 2.0 ** -126).all())
    big = a.abs() >= 3.4028235677973366e38
    assert bool((got[big] == want[big]).all())
    rest = ~(small | big | a.isnan())
    up = torch.nextafter(want[rest].float(), want[rest].float() * 4).double()
    tie = (a[rest] - want[rest]).abs() * 2 == (up - want[rest]).abs()
    assert bool(((got[rest] == want[rest]) | tie).all())
    assert bool(((got[rest] - a[rest]).abs() <= (want[rest] - a[rest]).abs()).all())
    assert bool(got[a.isnan()].isnan().all())
    ctx.close()


def test_arguments_are_checked():
    require_gpu()
    from paper_2111_02534_gb300 import tps
    ctx = tps.Context(1, 0)
    x = torch.zeros(2, 64, dtype=torch.float64, device="cuda")
    p = x.data_ptr()
    good = dict(A=p, lda=64, bsa=0, p=1, Y=p, bsy=17, C=p, bsc=64, nrows=64, gram=1, G=p, bsg=17,
                batch=1)
    for bad in ({"p": 0}, {"p": 17}, {"lda": 8}, {"Y": None}, {"batch": 0}, {"nrows": 0},
                {"bsc": 63}, {"p": 2, "bsg": 1}):
        args = {**good, **bad}.values()
        assert tps._lib.tps_selftest_arnoldi_pass(ctx._h, *args, None) == tps.ERR_INVALID_ARG, bad
    ctx.close()
