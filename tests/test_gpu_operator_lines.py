"""GPU checks of the operator line by line: the rows of the periodic second derivative, and the
tensor-core H-apply on lines of very different size, each against its own scale, and on more
vectors than one launch takes.
"""
import math

import numpy as np
import pytest

from gpu_common import torch, require_gpu, make_ctx_1d, make_ctx_2d

pytestmark = pytest.mark.gpu
FAR = 1e20  # a box so long that the mode's products vanish beside the smallest line's rounding


def _random(nvec, N, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(nvec, N, generator=g, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [64, 66, 130, 512, 1024])
def test_rows_of_the_second_derivative_vanish_on_constants(n):
    # unit vectors give the entries to the bit (FP64 products with 0 and 1; the other mode's are
    # below half a unit of the diagonal).  Two entries of a row, at distance four, hold what the
    # rounding of the others left: each is rounded once, so a row sums to at most their unit
    require_gpu()
    from paper_2111_02534_gb300 import tps
    ctx = make_ctx_1d(20.0, 1.0, (4, n), (FAR, 20.0), 1.0, 1.0, V=np.zeros(4 * n))
    psi = torch.zeros(n, 4, n, dtype=torch.float64, device="cuda")
    psi[:, 0] = torch.eye(n, dtype=torch.float64, device="cuda")
    out = torch.empty_like(psi)
    ctx.apply_h(psi.view(n, -1), out.view(n, -1), 0.0, dtype=tps.F64)
    K = out[:, 0].T.cpu().numpy()
    ctx.close()
    assert np.array_equal(K, K.T)
    assert np.array_equal(K, np.roll(K, (1, 1), (0, 1)))  # circulant
    assert abs(math.fsum(K[0])) <= 1.001 * np.spacing(abs(K[0, 4]))


# FP64's own rounding is what the bounds of the next two cover: at most n / 8 + 8 terms in a run,
# 2^-53 of a row's absolute sum each, so 1e-14 of ||H|| times the line's largest entry
SCALES = 2.0 ** -(37 * torch.arange(1024, dtype=torch.float64) % 59)


@pytest.mark.parametrize("nx,ny", [(60, 130), (290, 12), (580, 16), (146, 34), (64, 66), (12, 10),
                                   (256, 128), (8, 294), (16, 584)])
@pytest.mark.parametrize("mode", ["y", "x"])
def test_1d_lines_have_their_own_scale(nx, ny, mode):
    require_gpu()
    from paper_2111_02534_gb300 import tps
    L = (FAR, 15.0) if mode == "y" else (15.0, FAR)
    ctx = make_ctx_1d(20.0, 1.0, (nx, ny), L, 1.0, 1.0, V=np.zeros(nx * ny))
    hn = ctx.info()[1]
    psi = _random(2, nx * ny, 3).view(2, nx, ny)
    s = SCALES.cuda()
    psi *= s[:nx, None] if mode == "y" else s[:ny]
    psi[1] = psi[1].flip(0, 1)
    out, ref = torch.empty_like(psi), torch.empty_like(psi)
    ctx.apply_h(psi.view(2, -1), out.view(2, -1), 0.0, dtype=tps.F64_TC)
    ctx.apply_h(psi.view(2, -1), ref.view(2, -1), 0.0, dtype=tps.F64)
    ctx.device_status()
    d = 2 if mode == "y" else 1
    assert bool(((out - ref).abs().amax(d) <= 1e-14 * hn * psi.abs().amax(d)).all())
    ctx.close()


@pytest.mark.parametrize("nx,ny", [(6, 18), (18, 6), (8, 48), (50, 8), (64, 4), (4, 66), (66, 4)])
@pytest.mark.parametrize("mode", ["y", "x"])
def test_2d_lines_have_their_own_scale(nx, ny, mode):
    # the fibers of the two modes of one particle share a scale, all others have their own
    require_gpu()
    from paper_2111_02534_gb300 import tps
    L = (FAR, FAR, 8.0, 8.0) if mode == "y" else (8.0, 8.0, FAR, FAR)
    n = (nx, nx, ny, ny)
    ctx = make_ctx_2d(20.0, 1.0, n, L, 2.0, 1.0)
    ctx.set_potential(np.zeros(nx * nx * ny * ny))
    hn = ctx.info()[1]
    psi = _random(2, nx * nx * ny * ny, 7).view(2, nx * nx, ny * ny)
    s = SCALES.cuda().repeat(5)
    psi *= s[:nx * nx, None] if mode == "y" else s[:ny * ny]
    out, ref = torch.empty_like(psi), torch.empty_like(psi)
    ctx.apply_h(psi.view(2, -1), out.view(2, -1), 0.0, dtype=tps.F64_TC)
    ctx.apply_h(psi.view(2, -1), ref.view(2, -1), 0.0, dtype=tps.F64)
    ctx.device_status()
    d = 2 if mode == "y" else 1
    assert bool(((out - ref).abs().amax(d) <= 1e-14 * hn * psi.abs().amax(d)).all())
    ctx.close()


@pytest.mark.parametrize("n,nvec", [((12, 10), 130), ((66, 50), 70), ((512, 512), 30),
                                    ((8, 294), 67), ((6, 6, 8, 8), 130), ((4, 4, 66, 66), 66)])
def test_blocks_of_more_vectors_than_a_launch_takes(n, nvec):
    # whole numbers inside: a vector's result is the same to the bit in any block
    require_gpu()
    from paper_2111_02534_gb300 import tps
    L = (9.0,) * len(n)
    make = make_ctx_1d if len(n) == 2 else make_ctx_2d
    ctx = make(20.0, 1.0, n, L, 1.0, 1.0)
    N = ctx.info()[0]
    psi = _random(nvec, N, 9)
    out, one = torch.empty_like(psi), torch.empty(1, N, dtype=torch.float64, device="cuda")
    ctx.apply_h(psi, out, -0.3, dtype=tps.F64_TC)
    for v in (0, 1, 22, 63, 64, nvec - 1):
        if v < nvec:
            ctx.apply_h(psi[v:v + 1], one, -0.3, dtype=tps.F64_TC)
            ctx.device_status()
            assert torch.equal(out[v], one[0]), v
    ctx.close()


@pytest.mark.parametrize("n", [(64, 66), (60, 130), (12, 12, 18, 18), (6, 6, 48, 48)])
@pytest.mark.parametrize("k", [-1015, -1000, -960, -940, 870, 900, 930, 1000])
def test_results_near_the_ends_of_the_range(n, k):
    # the recombination scales by exponent arithmetic, near the ends of FP64's range in two factors:
    # a wave function times 2^k against the plain one, whose sums are the same integers.  The mode
    # products count subnormals as zero; the potential term takes them as they are
    require_gpu()
    from paper_2111_02534_gb300 import tps
    L = (9.0,) * len(n)
    ctx = (make_ctx_1d if len(n) == 2 else make_ctx_2d)(20.0, 1.0, n, L, 1.0, 1.0)
    N, hn = ctx.info()
    assert hn < 2.0 ** 12
    V = -np.random.default_rng(5).random(N)
    ctx.set_potential(V)
    psi = _random(2, N, 11)
    ref, out = torch.empty_like(psi), torch.empty_like(psi)
    big = psi * 2.0 ** k
    kept = torch.where(big.abs() >= 2.0 ** -1022, psi, 0.0)
    ctx.apply_h(kept, ref, -0.3, dtype=tps.F64_TC)
    ref += (torch.from_numpy(V).cuda() + 0.3) * (psi - kept)
    ctx.apply_h(big, out, -0.3, dtype=tps.F64_TC)
    ctx.device_status()
    # below 2^-1022 a result has 2^-1074 left, 2^-59 of the scale here
    bound = 1e-14 * hn * float(psi.abs().max())
    assert bool(out.isfinite().all())
    assert bool(((out * 2.0 ** -k - ref).abs() <= bound).all())
    ctx.close()
