"""The FP64-class products of exact slices hold every sum as closely as
double-float does, however far its entries lie below the largest ones: the
guards find the sums that the slices would lose digits of.  Measured against the
same call on the FP32 pipes in double-float."""
import pytest

pytestmark = pytest.mark.gpu


def _context(Nd, Nx, Ny, Nt, B, F, Fq, noise):
    from paper_2504_16344_gb300 import tw
    ctx = tw.Context(Nd, Fq.shape[1], Nx, Ny, Nt, keep=tw.KEEP_FP64)
    ctx.set_prior(1.0, 0.1, 1.0)
    ctx.set_block_column(tw.MAP_F, 0, F)
    ctx.set_block_column(tw.MAP_FQ, 0, Fq)
    ctx.factor_K(noise)
    ctx.reserve_batch(B)
    return tw, ctx


def _randn(seed, *shape):
    import torch
    return torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(seed), dtype=torch.float64,
                       device="cuda")


# rows: part of a 16-row step, one exact chunk, two; columns: below a tile, a full
# one, one more; grid points past a tile of 128.  spread: powers of two by which one
# sensor's rows lie above the others', and its data below theirs
@pytest.mark.parametrize("spread", [0, 24, 40])
@pytest.mark.parametrize("Nd,Nx,Ny,B", [(5, 5, 7, 3), (20, 9, 15, 32), (110, 13, 10, 33)])
def test_adjoint_of_wide_range(Nd, Nx, Ny, B, spread):
    import torch
    Nt = 5
    F, Fq = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, 2, Nx * Ny)
    F[:, 1] *= 2.0 ** spread
    F[:, :, 3] = 0.0                                   # a point that no sensor sees
    # noise far above the signal: y is the data, scaled
    tw, ctx = _context(Nd, Nx, Ny, Nt, B, F, Fq, 1e6 * Nx * Ny * 4.0 ** spread)
    d = _randn(3, B, Nt, Nd)
    d[:, :, 1] *= 2.0 ** -spread
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    win[B - 1] = 0                                     # an empty slot beside them
    m = {}
    for rw in (0, 4):
        ctx.set_batch_tiles(8, rw, 1)
        m[rw], _ = ctx.infer_batch(tw.PREC_FP64, d, win)
    ctx.set_batch_tiles(8, 0, 1)
    one, _ = ctx.infer_batch(tw.PREC_FP64, d[1:2].contiguous(), win[1:2].contiguous())
    bad = d.clone()
    bad[0, 0, 0] = float("nan")
    mates, _ = ctx.infer_batch(tw.PREC_FP64, bad, win)
    ctx.check()
    ctx.close()
    # n roundings of 2^-47 of the terms' sum, which is sqrt(n) times a sum of random sign
    n = 2 * Nd
    for b in range(B - 1):
        e = (m[0][b] - m[4][b]).norm() / m[4][b].norm()
        assert e < 2.0 ** -47 * n ** 1.5, (b, float(e))
    assert not m[0][B - 1].any()
    # no column depends on its batch mates
    assert torch.equal(one[0], m[0][1])
    assert torch.equal(mates[1:], m[0][1:]) and torch.isnan(mates[0]).all()


# several tiles per CTA (2 x 81 frequencies x 2 column tiles on 152 SMs): an odd
# number of stages, and two exact chunks
@pytest.mark.parametrize("Nd,B", [(20, 33), (110, 32)])
def test_adjoint_over_several_tiles_per_cta(Nd, B):
    import torch
    Nx, Ny, Nt = 15, 25, 80
    F, Fq = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, 2, Nx * Ny)
    tw, ctx = _context(Nd, Nx, Ny, Nt, B, F, Fq, 1e6 * Nx * Ny)
    d = _randn(3, B, Nt, Nd)
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    m = {}
    for rw in (0, 4):
        ctx.set_batch_tiles(8, rw, 1)
        m[rw], _ = ctx.infer_batch(tw.PREC_FP64, d, win)
    ctx.check()
    ctx.close()
    for b in range(B):
        e = (m[0][b] - m[4][b]).norm() / m[4][b].norm()
        assert e < 2.0 ** -47 * (2 * Nd) ** 1.5, (b, float(e))
