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


# a forecast of fields that are large where the map is small.  Rows: X^ on the MMA
# rows (16 and 32 columns), F^ on them (100 rows); grid points: two ranges, the
# second of 32; columns: part of a tile and more than one
@pytest.mark.parametrize("spread", [0, 24, 40])
@pytest.mark.parametrize("Nq,B", [(2, 2), (20, 70), (100, 33)])
def test_forward_of_wide_range(Nq, B, spread):
    import torch
    Nd, Nx, Ny, Nt = 2, 65, 64, 5
    F, Fq, m = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, Nq, Nx * Ny), _randn(3, B, Nt, Nx * Ny)
    Fq[:, 1:, 100:] *= 2.0 ** -spread                  # row 0 stays as it is
    m[:, :, :100] *= 2.0 ** -spread
    m[B - 1] = 0.0
    tw, ctx = _context(Nd, Nx, Ny, Nt, B, F, Fq, 1e6 * Nx * Ny)
    q = {}
    for rw in (0, 4):
        ctx.set_batch_tiles(8, rw, 1)
        q[rw] = ctx.forecast_batch(tw.PREC_FP64, m)
    ctx.set_batch_tiles(8, 0, 1)
    one = ctx.forecast_batch(tw.PREC_FP64, m[:1].contiguous())
    bad = m.clone()
    bad[1, 0, 7] = float("nan")
    mates = ctx.forecast_batch(tw.PREC_FP64, bad)
    ctx.check()
    ctx.close()
    # n terms of random sign: running sums grow as sqrt(k), n independent roundings of
    # 2^-48 of them come to sqrt(n / 2) 2^-48 of the result; four times that for each side
    tol = 8 * 2.0 ** -48 * (2 * Nx * Ny) ** 0.5
    for b in range(B - 1):
        e = ((q[0][b] - q[4][b]).norm(dim=0) / q[4][b].norm(dim=0)).max()        # every forecast point by itself
        assert e < tol, (b, float(e))
    assert not q[0][B - 1].any()
    assert torch.equal(one[0], q[0][0])
    keep = [b for b in range(B) if b != 1]
    assert torch.equal(mates[keep], q[0][keep]) and torch.isnan(mates[1]).all()


# sweeps in panels (132 block rows) whose loud right-hand sides meet small entries of
# the factor: half of the sensors measure 2^spread times less, and their data are
# that much larger, so the two halves' terms come out alike
@pytest.mark.parametrize("spread", [0, 24, 40])
@pytest.mark.parametrize("B", [64, 70])
def test_sweeps_of_wide_range(B, spread):
    import torch
    Nd, Nx, Ny, Nt = 200, 6, 5, 42
    F, Fq = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, 2, Nx * Ny)
    F[:, ::2] *= 2.0 ** -spread
    tw, ctx = _context(Nd, Nx, Ny, Nt, 1, F, Fq, 1.0 * Nx * Ny * Nt)
    d = _randn(3, B, Nt, Nd)
    d[:, :, ::2] *= 2.0 ** spread
    win = [1 + (7 * b + Nt - 1) % Nt for b in range(B)]
    ctx.reserve_batch(0)                               # single-vector solves
    ref = ctx.infer(tw.PREC_FP64, d, windows=win)
    ctx.reserve_batch(B)
    dev = torch.tensor(win, dtype=torch.int32, device="cuda")
    m, _ = ctx.infer_batch(tw.PREC_FP64, d, dev)
    one, _ = ctx.infer_batch(tw.PREC_FP64, d[B - 1:], dev[B - 1:])
    bad = d.clone()
    bad[1, 0, 0] = float("nan")
    mates, _ = ctx.infer_batch(tw.PREC_FP64, bad, dev)
    ctx.check()
    ctx.close()
    # two solves in 48-bit arithmetic, K's condition a few hundred: the bound of
    # test_batched_solves in test_gpu_slices.py
    for b in range(B):
        e = (m[b] - ref[b]).norm() / ref[b].norm()
        assert e < 1e-11, (b, float(e))
    assert torch.equal(one[0], m[B - 1])
    keep = [b for b in range(B) if b != 1]
    assert torch.equal(mates[keep], m[keep])


# several (frequency, range, tile) items per CTA: 81 x 2 of X^ on the MMA rows, 81 x 2
# x 2 of F^ on them
@pytest.mark.parametrize("Nq,B", [(20, 40), (100, 33)])
def test_forward_over_several_items_per_cta(Nq, B):
    import torch
    Nd, Nx, Ny, Nt = 2, 65, 64, 80
    F, Fq, m = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, Nq, Nx * Ny), _randn(3, B, Nt, Nx * Ny)
    tw, ctx = _context(Nd, Nx, Ny, Nt, B, F, Fq, 1e6 * Nx * Ny)
    q = {}
    for rw in (0, 4):
        ctx.set_batch_tiles(8, rw, 1)
        q[rw] = ctx.forecast_batch(tw.PREC_FP64, m)
    ctx.check()
    ctx.close()
    tol = 8 * 2.0 ** -48 * (2 * Nx * Ny) ** 0.5        # as above
    for b in range(B):
        e = ((q[0][b] - q[4][b]).norm(dim=0) / q[4][b].norm(dim=0)).max()
        assert e < tol, (b, float(e))


# more row and column tiles in the first panels' updates (85 x 2) than SMs
def test_sweeps_over_several_tiles_per_cta():
    import torch
    Nd, Nx, Ny, Nt, B = 200, 6, 5, 58, 65
    F, Fq = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, 2, Nx * Ny)
    tw, ctx = _context(Nd, Nx, Ny, Nt, 1, F, Fq, 1.0 * Nx * Ny * Nt)
    d = _randn(3, B, Nt, Nd)
    win = [1 + (7 * b + Nt - 1) % Nt for b in range(B)]
    ctx.reserve_batch(0)                               # single-vector solves
    ref = ctx.infer(tw.PREC_FP64, d, windows=win)
    ctx.reserve_batch(B)
    m, _ = ctx.infer_batch(tw.PREC_FP64, d, torch.tensor(win, dtype=torch.int32, device="cuda"))
    ctx.check()
    ctx.close()
    for b in range(B):
        e = (m[b] - ref[b]).norm() / ref[b].norm()
        assert e < 1e-11, (b, float(e))                # as above


def test_sweeps_can_be_kept_off_the_tensor_cores():
    """adj_rw 1, 2 or 4 set by the caller: one launch a sweep instead of panels, the same
    results within the solves' bound."""
    import torch
    Nd, Nx, Ny, Nt, B = 200, 6, 5, 42, 64
    F, Fq = _randn(1, Nt, Nd, Nx * Ny), _randn(2, Nt, 2, Nx * Ny)
    tw, ctx = _context(Nd, Nx, Ny, Nt, B, F, Fq, 1.0 * Nx * Ny * Nt)
    d = _randn(3, B, Nt, Nd)
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    m, q, count = {}, torch.empty((B, Nt, 2), dtype=torch.float64, device="cuda"), {}
    for rw in (0, 4):
        ctx.set_batch_tiles(8, rw, 1)
        m[rw] = torch.empty((B, Nt, Nx * Ny), dtype=torch.float64, device="cuda")
        with torch.cuda.stream(stream):
            ctx.infer_batch(tw.PREC_FP64, d, win, m[rw], q, stream=stream)
            stream.synchronize()
            with ctx.capture(stream) as cap:
                ctx.infer_batch(tw.PREC_FP64, d, win, m[rw], q, stream=stream)
            count[rw] = cap.graph.kernel_count()
            cap.graph.close()
    ctx.check()
    ctx.close()
    # eleven panels a sweep, five kernels each, against one
    assert count[4] < 30 and count[0] > count[4] + 80, count
    assert (m[0] - m[4]).norm() / m[4].norm() < 1e-11
