"""Products whose operands are cut into exact bf16 slices (tensor cores)
against the same call on the FP32 pipes in double-float, at the sizes where
tiles, chunks and columns end."""
import pytest

pytestmark = pytest.mark.gpu


def _context(Nd, Nx, Ny, Nt, B, keep_g=False):
    import torch
    from paper_2504_16344_gb300 import tw
    keep = tw.KEEP_FP64 | (tw.KEEP_G if keep_g else 0)
    ctx = tw.Context(Nd, 3, Nx, Ny, Nt, keep=keep)
    ctx.set_prior(1.0, 0.1, 1.0)
    g = torch.Generator(device="cuda").manual_seed(Nd + 7 * B)
    for which, rows in ((tw.MAP_F, Nd), (tw.MAP_FQ, 3)):
        col = torch.randn((Nt, rows, Nx * Ny), generator=g, dtype=torch.float64, device="cuda")
        ctx.set_block_column(which, 0, col)
    # noise far above the signal: K is well conditioned, F^T y hardly cancels
    ctx.factor_K(1e6 * Nx * Ny)
    ctx.reserve_batch(B)
    d = torch.randn((B, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    d *= 10.0 ** torch.arange(-3, B - 3, dtype=torch.float64, device="cuda")[:, None, None].clamp(max=3.0)
    win = torch.tensor([Nt - b % Nt for b in range(B)], dtype=torch.int32, device="cuda")
    return tw, ctx, d, win


# rows: one stage, an odd and an even number of stages, the last exact single
# chunk (102) and the first two-chunk sizes; grid points around the 128-row
# tile; right-hand sides around the tiles of 8, 16, 24, 32 and beyond
@pytest.mark.parametrize("Nd,Nx,Ny,B,keep_g", [
    (1, 5, 7, 1, False), (8, 16, 8, 8, False), (9, 3, 43, 9, True), (16, 16, 16, 16, False),
    (17, 11, 13, 24, False), (100, 10, 13, 32, True), (102, 16, 17, 33, False), (103, 9, 15, 25, False),
    (200, 12, 12, 40, False)])
def test_products_on_tensor_cores(Nd, Nx, Ny, B, keep_g):
    import torch
    tw, ctx, d, win = _context(Nd, Nx, Ny, 6, B, keep_g)
    out = {}
    for rw in (0, 4):
        ctx.set_batch_tiles(8, rw, 1)
        m, q = ctx.infer_batch(tw.PREC_FP64, d, win)
        # a sample's update of m_pr (a window of 0 leaves m_pr): F m_pr with all Nd rows
        z = torch.randn(m.shape, generator=torch.Generator(device="cuda").manual_seed(5), dtype=torch.float64,
                        device="cuda")
        zero = torch.zeros_like(d)
        s = ctx.sample_posterior_batch(tw.PREC_FP64, zero, z, zero, 1.0, win)
        s0 = ctx.sample_posterior_batch(tw.PREC_FP64, zero, z, zero, 1.0, torch.zeros_like(win))
        ctx.check()
        out[rw] = m.clone(), q.clone(), s - s0
    ctx.close()
    # both sums carry errors of a few 2^-48 of their terms, and n terms of random
    # sign sum to sqrt(n) of their size: n 2^-46 covers every term's worst case
    # (m: n = 2 Nd; q and the samples after it: 2 Nm).  The update of a sample is
    # read off as a difference of FP64 values, each rounded at 2^-53.
    n = 2 * max(Nd, Nx * Ny, 8)
    for k in range(3):
        for b in range(B):
            e = (out[0][k][b] - out[4][k][b]).norm() / out[4][k][b].norm()
            tol = 2.0 ** -46 * n + (2.0 ** -51 * s0[b].norm() / out[4][k][b].norm() if k == 2 else 0.0)
            assert e < tol, (k, b, float(e))


# one sweep with narrow slices (1 right-hand side, an odd number of them, one
# and several block rows), then panels: 132 block rows (11 full panels), 172 and
# 260 (part panels, odd pairs of blocks), right-hand sides that take tiles of 64,
# 48 and 32 columns (and 16, one alone), windows that end inside the panels
@pytest.mark.parametrize("Nd,Nt,B", [(7, 9, 1), (50, 33, 17), (49, 33, 40), (200, 42, 64), (200, 42, 65),
                                     (199, 55, 48), (200, 83, 32)])
def test_batched_solves(Nd, Nt, B):
    import torch
    from paper_2504_16344_gb300 import tw
    Nx, Ny = 6, 5
    ctx = tw.Context(Nd, 2, Nx, Ny, Nt, keep=tw.KEEP_FP64)
    ctx.set_prior(1.0, 0.1, 1.0)
    g = torch.Generator(device="cuda").manual_seed(Nd + Nt + B)
    ctx.set_block_column(tw.MAP_F, 0, torch.randn((Nt, Nd, Nx * Ny), generator=g, dtype=torch.float64,
                                                  device="cuda"))
    ctx.set_block_column(tw.MAP_FQ, 0, torch.randn((Nt, 2, Nx * Ny), generator=g, dtype=torch.float64,
                                                   device="cuda"))
    ctx.factor_K(1.0 * Nx * Ny * Nt)       # K's condition stays below a few hundred
    d = torch.randn((B, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    win = [1 + (7 * b + Nt - 1) % Nt for b in range(B)]
    ref = ctx.infer(tw.PREC_FP64, d, windows=win)          # single-vector solves: no batch is reserved
    ctx.reserve_batch(B)
    m, _ = ctx.infer_batch(tw.PREC_FP64, d, torch.tensor(win, dtype=torch.int32, device="cuda"))
    # the same right-hand sides one at a time: bitwise the same (no batch mates)
    one, _ = ctx.infer_batch(tw.PREC_FP64, d[B - 1:], torch.tensor(win[-1:], dtype=torch.int32, device="cuda"))
    ctx.check()
    assert torch.equal(one[0], m[B - 1])
    # two backward-stable solves in 48-bit arithmetic: condition x 2^-46 x a
    # modest growth, below 1e-11 as the library's FP64 bound
    for b in range(B):
        e = (m[b] - ref[b]).norm() / ref[b].norm()
        assert e < 1e-11, (b, float(e))
    ctx.close()
