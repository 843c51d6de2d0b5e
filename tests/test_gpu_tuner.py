"""The measured choice of the FP64-class products counts both products that it
decides about."""
import pytest

pytestmark = pytest.mark.gpu


def test_choice_counts_the_forward_product():
    """Two sensors and 40 forecast points: the adjoint is next to nothing in either form,
    the forward product twice as long on the FP32 pipes."""
    import torch
    from paper_2504_16344_gb300 import tw
    Nd, Nq, Nx, Ny, Nt, B = 2, 40, 100, 125, 60, 2
    g = torch.Generator(device="cuda").manual_seed(1)
    ctx = tw.Context(Nd, Nq, Nx, Ny, Nt, keep=tw.KEEP_FP64)
    ctx.set_prior(1.0, 0.1, 1.0)
    for which, rows in ((tw.MAP_F, Nd), (tw.MAP_FQ, Nq)):
        ctx.set_block_column(which, 0, torch.randn((Nt, rows, Nx * Ny), generator=g, dtype=torch.float64, device="cuda"))
    ctx.factor_K(1e3)
    tw.autotune_clear_cache()
    ctx.reserve_batch(B)
    chosen = ctx.batch_tiles()
    d = torch.randn((B, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    ms = {}
    for rw in (0, 1, 2, 4):
        ctx.set_batch_tiles(chosen.adj_tile, rw, chosen.fwd_lanes)
        for _ in range(3):
            ctx.infer_batch(tw.PREC_FP64, d, win)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            ctx.infer_batch(tw.PREC_FP64, d, win)
        b.record()
        torch.cuda.synchronize()
        ms[rw] = a.elapsed_time(b) / 10
    ctx.check()
    ctx.close()
    assert ms[chosen.adj_rw] < 1.3 * min(ms.values()), (chosen.adj_rw, ms)     # the others are 1.8 times as long
