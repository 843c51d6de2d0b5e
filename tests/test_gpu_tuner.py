"""The measured choice of the FP64-class products: each in the form that suits it."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nd,Nq", [(2, 40), (100, 1)])
def test_tuned_call_is_as_fast_as_the_fastest_fixed_choice(Nd, Nq):
    """Two sensors and 40 forecast points: the adjoint is next to nothing in either form,
    the forward product takes twice as long on the FP32 pipes; with 100 and one it is
    the other way round for the adjoint."""
    import torch
    from paper_2504_16344_gb300 import tw
    Nx, Ny, Nt, B = 100, 125, 60, 2
    g = torch.Generator(device="cuda").manual_seed(1)
    ctx = tw.Context(Nd, Nq, Nx, Ny, Nt, keep=tw.KEEP_FP64)
    ctx.set_prior(1.0, 0.1, 1.0)
    for which, rows in ((tw.MAP_F, Nd), (tw.MAP_FQ, Nq)):
        ctx.set_block_column(which, 0, torch.randn((Nt, rows, Nx * Ny), generator=g, dtype=torch.float64, device="cuda"))
    ctx.factor_K(1e3)
    tw.autotune_clear_cache()
    ctx.reserve_batch(B)
    tiles = ctx.batch_tiles()
    d = torch.randn((B, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    ms = {}
    for rw in ("tuned", 0, 1, 2, 4):
        if rw != "tuned":
            ctx.set_batch_tiles(tiles.adj_tile, rw, tiles.fwd_lanes)
        for _ in range(3):
            ctx.infer_batch(tw.PREC_FP64, d, win)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            ctx.infer_batch(tw.PREC_FP64, d, win)
        b.record()
        torch.cuda.synchronize()
        ms[rw] = a.elapsed_time(b) / 10
    print(Nd, Nq, ms)
    ctx.check()
    ctx.close()
    assert ms["tuned"] < 1.2 * min(ms.values()), ms
