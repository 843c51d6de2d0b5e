"""Batched calls on a forecast map of which only some rows are loaded: the
loaded rows come out as they do from the whole map."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reserve_first", [False, True])
def test_loaded_rows_of_a_partly_loaded_map(reserve_first):
    import torch
    from paper_2504_16344_gb300 import tw
    Nd, Nq, Nx, Ny, Nt, B = 5, 4, 9, 7, 6, 3
    g = torch.Generator(device="cuda").manual_seed(3)
    F, Fq = (torch.randn((Nt, n, Nx * Ny), generator=g, dtype=torch.float64, device="cuda") for n in (Nd, Nq))
    d = torch.randn((B, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    m = torch.randn((B, Nt, Nx * Ny), generator=g, dtype=torch.float64, device="cuda")
    win = torch.tensor([Nt, 2, 4], dtype=torch.int32, device="cuda")
    with_all, q = None, {}
    for rows in (Nq, 2):
        ctx = tw.Context(Nd, Nq, Nx, Ny, Nt, keep=tw.KEEP_FP64)
        ctx.set_prior(1.0, 0.1, 1.0)
        ctx.set_block_column(tw.MAP_F, 0, F)
        load = lambda: ctx.set_block_column(tw.MAP_FQ, 0, Fq[:, :rows].contiguous())
        if not reserve_first:
            load()
        ctx.factor_K(1e3)
        ctx.reserve_batch(B)
        if reserve_first:
            load()
        ctx.set_batch_tiles(8, 0, 1)          # the products on the tensor cores
        q[rows] = ctx.infer_batch(tw.PREC_FP64, d, win)[1][..., :2], ctx.forecast_batch(tw.PREC_FP64, m, win)[..., :2]
        ctx.check()
        ctx.close()
    for k in range(2):
        assert torch.equal(q[2][k], q[Nq][k])      # a row's sum does not depend on the other rows


def test_reloaded_rows_under_a_reservation():
    """New block columns after tw_reserve_batch: the sliced products read the
    operator that is loaded now (its entries 2^20 times the first one's)."""
    import torch
    from paper_2504_16344_gb300 import tw
    Nd, Nq, Nx, Ny, Nt, B = 5, 4, 9, 7, 6, 3
    g = torch.Generator(device="cuda").manual_seed(4)
    F, Fq = (torch.randn((Nt, n, Nx * Ny), generator=g, dtype=torch.float64, device="cuda") for n in (Nd, Nq))
    d = torch.randn((B, Nt, Nd), generator=g, dtype=torch.float64, device="cuda")
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    ctx = tw.Context(Nd, Nq, Nx, Ny, Nt, keep=tw.KEEP_FP64)
    ctx.set_prior(1.0, 0.1, 1.0)
    ctx.set_block_column(tw.MAP_F, 0, F)
    ctx.set_block_column(tw.MAP_FQ, 0, Fq)
    ctx.factor_K(1e3)
    ctx.reserve_batch(B)
    ctx.set_batch_tiles(8, 0, 1)
    m0, q0 = ctx.infer_batch(tw.PREC_FP64, d, win)
    ctx.set_block_column(tw.MAP_F, 2, (F[:, 2:] * 2.0 ** 20).contiguous())
    ctx.set_block_column(tw.MAP_F, 0, (F[:, :2] * 2.0 ** 20).contiguous())
    ctx.set_block_column(tw.MAP_FQ, 1, (Fq[:, 1:] * 2.0 ** 20).contiguous())
    m1, q1 = ctx.infer_batch(tw.PREC_FP64, d, win)
    ctx.check()
    ctx.close()
    # powers of two move exponents only
    assert torch.equal(m1, m0 * 2.0 ** 20)
    assert torch.equal(q1[..., 1:], q0[..., 1:] * 2.0 ** 40) and torch.equal(q1[..., 0], q0[..., 0] * 2.0 ** 20)
