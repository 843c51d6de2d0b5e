"""A reservation for which the sliced products' workspaces do not fit: the call
runs on the FP32 pipes and says so in its tiles."""
import pytest

pytestmark = pytest.mark.gpu

Nd, Nq, Nx, Ny, Nt, B = 200, 2, 16, 8, 20, 512


@pytest.fixture(scope="module")
def ctx():
    import torch
    from paper_2504_16344_gb300 import tw
    g = torch.Generator(device="cuda").manual_seed(1)
    c = tw.Context(Nd, Nq, Nx, Ny, Nt, keep=tw.KEEP_FP64)
    c.set_prior(1.0, 0.1, 1.0)
    for which, rows in ((tw.MAP_F, Nd), (tw.MAP_FQ, Nq)):
        c.set_block_column(which, 0, torch.randn((Nt, rows, Nx * Ny), generator=g, dtype=torch.float64, device="cuda"))
    c.factor_K(1e3)
    yield c
    c.close()


class Short:
    """The rest of the device's memory held, but for what a reservation takes less 90 MB
    (its slices are over 160 of some 350 MB, and come last)."""

    def __init__(self, ctx):
        import torch
        ctx.reserve_batch(0)
        torch.cuda.empty_cache()
        f = self.free()
        ctx.reserve_batch(B)
        self.need = f - self.free()
        ctx.reserve_batch(0)

    @staticmethod
    def free():
        import torch
        return torch.cuda.mem_get_info()[0]

    def __enter__(self):
        import torch
        self.held = []
        while self.free() > self.need + (64 << 30):
            self.held.append(torch.empty(60 << 30, dtype=torch.uint8, device="cuda"))
        self.held.append(torch.empty(self.free() - self.need + (90 << 20), dtype=torch.uint8, device="cuda"))

    def __exit__(self, *_):
        import torch
        self.held.clear()
        torch.cuda.empty_cache()


def test_reservation_without_room_for_the_slices(ctx):
    import torch
    from paper_2504_16344_gb300 import tw
    d = torch.randn((B, Nt, Nd), generator=torch.Generator(device="cuda").manual_seed(2), dtype=torch.float64,
                    device="cuda")
    win = torch.full((B,), Nt, dtype=torch.int32, device="cuda")
    m = torch.empty((B, Nt, Nx * Ny), dtype=torch.float64, device="cuda")
    q = torch.empty((B, Nt, Nq), dtype=torch.float64, device="cuda")
    short = Short(ctx)
    tw.autotune_clear_cache()
    with short:
        ctx.reserve_batch(B)
        tiles = ctx.batch_tiles()
        ctx.infer_batch(tw.PREC_FP64, d, win, m, q)
        m0, q0 = m.cpu(), q.cpu()
        ctx.check()
        ctx.reserve_batch(0)
    tw.autotune_clear_cache()
    assert tiles.adj_rw in (1, 2, 4)
    ctx.reserve_batch(B)
    ctx.set_batch_tiles(tiles.adj_tile, tiles.adj_rw, tiles.fwd_lanes)
    ctx.infer_batch(tw.PREC_FP64, d, win, m, q)
    ctx.check()
    # (set by hand, these tiles take the sweeps off the tensor cores too: the solves' bound)
    assert (m.cpu() - m0).norm() / m0.norm() < 1e-11 and (q.cpu() - q0).norm() / q0.norm() < 1e-11


def test_choice_without_the_slices_is_not_kept_for_others(ctx):
    """The measured tiles of such a reservation are not taken over by one with room,
    whose products run on the tensor cores (several times faster at this size)."""
    from paper_2504_16344_gb300 import tw
    short = Short(ctx)
    tw.autotune_clear_cache()
    with short:
        ctx.reserve_batch(B)
        tight = ctx.batch_tiles().adj_rw
        ctx.reserve_batch(0)
    ctx.reserve_batch(B)
    assert tight in (1, 2, 4) and ctx.batch_tiles().adj_rw == 0
