"""Scale refinement and loss with one H_in per head through the tensor-core products: heads that are no whole tiles of
128 rows, wide groups, groups of 32 columns (no tensor-core Yw), with and without the propagated-error term."""
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu

CD, ADAPT = 2, 1


@pytest.mark.parametrize("dh,gq,with_r,flags", [(64, 256, False, CD | ADAPT), (64, 128, True, CD | ADAPT), (40, 64, False, CD),
                                                (136, 0, False, CD), (64, 32, True, CD | ADAPT), (72, 128, True, 0)])
def test_heads_of_any_size(dh, gq, with_r, flags):
    prob = make_problem(70, 512, 3, dh, 1024, n_hin=3, with_r=with_r, hout="spd")
    compare(prob, run_gpu(prob, 4, gq, 8, flags), 4, gq, 8, flags, label=f"heads{dh}")


def test_groups_of_32_columns_shared_hessian():
    prob = make_problem(71, 512, 3, 64, 1024, with_r=True)
    compare(prob, run_gpu(prob, 3, 32, 16, CD | ADAPT), 3, 32, 16, CD | ADAPT, label="gq32")


# coordinates per head (rows x groups): 21, 256 (one group), 33 x 6, 128 x 8, 512 x 4 (the most), 64 x 16, 128 x 24 and 17
# heads of 128 x 8 (walked row by row)
@pytest.mark.parametrize("d,heads,dh,gq,iters", [(384, 2, 21, 0, 1), (256, 1, 256, 0, 2), (384, 3, 33, 64, 1), (512, 2, 64, 32, 1),
                                                 (1024, 1, 128, 128, 2), (512, 1, 512, 128, 1), (768, 1, 128, 32, 1),
                                                 (1024, 17, 128, 128, 1)])
def test_coordinates_per_head(d, heads, dh, gq, iters):
    prob = make_problem(72, d, heads, dh, 2048, hout="spd")
    compare(prob, run_gpu(prob, 3, gq, dh, CD | ADAPT, cd_iters=iters), 3, gq, dh, CD | ADAPT, cd_iters=iters, label=f"coords{dh}")


# heads walked row by row with the row's columns staged in shared memory: 16 and 32 groups, rows that end inside a block of 16
# and beyond a fold's 64, a cluster of one CTA and of several, a group of zeros (a coordinate that is skipped)
@pytest.mark.parametrize("d,heads,dh,gq,iters", [(1024, 2, 21, 64, 1), (2048, 3, 150, 64, 2), (1152, 1, 97, 128, 1),
                                                 (2048, 30, 16, 64, 1)])
def test_rows_staged_in_shared_memory(d, heads, dh, gq, iters):
    prob = make_problem(73, d, heads, dh, 2048, hout="spd")
    prob["W"][3, :gq] = 0.0
    compare(prob, run_gpu(prob, 3, gq, dh, CD | ADAPT, cd_iters=iters), 3, gq, dh, CD | ADAPT, cd_iters=iters, label=f"staged{dh}")


def test_more_rows_than_a_grid_dimension_holds():
    """66 560 rows with one scale each in one batch: heads at the beginning, past row 65 535 and at the end."""
    prob = make_problem(74, 128, 520, 128, 512, hout="spd")
    flags = CD | ADAPT
    gpu = run_gpu(prob, 3, 0, 32, flags)
    compare(prob, gpu, 3, 0, 32, flags, heads=[0, 511, 512, 519], label="rows66560")


@pytest.mark.parametrize("with_r", [False, True])
def test_heads_whose_pieces_go_through_in_two_launches(with_r):
    """12 heads of 8192 columns, 10 to a launch: every head has the same H_in, so the result is that of the shared one (the
    products per head are the same, only the launches differ)."""
    import torch
    import paper_2602_04929_b200 as tb
    H, dh, d, dev = 12, 8, 8192, "cuda:0"
    g = torch.Generator(device=dev).manual_seed(9)
    V = torch.randn(d, 16, generator=g, device=dev) / 16
    Hin = V @ V.T
    Hin = 0.5 * (Hin + Hin.T)
    Hin.diagonal().add_(1.0)
    U, info = tb.tb_factor(Hin)
    W = 0.02 * torch.randn(H * dh, d, generator=g, device=dev)
    Ho = torch.eye(dh, device=dev) + 0.3
    Hout = Ho.expand(H, dh, dh).contiguous()
    Uout, _ = tb.tb_factor(Hout)
    ops = [None] * 3
    if with_r:
        R = 0.05 * torch.randn(d, d, generator=g, device=dev) / d ** 0.5
        ops = [R, *tb.tb_prepare_correction(R, U)]

    def run(n_hin):
        def per(t):
            return None if t is None else t.expand(n_hin, d, d).contiguous()
        desc = tb.layer_desc(H * dh, d, H, dh, 3, 128, 8, n_hin=n_hin, flags=CD | ADAPT)
        out = tb.tb_quantize_layer(desc, W, per(Hin), per(U), Hout, Uout, *[per(t) for t in ops], want_loss=False)
        torch.cuda.synchronize()
        return out

    one, many = run(1), run(H)
    assert torch.equal(one.codes, many.codes) and torch.equal(one.zeros, many.zeros)
    assert float((one.scales - many.scales).norm() / one.scales.norm()) <= 1e-6
