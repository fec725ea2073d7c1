"""Scale refinement and loss with one H_in per head: heads that are and are no whole tiles of 128 rows (the tensor-core
products, and double), wide groups, groups of 32 columns, with and without the propagated-error term."""
import numpy as np
import pytest

from parity_util import compare, make_problem, run_gpu, run_oracle

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


# groups that are no multiple of 64 columns; with one H_in per head groups wider than 128, and heads that are no multiple of
# 128 rows (with refinement, and the loss alone)
@pytest.mark.parametrize("d,heads,dh,n_hin,gq,with_r,flags", [
    (512, 3, 64, 1, 32, True, CD | ADAPT), (1152, 2, 64, 1, 96, False, CD | ADAPT), (512, 3, 64, 3, 256, False, CD | ADAPT),
    (512, 3, 128, 3, 0, True, CD), (512, 3, 40, 3, 64, True, CD), (512, 3, 72, 3, 128, True, 0), (512, 12, 8, 12, 32, False, CD),
])
def test_refinement_and_loss_in_double(d, heads, dh, n_hin, gq, with_r, flags):
    """What is formed in double: scales are the oracle's, rounded to float once (but for ties of that rounding), the loss
    agrees to sums in another order (512 .. 1152 terms of 2^-53 each way, a cancellation of up to 100)."""
    prob = make_problem(77, d, heads, dh, 1024, n_hin=n_hin, with_r=with_r, hout="spd")
    gpu = run_gpu(prob, 4, gq, 8, flags)
    rep = compare(prob, gpu, 4, gq, 8, flags, label=f"double{dh}")
    res, _ = run_oracle(prob, gpu, 4, gq, 8, flags)
    assert np.count_nonzero(gpu["scales"] != res.scales.astype(np.float32)) <= 1
    assert rep["loss_rel"] <= 1e-13
