"""Column sweep: every way rows are dealt to CTAs (clusters of 8, 4 and 2 CTAs, 8, 16 and 32 rows per CTA), ragged
rows, one to several blocks of 128 columns, values far outside the grid, and the propagated-error term."""
import numpy as np
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu

ADAPT = 1


def _case(prob, bits, gq, g, flags=ADAPT):
    return compare(prob, run_gpu(prob, bits, gq, g, flags), bits, gq, g, flags, label=f"sweep g{g}")


# rows of a step: 5 (cluster of 8), 150 (4 CTAs), 300 (4), 590 (2), 900 (8 rows a CTA), 1300 (16), 2500 (32)
@pytest.mark.parametrize("heads,dh", [(1, 5), (6, 25), (12, 25), (10, 59), (18, 50), (13, 100), (25, 100)])
@pytest.mark.parametrize("with_r", [False, True])
def test_rows_per_cta(heads, dh, with_r):
    prob = make_problem(60, 512, heads, dh, 1024, with_r=with_r, hout="spd" if dh < 60 else None)
    _case(prob, 3, 128, dh)


@pytest.mark.parametrize("d", [128, 256, 1152])
def test_blocks(d):
    prob = make_problem(61, d, 3, 24, 1024, hout="spd")
    _case(prob, 2, 32, 8)


@pytest.mark.parametrize("n_hin", [3])
def test_one_hessian_per_head(n_hin):
    prob = make_problem(62, 384, 3, 40, 1024, n_hin=n_hin, with_r=True, hout="spd")
    _case(prob, 4, 64, 20)


def test_values_beyond_the_integer_range():
    """A row whose later columns are 2^40 times its grid (all-zero first group, fixed grid of another group) saturates
    like the oracle's clamp: the walk's range test has to see it."""
    prob = make_problem(63, 256, 2, 16, 1024, hout="spd")
    W = prob["W"]
    W[3, :] *= 1e-9
    W[3, 128:] *= 1e3
    W[5, 0:32] = 0.0
    W[5, 7] = 1e-12
    _case(prob, 2, 32, 16, flags=0)
