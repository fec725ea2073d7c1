"""Column sweep: every way rows are dealt to CTAs (clusters of 8, 4 and 2 CTAs, 8, 16 and 32 rows per CTA), ragged
rows, one to several blocks of 128 columns, values far outside the grid, and the propagated-error term."""
import numpy as np
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu

ADAPT = 1


def _case(prob, bits, gq, g, flags=ADAPT):
    return compare(prob, run_gpu(prob, bits, gq, g, flags), bits, gq, g, flags, label=f"sweep g{g}")


# rows of a step: 5 (cluster of 8), 150 (4 CTAs), 300 and 590 (2), 900 (8 rows a CTA), 1300 (16), 2500 (32)
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


# the sweep after an update of few rows: 48 CTAs, launched ahead of the update's own wait, and 96, which are not
@pytest.mark.parametrize("n_hin", [3, 12])
@pytest.mark.parametrize("with_r", [False, True])
def test_one_hessian_per_head_beyond_512_columns(n_hin, with_r):
    prob = make_problem(67, 768, n_hin, 32, 1024, n_hin=n_hin, with_r=with_r, hout="spd")
    _case(prob, 3, 128, 16)


def test_one_hessian_per_head_and_many_rows():
    """As many rows of as many columns as take digit products with a shared factor: with one per head they do not."""
    prob = make_problem(66, 640, 2, 1920, 1024, n_hin=2, hout=None)
    _case(prob, 3, 128, 1920)


# one big factor entry a column, so that the rounding error of the first column drives every later one to a chosen magnitude
# in units of its grid, 2^31 and far beyond, in both directions; columns of the first piece of 16, of the first block of 128
# and of the second
@pytest.mark.parametrize("flags", [0, 4])
def test_values_beyond_the_integer_range(flags):
    """The walk's range test has to see them, and the code is the end of the grid that the value lies beyond."""
    d, gq, bits = 256, 128, 4
    prob = make_problem(63, d, 3, 16, 1024, hout=None)
    rng = np.random.default_rng(5)
    U = np.eye(d)
    cols = np.r_[1:16, 20:128:3, 130:256:2] if flags == 0 else np.r_[1:16, 20:128:3]
    # x = w / s + z - e U[0][c] / s: e is up to s / 2, so the magnitudes below reach both sides of 6.8e15 and 1.4e16
    U[0, cols] = rng.choice([-1.0, 1.0], len(cols)) * 10.0 ** rng.uniform(8.0, 18.0, len(cols))
    prob["Uin"] = U[None].astype(np.float32)
    gpu = run_gpu(prob, bits, gq, 16, flags)
    rep = compare(prob, gpu, bits, gq, 16, flags, label=f"beyond{flags}")
    assert rep["code_mismatch"] == 0
    W, u = prob["W"].astype(np.float64), prob["Uin"][0].astype(np.float64)
    sc, z = np.repeat(gpu["scales"], gq, 1).astype(np.float64), np.repeat(gpu["zeros"], gq, 1)
    e = W[:, 0] - sc[:, 0] * (gpu["codes"][:, 0].astype(np.float64) - z[:, 0])
    x = (W - e[:, None] * u[0][None, :]) / sc + z
    assert np.any(x[:, cols] > 2.0 ** 31) and np.any(x[:, cols] < -2.0 ** 31)
    assert np.any((x[:, cols] > -1.35e16) & (x[:, cols] < -6.8e15))


# few rows (rank-512 updates straight from the factor) and many (digit products)
@pytest.mark.parametrize("heads,dh", [(2, 12), (16, 128)])
def test_a_weight_that_is_no_number(heads, dh):
    """Everything behind it in its row is no number either and takes code 0; no other row notices."""
    prob = make_problem(64, 640, heads, dh, 1024, hout=None)
    clean = run_gpu(prob, 3, 128, dh, 0, want_loss=False)
    prob["W"][5, 40] = np.nan
    gpu = run_gpu(prob, 3, 128, dh, 0, want_loss=False)
    assert np.all(gpu["codes"][5, 40:] == 0)
    others = np.arange(heads * dh) != 5
    for k in ("codes", "scales", "zeros", "cand"):
        assert np.array_equal(gpu[k][others], clean[k][others]), k


def test_more_rows_than_a_grid_dimension_holds():
    """66 000 rows in one step, and columns beyond the first 512: the last rows against the oracle."""
    n, d = 66000, 640
    prob = make_problem(65, d, 1, 48, 1024, hout=None)
    reps = n // 48
    big = dict(prob, W=np.tile(prob["W"], (reps, 1)), d_out=n, d_head=n)
    gpu = run_gpu(big, 3, 128, n, ADAPT, want_loss=False)
    rows = np.r_[0:48, 65520:65568, n - 48:n].reshape(3, 48)
    for r in rows:
        part = {k: (v[r] if k in ("codes", "scales", "zeros", "cand", "w_hat", "w_comp") else v) for k, v in gpu.items()}
        compare(prob, part, 3, 128, 48, ADAPT, label=f"rows{r[0]}")
