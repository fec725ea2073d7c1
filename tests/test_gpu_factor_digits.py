"""tb_factor from 1024 columns on, where the wide products run on the integer tensor cores: sizes at the edges of its
blocks (64, 256, 512 columns and their powers of two), rows of very different scale, and the info words."""
import numpy as np
import pytest

import oracle
import tb_inputs
from parity_util import rel_fro

pytestmark = pytest.mark.gpu


def _factor(H, **kw):
    import torch
    import paper_2602_04929_b200 as tb
    out = tb.tb_factor(torch.from_numpy(H).to("cuda:0"), **kw)
    torch.cuda.synchronize()
    assert tb.tb_device_error_flag() == 0
    return [t.cpu().numpy() for t in out]


# below the switch with a short last block; the smallest size above it; a last block of 64, of 128 and a half; more
# than one level above 512 with a short second half at each
@pytest.mark.parametrize("d,n_batch", [(700, 1), (961, 1), (1090, 2), (1664, 1), (2120, 1), (2600, 1)])
def test_factor_sizes(d, n_batch):
    """The factor is formed in double precision and rounded once: half an ulp of float is 6e-8."""
    H = np.stack([tb_inputs.spd_matrix(40 + b, d, cond=1e4) for b in range(n_batch)])
    U, info, Hinv = _factor(H, want_inverse=True)
    assert info.tolist() == [0] * n_batch
    for b in range(n_batch):
        assert np.all(np.tril(U[b], -1) == 0.0)
        assert rel_fro(U[b], oracle.factor_upper(H[b:b + 1])[0]) <= 6e-8
        assert rel_fro(Hinv[b], np.linalg.inv(H[b].astype(np.float64))) <= 1e-6


def test_factor_of_rows_of_very_different_scale():
    """H = S A S with S from 1e-6 to 1e6 (powers of two): U is the factor of A with scaled columns, bit for bit."""
    d = 1100
    A = tb_inputs.spd_matrix(50, d, cond=1e4)
    s = np.exp2(np.random.default_rng(1).integers(-20, 21, d)).astype(np.float32)
    U0, _ = _factor(A)
    U1, info = _factor(A * s[:, None] * s[None, :])
    assert info.tolist() == [0]
    assert np.array_equal(U1 * s[None, :], U0)


@pytest.mark.parametrize("what", ["negative", "nan", "inf"])
def test_factor_names_the_first_bad_pivot(what):
    """Row r of the elimination order is row d - 1 - r: a negative diagonal entry, or an entry that is no number in
    the second block of columns to the left of pivot 900, is reported there."""
    d, r = 1100, 900
    H = tb_inputs.spd_matrix(51, d, cond=1e3)
    if what == "negative":
        H[d - 1 - r, d - 1 - r] = -1.0
    else:
        bad = np.float32(what)
        H[d - 1 - r, d - 1 - 300] = H[d - 1 - 300, d - 1 - r] = bad
    _, info = _factor(H)
    assert info.tolist() == [r + 1]


def test_factor_of_the_largest_diagonal():
    """Diagonal entries up to the largest float are pivots like any other, whatever stands beside them."""
    d, top = 1024, np.float64(np.finfo(np.float32).max)
    H = np.diag(np.full(d, top))
    H[10, 700] = H[700, 10] = 0.5 * top
    U, info = _factor(H.astype(np.float32))
    assert info.tolist() == [0]
    # the pair's block of H^-1 is 4/3 [[1, -1/2], [-1/2, 1]] / top = U^T U
    want = np.diag(np.full(d, top ** -0.5))
    want[10, 10] *= (4.0 / 3.0) ** 0.5
    want[10, 700] = -0.5 * want[10, 10]
    assert rel_fro(U, want) <= 6e-8


def test_factor_wider_than_a_digit_product_contracts():
    """33 000 columns: a doubling step of 32 768, beyond the 16 384 steps that an int32 sum of digit products holds.
    H = S (1 + V V^T) S, and U H U^T x = x for random x, in double; U is rounded to float (6e-8 an entry, each way) on a
    matrix whose condition number is about 10, so the residual stays below 1e-6 or so; a block that is off by one part in a
    thousand shows."""
    import torch
    import paper_2602_04929_b200 as tb
    d, dev = 33000, "cuda:0"
    g = torch.Generator(device=dev).manual_seed(3)
    V = torch.randn(d, 8, generator=g, device=dev) * (3.0 / d ** 0.5)
    s = torch.exp2(torch.randint(-8, 9, (d,), generator=g, device=dev).float())
    H = V @ V.T
    H = 0.5 * (H + H.T)
    H.diagonal().add_(1.0)
    H *= s[:, None]
    H *= s[None, :]
    U, info = tb.tb_factor(H)
    torch.cuda.synchronize()
    assert tb.tb_device_error_flag() == 0 and info.tolist() == [0]

    def times(A, x, transposed=False):  # in double, 2048 rows of A at a time
        y = torch.zeros_like(x)
        for r in range(0, d, 2048):
            a = A[r:r + 2048].double()
            if transposed:
                y += a.T @ x[r:r + 2048]
            else:
                y[r:r + 2048] = a @ x
        return y

    x = torch.randn(d, 4, generator=g, device=dev, dtype=torch.float64)
    y = times(U, times(H, times(U, x, True)))
    assert float((y - x).norm() / x.norm()) <= 1e-5
    assert torch.count_nonzero(torch.tril(U[32000:], 31999)).item() == 0
