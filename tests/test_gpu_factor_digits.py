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
