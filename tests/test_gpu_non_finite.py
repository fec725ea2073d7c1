"""Operands with entries that are no finite numbers in the products on the integer tensor cores: what they touch is no number."""
import numpy as np
import pytest

from parity_util import make_problem, run_gpu

pytestmark = pytest.mark.gpu


def _correction(R, U):
    import torch
    import paper_2602_04929_b200 as tb
    P, C = tb.tb_prepare_correction(torch.from_numpy(R).to("cuda:0"), torch.from_numpy(U).to("cuda:0"))
    torch.cuda.synchronize()
    return P.cpu().numpy(), C.cpu().numpy()


@pytest.mark.parametrize("what", ["nan", "inf", "-inf"])
def test_correction_operands(what):
    """P = ((R U^T) masked) U and C = R U^T U: a row of R with such an entry spoils its row of both and no other; an entry
    of U in column n spoils column n of C."""
    prob = make_problem(80, 256, 1, 8, 1024, with_r=True)
    R, U = prob["R"][0].copy(), prob["Uin"][0].copy()
    P0, C0 = _correction(R, U)
    R1 = R.copy()
    R1[37, 255] = np.float32(what)
    P, C = _correction(R1, U)
    assert not np.any(np.isfinite(C[37])) and not np.any(np.isfinite(P[37, 38:]))
    rest = np.arange(256) != 37
    assert np.array_equal(P[rest], P0[rest]) and np.array_equal(C[rest], C0[rest])
    U1 = U.copy()
    U1[3, 200] = np.float32(what)
    P, C = _correction(R, U1)
    assert not np.any(np.isfinite(C[:, 200]))


@pytest.mark.parametrize("what", ["nan", "inf"])
def test_joint_compensation(what):
    """E - W0 C with such a weight in a row of the step: the rows of its head that are still to come are spoilt in every
    column, the other head is not touched."""
    prob = make_problem(81, 256, 2, 32, 1024, with_r=True, hout="spd")
    clean = run_gpu(prob, 3, 128, 8, 0, want_loss=False)
    prob["W"][3, 40] = np.float32(what)
    gpu = run_gpu(prob, 3, 128, 8, 0, want_loss=False)
    assert not np.any(np.isfinite(gpu["w_comp"][8:32]))
    assert np.array_equal(gpu["w_comp"][32:], clean["w_comp"][32:]) and np.array_equal(gpu["codes"][32:], clean["codes"][32:])
