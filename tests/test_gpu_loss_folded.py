"""The loss formed from the triangle that H_in folds into, against the loss formed in double from all of H_in: the same rows
with and without four rows of zeros (those lose nothing, and only a multiple of eight rows takes the split products)."""
import numpy as np
import pytest
import torch

import paper_2602_04929_b200 as tb
from parity_util import TOL_LOSS, make_problem

pytestmark = pytest.mark.gpu


def _loss(W, H, U, Hout, Uout, bits, gq, R=None, P=None, C=None):
    dev = torch.device("cuda:0")
    t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(dev)
    rows, d = W.shape
    desc = tb.layer_desc(rows, d, 1, rows, bits, gq, rows, flags=1)
    out = tb.empty_result(desc, dev)
    ws = torch.empty(tb.tb_quantize_layer_workspace(desc, R is not None, True), dtype=torch.uint8, device=dev)
    tb.tb_quantize_layer(desc, t(W), t(H), t(U), t(Hout), t(Uout), t(R), t(P), t(C), ws=ws, out=out)
    return out.codes.cpu().numpy(), float(out.loss[0])


# widths of one column tile and of several, whole and not; rows of one row tile and of several
@pytest.mark.parametrize("d,rows", [(128, 12), (384, 124), (640, 140), (1152, 260)])
@pytest.mark.parametrize("hout", [None, "spd"])
@pytest.mark.parametrize("with_r", [False, True])
def test_folded_loss(d, rows, hout, with_r):
    prob = make_problem(71, d, 1, rows, 1024, with_r=with_r, hout=hout)

    def padded(a, eye=False):
        if a is None:
            return None
        b = np.eye(rows + 4, dtype=a.dtype)[None] if eye else np.zeros((rows + 4, d), a.dtype)
        if eye:
            b[0, :rows, :rows] = a[0]
        else:
            b[:rows] = a
        return b

    pr = {k: prob.get(k) for k in ("R", "P", "C")}
    c0, want = _loss(prob["W"], prob["Hin"], prob["Uin"], prob.get("Hout"), prob.get("Uout"), 3, 128, **pr)
    c1, got = _loss(padded(prob["W"]), prob["Hin"], prob["Uin"], padded(prob.get("Hout"), True), padded(prob.get("Uout"), True), 3, 128, **pr)
    assert np.array_equal(c0, c1[:rows])
    # eight truncating float accumulations a chunk of 128 steps, in steps of 2^-23 of a sum whose halves cancel about fourfold;
    # W R takes the other form of the product and cancels against the rest
    assert abs(got - want) <= (TOL_LOSS if with_r else 8 * 2.0 ** -23 * 4) * abs(want)
