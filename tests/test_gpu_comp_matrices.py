"""Compensation matrices: more remaining rows than a pass over them takes, steps whose factor rows fit shared memory and steps
whose do not, a step of one row, a ragged last quarter of a dot product."""
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dh,g", [(300, 20), (256, 128), (131, 1), (45, 15)])
def test_compensation_matrices(dh, g):
    prob = make_problem(75, 128, 2, dh, 512, hout="spd")
    compare(prob, run_gpu(prob, 3, 64, g, 0), 3, 64, g, 0, label=f"comp{dh}")


# launches of few CTAs, which fetch the rows to be updated ahead, and of many, which do not: steps that take the group in one
# pass of 32 rows and in two, remaining rows that are no whole tile
@pytest.mark.parametrize("d,heads,dh,g,with_r", [(256, 3, 90, 45, False), (1152, 64, 96, 48, False), (1152, 64, 69, 23, False),
                                                 (256, 3, 90, 45, True), (640, 40, 90, 45, True), (640, 40, 81, 9, True)])
def test_compensation_of_few_and_many_rows(d, heads, dh, g, with_r):
    prob = make_problem(77, d, heads, dh, 1024, with_r=with_r, hout="spd")
    compare(prob, run_gpu(prob, 3, 128, g, 0), 3, 128, g, 0, heads=[0, heads // 2, heads - 1], label=f"comp{heads}")


def test_codes_at_an_odd_address():
    """The codes may lie anywhere: the joint compensation reads them back a byte at a time."""
    import torch
    import paper_2602_04929_b200 as tb
    prob = make_problem(76, 256, 2, 24, 512, hout="spd")
    dev = "cuda:0"
    desc = tb.layer_desc(48, 256, 2, 24, 4, 64, 8)
    args = [torch.from_numpy(prob[k]).to(dev) for k in ("W", "Hin", "Uin", "Hout", "Uout")]
    ref = tb.tb_quantize_layer(desc, *args, want_loss=False)
    out = tb.tb_quantize_layer(desc, *args, want_loss=False)
    buf = torch.zeros(48 * 256 + 1, dtype=torch.uint8, device=dev)
    out.codes = buf[1:].view(48, 256)
    assert out.codes.data_ptr() % 2 == 1
    tb.tb_quantize_layer(desc, *args, want_loss=False, out=out)
    torch.cuda.synchronize()
    assert torch.equal(out.codes, ref.codes) and torch.equal(out.w_hat, ref.w_hat)
