"""Dynamic-grid sweep: group widths between a piece of 16 columns and 128, rows that end inside a CTA's eight and inside an
update tile's 64, one H_in per head, with and without the propagated-error term, codes far outside the grid."""
import numpy as np
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu

DYN = 4


@pytest.mark.parametrize("d,heads,dh,n_hin,gq,g,bits,with_r", [
    (384, 3, 20, 1, 96, 20, 3, False),   # 60 rows, two pieces of a group left over
    (384, 3, 25, 3, 32, 5, 4, True),     # 5 rows a unit
    (640, 2, 70, 2, 128, 70, 2, True),   # 70 rows a unit: a second tile of six rows
    (256, 1, 1, 1, 64, 1, 8, False),     # a single row
    (768, 5, 128, 1, 64, 128, 3, False),
])
def test_dynamic_panel_edges(d, heads, dh, n_hin, gq, g, bits, with_r):
    prob = make_problem(23, d, heads, dh, 1500, with_r=with_r, n_hin=n_hin)
    prob["W"][0, 1] = np.float32(3.0e3) * prob["W"].max()  # the other codes of its group all round to one
    compare(prob, run_gpu(prob, bits, gq, g, DYN), bits, gq, g, DYN, label=f"dyn{gq}")
