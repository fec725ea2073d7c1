"""Compensation matrices: more remaining rows than a pass over them takes, steps whose factor rows fit shared memory and steps
whose do not, a step of one row, a ragged last quarter of a dot product."""
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dh,g", [(300, 20), (256, 128), (131, 1), (45, 15)])
def test_compensation_matrices(dh, g):
    prob = make_problem(75, 128, 2, dh, 512, hout="spd")
    compare(prob, run_gpu(prob, 3, 64, g, 0), 3, 64, g, 0, label=f"comp{dh}")
