"""Grid search of column groups wider than 128 columns: both tile sizes, ragged column and row tiles,
candidate counts from 1 to 32, one H_in per head, and rows that go through in several chunks of scratch."""
import pytest

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu

ADAPT = 1


@pytest.mark.parametrize("d,heads,dh,n_hin,gq,g,flags,n_cand", [
    (640, 8, 64, 1, 0, 16, 0, 16),      # 128 x 128 tiles, several chunks of rows
    (640, 8, 64, 1, 0, 1, 0, 16),       # the same rows with scratch for few: 32 x 32 tiles
    (640, 3, 20, 1, 160, 20, ADAPT, 16),  # groups that end inside a column tile, ragged rows
    (384, 2, 32, 1, 0, 32, ADAPT, 32),  # one row per narrow tile
    (384, 2, 32, 1, 192, 8, ADAPT, 1),  # a single candidate
    (512, 3, 64, 3, 256, 16, ADAPT, 5),  # one H_in per head
    (512, 3, 64, 3, 0, 4, 0, 16),       # one H_in per head, chunks inside a head
    (384, 1, 4, 1, 0, 1, ADAPT, 20),    # steps of one row, more than 16 candidates
    (256, 1, 6, 1, 0, 1, 0, 32),        # the fixed grid with scratch for one row
])
def test_wide_groups(d, heads, dh, n_hin, gq, g, flags, n_cand):
    prob = make_problem(21, d, heads, dh, 1024, n_hin=n_hin)
    compare(prob, run_gpu(prob, 3, gq, g, flags, n_cand=n_cand), 3, gq, g, flags, n_cand=n_cand, label=f"wide{gq}")
