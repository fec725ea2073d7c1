"""Grid search with many rows (integer tensor cores): the chosen candidates are those of the score evaluated directly in
double, over group widths below, at and beyond a column tile, bit widths (8: the integers do not fit a byte),
candidate counts, ragged tiles, one H_in per head, and groups in which no candidate can be told apart by the bounds."""
import pytest
import torch

from parity_util import compare, make_problem, run_gpu

pytestmark = pytest.mark.gpu


def direct_scores(W, H, seg, maxq, n_cand):
    """[rows, groups, candidates] of (e H e^T) / 2, all in double."""
    rows, d = W.shape
    W = W.double().view(rows, d // seg, seg)
    mn, mx = W.amin(2).clamp(max=0), W.amax(2).clamp(min=0)
    out = []
    for k in range(n_cand):
        pk = 1.0 - k / 32.0
        s = (pk * mx - pk * mn) / maxq
        s = torch.where(s == 0, torch.ones_like(s), s)
        z = torch.round(-(pk * mn) / s).clamp(0, maxq)
        q = torch.round(W / s[..., None] + z[..., None]).clamp(0, maxq)
        e = W - s[..., None] * (q - z[..., None])
        out.append(torch.stack([0.5 * ((e[:, g] @ H[g * seg:(g + 1) * seg, g * seg:(g + 1) * seg].double()) * e[:, g]).sum(1)
                                for g in range(d // seg)], 1))
    return torch.stack(out, 2)


@pytest.mark.parametrize("rows,d,seg,bits,n_cand,heads,outlier", [
    (4096, 512, 32, 4, 16, 1, False),
    (2600, 1152, 96, 2, 16, 1, False),      # ragged row tiles
    (8192, 1024, 64, 3, 3, 1, False),       # four candidates to a group of lanes, one of them empty
    (4096, 1024, 128, 8, 16, 1, False),     # integers beyond a byte
    (2048, 1024, 128, 7, 32, 4, False),     # one H_in per head, 32 candidates
    (40000, 128, 128, 4, 16, 1, False),     # several chunks of rows
    (1000, 1664, 0, 4, 16, 1, False),       # one group of 13 column tiles
    (777, 1280, 160, 8, 5, 1, False),       # groups that end inside a column tile
    (300, 1024, 0, 3, 16, 3, False),        # wide, one H_in per head
    (2048, 1024, 128, 4, 16, 1, True),      # every (row, group) goes to the direct evaluation
    (300, 2048, 0, 4, 16, 1, True),
])
def test_candidates_are_those_of_the_direct_score(rows, d, seg, bits, n_cand, heads, outlier):
    import paper_2602_04929_b200 as tb

    g = torch.Generator(device="cuda").manual_seed(rows + d)
    n_hin = heads
    rows -= rows % heads
    X = torch.randn(n_hin, 2 * d, d, generator=g, device="cuda", dtype=torch.float64)
    X = X * torch.exp(torch.randn(n_hin, 1, d, generator=g, device="cuda", dtype=torch.float64))
    H = (X.transpose(1, 2) @ X / (2 * d) + 0.01 * torch.eye(d, device="cuda", dtype=torch.float64)).float()
    W = torch.randn(rows, d, generator=g, device="cuda")
    W[5::7, : (seg or d)] = 0.0             # groups of zeros
    if outlier:                             # a huge diagonal that no error meets: the bounds say nothing
        H[:, 3::32, :] = 0.0
        H[:, :, 3::32] = 0.0
        H[:, torch.arange(3, d, 32), torch.arange(3, d, 32)] = 1e20
        W[:, 3::32] = 0.0
    H = (H + H.transpose(1, 2)) / 2
    U, info = tb.tb_factor(H.contiguous())[:2]
    desc = tb.layer_desc(rows, d, heads, rows // heads, bits, seg, rows // heads, n_hin=n_hin, n_cand=n_cand, cd_iters=0, flags=0)
    res = tb.tb_quantize_layer(desc, W, H.contiguous(), U, None, None, None, None, None)
    torch.cuda.synchronize()
    assert tb.tb_device_error_flag() == 0
    sg, per = seg or d, rows // heads
    J = torch.cat([direct_scores(W[h * per:(h + 1) * per], H[h], sg, 2 ** bits - 1, n_cand) for h in range(heads)])
    got = torch.gather(J, 2, res.cand.long().view(rows, d // sg, 1))[..., 0]
    best, arg = J.min(2)
    # the two evaluations differ by rounding alone: seg terms of 2^-53 relative to sums of one sign in H's norm
    assert bool((got <= best * (1 + 1e-11)).all())
    second = J.scatter(2, arg[..., None], float("inf")).min(2).values
    clear = second > best * (1 + 1e-11)
    assert bool((arg == res.cand.view(rows, -1))[clear].all())
    assert bool((res.cand.view(rows, -1)[5::7, 0] == 0).all())


def test_steps_of_an_adaptive_grid():
    prob = make_problem(21, 1024, 4, 64, 2048)
    compare(prob, run_gpu(prob, 3, 0, 16, 1), 3, 0, 16, 1, label="digits")
