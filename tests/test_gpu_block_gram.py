"""Out-channel Hessians from per-block Grams: row counts around a tile of 64, a contraction in one and in many parts, widths
that are no multiple of a step, blocks shared by heads and heads of several blocks."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_heads,g_heads,dh,d,with_sum", [
    (1, 1, 1, 40, False), (2, 1, 63, 1000, True), (1, 4, 64, 4096, True), (3, 3, 65, 777, False),
    (2, 6, 130, 2080, True), (40, 40, 128, 512, False), (1, 1, 128, 8192, False),
])
def test_block_gram(n_heads, g_heads, dh, d, with_sum):
    import paper_2602_04929_b200 as tb

    g = torch.Generator(device="cuda").manual_seed(d + dh)
    G = torch.randn(g_heads * dh, d, generator=g, device="cuda")
    H = None
    if with_sum:
        X = torch.randn(d, d, generator=g, device="cuda")
        H = X @ X.t() / d + torch.eye(d, device="cuda")
    got = tb.tb_build_hout(G, H, n_heads, dh, 0.01)
    Gb = G.double().view(g_heads, dh, d)
    C = (Gb @ H.double() if with_sum else Gb) @ Gb.transpose(1, 2)
    if g_heads >= n_heads:
        C = C.view(n_heads, g_heads // n_heads, dh, dh).sum(1)
    else:
        C = C.repeat_interleave(n_heads // g_heads, 0)
    C = C + 0.01 * C.diagonal(dim1=1, dim2=2).mean(1)[:, None, None] * torch.eye(dh, device="cuda", dtype=torch.float64)
    # the result is rounded to float; G Hsum is float-accurate (24-bit pieces), d terms
    scale = C.diagonal(dim1=1, dim2=2).abs().amax()
    assert float((got.double() - C).abs().max() / scale) < (4e-6 if with_sum else 2e-7)
