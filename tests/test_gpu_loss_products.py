"""The loss from split products on the tensor cores against the loss formed in double: the same rows with and without four
rows of zeros a head (those lose nothing, and only a multiple of eight rows, of 128 a head with one H_in per head, takes the
split products), or the sum formed here from the codes and scales that came back."""
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
def test_loss_of_padded_rows(d, rows, hout, with_r):
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
    # a chunk's truncating float accumulations, and W R, which cancels against the rest
    assert abs(got - want) <= (TOL_LOSS if with_r else 8 * 2.0 ** -23 * 4) * abs(want)


# ---- inputs whose channels share a strong component ----
# The products sum 128 columns at a time in float, 48 truncating accumulations of at most a last place each, and the chunks in
# double.  Where a chunk's partial sums stay below its result, its relative error is at most this; dW makes the strong
# component cancel inside dW H_in, so the sum over the chunks and rows keeps it.  With R both terms of the loss, tr(H_out dW H_in
# dW^T) and 2 tr(H_out W R dW^T), have that error and they cancel against one another: the bound is on their magnitudes.
# (Seen: up to 4.3e-6 of the loss without R.  A loss from the triangle that H_in folds into, where the component cancels after
# the products, is off by 0.6e-5 to 1.5e-5 with 8 bits.)
TRUNCATION = 48 * 2.0 ** -23


def _upper_factor(h):
    low = torch.linalg.cholesky(h.double().flip(-2, -1)).flip(-2, -1)
    eye = torch.eye(h.shape[-1], device=h.device, dtype=torch.float64)
    return torch.linalg.solve_triangular(low, eye.expand_as(low), upper=True).triu().float().contiguous()


def _correlated(d, heads, d_head, n_hin, hout, with_r, damp):
    """Activations with a rank-16 common factor of about 20 times the rest of a channel."""
    g = torch.Generator(device="cuda:0").manual_seed(73)
    rand = lambda *s: torch.randn(s, generator=g, device="cuda:0", dtype=torch.float64)
    H, R, P, C = [], [], [], []
    for _ in range(n_hin):
        x = (rand(2 * d + 500, d) + 5.0 * rand(2 * d + 500, 16) @ rand(16, d)) * torch.exp(0.5 * rand(2 * d + 500, 1))
        h = x.T @ x / x.shape[0]
        h.diagonal().add_(damp * h.diagonal().mean())
        H.append(h.float())
        if with_r:
            r = (0.025 * rand(*x.shape).T @ x / x.shape[0]).float()
            u = _upper_factor(H[-1]).double()
            R.append(r)
            P.append(((r.double() @ u.T).triu(1) @ u).float())
            C.append((r.double() @ u.T @ u).float())
    H = torch.stack(H)
    Hout = Uout = None
    if hout:
        q = torch.linalg.qr(rand(heads, d_head, d_head))[0]
        Hout = ((q * torch.logspace(0, -3, d_head, device=q.device, dtype=q.dtype)) @ q.mT).float()
        Hout = (0.5 * (Hout + Hout.mT)).contiguous()
        Uout = _upper_factor(Hout)
    st = lambda a: torch.stack(a).contiguous() if a else None
    return dict(W=0.02 * rand(heads * d_head, d).float(), H=H, U=_upper_factor(H), Hout=Hout, Uout=Uout, R=st(R), P=st(P), C=st(C))


def _quantized(p, heads, bits, gq, flags):
    rows, d = p["W"].shape
    desc = tb.layer_desc(rows, d, heads, rows // heads, bits, gq, rows // heads, n_hin=p["H"].shape[0], flags=flags)
    out = tb.empty_result(desc, p["W"].device)
    ws = torch.empty(tb.tb_quantize_layer_workspace(desc, p["R"] is not None, True), dtype=torch.uint8, device=p["W"].device)
    tb.tb_quantize_layer(desc, p["W"], p["H"], p["U"], p["Hout"], p["Uout"], p["R"], p["P"], p["C"], ws=ws, out=out)
    assert tb.tb_device_error_flag() == 0
    return out


def _loss_terms(p, out, heads, gq):
    """The loss's two terms for every head, in double from the codes and scales."""
    D = out.scales.double().repeat_interleave(gq, 1) * (out.codes.double() - out.zeros.double().repeat_interleave(gq, 1))
    W = p["W"].double().view(heads, -1, D.shape[1])
    D = D.view_as(W) - W
    against = lambda Z: ((Z if p["Hout"] is None else p["Hout"].double() @ Z) * D).sum((1, 2))
    return against(D @ p["H"].double()), 0.0 if p["R"] is None else against(2.0 * W @ p["R"].double())


def _with_zero_rows(p, heads, d_head, extra):
    def eye(a):
        if a is None:
            return None
        b = torch.eye(d_head + extra, device=a.device).repeat(heads, 1, 1)
        b[:, :d_head, :d_head] = a
        return b.contiguous()

    W = torch.nn.functional.pad(p["W"].view(heads, d_head, -1), (0, 0, 0, extra)).reshape(heads * (d_head + extra), -1)
    return dict(p, W=W.contiguous(), Hout=eye(p["Hout"]), Uout=eye(p["Uout"]))


# one shared H_in, and one per head with several column tiles for each head's rows
@pytest.mark.parametrize("d,heads,n_hin,with_r", [(1024, 1, 1, False), (2048, 1, 1, False), (1024, 1, 1, True), (2048, 1, 1, True), (1024, 3, 3, False)])
@pytest.mark.parametrize("hout", [False, True])
@pytest.mark.parametrize("bits,damp", [(4, 1e-2), (8, 1e-4)])
def test_loss_of_correlated_channels(d, heads, n_hin, with_r, hout, bits, damp):
    p = _correlated(d, heads, 124, n_hin, hout, with_r, damp)
    a = _quantized(p, heads, bits, 128, 1)
    b = _quantized(_with_zero_rows(p, heads, 124, 4), heads, bits, 128, 1)
    assert torch.equal(a.codes.view(heads, 124, d), b.codes.view(heads, 128, d)[:, :124])
    terms = sum(abs(t) for t in _loss_terms(p, a, heads, 128))
    assert ((a.loss - b.loss).abs() <= TRUNCATION * terms).all(), (a.loss, b.loss, terms)


# W R kept from the refinement for the loss: all rows in one batch of the refinement, and in two
@pytest.mark.parametrize("d,heads,d_head,gq", [(1024, 1, 128, 128), (1024, 2, 64, 64), (4096, 17, 128, 64)])
@pytest.mark.parametrize("hout", [False, True])
def test_loss_after_refinement(d, heads, d_head, gq, hout):
    p = _correlated(d, heads, d_head, 1, hout, True, 1e-2)
    out = _quantized(p, heads, 4, gq, 3)
    terms = _loss_terms(p, out, heads, gq)
    assert ((out.loss - sum(terms)).abs() <= TRUNCATION * sum(abs(t) for t in terms)).all(), (out.loss, terms)


# Weights in the upper half of the float range: every step scales by powers of two (the sweep takes ratios of entries of U), so
# codes and loss are those of ordinary weights (up to pieces of small entries below the smallest bf16)
@pytest.mark.parametrize("hout", [False, True])
@pytest.mark.parametrize("flags", [1, 3])
@pytest.mark.parametrize("with_r", [False, True])
def test_loss_of_weights_near_the_float_range(hout, flags, with_r):
    p = _correlated(256, 1, 128, 1, hout, with_r, 1e-2)
    a = _quantized(p, 1, 4, 128, flags)
    w, h = 127 - int(torch.floor(torch.log2(p["W"].abs().max()))), -24
    q = dict(p, W=(p["W"].double() * 2.0 ** w).float(), H=p["H"] * 2.0 ** h)
    if with_r:
        q["R"] = p["R"] * 2.0 ** h
    assert 2.0 ** 127 <= float(q["W"].abs().max()) < 2.0 ** 128
    b = _quantized(q, 1, 4, 128, flags)
    assert torch.equal(a.codes, b.codes)
    want = a.loss * 2.0 ** (2 * w + h)
    assert ((b.loss - want).abs() <= TRUNCATION * want.abs()).all(), (b.loss, want)
