"""Packing and unpacking at the edges of a warp's piece (512 codes, 128 values) and of a CTA's turn (4096): bytes and
values equal to the oracle's bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 3, 5, 8])
@pytest.mark.parametrize("rows,d,group", [(1, 32, 0), (1, 544, 32), (3, 96, 96), (7, 608, 0), (129, 4096, 128), (2400, 2080, 416)])
def test_pack_unpack_edges(rows, d, group, bits):
    import paper_2602_04929_b200 as tb

    rng = np.random.default_rng(rows * d + bits)
    codes = rng.integers(0, 1 << bits, (rows, d)).astype(np.uint8)
    ng = d // (group or d)
    scales = rng.random((rows, ng), dtype=np.float32) + np.float32(0.1)
    zeros = rng.integers(0, 1 << bits, (rows, ng)).astype(np.int32)
    t = torch.from_numpy
    packed = tb.tb_pack_codes(t(codes).cuda(), bits)
    bitstream = np.unpackbits(codes.reshape(-1, 1), axis=1, bitorder="little")[:, :bits]
    want = np.packbits(bitstream.reshape(rows, -1), axis=1, bitorder="little").view("<i4")
    assert np.array_equal(packed.cpu().numpy(), want)
    ref = np.repeat(scales, d // ng, axis=1) * (codes.astype(np.int32) - np.repeat(zeros, d // ng, axis=1)).astype(np.float32)
    bad = codes.copy()
    bad[-1, -1] ^= 1
    got, w, miss = tb.tb_unpack_dequant(packed, t(scales).cuda(), t(zeros).cuda(), d, bits, group,
                                        codes_ref=t(bad).cuda(), w_hat_ref=t(ref).cuda())
    assert np.array_equal(got.cpu().numpy(), codes) and np.array_equal(w.cpu().numpy(), ref)
    assert list(miss) == [1, 0]
