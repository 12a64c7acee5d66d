"""Single kernels at the sizes where they can go wrong: tile edges, remainders, the ends of their ranges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bpd():
    import paper_1811_03115_b200 as b
    return b


# token tiles of 16..256 rows, K splits over clusters of 1, 2, 4 and 8 CTAs (with a short or an empty last split),
# feature counts that end inside a tile, inside a group of four, or take the scalar stores
@pytest.mark.parametrize("rows,in_f,out_f", [(1, 8, 4), (16, 64, 128), (17, 72, 130), (31, 584, 127), (33, 1024, 512), (96, 640, 1027),
                                             (257, 512, 256), (113, 4096, 516), (300, 2040, 64), (130, 328, 4100)])
def test_wide_projection_at_tile_edges(bpd, rows, in_f, out_f):
    import torch
    g = torch.Generator().manual_seed(rows + in_f)
    x = torch.randn(rows, in_f, generator=g).bfloat16()
    w = (torch.randn(out_f, in_f, generator=g) * 0.05).bfloat16()
    b = (torch.randn(out_f, generator=g) * 0.1).bfloat16()
    want = np.maximum(x.double().numpy() @ w.double().numpy().T + b.double().numpy(), 0)
    got = bpd.bpd_op_linear(x.cuda(), w.cuda(), b.cuda(), relu=True).cpu().numpy()
    np.testing.assert_allclose(got, want, atol=1e-5 * np.sqrt(in_f))
    idx, val = bpd.bpd_op_vocab_argmax(x[:, :1024].contiguous().cuda(), w[:, :1024].contiguous().cuda(), want_val=True)
    logits = x[:, :1024].double().numpy() @ w[:, :1024].double().numpy().T
    picked = logits[np.arange(rows), idx.cpu().numpy()]
    np.testing.assert_allclose(picked, logits.max(-1), atol=1e-4)
    np.testing.assert_allclose(val.cpu().numpy(), logits.max(-1), atol=1e-4)


# row tiles of 8, 16, 32 and 64 rows, K tiles of 64 columns, feature tiles of 32
@pytest.mark.parametrize("rows,in_f,out_f", [(1, 8, 1), (8, 64, 32), (9, 72, 33), (16, 1024, 31), (17, 136, 65), (64, 200, 96), (65, 64, 40),
                                             (129, 520, 7)])
def test_fp32_projection_at_tile_edges(bpd, rows, in_f, out_f):
    import torch
    g = torch.Generator().manual_seed(rows + in_f)
    x = torch.randn(rows, in_f, generator=g)
    w = torch.randn(out_f, in_f, generator=g) * 0.05
    b = torch.randn(out_f, generator=g) * 0.1
    want = x.double().numpy() @ w.double().numpy().T
    got = bpd.bpd_op_linear(x.cuda(), w.cuda(), b.cuda(), relu=True).cpu().numpy()
    np.testing.assert_allclose(got, np.maximum(want + b.double().numpy(), 0), atol=2e-6 * np.sqrt(in_f))
    idx, val = bpd.bpd_op_vocab_argmax(x.cuda(), w.cuda(), want_val=True)
    idx2, val2 = torch.zeros(rows, dtype=torch.int32, device="cuda"), torch.zeros(rows, device="cuda")
    bpd.bpd_op_vocab_argmax_noalloc(x.cuda(), w.cuda(), idx2, val2)
    for i, v in ((idx, val), (idx2, val2)):
        np.testing.assert_allclose(want[np.arange(rows), i.cpu().numpy()], want.max(-1), atol=1e-5)
        np.testing.assert_allclose(v.cpu().numpy(), want.max(-1), atol=1e-5)
