"""Edges of bakron_gram's block kernel: operands read straight from X (d a
multiple of 64, 16-byte aligned rows) or through a padded copy, partial last
column blocks, partial sample slots, and blocks split along the samples.

Tolerance as in test_gpu_gram.py, from the arithmetic: at most 256 exact (or
2^-21 accurate) products are summed in place (256 * 2^-23 of their absolute
sum), the groups in fp32.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2608_06291_gb300 as P


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()


# (k, d, column offset of X in a wider buffer, weighted, dtype, beta)
CASES = [(1, 64, 0, False, torch.bfloat16, 0.0),       # one row, half a block
         (63, 128, 0, False, torch.bfloat16, 1.0),     # a partial slot
         (65, 192, 0, False, torch.bfloat16, 0.0),     # 1.5 row blocks
         (4096, 64, 0, False, torch.bfloat16, 1.0),    # one block, split along the samples
         (2000, 320, 8, False, torch.bfloat16, -0.5),  # aligned view, uneven splits
         (2000, 320, 3, False, torch.bfloat16, 1.0),   # misaligned view: the copy
         (1500, 250, 0, False, torch.bfloat16, 0.0),   # d no multiple of 64: the copy
         (3000, 129, 0, False, torch.float32, 1.0),    # tf32, split
         (3000, 257, 1, True, torch.float32, 0.0),     # tf32 weighted, split, misaligned
         (3000, 384, 0, True, torch.bfloat16, 1.0)]    # one exact operand


@pytest.mark.parametrize("k,d,off,weighted,dtype,beta", CASES)
def test_gram_blocks(k, d, off, weighted, dtype, beta):
    g = torch.Generator().manual_seed(k + d)
    Xb = (torch.randn(k, d + 16, generator=g) * 1.5).to(dtype).cuda()
    X = Xb[:, off:off + d]
    w = (torch.rand(k, generator=g) + 0.5).cuda() if weighted else None
    G0 = torch.randn(d, d, generator=g)
    G0 = (G0 + G0.T).cuda()
    G = torch.full((d, d + 5), 7.0, device="cuda")
    G[:, :d] = G0
    P.bakron_gram(X, w, alpha=0.5, beta=beta, G=G[:, :d])
    torch.cuda.synchronize()
    assert torch.all(G[:, d:] == 7.0)
    got = G[:, :d].double()
    x = X.double()
    wx = x if w is None else x * w.double()[:, None]
    ref = 0.5 * (wx.T @ x) + beta * G0.double()
    bound = 2.0 ** -14 * 0.5 * (wx.abs().T @ x.abs()) + 2.0 ** -20 * abs(beta) * G0.double().abs()
    assert torch.all((got - ref).abs() <= bound + 1e-30)
    assert torch.equal(got, got.T)


def test_gram_small_workspace_is_not_split():
    """A workspace that holds one slot of samples: many chunks, no parts."""
    k, d = 700, 192
    X = torch.randn(k, d, generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
    ws = torch.empty(256 + 2 * 256 * 64, dtype=torch.uint8, device="cuda")
    G = P.bakron_gram(X, alpha=1.0, workspace=ws)
    ws3 = torch.empty(256 + 2 * 256 * 64, dtype=torch.uint8, device="cuda")
    Xm = torch.zeros(k, d + 1, dtype=torch.bfloat16, device="cuda")[:, 1:]
    Xm.copy_(X)
    G3 = P.bakron_gram(Xm, alpha=1.0, workspace=ws3)
    torch.cuda.synchronize()
    x = X.double()
    bound = 2.0 ** -14 * (x.abs().T @ x.abs())
    for g in (G, G3):
        assert torch.all((g.double() - x.T @ x).abs() <= bound)
    with pytest.raises(P.BakronError):
        P.bakron_gram(X, alpha=1.0, workspace=ws[:-1])
