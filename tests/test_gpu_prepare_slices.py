"""bakron_prepare's sliced products at the edges of their blocks: sides around
multiples of 64 and 128 (panels, tiles, uneven halves of the inverse), sides of
different size, and Grams whose rows and columns differ by many powers of two.

The factors are compared with an fp64 Cholesky and triangular inverse on the
host.  Tolerance: one rounding to fp32 (2^-24 relative, 6e-8) and the fp64-grade
factorisation, kappa * n * 2^-53 of the largest entry (kappa < 1e5, n < 1000:
1e-8), as in test_prepare_matches_oracle.
"""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as WL
from tests._helpers import to_np

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2608_06291_gb300 as P


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    P.build()
    P.lib()


def _check(A, B, damp):
    LA, LB, rA, rB = (t.cpu().numpy().astype(np.float64)
                      for t in P.bakron_get_factors(P.bakron_prepare(A.cuda(), B.cuda(), damp)))
    f = O.prepare(to_np(A), to_np(B), damp, via_inverse=False)
    for got, want in ((LA, f.LA), (LB, f.LB)):
        assert not np.triu(got, 1).any()
        np.testing.assert_array_equal(np.diag(got), 1.0)
        np.testing.assert_allclose(got, want, rtol=2e-7, atol=1e-8 * np.abs(want).max())
    np.testing.assert_allclose(rA, f.rA, rtol=2e-7)
    np.testing.assert_allclose(rB, f.rB, rtol=2e-7)


@pytest.mark.parametrize("m,n", [(127, 129), (128, 192), (191, 256), (257, 64), (1, 385), (640, 513)])
def test_prepare_block_edges(m, n):
    _, A, B = WL.small_problem(m, n, 77 + m + n)
    _check(A, B, 0.01)


def test_prepare_uneven_scales():
    """Row and column i scaled by 2^k_i, k_i in -30 .. 30: the factors scale with
    them exactly, so without damping the result is the unscaled one's."""
    n, m = 200, 70
    _, A, B = WL.small_problem(m, n, 5)
    A = A + 0.05 * A.diagonal().mean() * torch.eye(n)
    B = B + 0.05 * B.diagonal().mean() * torch.eye(m)
    g = torch.Generator().manual_seed(1)
    sa = torch.ldexp(torch.ones(n), torch.randint(-30, 31, (n,), generator=g))
    sb = torch.ldexp(torch.ones(m), torch.randint(-30, 31, (m,), generator=g))
    L0 = P.bakron_get_factors(P.bakron_prepare(A.cuda(), B.cuda(), 0.0))
    L1 = P.bakron_get_factors(P.bakron_prepare((sa[:, None] * A * sa).cuda(), (sb[:, None] * B * sb).cuda(), 0.0))
    # H -> D H D gives R -> R D and Lhat -> D^-1 Lhat D
    for k, s in ((0, sa.cuda()), (1, sb.cuda())):
        assert torch.equal(L1[k], L0[k] / s[:, None] * s)
        assert torch.equal(L1[k + 2], L0[k + 2] * s)
    _check(A, B, 0.0)


@pytest.mark.parametrize("spoil", ["indefinite", "large", "nan", "zero"])
def test_prepare_refuses(spoil):
    _, A, B = WL.small_problem(130, 200, 9)
    if spoil == "indefinite":      # an off-diagonal entry no positive definite matrix has
        A[150, 20] = A[20, 150] = 1.5 * A.diagonal().max()
    elif spoil == "large":
        A[150, 20] = A[20, 150] = 3e38
    elif spoil == "nan":
        A[199, 0] = float("nan")
    else:
        A.zero_()
    with pytest.raises(P.BakronError) as e:
        P.bakron_prepare(A.cuda(), B.cuda(), 0.0 if spoil == "zero" else 0.01)
    assert e.value.status == 2
